// gks_kernels.h -- device data views and kernel launchers of libgks.
#pragma once

#include <cuda_runtime.h>

#include <cstdint>

namespace gks {

// control block in device memory (doubles)
enum { CTRL_T = 0, CTRL_DT = 1, CTRL_DT_FIXED = 2, CTRL_T_END = 3, CTRL_N = 8 };
// per-block partial results of the update / time-step kernels
enum { PART_DTMIN = 0, PART_RES = 1, PART_N = 6 };
// device error flags
enum { ERR_STATE = 1, ERR_TIMEOUT = 2 };

constexpr int FLUX_FACES = 32;       // faces per flux block (3 threads each)
constexpr int FLUX_THREADS = 3 * FLUX_FACES;
constexpr int FLUX_THREADS_FP64 = 64;  // the small blocks of the FP64 flux (21 faces)
constexpr int CELL_THREADS = 128;    // threads per cell-kernel block
constexpr int CELLS_PER_BLOCK = 24;  // 4 warps x 6 cells, 5 lanes per cell
constexpr int FGEO = 24;             // reals per face geometry record
constexpr int POLY_STRIDE = 52;      // reals per cell reconstruction record, FP64 (50 used)
constexpr int XS = 20;               // reals per cell working-state record, FP64: W (5), grad W (15, 3q+i)
// FP32 bulk keeps each cell average as an unevaluated pair hi + lo of FP32
// numbers (the FP64 average to ~48 bits), so that differences between
// neighbouring averages stay exact to FP32 rounding of the difference:
//   working state [nc][28]: W hi (5), W lo (5), pad (2), grad W (15), pad (1):
//   the averages, which most gathers of a neighbour want alone, are three
//   16-byte vectors, the gradients four
//   reconstruction record [nc][60]: per component the constant R(centroid)
//   minus the average and the 9 slopes/curvatures (50), the average's hi (5)
//   and lo (5) parts
constexpr int XS32 = 28;
constexpr int XLO = 5;               // offset of the lo parts in an FP32 working-state record
// Face records, sums over the face's Gauss points with their weights w:
//   stage 1  per component: sum w Fh, sum w (2 Fh - D / 3), sum w W(t*),
//            sum w W(0); FP32: the flux and interface-state entries are
//            relative to the mean W_m of the face's two cell averages, and the
//            reference flux (dt / 2) A F_n(W_m) follows as hi and lo parts
//            (one aligned 128-byte record)
//   stage 2  per component: sum w 4/3 D, sum w dW
// The interface states enter a cell times the face's normal, which the
// update multiplies in: a third of the words that (sum w W n) would take.
// NR (40, 20) names the stage: the length of its record with the normal
// multiplied in, as gks_debug_face_records gives it.
// A component's entries (rec_entries of them) lie together, so that an update
// lane reads them as vectors.
template <typename T, int NR>
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int rec_entries() {
    return NR == 20 ? 2 : sizeof(T) == 4 ? 6 : 4;
}
template <typename T, int NR>
constexpr int rec_stride() {
    return NR == 20 ? 10 : sizeof(T) == 4 ? 32 : 20;
}
constexpr int POLY_STRIDE32 = 60;
constexpr int PHI = 50, PLO = 55;    // offsets of the average's hi / lo parts in an FP32 record
template <typename T>
struct Stride {
    static constexpr int xs = sizeof(T) == 4 ? XS32 : XS;
    static constexpr int xg = sizeof(T) == 4 ? 12 : 5;  // offset of grad W (row 3 q + i) in it
    static constexpr int poly = sizeof(T) == 4 ? POLY_STRIDE32 : POLY_STRIDE;
};
// Per-block tile of the reconstruction's static cell data, one contiguous
// record of TILE_ROWS values for each of the block's CELLS_PER_BLOCK cells: M2
// (144), M1 (12), central second moments (6), |Omega|^(2/3), |Omega|^(4/3),
// the largest |x|, |y|, |z| of the cell's 12 face Gauss points about its
// centroid (3, pad 1); these first TILE_COPY rows come into shared memory by
// one bulk copy.  The Gauss points themselves (36) stay in global memory:
// only cells that the bound from the largest offsets cannot clear read them.
// Consecutive rows of a cell lie together in 16-byte groups, so that a lane
// reads four (FP64: two) in one shared-memory access.
enum { TILE_M2 = 0, TILE_M1 = 144, TILE_MOM = 156, TILE_V23 = 162, TILE_V43 = 163, TILE_BND = 164, TILE_COPY = 168,
       TILE_G = 168, TILE_ROWS = 204 };
template <typename TO>
#ifdef __CUDACC__
__host__ __device__
#endif
constexpr int64_t tile_at(int row, int cell) {
    constexpr int V = 16 / (int)sizeof(TO);
    return ((int64_t)(row / V) * CELLS_PER_BLOCK + cell) * V + row % V;
}
// a wall-constrained operator slot: W2 [9][17] (P2 from [data (16); Q0])
// then W1 [3][5] (P1 slopes from [dQ_f (4); Q0])
enum { WOP_W1 = 153, WOP_STRIDE = 168 };

// The FP64 flux is bound by its pipe whatever the occupancy (218-238 registers,
// no spills), so a launch lasts as long as the SM with the most warps: blocks
// of 96 threads (32 faces, no lane idle) or of 64 (21 faces, one lane idle),
// whichever leaves the fullest of the device's SMs with fewer warps.  On 152
// SMs, 6,144 faces: 6 warps with blocks of 96, 4 with 64, a whole step 215 and
// 153 us; 49,280 faces: 33 and 32 warps, 1,242 and 1,188 us; from about 10^6
// faces the blocks of 96 win by their full lanes.
inline int64_t fullest_sm_warps(int64_t nf, int threads, int sms) {
    const int64_t blocks = (nf + threads / 3 - 1) / (threads / 3);
    return (blocks + sms - 1) / sms * (threads / 32);
}
inline bool flux_small_blocks(int64_t nf, int sms) {
    return fullest_sm_warps(nf, FLUX_THREADS_FP64, sms) < fullest_sm_warps(nf, FLUX_THREADS, sms);
}

template <typename T>
struct DevMesh {
    int64_t nc, nf;
    int32_t ncase;
    const int32_t* cell_case;  // [nc] case of each cell (ascending)
    const int32_t* nbr;    // [4][nc], -1 = none
    const int32_t* cface;  // [4][nc] face * 2 + side (side 1 = right)
    const double* inv_vol; // [nc]
    const T* dr;           // [nc]
    const T* M1;           // [12][nc]
    const T* tile;         // [blocks][TILE_ROWS * CELLS_PER_BLOCK] reconstruction data (tile_at)
    // FP32 bulk with FP64 stencil operators (precision 2): the same two in
    // FP64, M1 and tile NULL (else these are NULL)
    const double* M1d;
    const double* tiled;
    const int32_t* flr;    // [2][nf]
    const T* fgeo;         // [nf][FGEO]: n(3), w, XL(9), XR(9), pad
    const T* fnw;          // [nf][4]: n(3), w once more, apart from the rest for the updates
    const float* fan;      // FP32 bulk: [nf][6] face area vectors A n as FP32 hi / lo pairs (NULL in FP64)
    const T* fixed;        // [nc][Stride<T>::xs] state held by fixed boundary faces (NULL: none)
    // Sec. 4.4 wall-constrained momentum stencils (NULL: none): slot of each
    // cell (-1: none) and per slot W2 [9][17] at 0, W1 [3][5] at WOP_W1, in
    // the operator precision (wop; precision 2: wopd)
    const int32_t* wslot;
    const T* wop;
    const double* wopd;
    int32_t xwalls;        // 1: the mesh has isothermal or moving wall faces
    int32_t sms;           // the device's SMs (flux_small_blocks)
};

template <typename T>
struct DevState {
    double* Wd;   // [5][nc] master cell averages (FP64)
    T* X;         // [nc][Stride<T>::xs] working state W^n, grad W^n (cell-major for neighbour gathers)
    T* Xs;        // [nc][Stride<T>::xs] stage state W*, grad W*
    double* S;    // [nc][5] saved stage-1 flux term
    T* G;         // [nc][15] saved stage-1 gradient term
    T* slopes;    // [nc][5] |b|^2 of the P1 slopes (slopes pass), or [nc][15] the slopes (diagnostics)
    T* poly;      // [nc][Stride<T>::poly]
    T* rec;       // [nf][rec_stride]
    double* ctrl; // [CTRL_N] global controls (dt_fixed, t_end)
    double* case_t;   // [ncase] time of each case
    double* case_dt;  // [ncase] step of each case for the current step
    unsigned long long* case_dtmin;  // [ncase] bits of the minimum local dt (atomicMin)
    double* part; // [n_part_blocks][PART_N] residual sums per block
    int32_t* err;
};

struct HostPhys {
    double gamma, cfl, mu, eps_weno, tau_eps, tau_c;
    int weno, order, smooth, viscous;
    double prf;    // Pr fix factor 1/Pr - 1 (0: none)
    double twall;     // isothermal wall temperature
    double uwall[3];  // moving wall velocity
};

template <typename T>
struct Launch {
    // stage pieces
    // fin (may be NULL): block 0 first turns the per-block minima into the
    // step's dt (the time-step rule's global minimum, t_end clipping)
    struct Finalize {
        unsigned long long* dtmin;
        double* case_t;
        double* case_dt;
        int32_t ncase;
        double cfl;
        const double* ctrl;
    };
    // step 1 of the reconstruction: |b|^2 of every cell's P1 slopes, s2[nc][5]
    static cudaError_t slopes(const DevMesh<T>& m, const T* X, T* s2, const Finalize* fin,
                              cudaStream_t s);
    // s2_in (may be NULL): the slopes pass's result; without it the kernel
    // computes its neighbours' slopes itself.
    // slopes_out (may be NULL) receives the cell's own step-1 slopes.
    // err: ERR_TIMEOUT is or-ed in if a block's bounded wait for its tile
    // gave up
    static cudaError_t recon(const DevMesh<T>& m, const HostPhys& p, const T* X, const T* s2_in,
                             T* slopes_out, T* poly, int32_t* fallback, const Finalize* fin,
                             int32_t* err, cudaStream_t s);
    // case_dt: per-case step (NULL: dt_override for every face)
    // variant (FP32): 1 = more resident warps, 0 = more registers; ignored in FP64
    static cudaError_t flux(const DevMesh<T>& m, const HostPhys& p, const T* X, const T* poly, T* rec,
                            const double* case_dt, double dt_override, int stage, cudaStream_t s,
                            int variant = 1);
    static cudaError_t update1(const DevMesh<T>& m, const HostPhys& p, const DevState<T>& st, cudaStream_t s);
    static cudaError_t update2(const DevMesh<T>& m, const HostPhys& p, const DevState<T>& st,
                               cudaStream_t s);
    static cudaError_t dt_partials(const DevMesh<T>& m, const HostPhys& p, const T* X,
                                   double* part, cudaStream_t s);
    // X (and, where not NULL, the master averages Wd and the per-case minima of
    // the local time-step limits dtmin, reset before) from FP64
    // component-major W[5][nc], dW[15][nc] (cperm, may be NULL: device cell ->
    // cell of W, dW)
    static cudaError_t pack(const DevMesh<T>& m, const HostPhys& p, const double* W, const double* dW, T* X,
                            double* Wd, unsigned long long* dtmin, cudaStream_t s, const int32_t* cperm = nullptr);
    // FP64 component-major W[5][nc] from Wd (NULL: from the FP64 state X) and
    // dW[15][nc] from X, in the order of cperm's cells; W, dW may be NULL
    static cudaError_t unpack(const double* Wd, const T* X, double* W, double* dW, int64_t nc, cudaStream_t s,
                              const int32_t* cperm = nullptr);
    // conversions for diagnostics
    static cudaError_t to_double(const T* in, double* out, int64_t n, cudaStream_t s);
    // face records in device order -> FP64 in canonical order (perm: device -> canonical),
    // the interface-state entries times the mesh's normals.
    // FP32 stage-1 records hold the interface states and fluxes relative to
    // the mean W_m of the two cells' averages (Stride comment above): W_m
    // sum_k w_k n from the state X, and the records' own flux terms
    // (dt / 2) A F_n(W_m), dt A F_n(W_m), are added back so that the output is
    // the record of the definition.
    static cudaError_t rec_to_double(const DevMesh<T>& m, const T* rec, const int32_t* perm, double* out, int nr,
                                     const T* X, cudaStream_t s);
    // padded reconstruction records -> compact FP64 [nc][50] in centroid-monomial form
    // (rows in the order of cperm's cells)
    static cudaError_t poly_to_double(const T* in, double* out, int64_t nc, cudaStream_t s,
                                      const int32_t* cperm = nullptr);
};

// Local time-step limit of one cell (Sec. 5, Eq. time-step, without C_CFL):
// dr / (|U| + a), and dr^2 / (3 nu) if viscous, from its averages Wv[5],
// in the working precision T.  The constants are rounded to T on the host:
// done in the kernel, each costs every warp FP64 instructions.
template <typename T>
struct DtPhys {
    T gamma, gm1, mu3;  // mu3 = 3 mu (0: inviscid)
    explicit DtPhys(const HostPhys& p)
        : gamma((T)p.gamma), gm1((T)(p.gamma - 1.0)), mu3((T)(p.viscous && p.mu > 0.0 ? 3.0 * p.mu : 0.0)) {}
};
#ifdef __CUDACC__
template <typename T>
__device__ __forceinline__ T local_dt(const T* Wv, T dr, const DtPhys<T>& p) {
    const T ir = T(1) / Wv[0];
    const T u = Wv[1] * ir, v = Wv[2] * ir, w = Wv[3] * ir;
    const T q = u * u + v * v + w * w;
    const T pr = p.gm1 * (Wv[4] - T(0.5) * Wv[0] * q);
    const T a = sqrt(p.gamma * pr * ir);
    T d = dr / (sqrt(q) + a);
    if (p.mu3 > T(0)) {
        const T dv = dr * dr * Wv[0] / p.mu3;
        d = d < dv ? d : dv;
    }
    return d;
}
#endif

// Device buffers of the adjoint sweep (FP64): the two stages' reconstruction
// records, the per-cell record adjoints (up to 40), the per-face adjoints of
// both cells' reconstruction coefficients [nf][2][50] (through the point
// input adjoints [40][nf][3]), their per-cell sums
// [nc][50], stencil adjoints [nc][5][16] and own parts [nc][5], the working
// state adjoints of the stage and of the step [nc][XS], the reverse face
// slots [4][nc] and the positivity-fallback flags of both stages [2][nc].
struct AdjBuffers {
    const double* poly1;
    const double* poly2;
    double *src, *lx, *lpf, *lp, *ld, *own, *lXs, *lX1;
    double *lbn, *lds;  // WENO only: neighbour-slope adjoints [nc][5][4][3], [nc][5][4]
    double* lwo;        // open-face ghost adjoints [nf][5]
    int8_t* rev;
    int32_t* fallback;
};
// out row r = in row map[r] for rows of width_words 4-byte words
cudaError_t launch_rows_gather(const void* in, void* out, int64_t nrows, int width_words, const int32_t* map,
                               cudaStream_t s);
// the one-launch stage's grid barrier on a barrier nothing completes: each
// of two blocks polls `limit` times, gives up and sets ERR_TIMEOUT
cudaError_t launch_grid_barrier_probe(unsigned* gbar, int32_t* err, int limit, cudaStream_t s);
// one stage of the FP32-bulk step (reconstruction with the neighbours'
// slopes recomputed, face flux, cell update) as one persistent launch with
// grid-wide barriers; gbar: 2 unsigned words of device scratch (reset by the
// launch); fin (stage 1, may be NULL) as for the reconstruction
cudaError_t launch_stage(const DevMesh<float>& m, const HostPhys& p, const DevState<float>& st, int stage,
                         const Launch<float>::Finalize* fin, unsigned* gbar, cudaStream_t s);
// a bounded mbarrier wait that gives up (nothing completes it): sets ERR_TIMEOUT
cudaError_t launch_wait_probe(int32_t* err, int tries, cudaStream_t s);

// lambda (W^n, grad W^n) from lambda (W^{n+1}, grad W^{n+1}) for one step
// with the frozen time step dt (public [component][cell] FP64 layouts)
cudaError_t adjoint_reverse(const DevMesh<double>& m, const HostPhys& p, double dt, const AdjBuffers& b,
                            const double* X1, const double* X2, const double* lW, const double* ldW, double* oW,
                            double* odW, cudaStream_t s);

// sets dt_fixed and t_end; with reset_time also zeroes the case times and
// steps and sets the case minima to +inf; err (may be NULL) is cleared
cudaError_t launch_set_control(double* ctrl, double* case_t, double* case_dt,
                               unsigned long long* case_dtmin, int32_t ncase, double dt_fixed,
                               double t_end, int reset_time, int32_t* err, cudaStream_t s);
int update_blocks(int64_t nc);  // blocks of CELLS_PER_BLOCK cells

}  // namespace gks
