// gks_kernels.cu -- cell-update and bookkeeping kernels of one two-stage step
// (sm_103a, FP64 and FP32-bulk instantiations).  The reconstruction kernels
// are in gks_recon.cu, the face flux in gks_flux.cu.
//
//   k_update1  cell-ordered gather of the 4 face records (CSR, signed):
//              W*, grad W* and the saved stage-1 terms
//   k_update2  W^{n+1}, grad W^{n+1}; per-case minima of the next step's
//              local time-step limits (Sec. 5) and residual sums
//   k_dt_*     time-step rule of Sec. 5 (deterministic per-block minima)
//   k_pack / k_unpack   public [component][cell] FP64 state <-> the
//              cell-major working state
//
// No atomics on data: every sum has a fixed order, so results are
// reproducible run to run (the per-case minima use atomicMin, which is
// exact).
#include <cuda_runtime.h>

#include <algorithm>

#include "gks_update.cuh"

namespace gks {

constexpr int PACK_THREADS = 128;  // threads (cells) a block of k_pack, k_unpack

template <typename T>
__global__ void __launch_bounds__(CELL_THREADS) k_update1(DevMesh<T> m, DevState<T> st) {
    update1_cells<T>(m, st, blockIdx.x, threadIdx.x);
}

template <typename T>
__global__ void __launch_bounds__(CELL_THREADS) k_update2(DevMesh<T> m, DtPhys<T> p, DevState<T> st) {
    __shared__ T red[CELL_THREADS / 32][5];
    update2_cells<T>(m, p, st, blockIdx.x, threadIdx.x, 0, red);
}

// local limit of one cell from the averages in X, one thread per cell
template <typename T>
__device__ __forceinline__ T cell_dt(const DevMesh<T>& m, const DtPhys<T>& p, const T* __restrict__ X, int64_t c) {
    T Wv[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) Wv[q] = X[c * Stride<T>::xs + q];
    return local_dt(Wv, m.dr[c], p);
}

// block b: the minimum over its CELLS_PER_BLOCK cells (one warp of the block
// size that update_blocks counts)
template <typename T>
__global__ void __launch_bounds__(32) k_dt_partials(DevMesh<T> m, DtPhys<T> p, const T* __restrict__ X,
                                                    double* __restrict__ part) {
    const int64_t c = (int64_t)blockIdx.x * CELLS_PER_BLOCK + threadIdx.x;
    T mn = T(INFINITY);
    if (threadIdx.x < CELLS_PER_BLOCK && c < m.nc) mn = cell_dt(m, p, X, c);
    if (!(mn < T(INFINITY))) mn = T(INFINITY);
    mn = warp_min(mn);
    if (threadIdx.x == 0) part[(int64_t)blockIdx.x * PART_N + PART_DTMIN] = (double)mn;
}

__global__ void k_set_control(double* ctrl, double* case_t, double* case_dt, unsigned long long* dtmin,
                              int32_t ncase, double dt_fixed, double t_end, int reset, int32_t* err) {
    if (threadIdx.x == 0 && blockIdx.x == 0) {
        ctrl[CTRL_DT_FIXED] = dt_fixed;
        ctrl[CTRL_T_END] = t_end;
        if (err) *err = 0;
    }
    if (reset)
        for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < ncase; k += gridDim.x * blockDim.x) {
            case_t[k] = 0.0;
            case_dt[k] = 0.0;
            dtmin[k] = (unsigned long long)__double_as_longlong(INFINITY);
        }
}

template <typename A, typename B>
__global__ void k_convert(const A* __restrict__ in, B* __restrict__ out, int64_t n) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
        out[i] = (B)in[i];
}

// One thread per cell: rows of the caller's [component][cell] arrays are read
// (written) in full lines, records as 16-byte vectors.  cperm (may be NULL):
// device cell -> the caller's cell of W, dW.  Bound by memory: with one thread
// per word of the record, each reading another row, an initialisation and a
// read-back of 1.57 M cells in FP32 took about 1.17 ms, 0.40 ms this way.
//
// k_pack also writes (where not NULL) the FP64 master averages Wd and each
// case's minimum of the local time-step limits into dtmin; k_unpack takes the
// averages from Wd (NULL: from the FP64 working state): one launch each, where
// copies, conversions, a memset and a kernel for the minima were five and two
// (a run of two steps on 24,576 cells in FP32, start to end: 277 -> 261 us).
template <typename T>
__global__ void __launch_bounds__(PACK_THREADS) k_pack(DevMesh<T> m, DtPhys<T> p, const double* __restrict__ W,
                                                       const double* __restrict__ dW, T* __restrict__ X,
                                                       double* __restrict__ Wd,
                                                       unsigned long long* __restrict__ dtmin,
                                                       const int32_t* __restrict__ cperm) {
    constexpr int XSR = Stride<T>::xs;
    const int64_t nc = m.nc, d0 = (int64_t)blockIdx.x * PACK_THREADS + threadIdx.x;
    const bool active = d0 < nc;
    const int64_t d = active ? d0 : nc - 1;
    const int64_t c = cperm ? (int64_t)cperm[d] : d;
    T x[XSR];
#pragma unroll
    for (int j = 0; j < XSR; ++j) x[j] = T(0);
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const double w = W[q * nc + c];
        if (Wd && active) Wd[q * nc + d] = w;
        if constexpr (sizeof(T) == 4)
            split_pair(w, x[q], x[XLO + q]);
        else
            x[q] = w;
    }
#pragma unroll
    for (int j = 0; j < 15; ++j) {
        if constexpr (sizeof(T) == 4)
            x[Stride<T>::xg + j] = narrow(dW[j * nc + c]);
        else
            x[Stride<T>::xg + j] = dW[j * nc + c];
    }
    if (active) store_vec<XSR>(X + d * XSR, x);
    if (dtmin) warp_case_min(active ? local_dt(x, m.dr[d], p) : T(INFINITY), m.cell_case[d], dtmin);
}

template <typename T>
__global__ void __launch_bounds__(PACK_THREADS) k_unpack(const double* __restrict__ Wd, const T* __restrict__ X,
                                                         double* __restrict__ W, double* __restrict__ dW,
                                                         int64_t nc, const int32_t* __restrict__ cperm) {
    constexpr int XSR = Stride<T>::xs;
    const int64_t d = (int64_t)blockIdx.x * PACK_THREADS + threadIdx.x;
    if (d >= nc) return;
    const int64_t c = cperm ? (int64_t)cperm[d] : d;
    T x[XSR];
    if (dW || !Wd) load_vec<XSR>(X + d * XSR, x);
    if (W)
#pragma unroll
        for (int q = 0; q < 5; ++q) W[q * nc + c] = Wd ? Wd[q * nc + d] : widen(x[q]);
    if (dW)
#pragma unroll
        for (int j = 0; j < 15; ++j) dW[j * nc + c] = widen(x[Stride<T>::xg + j]);
}

// out row r = in row map[r], rows of `width` words of 4 bytes
__global__ void k_rows_gather(const uint32_t* __restrict__ in, uint32_t* __restrict__ out, int64_t nrows, int width,
                              const int32_t* __restrict__ map) {
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nrows * width; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t r = i / width;
        out[i] = in[(int64_t)map[r] * width + (i - r * width)];
    }
}

template <typename T>
__global__ void k_rec_out(DevMesh<T> m, const T* __restrict__ rec, const int32_t* __restrict__ perm,
                          double* __restrict__ out, int nr, const T* __restrict__ X) {
    constexpr int XSR = Stride<T>::xs;
    const int64_t nf = m.nf;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nf * nr; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t d = i / nr;
        const int j = (int)(i - d * nr);
        // the public record has the interface-state entries times the normal
        const int nflux = nr == 40 ? 10 : 5;
        const T* r = rec + d * (nr == 40 ? rec_stride<T, 40>() : rec_stride<T, 20>());
        const int je = j - nflux;
        const int J = nr == 40 ? rec_entries<T, 40>() : rec_entries<T, 20>();
        double v = j < nflux ? (double)r[(j % 5) * J + j / 5]
                             : (double)r[((je % 15) / 3) * J + nflux / 5 + je / 15] *
                                   (double)m.fnw[d * 4 + (je % 15) % 3];
        if (sizeof(T) == 4 && nr == 40 && j < 10) {
            // the reference flux (dt / 2) A F_n(W_m), twice in the S entries
            const double ref = (double)r[(j % 5) * J + 4] + (double)r[(j % 5) * J + 5];
            v += j < 5 ? ref : 2.0 * ref;
        }
        if (sizeof(T) == 4 && nr == 40 && j >= 10) {
            // the mean of the two averages (the interior one on a boundary
            // face) times sum_k w_k n = 3 w n
            const int k = (j - 10) % 15, q = k / 3, dir = k - 3 * q;
            const int L = m.flr[d], R = m.flr[m.nf + d];
            auto avg = [&](int c) { return (double)X[(int64_t)c * XSR + q] + (double)X[(int64_t)c * XSR + XLO + q]; };
            const double wm = (L >= 0 && R >= 0) ? 0.5 * (avg(L) + avg(R)) : avg(L >= 0 ? L : R);
            const T* nw = m.fnw + d * 4;
            v += wm * 3.0 * (double)nw[3] * (double)nw[dir];
        }
        out[(int64_t)perm[d] * nr + j] = v;
    }
}

template <typename T>
__global__ void k_poly_out(const T* __restrict__ in, double* __restrict__ out, int64_t nc,
                           const int32_t* __restrict__ cperm) {
    constexpr int PS = Stride<T>::poly;
    for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < nc * 50; i += (int64_t)gridDim.x * blockDim.x) {
        const int64_t c = i / 50;
        const int k = (int)(i - c * 50);
        const int64_t o = (cperm ? (int64_t)cperm[c] : c) * 50 + k;
        double v = (double)in[c * PS + k];
        if (sizeof(T) == 4 && k % 10 == 0) {
            // FP32 records hold R(centroid) minus the average: add the average back
            const int q = k / 10;
            v += (double)in[c * PS + PHI + q] + (double)in[c * PS + PLO + q];
        }
        out[o] = v;
    }
}

// --------------------------------------------------------------------------
// launchers
// --------------------------------------------------------------------------
int update_blocks(int64_t nc) { return (int)cell_grid(nc); }

template <typename T>
cudaError_t Launch<T>::update1(const DevMesh<T>& m, const HostPhys& p, const DevState<T>& st, cudaStream_t s) {
    if (m.nc == 0) return cudaSuccess;
    k_update1<T><<<cell_grid(m.nc), CELL_THREADS, 0, s>>>(m, st);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::update2(const DevMesh<T>& m, const HostPhys& p, const DevState<T>& st,
                               cudaStream_t s) {
    if (m.nc == 0) return cudaSuccess;
    k_update2<T><<<cell_grid(m.nc), CELL_THREADS, 0, s>>>(m, DtPhys<T>(p), st);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::dt_partials(const DevMesh<T>& m, const HostPhys& p, const T* X,
                                   double* part, cudaStream_t s) {
    if (m.nc == 0) return cudaSuccess;
    k_dt_partials<T><<<cell_grid(m.nc), 32, 0, s>>>(m, DtPhys<T>(p), X, part);
    return cudaGetLastError();
}

static inline unsigned pack_grid(int64_t nc) { return (unsigned)((nc + PACK_THREADS - 1) / PACK_THREADS); }

static inline unsigned ew_grid(int64_t n) { return (unsigned)((n + 255) / 256 < 8192 ? (n + 255) / 256 : 8192); }

template <typename T>
cudaError_t Launch<T>::pack(const DevMesh<T>& m, const HostPhys& p, const double* W, const double* dW, T* X,
                            double* Wd, unsigned long long* dtmin, cudaStream_t s, const int32_t* cperm) {
    if (m.nc == 0) return cudaSuccess;
    k_pack<T><<<pack_grid(m.nc), PACK_THREADS, 0, s>>>(m, DtPhys<T>(p), W, dW, X, Wd, dtmin, cperm);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::unpack(const double* Wd, const T* X, double* W, double* dW, int64_t nc, cudaStream_t s,
                              const int32_t* cperm) {
    if (nc == 0) return cudaSuccess;
    k_unpack<T><<<pack_grid(nc), PACK_THREADS, 0, s>>>(Wd, X, W, dW, nc, cperm);
    return cudaGetLastError();
}

cudaError_t launch_rows_gather(const void* in, void* out, int64_t nrows, int width_words, const int32_t* map,
                               cudaStream_t s) {
    if (nrows == 0) return cudaSuccess;
    k_rows_gather<<<ew_grid(nrows * width_words), 256, 0, s>>>(static_cast<const uint32_t*>(in),
                                                               static_cast<uint32_t*>(out), nrows, width_words, map);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::to_double(const T* in, double* out, int64_t n, cudaStream_t s) {
    if (n == 0) return cudaSuccess;
    k_convert<T, double><<<(unsigned)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096), 256, 0, s>>>(in, out, n);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::rec_to_double(const DevMesh<T>& m, const T* rec, const int32_t* perm, double* out, int nr,
                                     const T* X, cudaStream_t s) {
    if (m.nf == 0) return cudaSuccess;
    const int64_t n = m.nf * nr;
    k_rec_out<T><<<(unsigned)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096), 256, 0, s>>>(m, rec, perm, out, nr, X);
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::poly_to_double(const T* in, double* out, int64_t nc, cudaStream_t s, const int32_t* cperm) {
    if (nc == 0) return cudaSuccess;
    const int64_t n = nc * 50;
    k_poly_out<T><<<(unsigned)((n + 255) / 256 < 4096 ? (n + 255) / 256 : 4096), 256, 0, s>>>(in, out, nc, cperm);
    return cudaGetLastError();
}

cudaError_t launch_set_control(double* ctrl, double* case_t, double* case_dt, unsigned long long* case_dtmin,
                               int32_t ncase, double dt_fixed, double t_end, int reset_time, int32_t* err,
                               cudaStream_t s) {
    const int grid = reset_time ? (int)((ncase + 255) / 256 < 1024 ? (ncase + 255) / 256 : 1024) : 1;
    k_set_control<<<grid < 1 ? 1 : grid, 256, 0, s>>>(ctrl, case_t, case_dt, case_dtmin, ncase, dt_fixed,
                                                      t_end, reset_time, err);
    return cudaGetLastError();
}


#define GKS_CELLS_INST(T)                                                                                   \
    template cudaError_t Launch<T>::update1(const DevMesh<T>&, const HostPhys&, const DevState<T>&,         \
                                            cudaStream_t);                                                  \
    template cudaError_t Launch<T>::update2(const DevMesh<T>&, const HostPhys&, const DevState<T>&,         \
                                            cudaStream_t);                                                  \
    template cudaError_t Launch<T>::dt_partials(const DevMesh<T>&, const HostPhys&, const T*, double*,      \
                                                cudaStream_t);                                              \
    template cudaError_t Launch<T>::pack(const DevMesh<T>&, const HostPhys&, const double*, const double*, T*, \
                                         double*, unsigned long long*, cudaStream_t, const int32_t*);       \
    template cudaError_t Launch<T>::unpack(const double*, const T*, double*, double*, int64_t, cudaStream_t, \
                                           const int32_t*);                                                 \
    template cudaError_t Launch<T>::to_double(const T*, double*, int64_t, cudaStream_t);                    \
    template cudaError_t Launch<T>::rec_to_double(const DevMesh<T>&, const T*, const int32_t*, double*, int, \
                                                  const T*, cudaStream_t);                                  \
    template cudaError_t Launch<T>::poly_to_double(const T*, double*, int64_t, cudaStream_t, const int32_t*);
GKS_CELLS_INST(double)
GKS_CELLS_INST(float)

}  // namespace gks
