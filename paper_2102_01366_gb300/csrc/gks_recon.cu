// gks_recon.cu -- reconstruction kernels (Sec. 4.1-4.3), sm_103a, FP64 and
// FP32-bulk instantiations.
//
//   k_slopes   reconstruction step 1: |b|^2 of the P1 slopes (Sec. 4.3)
//   k_recon    reconstruction step 2: P2 by the 9x16 operator, smoothness
//              indicators, two-step beta_0, nonlinear weights, positivity
//              (Sec. 4.1-4.3); R written about the centroid in monomial form
//
// The first kernel of a step (block 0) also turns the per-case minima of
// the local time-step limits into each case's step (Sec. 5).
#include <cuda_runtime.h>

#include "gks_recon.cuh"

namespace gks {

constexpr int SLOPES_THREADS = 64;  // threads (cells) a block of k_slopes

// reconstruction step 1: |b|^2 of the P1 slopes b = M1 (Q_nb - Q_0), Sec.
// 4.3, the products in the operator precision TO; beta_0 of the cells around
// (Eq. p0-non-linear-weight) takes the slopes in this form only.  One thread
// per cell: the averages of a cell are whole 16-byte vectors and M1 is read
// in full lines (both stages, FP32: 409,644 cells 74 -> 54 us, 580,320 cells
// 110 -> 71 us against five lanes a cell).  The arithmetic is that of p1_slope.
template <typename T, typename TO>
__global__ void __launch_bounds__(SLOPES_THREADS) k_slopes(DevMesh<T> m, const T* __restrict__ X,
                                                            T* __restrict__ s2, FinArg<T> fin) {
    if (fin.dtmin && blockIdx.x == 0) finalize_cases(fin.dtmin, fin.case_t, fin.case_dt, fin.ncase, fin.cfl, fin.ctrl);
    const int64_t c = (int64_t)blockIdx.x * SLOPES_THREADS + threadIdx.x, nc = m.nc;
    if (c >= nc) return;
    constexpr bool F32 = sizeof(T) == 4;
    constexpr int XSR = Stride<T>::xs, NA = F32 ? 12 : 6;  // words that hold the averages
    int nb[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) nb[f] = m.nbr[f * nc + c];
    T own[NA], x[4][NA];
    load_vec<NA>(X + c * XSR, own);
#pragma unroll
    for (int f = 0; f < 4; ++f) load_vec<NA>(X + (nb[f] >= 0 ? (int64_t)nb[f] : c) * XSR, x[f]);
    TO op[12];
#pragma unroll
    for (int k = 0; k < 12; ++k) op[k] = m1_at<T, TO>(m, k, c);
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const TO* wo = wall_ops<T, TO>(m, c, q);  // the wall-constrained slopes of Sec. 4.4
        TO s[3] = {TO(0), TO(0), TO(0)};
#pragma unroll
        for (int f = 0; f < 4; ++f) {
            if (nb[f] < 0) continue;
            TO dq;
            if constexpr (F32)
                dq = (to_op<TO>(x[f][q]) - to_op<TO>(own[q])) + (to_op<TO>(x[f][XLO + q]) - to_op<TO>(own[XLO + q]));
            else
                dq = x[f][q] - own[q];
#pragma unroll
            for (int i = 0; i < 3; ++i) s[i] += (wo ? wo[WOP_W1 + i * 5 + f] : op[i * 4 + f]) * dq;
        }
        if (wo) {
            const TO q0 = avg_at<T, TO>(X, c, q);
#pragma unroll
            for (int i = 0; i < 3; ++i) s[i] += wo[WOP_W1 + i * 5 + 4] * q0;
        }
        const T b[3] = {from_op<T>(s[0]), from_op<T>(s[1]), from_op<T>(s[2])};
        s2[c * 5 + q] = slope_sq(b);
    }
}

template <typename T, typename TO, bool WALL>
__global__ void __launch_bounds__(CELL_THREADS) k_recon(DevMesh<T> m, ReconConst<T> rc,
                                                         const T* __restrict__ X,
                                                         const T* __restrict__ s2_in,
                                                         T* __restrict__ slopes_out,
                                                         T* __restrict__ poly,
                                                         int32_t* __restrict__ fallback,
                                                         FinArg<T> fin, int32_t* __restrict__ err) {
    __shared__ alignas(128) Tile<TO> sT;
    __shared__ alignas(8) unsigned long long bar;
    if (threadIdx.x == 0) mbar_init(&bar, 1);
    __syncthreads();  // the barrier exists before anyone waits on it
    if (fin.dtmin && blockIdx.x == 0) finalize_cases(fin.dtmin, fin.case_t, fin.case_dt, fin.ncase, fin.cfl, fin.ctrl);
    recon_cells<T, TO, WALL>(m, rc, X, s2_in, slopes_out, poly, fallback, err, blockIdx.x, threadIdx.x, sT, &bar,
                             0);
}

// --------------------------------------------------------------------------
// launchers
// --------------------------------------------------------------------------
template <typename T>
static FinArg<T> fin_arg(const typename Launch<T>::Finalize* fin) {
    FinArg<T> a;
    a.dtmin = fin ? fin->dtmin : nullptr;
    a.case_t = fin ? fin->case_t : nullptr;
    a.case_dt = fin ? fin->case_dt : nullptr;
    a.ncase = fin ? fin->ncase : 0;
    a.cfl = fin ? fin->cfl : 0.0;
    a.ctrl = fin ? fin->ctrl : nullptr;
    return a;
}

template <typename T>
cudaError_t Launch<T>::slopes(const DevMesh<T>& m, const T* X, T* s2, const Finalize* fin,
                              cudaStream_t s) {
    if (m.nc == 0) return cudaSuccess;
    const unsigned grid = (unsigned)((m.nc + SLOPES_THREADS - 1) / SLOPES_THREADS);
    if (m.M1d && sizeof(T) == 4)
        k_slopes<T, double><<<grid, SLOPES_THREADS, 0, s>>>(m, X, s2, fin_arg<T>(fin));
    else
        k_slopes<T, T><<<grid, SLOPES_THREADS, 0, s>>>(m, X, s2, fin_arg<T>(fin));
    return cudaGetLastError();
}

template <typename T>
cudaError_t Launch<T>::recon(const DevMesh<T>& m, const HostPhys& p, const T* X, const T* s2_in,
                             T* slopes, T* poly, int32_t* fallback, const Finalize* fin, int32_t* err,
                             cudaStream_t s) {
    if (m.nc == 0) return cudaSuccess;
    ReconConst<T> rc;
    rc.gm1 = (T)(p.gamma - 1.0);
    rc.eps = (T)p.eps_weno;
    rc.weno = p.weno;
    rc.order = p.order;
    // the wall-constrained instances only where the mesh has such cells
    auto go = [&](auto kernel) {
        kernel<<<cell_grid(m.nc), CELL_THREADS, 0, s>>>(m, rc, X, s2_in, slopes, poly, fallback, fin_arg<T>(fin),
                                                         err);
    };
    if (m.tiled && sizeof(T) == 4)
        m.wslot ? go(k_recon<T, double, true>) : go(k_recon<T, double, false>);
    else
        m.wslot ? go(k_recon<T, T, true>) : go(k_recon<T, T, false>);
    return cudaGetLastError();
}


#define GKS_RECON_INST(T)                                                                                  \
    template cudaError_t Launch<T>::slopes(const DevMesh<T>&, const T*, T*, const Launch<T>::Finalize*,     \
                                           cudaStream_t);                                                  \
    template cudaError_t Launch<T>::recon(const DevMesh<T>&, const HostPhys&, const T*, const T*, T*, T*,   \
                                          int32_t*, const Launch<T>::Finalize*, int32_t*, cudaStream_t);
GKS_RECON_INST(double)
GKS_RECON_INST(float)

// The bounded wait's failure path without a fault: an mbarrier that expects
// bytes no copy will deliver (nothing is in flight), polled `tries` times by
// the same try_wait as the reconstruction's tile wait; giving up sets
// ERR_TIMEOUT exactly as a stalled tile copy would.
__global__ void k_wait_probe(int32_t* __restrict__ err, int tries) {
    __shared__ alignas(8) unsigned long long bar;
    if (threadIdx.x == 0) mbar_init(&bar, 1);
    __syncthreads();
    if (threadIdx.x == 0) mbar_arrive_expect_tx(&bar, 16);
    __syncthreads();
    bool ok = false;
    for (int i = 0; i < tries && !ok; ++i) ok = mbar_try_wait(&bar, 0);
    if (!ok && (threadIdx.x & 31) == 0) atomicOr(err, ERR_TIMEOUT);
}

cudaError_t launch_wait_probe(int32_t* err, int tries, cudaStream_t s) {
    k_wait_probe<<<1, 64, 0, s>>>(err, tries);
    return cudaGetLastError();
}

}  // namespace gks
