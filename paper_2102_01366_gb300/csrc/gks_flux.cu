// gks_flux.cu -- face flux kernels (Sec. 2.2, 3, 4.4, 4.5), sm_103a, FP64 and
// FP32-bulk instantiations.
//
//   k_flux         face-ordered, 6 threads per face (3 Gauss points x 2
//                  sides): R of both cells at the Gauss points, face frame,
//                  kinetic solution (Eq. 2nd-flux with the equilibrium state
//                  of Eq. new-equ-part), weighted face record of the stage
//                  (Sec. 3 Eqs. linear-system, s2o4, step-du); FP32
//   k_flux_single  the same with one thread per Gauss point; FP64
//
// Boundary faces take their ghost side from the face's kind (Sec. 4.4 slip
// wall, a fixed state, or zeroth-order extrapolation).
#include <cuda_runtime.h>

#include "gks_flux.cuh"
#include "gks_kinetic.cuh"

namespace gks {

// --------------------------------------------------------------------------
// face flux
// --------------------------------------------------------------------------


// 3 threads per face, one Gauss point each (FP64).  The kinetic solution's
// sums over the two sides are accumulated in one loop body, so only one
// side's state and moments are live at a time.  VISC: the time slopes of
// viscous flow.
//
// Bound by the FP64 pipe (2 lanes an SM: 16 cycles a warp instruction), so
// what counts is the number of FP64 instructions: 1,601 a Gauss point here
// against about 3,000 with the moment tables, 896 -> 484 us on 49,280 faces
// (stage 1, inviscid; pipe 86 % busy).  Occupancy does not matter: 2 blocks
// an SM (232 registers, no spills) take 494 us, 5 blocks (128 registers)
// 497 us.
template <typename T, int NR, bool VISC>
__global__ void __launch_bounds__(3 * FLUX_FACES, 2)
    k_flux_single(DevMesh<T> m, Phys<T> ph, const T* __restrict__ Wavg, const T* __restrict__ poly,
                  T* __restrict__ rec, const double* __restrict__ ctrl, double dt_override) {
    __shared__ T red[FLUX_FACES * 3 * NR];
    const int lf = threadIdx.x / 3;
    const int k = threadIdx.x - 3 * lf;
    const int64_t f = (int64_t)blockIdx.x * FLUX_FACES + lf;
    T* mine = red + (lf * 3 + k) * NR;
    if (f < m.nf) {
        const int L = m.flr[f], Rc = m.flr[m.nf + f];
        const double dtc = ctrl ? ctrl[m.cell_case[L >= 0 ? L : Rc]] : dt_override;
        const T dt = dtc > 0.0 ? (T)dtc : T(1);
        const T* geo = m.fgeo + f * FGEO;
        const T n[3] = {geo[0], geo[1], geo[2]};
        T Rm[3][3];
        face_frame(n, Rm);
        KSums<T> S;
        S.init();
        T pl = T(0), pr = T(0);
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {
            T tW[5], tg[3][5];
            side_state<T, true>(m, ph, Wavg, poly, geo, Rm, L, Rc, side, k, tW, tg);
            pl = pr;
            pr = kin_side<VISC>(ph, tW, tg, side == 0 ? +1 : -1, S);
        }
        T Wc[5], Fh[5], D[5], W0[5], dWt[5];
        finish_point<VISC, false>(ph, S, pl, pr, dt, Wc, Fh, D, W0, dWt);
        to_global(Rm, Fh);
        to_global(Rm, D);
        to_global(Rm, W0);
        to_global(Rm, dWt);
        const T w = geo[3];
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            if (NR == 40) {
                mine[q] = w * Fh[q];
                mine[5 + q] = w * (T(2) * Fh[q] - D[q] * T(1.0 / 3.0));
                const T ws = w * (W0[q] + T(0.5) * dWt[q]);
                const T w0 = w * W0[q];
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    mine[10 + 3 * q + i] = ws * n[i];
                    mine[25 + 3 * q + i] = w0 * n[i];
                }
            } else {
                mine[q] = w * T(4.0 / 3.0) * D[q];
                const T dg = w * dWt[q];
#pragma unroll
                for (int i = 0; i < 3; ++i) mine[5 + 3 * q + i] = dg * n[i];
            }
        }
    }
    __syncthreads();
    const int64_t base = (int64_t)blockIdx.x * FLUX_FACES;
    for (int idx = threadIdx.x; idx < FLUX_FACES * NR; idx += 3 * FLUX_FACES) {
        const int fl = idx / NR, j = idx - fl * NR;
        if (base + fl < m.nf) {
            const T* r = red + fl * 3 * NR + j;
            rec[(base + fl) * NR + j] = (r[0] + r[NR]) + r[2 * NR];
        }
    }
}

// --------------------------------------------------------------------------
// launcher
// --------------------------------------------------------------------------


template <typename T>
cudaError_t Launch<T>::flux(const DevMesh<T>& m, const HostPhys& p, const T* W, const T* poly, T* rec,
                            const double* ctrl, double dt_override, int stage, cudaStream_t s, int variant) {
    // ctrl is the per-case step array (NULL: dt_override everywhere)
    if (m.nf == 0) return cudaSuccess;
    const unsigned grid = (unsigned)((m.nf + FLUX_FACES - 1) / FLUX_FACES);
    const Phys<T> ph = make_phys<T>(p);
    if constexpr (sizeof(T) == 4) {
        // FP32: the two sides of each Gauss point in separate warps; variant
        // 1 trades registers for occupancy (3 blocks per SM), variant 0 keeps
        // 2 blocks per SM without spills; the Pr fix has its own instances
        const bool prf = p.prf != 0.0;
        // meshes with isothermal or moving walls: the instances that carry
        // their ghosts (gks_flux_xw.cu)
        if (m.xwalls) return launch_flux_xw(m, ph, W, poly, rec, ctrl, dt_override, stage, s, variant, prf);
        auto go = [&](auto kernel) { kernel<<<grid, 2 * FP_GP, 0, s>>>(m, ph, W, poly, rec, ctrl, dt_override); };
        if (variant == 1) {
            if (stage == 1)
                prf ? go(k_flux<T, 40, 3, true, false>) : go(k_flux<T, 40, 3, false, false>);
            else
                prf ? go(k_flux<T, 20, 3, true, false>) : go(k_flux<T, 20, 3, false, false>);
        } else {
            if (stage == 1)
                prf ? go(k_flux<T, 40, 2, true, false>) : go(k_flux<T, 40, 2, false, false>);
            else
                prf ? go(k_flux<T, 20, 2, true, false>) : go(k_flux<T, 20, 2, false, false>);
        }
    } else {
        auto go = [&](auto kernel) { kernel<<<grid, 3 * FLUX_FACES, 0, s>>>(m, ph, W, poly, rec, ctrl, dt_override); };
        if (stage == 1)
            p.viscous ? go(k_flux_single<T, 40, true>) : go(k_flux_single<T, 40, false>);
        else
            p.viscous ? go(k_flux_single<T, 20, true>) : go(k_flux_single<T, 20, false>);
    }
    return cudaGetLastError();
}


template cudaError_t Launch<double>::flux(const DevMesh<double>&, const HostPhys&, const double*, const double*,
                                          double*, const double*, double, int, cudaStream_t, int);
template cudaError_t Launch<float>::flux(const DevMesh<float>&, const HostPhys&, const float*, const float*,
                                         float*, const double*, double, int, cudaStream_t, int);

}  // namespace gks
