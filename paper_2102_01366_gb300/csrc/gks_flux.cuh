// gks_flux.cuh -- the face flux of one block of faces (Sec. 2.2, 3, 4.4,
// 4.5), FP64 and FP32 bulk, shared by the standalone flux kernel and the
// persistent stage kernel.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "gks_cells.cuh"
#include "gks_device.cuh"
#include "gks_face.cuh"
#include "gks_kernels.h"
#include "gks_kinetic.cuh"

namespace gks {

// A block of FLUX_FACES faces is worked on by FLUX_THREADS threads, one per
// Gauss point.  A thread takes the two sides of its point in turn: R at the
// point, face frame, primitive derivatives, and the sums over both sides
// (KSums), from which the point's outputs follow; nothing is exchanged
// between threads until the three points of a face are added up.  Outputs
// stay in the face frame until then, so the rotation back and the weights are
// done once per face.
//
// FP32 is bound by instruction issue, with the gathers of the two 240-byte
// reconstruction records behind it; the faster layout is therefore the one
// with the fewest instructions and barriers.  Stage 1 / stage 2 on 3.15 M
// faces 905 / 594 us, on 49,280 faces 22.1 / 18.5 us.  Against it: two threads
// a point (one a side, in two warps), which repeat the frame and meet four
// times at a barrier through 60 KB of shared memory, 2,087 / 1,335 us and 40.6 /
// 28.7 us; persistent blocks that fetch the next block's records into shared
// memory, which hides the gathers but has a block's three warps wait for each
// other, stage 1 1,207 us (the present layout at that time 1,108).
// FP64 is bound by its pipe (16 cycles a warp instruction): rotating and
// weighting per face instead of per point took 484 -> 450 us on 49,280 faces.

// Fh, D, W0, dW of a point (stage 2: D, dW); rows padded to an odd length
// so that the threads of a warp write to different banks
template <int NR>
constexpr int flux_vals() { return NR == 40 ? 20 : 10; }

// FP32 stage 2 has its faces' records and geometry copied to shared memory
// while it forms the face frames: one barrier, but no wait for a gather in
// either side's turn (stage 2 on 3.15 M faces 679 -> 631 us, viscous on 1.16 M
// 287 -> 255 us).  In stage 1, whose longer output leaves the L1 less room and
// which prefetches the right side, it cost 975 -> 1,018 us.
template <typename T, int NR>
constexpr bool flux_copies() { return sizeof(T) == 4 && NR == 20; }

template <typename T, int NR, int TH = FLUX_THREADS>
struct FluxSmem {
    // FP32 stage 2: both sides' reconstruction records and the geometry of each face
    alignas(16) T poly[flux_copies<T, NR>() ? (TH + 2) / 3 : 1][2][flux_copies<T, NR>() ? Stride<T>::poly : 4];
    alignas(16) T geo[flux_copies<T, NR>() ? (TH + 2) / 3 : 1][flux_copies<T, NR>() ? FGEO : 4];
    T out[TH][flux_vals<NR>() + 1];
    T frame[(TH + 2) / 3][7];                                 // tangents of the face frame
    T rec[sizeof(T) == 4 && NR == 40 ? (TH + 2) / 3 : 1][33];  // the block's records (FP32 stage 1)
};

// hi (5) and lo (5) parts of a record's cell average, in whole vectors: ten
// single loads each went to as many lines as the warp has faces
__device__ __forceinline__ void load_average(const float* P, float* hi, float* lo) {
    static_assert(PHI == 50 && PLO == 55 && POLY_STRIDE32 == 60, "the averages end the record");
    float v[12];
    load_vec<12>(P + 48, v);
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        hi[q] = v[2 + q];
        lo[q] = v[7 + q];
    }
}

// Stage 1, FP32: the interface state W^c of Eq. new-equ-part relative to W_m,
// the mean of the two cells' averages (the interior cell's average on a
// boundary face), into dW, and F_1(W^c) - F_1(W_m) into dF (face frame).
// The gradient records sum w W(0) n over a cell's faces, where the O(|W|)
// parts cancel to |Omega| grad W, and the flux records likewise to |Omega|
// div F: an FP32 W^c or F would leave its rounding, eps |W|, in each face
// term, an error ~ eps |W| / dr in the gradient.  Taken relative to W_m
// (exact differences of the hi / lo averages) and by the half-difference
// rules, both carry rounding relative to themselves only.  Interior and open
// faces; wall and fixed faces subtract directly.
//   al, ar       the sides' records (a missing side's: the interior cell's)
//   dsum, ddiff  sum and difference (left - right) of the sides' R - average
//   hl, hr       the sides' half-space moments
__device__ __forceinline__ void interface_deviation(const float* al, const float* ar, int L, int Rc,
                                                    const float (*Rm)[3], const float* dsum, const float* ddiff,
                                                    const HalfSpace<float>& hl, const HalfSpace<float>& hr,
                                                    const float* Wc, float gm1, float* dW,
                                                    float* dF) {
    const bool pair = (L >= 0 || L == FLR_OPEN) && (Rc >= 0 || Rc == FLR_OPEN);
    float Wm[5], sg[5], hg[5], ql[5], ll[5], qr[5], lr[5];
    load_average(al, ql, ll);
    load_average(ar, qr, lr);
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        Wm[q] = 0.5f * (ql[q] + qr[q]);
        sg[q] = 0.5f * dsum[q];
        hg[q] = 0.5f * (((ql[q] - qr[q]) + (ll[q] - lr[q])) + ddiff[q]);
    }
    float tm[5] = {Wm[0], 0, 0, 0, Wm[4]};
    rotate_vec(Rm, Wm + 1, tm + 1);
    if (pair) {
        float ts[5] = {sg[0], 0, 0, 0, sg[4]}, th[5] = {hg[0], 0, 0, 0, hg[4]}, tl[5], tr[5];
        rotate_vec(Rm, sg + 1, ts + 1);
        rotate_vec(Rm, hg + 1, th + 1);
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            tl[q] = tm[q] + (ts[q] + th[q]);
            tr[q] = tm[q] + (ts[q] - th[q]);
        }
        psi_half_difference(tl, tr, th, gm1, hl, hr, dW);
#pragma unroll
        for (int q = 0; q < 5; ++q) dW[q] += ts[q];
        flux1_difference(Wc, tm, dW, gm1, dF);
    } else {
        // both records are the interior cell's: W_m = hi + lo
        float tlo[5], Fc[5], Fm[5];
        tlo[0] = ll[0];
        tlo[4] = ll[4];
        rotate_vec(Rm, ll + 1, tlo + 1);
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            dW[q] = (Wc[q] - tm[q]) - tlo[q];
            tm[q] += tlo[q];
        }
        euler_flux1(Wc, gm1, Fc);
        euler_flux1(tm, gm1, Fm);
#pragma unroll
        for (int q = 0; q < 5; ++q) dF[q] = Fc[q] - Fm[q];
    }
}

// The reference flux (dt / 2) A F_n(W_m) of a face (FP32 stage 1): W_m from
// the hi / lo averages and the face's area vector A n taken exactly (its sum
// over a closed cell vanishes to FP64 rounding, where the FP32 weights and
// normals leave eps A), in FP32 pairs, stored as the record's hi and lo parts; entering
// both cells with opposite signs, it keeps the update exactly conservative.
__device__ __forceinline__ void reference_flux(const float* al, const float* ar, const float* __restrict__ an,
                                               float gm1, float dt, float* __restrict__ out) {
    F2 Wm[5], ref[5];
    float ql[5], ll[5], qr[5], lr[5];
    load_average(al, ql, ll);
    load_average(ar, qr, lr);
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const F2 a = f2_add({ql[q], ll[q]}, {qr[q], lr[q]});
        Wm[q] = {0.5f * a.hi, 0.5f * a.lo};
    }
    const F2 A[3] = {{an[0], an[1]}, {an[2], an[3]}, {an[4], an[5]}};
    const F2 mn = f2_add(f2_add(f2_mul(Wm[1], A[0]), f2_mul(Wm[2], A[1])), f2_mul(Wm[3], A[2]));
    const F2 un = f2_div(mn, Wm[0]);  // A u.n
    const F2 mm = f2_add(f2_add(f2_mul(Wm[1], Wm[1]), f2_mul(Wm[2], Wm[2])), f2_mul(Wm[3], Wm[3]));
    const F2 ke = f2_div(f2_scale(0.5f, mm), Wm[0]);
    const F2 pm = f2_scale(gm1, f2_add(Wm[4], {-ke.hi, -ke.lo}));
    const float hd = 0.5f * dt;
    ref[0] = f2_scale(hd, mn);
#pragma unroll
    for (int j = 0; j < 3; ++j) ref[1 + j] = f2_scale(hd, f2_add(f2_mul(Wm[1 + j], un), f2_mul(pm, A[j])));
    ref[4] = f2_scale(hd, f2_mul(f2_add(Wm[4], pm), un));
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        out[6 * q + 4] = ref[q].hi;
        out[6 * q + 5] = ref[q].lo;
    }
    out[30] = out[31] = 0.0f;
}

// asynchronous copy of 16 bytes to shared memory
__device__ __forceinline__ void copy16(float* to, const float* from) {
    asm volatile("cp.async.ca.shared.global [%0], [%1], 16;" ::"r"((unsigned)__cvta_generic_to_shared(to)), "l"(from)
                 : "memory");
}

// One block of TH / 3 faces (block index fb) by TH threads (tid; one may be
// left over, which computes and stores nothing): sm its shared memory, bar_id the barrier of its threads (0: the
// whole thread block).  VISC: viscous flow (time slopes, Pr fix).  XW: the
// mesh may have isothermal or moving wall faces (their ghosts are compiled
// only into those instances).
template <typename T, int NR, bool VISC, bool XW, int TH = FLUX_THREADS>
__device__ __forceinline__ void flux_faces(const DevMesh<T>& m, const Phys<T>& ph, const T* __restrict__ Wavg,
                                           const T* __restrict__ poly, T* __restrict__ rec,
                                           const double* __restrict__ ctrl, double dt_override, int64_t fb, int tid,
                                           FluxSmem<T, NR, TH>& sm, int bar_id) {
    constexpr bool REL = sizeof(T) == 4 && NR == 40, COPY = flux_copies<T, NR>();
    constexpr int FACES = TH / 3;
    static_assert(REL ? FACES == 32 : 2 * FACES <= TH, "a thread per face and job");
    {
        const int lf = tid / 3, k = tid - 3 * lf;
        const int64_t f0 = fb * FACES + lf;
        const int64_t f = f0 < m.nf ? f0 : m.nf - 1;  // idle points compute a valid face, store nothing
        const int L = m.flr[f], Rc = m.flr[m.nf + f];
        const T* geo = m.fgeo + f * FGEO;
        const T n[3] = {geo[0], geo[1], geo[2]};
        if constexpr (COPY) {
            // both sides' records on their way to shared memory, 16 bytes a
            // copy, a third of each by each of the face's threads
#pragma unroll
            for (int side = 0; side < 2; ++side) {
                const T* p = poly + side_cell(L, Rc, side) * Stride<T>::poly;
#pragma unroll
                for (int j = 4 * k; j < Stride<T>::poly; j += 12) copy16(&sm.poly[lf][side][j], p + j);
            }
#pragma unroll
            for (int j = 4 * k; j < FGEO; j += 12) copy16(&sm.geo[lf][j], geo + j);
        }
        T Rm[3][3];
        face_frame(n, Rm);
        if (k == 0) {
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                sm.frame[lf][i] = Rm[1][i];
                sm.frame[lf][3 + i] = Rm[2][i];
            }
        }
        if constexpr (REL) {
            // the right side's record on its way to L1 while the left side is
            // worked on: the face's three threads take its (at most three)
            // lines.  Stage 1, 3.15 M faces: 1,160 -> 1,108 us.
            const T* rr = poly + side_cell(L, Rc, 1) * Stride<T>::poly;
            asm volatile("prefetch.global.L1 [%0];" ::"l"(rr + (k < 2 ? 32 * k : Stride<T>::poly - 1)));
        }
        if constexpr (COPY) {
            asm volatile("cp.async.wait_all;" ::: "memory");
            group_barrier(bar_id, TH);
        }
        KSums<T> S;
        S.init();
        T pl = T(0), pr = T(0), dsum[5], ddiff[5];
        HalfSpace<T> hl{}, hr{};
#pragma unroll
        for (int q = 0; q < 5; ++q) dsum[q] = ddiff[q] = T(0);
#pragma unroll 1
        for (int side = 0; side < 2; ++side) {
            T tW[5], tg[3][5], dev[5];
            const T* P = COPY ? &sm.poly[lf][side][0] : poly + side_cell(L, Rc, side) * Stride<T>::poly;
            const T* G = COPY ? &sm.geo[lf][0] : geo;
            side_state<T, XW>(m, ph, Wavg, P, G, Rm, L, Rc, side, k, tW, tg, REL ? dev : nullptr);
            pl = pr;
            hl = hr;
            pr = kin_side<VISC>(ph, tW, tg, side == 0 ? +1 : -1, S, &hr);
            if constexpr (REL) {
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    dsum[q] += dev[q];
                    ddiff[q] = dev[q] - ddiff[q];  // right minus left after both sides
                }
            }
        }
        // the face's case step; a finished case (dt = 0) computes with a dummy
        // step and its cells ignore the record
        const double dtc = ctrl ? ctrl[m.cell_case[L >= 0 ? L : Rc]] : dt_override;
        const T dt = dtc > 0.0 ? (T)dtc : T(1);
        T Wc[5], Fh[5], D[5], W0[5], dWt[5];
        finish_point<VISC, REL>(ph, S, pl, pr, dt, Wc, Fh, D, W0, dWt);
        if constexpr (REL) {
#pragma unroll
            for (int q = 0; q < 5; ++q) ddiff[q] = -ddiff[q];
            T dW[5], dF[5];
            interface_deviation(poly + side_cell(L, Rc, 0) * Stride<T>::poly,
                                poly + side_cell(L, Rc, 1) * Stride<T>::poly, L, Rc, Rm, dsum, ddiff, hl, hr, Wc, ph.gm1, dW, dF);
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                Fh[q] += T(0.5) * dt * dF[q];
                W0[q] += dW[q];
            }
        }
        T* o = sm.out[tid];
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            if constexpr (NR == 40) {
                o[q] = Fh[q];
                o[5 + q] = D[q];
                o[10 + q] = W0[q];
                o[15 + q] = dWt[q];
            } else {
                o[q] = D[q];
                o[5 + q] = dWt[q];
            }
        }
    }
    group_barrier(bar_id, TH);
    // per face, a thread each (with 32 faces a warp each): the flux entries,
    // the interface-state entries and (FP32 stage 1) the reference flux
    const int job = tid / FACES, lf = tid - FACES * job;
    const int64_t f = fb * FACES + lf;
    constexpr int VALS = flux_vals<NR>(), RS = rec_stride<T, NR>(), J = rec_entries<T, NR>();
    if (f < m.nf && job < 2) {
        T Rm[3][3], n[4];
        load_vec<4>(COPY ? &sm.geo[lf][0] : m.fgeo + f * FGEO, n);
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            Rm[0][i] = n[i];
            Rm[1][i] = sm.frame[lf][i];
            Rm[2][i] = sm.frame[lf][3 + i];
        }
        const T w = n[3];
        auto sum = [&](int at, T* v) {
#pragma unroll
            for (int q = 0; q < 5; ++q)
                v[q] = w * ((sm.out[3 * lf][at + q] + sm.out[3 * lf + 1][at + q]) + sm.out[3 * lf + 2][at + q]);
            to_global(Rm, v);
        };
        // FP32 stage 1: by way of shared memory
        T* r = REL ? sm.rec[lf] : rec + f * RS;
        T a[5], b[5];
        sum((VALS / 2) * job, a);
        if constexpr (NR == 40) {
            sum(10 * job + 5, b);
#pragma unroll
            for (int q = 0; q < 5; ++q) {
                // dt L + dt^2/6 L_t = 8/3 Fh - 1/3 F = 2 Fh - D / 3 (Eqs. linear-system, s2o4)
                // f* = f^n + dt/2 f_t^n
                r[J * q + 2 * job] = job == 0 ? a[q] : a[q] + T(0.5) * b[q];
                r[J * q + 2 * job + 1] = job == 0 ? T(2) * a[q] - b[q] * T(1.0 / 3.0) : a[q];
            }
        } else {
#pragma unroll
            for (int q = 0; q < 5; ++q)
                // dt^2/3 L_t(W*) = 4/3 (F* - 2 Fh*); f^{n+1} = f^n + dt f_t^*
                r[J * q + job] = job == 0 ? T(4.0 / 3.0) * a[q] : a[q];
        }
    }
    if constexpr (REL) {
        if (f < m.nf && job == 2) {
            const int L = m.flr[f], Rc = m.flr[m.nf + f];
            const double dtc = ctrl ? ctrl[m.cell_case[L >= 0 ? L : Rc]] : dt_override;
            reference_flux(poly + side_cell(L, Rc, 0) * Stride<T>::poly, poly + side_cell(L, Rc, 1) * Stride<T>::poly,
                           m.fan + 6 * f, ph.gm1, dtc > 0.0 ? (T)dtc : T(1), sm.rec[lf]);
        }
        group_barrier(bar_id, TH);
        // the block's records are one stretch of memory: whole vectors by all
        // threads, where a thread per face wrote each of its 10 words to a line
        // of its own (L1's data pipe 67 % busy).  Stage 1, 3.15 M faces: 1,071
        // -> 907 us.  Stage 2's short records lost more by the second barrier
        // (687 -> 733 us) and FP64 has its pipe as bound: these write directly.
        const int64_t left = m.nf - fb * FACES;
        const int words = (int)(left < FACES ? left : FACES) * (RS / 4);
        for (int i = tid; i < words; i += TH) {
            const int face = i / (RS / 4), e = 4 * (i - face * (RS / 4));
            T v[4];
#pragma unroll
            for (int k = 0; k < 4; ++k) v[k] = sm.rec[face][e + k];
            store_vec<4>(rec + fb * FACES * RS + 4 * (int64_t)i, v);
        }
    }
}

template <typename T>
inline Phys<T> make_phys(const HostPhys& p) {
    Phys<T> ph;
    ph.gamma = (T)p.gamma;
    ph.gm1 = (T)(p.gamma - 1.0);
    ph.K = (T)((5.0 - 3.0 * p.gamma) / (p.gamma - 1.0));
    ph.tau_eps = (T)p.tau_eps;
    ph.tau_c = (T)p.tau_c;
    ph.mu = (T)p.mu;
    ph.eps_w = (T)p.eps_weno;
    ph.viscous = p.viscous;
    ph.smooth = p.smooth;
    ph.prf = (T)p.prf;
    ph.twall = (T)p.twall;
    for (int i = 0; i < 3; ++i) ph.uwall[i] = (T)p.uwall[i];
    return ph;
}


// the flux kernel: one block of TH / 3 faces per thread block; MINB resident
// blocks an SM
template <typename T, int NR, int TH, int MINB, bool VISC, bool XW>
__global__ void __launch_bounds__(TH, MINB) k_flux(DevMesh<T> m, Phys<T> ph, const T* __restrict__ Wavg,
                                                   const T* __restrict__ poly, T* __restrict__ rec,
                                                   const double* __restrict__ ctrl, double dt_override) {
    __shared__ FluxSmem<T, NR, TH> sm;
    flux_faces<T, NR, VISC, XW, TH>(m, ph, Wavg, poly, rec, ctrl, dt_override, blockIdx.x, threadIdx.x, sm, 0);
}

// Threads a block and resident blocks an SM, hence registers.  FP32 variant
// 1: the most blocks that spill nothing, 5 (15 warps, 128 registers), in
// inviscid stage 2 6 (96 registers).  Variant 0: 4 blocks; the faster one where
// a launch has too few blocks to use the warps (a step of 1,536 cells 33.0 us
// with variant 1, 31.0-32.2 with 0; 2,592 viscous cells 35.1 and 33.0; from 3,330
// cells on the same or slower).  Measured, with 4 / 5 / 6 / 8 blocks an SM:
//   3.15 M faces, inviscid, stage 1   1,069 / 905 / 948 / 1,020 us
//                           stage 2     612 / 629 / 594 / 634
//   1.16 M faces, viscous,  stage 1     436 / 381 / 451 / 486
//                           stage 2     300 / 252 / 260 / 322
constexpr int FLUX_BLOCKS_V1 = 5, FLUX_BLOCKS_V1_STAGE2 = 6, FLUX_BLOCKS_V0 = 4;
template <typename T, bool XW>
static cudaError_t launch_flux(const DevMesh<T>& m, const HostPhys& p, const T* W, const T* poly, T* rec,
                               const double* ctrl, double dt_override, int stage, cudaStream_t s, int variant) {
    const Phys<T> ph = make_phys<T>(p);
    auto blocks = [&](auto threads, auto minb) {
        constexpr int TH = decltype(threads)::value, B = decltype(minb)::value;
        const unsigned grid = (unsigned)((m.nf + TH / 3 - 1) / (TH / 3));
        auto go = [&](auto kernel) { kernel<<<grid, TH, 0, s>>>(m, ph, W, poly, rec, ctrl, dt_override); };
        if (stage == 1)
            p.viscous ? go(k_flux<T, 40, TH, B, true, XW>) : go(k_flux<T, 40, TH, B, false, XW>);
        else
            p.viscous ? go(k_flux<T, 20, TH, B, true, XW>)
                      : go(k_flux<T, 20, TH, B == FLUX_BLOCKS_V1 ? FLUX_BLOCKS_V1_STAGE2 : B, false, XW>);
    };
    using std::integral_constant;
    if constexpr (sizeof(T) == 8) {
        if (flux_small_blocks(m.nf, m.sms))
            blocks(integral_constant<int, FLUX_THREADS_FP64>{}, integral_constant<int, 4>{});
        else
            blocks(integral_constant<int, FLUX_THREADS>{}, integral_constant<int, 2>{});
    } else if (variant == 1)
        blocks(integral_constant<int, FLUX_THREADS>{}, integral_constant<int, FLUX_BLOCKS_V1>{});
    else
        blocks(integral_constant<int, FLUX_THREADS>{}, integral_constant<int, FLUX_BLOCKS_V0>{});
    return cudaGetLastError();
}

// the launch on a mesh with isothermal or moving wall faces (the instances
// with their ghosts, in a translation unit of their own)
template <typename T>
cudaError_t launch_flux_xw(const DevMesh<T>& m, const HostPhys& p, const T* W, const T* poly, T* rec,
                           const double* ctrl, double dt_override, int stage, cudaStream_t s, int variant);

}  // namespace gks
