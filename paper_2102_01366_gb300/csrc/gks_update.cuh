// gks_update.cuh -- the cell updates of one block of cells (Sec. 3) and the
// block reductions of the time-step rule (Sec. 5), shared by the
// standalone kernels and the persistent stage kernel.
#pragma once

#include <cuda_runtime.h>

#include <type_traits>

#include "gks_cells.cuh"
#include "gks_device.cuh"
#include "gks_kernels.h"

namespace gks {

__device__ __forceinline__ float warp_min(float v) {
    // non-negative floats order like their bit patterns
    return __uint_as_float(__reduce_min_sync(0xffffffffu, __float_as_uint(v)));
}

__device__ __forceinline__ double warp_min(double v) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmin(v, __shfl_xor_sync(0xffffffffu, v, o));
    return v;
}

// Per-case minimum of the local limits of a warp's cells into dtmin (bits of
// non-negative doubles, which order like the doubles); v counts where it is
// finite.  A warp's cells are mostly of one case: then one lane brings the
// warp's minimum, and only if it is below the current one, so that the
// atomics on a case's word die out after its first few blocks (the minimum is
// exact, so neither order nor a stale reading changes it).  All 32 lanes call.
//
// A thread scanning the block's 24 limits in shared memory and one
// unconditional atomicMin a block made this most of the stage-2 update: on
// 1.57 M cells (FP32) 707 us, 303 us with the warp's minimum.
template <typename T>
__device__ __forceinline__ void warp_case_min(T v, int32_t cas, unsigned long long* dtmin) {
    if (!(v < T(INFINITY))) v = T(INFINITY);
    const bool valid = v < T(INFINITY);
    auto commit = [&](T x) {
        const unsigned long long bits = (unsigned long long)__double_as_longlong(widen(x));
        if (bits < __ldcg(dtmin + cas)) atomicMin(dtmin + cas, bits);
    };
    const int32_t c0 = __shfl_sync(0xffffffffu, cas, 0);
    if (__all_sync(0xffffffffu, cas == c0 || !valid)) {
        const T mn = warp_min(v);
        if ((threadIdx.x & 31) == 0 && mn < T(INFINITY)) commit(mn);
    } else if (valid) {
        commit(v);
    }
}

// x > 0 of a finite double, on the integer pipe
__device__ __forceinline__ bool positive(double x) { return __double_as_longlong(x) > 0; }

// --------------------------------------------------------------------------
// cell updates, five lanes per cell (one per component).  Bound by the
// latency of two dependent gathers (face list, then face records), so all of
// a cell's gathers are issued before the first is used, the normals lie apart
// from the Gauss points and a component's record entries together; in FP32
// bulk next by the FP64 pipe, so FP32 <-> FP64 conversions go through the
// integer pipe (widen, split_pair).  1.57 M cells, FP32, stage 1 / stage 2: 254 /
// 171 us; 393 / 707 with dependent loads, a block's serial time-step minimum and
// component-major S and G; 306 / 303 without the integer conversions and the
// normals apart.  One thread per cell with 16-byte gathers, when five lanes took
// 281 / 171, took 349 / 236 (too few warps in flight) and twice the time on 1,536
// to 3,072 cells.
// --------------------------------------------------------------------------

// N values of a record (8- or 16-byte aligned) as vectors of two
template <int N, typename T>
__device__ __forceinline__ void load_pairs(const T* __restrict__ p, T* v) {
    using T2 = std::conditional_t<sizeof(T) == 4, float2, double2>;
#pragma unroll
    for (int i = 0; i < N / 2; ++i) {
        const T2 x = reinterpret_cast<const T2*>(p)[i];
        v[2 * i] = x.x;
        v[2 * i + 1] = x.y;
    }
}

// the face's unit normal and w = area / 3, one 16-byte (FP64: two) load
template <typename T>
__device__ __forceinline__ void load_normal(const DevMesh<T>& m, int64_t face, T* n) {
    load_vec<4>(m.fnw + face * 4, n);
}

template <typename T>
__device__ __forceinline__ void update1_cells(const DevMesh<T>& m, const DevState<T>& st, int64_t vb, int tid) {
    const CellLane cl = cell_lane(m.nc, vb, tid);
    if (!cl.active) return;
    const int64_t nc = m.nc, c = cl.c;
    const int q = cl.q;
    constexpr int RS = rec_stride<T, 40>(), J = rec_entries<T, 40>(), XSR = Stride<T>::xs;
    constexpr bool F32 = sizeof(T) == 4;
    int e[4], nb[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        e[f] = m.cface[f * nc + c];
        nb[f] = F32 ? m.nbr[f * nc + c] : 0;
    }
    const double dtd = st.case_dt[m.cell_case[c]];
    const double iv = m.inv_vol[c], w0d = st.Wd[q * nc + c];
    T r[4][J], n[4][4], nx[4][2], own[2] = {T(0), T(0)};
    if constexpr (F32) {
        own[0] = st.X[c * XSR + q];
        own[1] = st.X[c * XSR + XLO + q];
    }
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        load_pairs<J>(st.rec + (int64_t)(e[f] >> 1) * RS + q * J, r[f]);
        load_normal(m, e[f] >> 1, n[f]);
        if constexpr (F32) {
            // a missing neighbour reads the cell itself
            const T* x = st.X + (nb[f] >= 0 ? (int64_t)nb[f] : c) * XSR + q;
            nx[f][0] = x[0];
            nx[f][1] = x[XLO];
        }
    }
    if (!positive(dtd)) return;  // finished case
    CSum<T> fh, s1;
    fh.init();
    s1.init();
    T gs[3] = {T(0), T(0), T(0)}, g0[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        const T s = (e[f] & 1) ? T(-1) : T(1);
        fh.add(s * r[f][0]);
        s1.add(s * r[f][1]);
        T ws = s * r[f][2], w0 = s * r[f][3];
        if constexpr (F32) {
            // the reference flux (dt / 2) A F_n(W_m) of the face, hi + lo; the
            // S entry takes it twice (2 Fh - D / 3)
            fh.add(s * r[f][4]);
            fh.add(s * r[f][5]);
            s1.add(T(2) * s * r[f][4]);
            s1.add(T(2) * s * r[f][5]);
            // FP32 records hold the interface states relative to the mean of
            // the face's two cell averages W_m (the interior cell's average on
            // a boundary face).  The cell needs sum_f s_f W_m A_f n_f back; as
            // sum_f s_f A_f n_f = 0 over a closed cell, that is
            // 1/2 sum_f s_f (W_nb - W_c) A_f n_f over its interior faces,
            // formed from the exact differences of the hi / lo pairs (A = 3 w).
            const T a = s * T(1.5) * n[f][3] * ((nx[f][0] - own[0]) + (nx[f][1] - own[1]));
            ws += a;
            w0 += a;
        }
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            gs[i] += ws * n[f][i];
            g0[i] += w0 * n[f][i];
        }
    }
    T* xs = st.Xs + c * XSR;
    // W* = W^n - (1/|Omega|) sum s sum_k w Fh  (Eq. s2o4, first stage)
    const double wstar = w0d - fh.value() * iv;
    T ivr;
    if constexpr (F32) {
        split_pair(wstar, xs[q], xs[XLO + q]);
        ivr = narrow(iv);
    } else {
        xs[q] = wstar;
        ivr = iv;
    }
    st.S[c * 5 + q] = s1.value();
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        xs[Stride<T>::xg + 3 * q + i] = gs[i] * ivr;  // Eq. gauss-formula at t* (Eq. step-du)
        st.G[c * 15 + 3 * q + i] = g0[i];
    }
}

// vb: the block of CELLS_PER_BLOCK cells (its residual sums go to part[vb]),
// tid the thread in its CELL_THREADS, bar_id their barrier (0: the whole
// thread block), red their [CELL_THREADS / 32][5] of shared memory
template <typename T>
__device__ __forceinline__ void update2_cells(const DevMesh<T>& m, const DtPhys<T>& p, const DevState<T>& st,
                                              int64_t vb, int tid, int bar_id, T (*red)[5]) {
    const CellLane cl = cell_lane(m.nc, vb, tid);
    const int64_t nc = m.nc, c = cl.c;
    const int q = cl.q;
    constexpr int RS = rec_stride<T, 20>(), XSR = Stride<T>::xs;
    int e[4];
#pragma unroll
    for (int f = 0; f < 4; ++f) e[f] = m.cface[f * nc + c];
    const int32_t cas = m.cell_case[c];
    const double dtd = st.case_dt[cas];
    const double iv = m.inv_vol[c], w0d = st.Wd[q * nc + c], s0d = st.S[c * 5 + q];
    T g0[3], r[4][2], n[4][4];
#pragma unroll
    for (int i = 0; i < 3; ++i) g0[i] = st.G[c * 15 + 3 * q + i];
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        load_pairs<2>(st.rec + (int64_t)(e[f] >> 1) * RS + q * 2, r[f]);
        load_normal(m, e[f] >> 1, n[f]);
    }
    const bool live = cl.active && positive(dtd);  // finished cases keep their state
    CSum<T> f2;
    f2.init();
    T dg[3] = {T(0), T(0), T(0)};
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        const T s = (e[f] & 1) ? T(-1) : T(1);
        f2.add(s * r[f][0]);
        const T dw = s * r[f][1];
#pragma unroll
        for (int i = 0; i < 3; ++i) dg[i] += dw * n[f][i];
    }
    // W^{n+1} |Omega| = W^n |Omega| - [dt F + dt^2/6 F_t](W^n) - [dt^2/3 F_t](W*)
    // (Eq. s2o4, second stage)
    const double inc = live ? (s0d + widen(f2.hi) + widen(f2.lo)) * iv : 0.0;
    const double wn = w0d - inc;
    T Wq, Wlo = T(0), ivr, incr, dtr, mn = T(INFINITY), res = T(0);
    if constexpr (sizeof(T) == 4) {
        split_pair(wn, Wq, Wlo);
        ivr = narrow(iv);
        incr = narrow(inc);
        dtr = narrow(dtd);
    } else {
        Wq = wn;
        ivr = iv;
        incr = inc;
        dtr = dtd;
    }
    if (live) {
        st.Wd[q * nc + c] = wn;
        T* x = st.X + c * XSR;
        x[q] = Wq;
        if constexpr (sizeof(T) == 4) x[XLO + q] = Wlo;
#pragma unroll
        for (int i = 0; i < 3; ++i) x[Stride<T>::xg + 3 * q + i] = (g0[i] + dg[i]) * ivr;
        // squared rates of change (W^{n+1} - W^n) / dt for the residual
        const T ti = incr / dtr;
        res = ti * ti;
    }
    // the cell's new state, gathered from its 5 lanes, for the positivity flag
    // and the next step's local time-step limit
    T Wn[5];
#pragma unroll
    for (int k = 0; k < 5; ++k) Wn[k] = __shfl_sync(0xffffffffu, Wq, cl.base + k);
    if (cl.active && q == 0) {
        const T pr = p.gm1 * (Wn[4] - T(0.5) * (Wn[1] * Wn[1] + Wn[2] * Wn[2] + Wn[3] * Wn[3]) / Wn[0]);
        if (!(Wn[0] > T(0)) || !(pr > T(0))) atomicOr(st.err, ERR_STATE);
        else mn = local_dt(Wn, m.dr[c], p);
    }
    warp_case_min(mn, cas, st.case_dtmin);
    // residual sums per component over the block's cells in a fixed order:
    // the warp's six cells (lanes q, q + 5, ..., q + 25), then the warps
    res += __shfl_down_sync(0xffffffffu, res, 15);
    res += __shfl_down_sync(0xffffffffu, res, 5) + __shfl_down_sync(0xffffffffu, res, 10);
    if ((tid & 31) < 5) red[tid >> 5][tid & 31] = res;
    group_barrier(bar_id, CELL_THREADS);
    if (tid < 5) {
        T sum = red[0][tid];
        for (int w = 1; w < CELL_THREADS / 32; ++w) sum += red[w][tid];
        st.part[vb * PART_N + PART_RES + tid] = widen(sum);
    }
}

}  // namespace gks
