// gks_kinetic.cuh -- the time-dependent kinetic solution at one Gauss point
// (Eq. 2nd-flux / Eq. 2nd-smooth-flux with the equilibrium state of Eq.
// new-equ-part) from closed forms of the velocity moments and of their
// derivatives.
//
// The micro-slope product g (a_i . psi) is the derivative of the Maxwellian
// g along x_i (Eq. co), so every moment of it is the derivative of a moment
// of g, rho <(a_i . psi) phi> = d_i (rho <phi>), over the whole space and
// over a half space alike (the half space is fixed).  With h = p / rho =
// 1 / (2 lambda), R_k = rho <u^k> (half or whole space) and
// q = V^2 + W^2 + (K + 2) h, the moments used are
//   A_a = rho <u^a psi>   = (R_a, R_a+1, V R_a, W R_a, (R_a+2 + q R_a) / 2)
//   B_a = rho <u^a v psi> = (V R_a, V R_a+1, (V^2 + h) R_a, V W R_a,
//                            V (R_a+2 + (q + 2 h) R_a) / 2)
// and B_a's counterpart in w; their derivatives follow from
//   d <u^k> = k <u^(k-1)> dU + k (k - 1) / 2 <u^(k-2)> dh     (k >= 2),
//   d <u>   = <u^0> dU + f dh / 2,   d <u^0> = f (dU - U dh / (2 h)),
// f the signed density of u at the half space's edge u = 0 (0 for the whole
// space).  Against summing a_m <psi_m psi_k phi> over the 5 x 5 moment
// matrix this needs no micro-slopes, no moment beyond u^4 and about a third
// of the operations, and it has no cancellation between the terms of a.psi.
//
// Energies (last entries) are carried doubled until finish_point.
#pragma once

#include "gks_device.cuh"

namespace gks {

// primitive state: h = p / rho, ge = (gamma - 1) E / rho
template <typename T>
struct KState {
    T rho, ir, U, V, W, h, p, ge;
};

// derivative of a primitive state: r = d rho / rho
template <typename T>
struct KGrad {
    T r, U, V, W, h;
};

template <typename T>
__device__ __forceinline__ KState<T> kin_state(const T* W, T gm1) {
    KState<T> s;
    s.rho = W[0];
    s.ir = T(1) / W[0];
    s.U = W[1] * s.ir;
    s.V = W[2] * s.ir;
    s.W = W[3] * s.ir;
    s.p = gm1 * (W[4] - T(0.5) * (W[1] * s.U + W[2] * s.V + W[3] * s.W));
    s.h = s.p * s.ir;
    s.ge = gm1 * W[4] * s.ir;
    return s;
}

// the primitive derivative of a conservative one, g[5]
template <typename T>
__device__ __forceinline__ KGrad<T> kin_grad(const KState<T>& s, const T* g, T gm1) {
    KGrad<T> d;
    d.r = g[0] * s.ir;
    d.U = g[1] * s.ir - s.U * d.r;
    d.V = g[2] * s.ir - s.V * d.r;
    d.W = g[3] * s.ir - s.W * d.r;
    d.h = gm1 * (g[4] * s.ir - (s.U * d.U + s.V * d.V + s.W * d.W)) - s.ge * d.r;
    return d;
}

// time derivative from the space derivatives by the Euler equations (the
// compatibility condition of A, Eq. co)
template <typename T>
__device__ __forceinline__ KGrad<T> kin_time(const KState<T>& s, const KGrad<T>* d, T gm1) {
    const T div = d[0].U + d[1].V + d[2].W;
    KGrad<T> t;
    t.r = -(s.U * d[0].r + s.V * d[1].r + s.W * d[2].r + div);
    t.U = -(s.U * d[0].U + s.V * d[1].U + s.W * d[2].U + s.h * d[0].r + d[0].h);
    t.V = -(s.U * d[0].V + s.V * d[1].V + s.W * d[2].V + s.h * d[1].r + d[1].h);
    t.W = -(s.U * d[0].W + s.V * d[1].W + s.W * d[2].W + s.h * d[2].r + d[2].h);
    t.h = -(s.U * d[0].h + s.V * d[1].h + s.W * d[2].h + gm1 * s.h * div);
    return t;
}

// R_k, k < 5, the multiples of them that the derivatives take (one set for
// the three directions), and (half space) F = rho f, F / 2, Uh = U / (2 h)
template <bool HALF, typename T>
struct KMom {
    T R[5], R1x2, R1x3, R2x3, R2x6, R3x4, F, Fh, Uh, q;
};

// half: +1 restricts u > 0, -1 u < 0 (HALF only).  hs (may be NULL): what the
// FP32 interface deviation takes of the half space.
template <bool HALF, typename T>
__device__ __forceinline__ KMom<HALF, T> kin_moments(const KState<T>& s, T K, int half,
                                                            HalfSpace<T>* hs = nullptr) {
    KMom<HALF, T> k;
    k.q = s.V * s.V + s.W * s.W + (K + T(2)) * s.h;
    if constexpr (HALF) {
        const T sg = half > 0 ? T(1) : T(-1);
        const T rs = d_rsqrt(T(2) * s.h);  // sqrt(lambda)
        const T x = s.U * rs;
        const T ex = d_exp(-x * x);
        const T u0 = half_erfc(-sg * x, ex);
        if (hs) *hs = {u0, rs, ex};
        k.F = sg * s.rho * T(0.56418958354775628695) * rs * ex;  // 1 / sqrt(pi)
        k.Uh = x * rs;
        k.R[0] = s.rho * u0;
        k.R[1] = s.U * k.R[0] + s.h * k.F;
        k.Fh = T(0.5) * k.F;
    } else {
        k.F = k.Fh = k.Uh = T(0);
        k.R[0] = s.rho;
        k.R[1] = s.U * s.rho;
    }
    k.R[2] = s.U * k.R[1] + s.h * k.R[0];
    k.R1x2 = T(2) * k.R[1];
    k.R1x3 = T(3) * k.R[1];
    k.R2x3 = T(3) * k.R[2];
    k.R2x6 = T(6) * k.R[2];
    k.R[3] = s.U * k.R[2] + s.h * k.R1x2;
    k.R3x4 = T(4) * k.R[3];
    k.R[4] = s.U * k.R[3] + s.h * k.R2x3;
    return k;
}

// d R_k along d
template <int N, bool HALF, typename T>
__device__ __forceinline__ T kin_dR(const KMom<HALF, T>& k, const KGrad<T>& d) {
    T v = d.r * k.R[N];
    if constexpr (N == 0) {
        if constexpr (HALF) v += k.F * (d.U - k.Uh * d.h);
    } else if constexpr (N == 1) {
        v += k.R[0] * d.U;
        if constexpr (HALF) v += k.Fh * d.h;
    } else if constexpr (N == 2) {
        v += k.R1x2 * d.U + k.R[0] * d.h;
    } else if constexpr (N == 3) {
        v += k.R2x3 * d.U + k.R1x3 * d.h;
    } else {
        v += k.R3x4 * d.U + k.R2x6 * d.h;
    }
    return v;
}

// out += A_a
template <int a, bool HALF, typename T>
__device__ __forceinline__ void kin_A(const KState<T>& s, const KMom<HALF, T>& k, T* out) {
    out[0] += k.R[a];
    out[1] += k.R[a + 1];
    out[2] += s.V * k.R[a];
    out[3] += s.W * k.R[a];
    out[4] += k.R[a + 2] + k.q * k.R[a];
}

// out += d A_a, given dR[a .. a + 2] (dR indexed by power) and dq
template <int a, bool HALF, typename T>
__device__ __forceinline__ void kin_dA(const KState<T>& s, const KMom<HALF, T>& k, const KGrad<T>& d, const T* dR,
                                       T dq, T* out) {
    out[0] += dR[a];
    out[1] += dR[a + 1];
    out[2] += s.V * dR[a] + d.V * k.R[a];
    out[3] += s.W * dR[a] + d.W * k.R[a];
    out[4] += dR[a + 2] + k.q * dR[a] + dq * k.R[a];
}

// out += d B_a; Y the transverse velocity of B (v: component 2 of out, w: 3),
// Z the other one
template <int a, int YC, bool HALF, typename T>
__device__ __forceinline__ void kin_dB(const KState<T>& s, const KMom<HALF, T>& k, const KGrad<T>& d, const T* dR,
                                       T dq, T* out) {
    constexpr int ZC = 5 - YC;
    const T Y = YC == 2 ? s.V : s.W, dY = YC == 2 ? d.V : d.W;
    const T Z = YC == 2 ? s.W : s.V, dZ = YC == 2 ? d.W : d.V;
    const T Ra = k.R[a], YR = Y * Ra;
    const T X = Y * dR[a] + dY * Ra;
    const T q2 = k.q + T(2) * s.h, dq2 = dq + T(2) * d.h;
    out[0] += X;
    out[1] += Y * dR[a + 1] + dY * k.R[a + 1];
    out[YC] += Y * X + dY * YR + (s.h * dR[a] + d.h * Ra);
    out[ZC] += Z * X + dZ * YR;
    out[4] += dY * (k.R[a + 2] + q2 * Ra) + Y * (dR[a + 2] + q2 * dR[a] + dq2 * Ra);
}

// sums over the two sides of a point (half spaces):
//   w = rho <psi> (W^c, Eq. new-equ-part), f0 = rho <u psi>, d[i] = rho <(a_i.psi) psi>,
//   r1 = rho sum_i <u_i (a_i.psi) psi>, f1 = rho sum_i <u u_i (a_i.psi) psi>,
//   r2 = rho <(A.psi) psi>, f2 = rho <u (A.psi) psi> (viscous only)
template <typename T>
struct KSums {
    T w[5], d[3][5], f0[5], f1[5], r1[5], f2[5], r2[5];
    __device__ __forceinline__ void init() {
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            w[q] = f0[q] = f1[q] = r1[q] = f2[q] = r2[q] = T(0);
            d[0][q] = d[1][q] = d[2][q] = T(0);
        }
    }
};

// the space-derivative sums of one state: d (half space only), r1, f1
template <bool HALF, typename T>
__device__ __forceinline__ void kin_conv(const KState<T>& s, const KMom<HALF, T>& k, const KGrad<T>* g, T K,
                                         T (*d)[5], T* r1, T* f1) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const KGrad<T>& e = g[i];
        T dR[5];
        dR[0] = kin_dR<0>(k, e);
        dR[1] = kin_dR<1>(k, e);
        dR[2] = kin_dR<2>(k, e);
        dR[3] = kin_dR<3>(k, e);
        const T dq = T(2) * (s.V * e.V + s.W * e.W) + (K + T(2)) * e.h;
        if constexpr (HALF) kin_dA<0>(s, k, e, dR, dq, d[i]);
        if (i == 0) {
            dR[4] = kin_dR<4>(k, e);
            kin_dA<1>(s, k, e, dR, dq, r1);
            kin_dA<2>(s, k, e, dR, dq, f1);
        } else if (i == 1) {
            kin_dB<0, 2>(s, k, e, dR, dq, r1);
            kin_dB<1, 2>(s, k, e, dR, dq, f1);
        } else {
            kin_dB<0, 3>(s, k, e, dR, dq, r1);
            kin_dB<1, 3>(s, k, e, dR, dq, f1);
        }
    }
}

// adds one side (face-frame state W, gradients g[i]; half +1 left, -1 right)
// to the sums; returns its pressure
template <bool VISC, typename T>
__device__ __forceinline__ T kin_side(const Phys<T>& ph, const T* W, const T (*g)[5], int half, KSums<T>& S,
                                      HalfSpace<T>* hs = nullptr) {
    const KState<T> s = kin_state(W, ph.gm1);
    KGrad<T> d[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) d[i] = kin_grad(s, g[i], ph.gm1);
    const KMom<true, T> k = kin_moments<true>(s, ph.K, half, hs);
    kin_A<0>(s, k, S.w);
    kin_A<1>(s, k, S.f0);
    kin_conv<true>(s, k, d, ph.K, S.d, S.r1, S.f1);
    if constexpr (VISC) {
        const KGrad<T> e = kin_time(s, d, ph.gm1);
        T dR[4];
        dR[0] = kin_dR<0>(k, e);
        dR[1] = kin_dR<1>(k, e);
        dR[2] = kin_dR<2>(k, e);
        dR[3] = kin_dR<3>(k, e);
        const T dq = T(2) * (s.V * e.V + s.W * e.W) + (ph.K + T(2)) * e.h;
        kin_dA<0>(s, k, e, dR, dq, S.r2);
        kin_dA<1>(s, k, e, dR, dq, S.f2);
    }
    return s.p;
}

// The point's outputs from the sums over its sides:
//   Fh = int_0^{dt/2} F dt,  D = int_0^dt F dt - 2 Fh   (second-order part)
//   W0 = W(0),               dW = W(dt) - W(0)
// D and dW come from differences of the time coefficients, in which the
// leading terms cancel exactly.  REL: Fh without (dt / 2) F(W^c) and W0
// without W^c (FP32 stage-1 records take those relative to the mean of the
// two cell averages).  Wc receives the interface state.
template <bool VISC, bool REL, typename T>
__device__ __forceinline__ void finish_point(const Phys<T>& ph, const KSums<T>& S, T pl, T pr, T dt, T* Wc, T* Fh,
                                             T* D, T* W0, T* dW) {
#pragma unroll
    for (int q = 0; q < 4; ++q) Wc[q] = S.w[q];
    Wc[4] = T(0.5) * S.w[4];
    const KState<T> s = kin_state(Wc, ph.gm1);
    KGrad<T> d[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const T g[5] = {S.d[i][0], S.d[i][1], S.d[i][2], S.d[i][3], T(0.5) * S.d[i][4]};
        d[i] = kin_grad(s, g, ph.gm1);
    }
    const KMom<false, T> k = kin_moments<false>(s, ph.K, 0);
    T f0[5] = {0, 0, 0, 0, 0}, f1[5] = {0, 0, 0, 0, 0}, f2[5] = {0, 0, 0, 0, 0}, r1[5] = {0, 0, 0, 0, 0};
    kin_A<1>(s, k, f0);
    kin_conv<false, T>(s, k, d, ph.K, nullptr, r1, f1);
    {
        const KGrad<T> e = kin_time(s, d, ph.gm1);
        T dR[4];
        dR[1] = kin_dR<1>(k, e);
        dR[2] = kin_dR<2>(k, e);
        dR[3] = kin_dR<3>(k, e);
        const T dq = T(2) * (s.V * e.V + s.W * e.W) + (ph.K + T(2)) * e.h;
        kin_dA<1>(s, k, e, dR, dq, f2);
    }
    const TimeCoef<T> tc = time_coefs(ph, pl, pr, s.p, dt);
    const T tau = tc.tau, hd = T(0.5) * dt;
    T IWh[5], IWd[5];  // state integrals over [0, dt/2] and their differences (Pr fix only)
    if (ph.smooth) {
        // f = g^c - tau (a^c.u + A^c) g^c + A^c g^c t, Eq. 2nd-smooth-flux
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            Fh[q] = (REL ? T(0) : hd * f0[q]) - tau * hd * f1[q] + (T(0.5) * hd * hd - tau * hd) * f2[q];
            D[q] = T(0.25) * dt * dt * f2[q];
            W0[q] = REL ? T(0) : S.w[q];  // the tau terms cancel: <(a.u + A) psi> = 0
            dW[q] = -dt * r1[q];
            if constexpr (VISC) {
                IWh[q] = hd * S.w[q] - T(0.5) * hd * hd * r1[q];
                IWd[q] = -T(0.25) * dt * dt * r1[q];
            }
        }
    } else {
        const T c1 = tau * tc.k0 + tc.k1, dc1 = tau * tc.dk0 + tc.dk1;
        const T omE = T(1) - tc.E;
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            // kinetic minus equilibrium moments under the kinetic factors
            // (C1's is dt/2 - k0, C2's k1 + tau k0 - tau dt/2)
            const T e0 = S.f0[q] - f0[q], e1 = S.f1[q] - f1[q];
            Fh[q] = tc.k0 * e0 - c1 * e1 + tc.q3 * f2[q];
            if (!REL) Fh[q] += hd * f0[q];
            D[q] = tc.dk0 * e0 - dc1 * e1 + tc.dq3 * f2[q];
            W0[q] = REL ? T(0) : S.w[q];
            if constexpr (VISC) {
                Fh[q] -= tau * (hd * f1[q] + tc.k0 * S.f2[q]);
                D[q] -= tau * tc.dk0 * S.f2[q];
                W0[q] -= tau * (S.r1[q] + S.r2[q]);
                dW[q] = (tau - (tau + dt) * tc.E) * S.r1[q] + tau * omE * S.r2[q] - dt * omE * r1[q];
                IWh[q] = hd * S.w[q] - c1 * S.r1[q] - tau * tc.k0 * S.r2[q] + (tc.q2 - tc.q3) * r1[q];
                IWd[q] = -dc1 * S.r1[q] - tau * tc.dk0 * S.r2[q] + (tc.dq2 - tc.dq3) * r1[q];
            } else {
                dW[q] = -dt * (tc.E * S.r1[q] + omE * r1[q]);
            }
        }
    }
    Fh[4] *= T(0.5);
    D[4] *= T(0.5);
    W0[4] *= T(0.5);
    dW[4] *= T(0.5);
    if constexpr (VISC) {
        if (ph.prf != T(0)) {
            IWh[4] *= T(0.5);
            IWd[4] *= T(0.5);
            const T U[3] = {s.U, s.V, s.W};
            if constexpr (REL) {
                // the fix acts on the whole flux: only its change is kept
                T F[5];
#pragma unroll
                for (int q = 0; q < 5; ++q) F[q] = Fh[q] + hd * (q == 4 ? T(0.5) : T(1)) * f0[q];
                const T before = F[4];
                prandtl_fix(ph.prf, U, IWh, F);
                Fh[4] += F[4] - before;
            } else {
                prandtl_fix(ph.prf, U, IWh, Fh);
            }
            prandtl_fix(ph.prf, U, IWd, D);
        }
    }
}

}  // namespace gks
