// gks_point_adj.cuh -- reverse-mode (adjoint) derivative of the kinetic
// solution at one Gauss point, FP64, inviscid or viscous.
//
// gks_point_adj recomputes the closed forms of gks_kinetic.cuh (both sides'
// sums, the interface equilibrium and its sums) and carries the output
// adjoints (of Fh, D, W0, dW) back through each of them in reverse order;
// every building block there has its transpose here (adj_*).  A point's
// outputs depend on the two sides only through the sums over both (KSums) and
// the pressures, so each side's reverse pass is on its own: its moments are
// formed once more (with the two transcendental ones kept), and no more than
// one side is live at a time.
//
// Bound by the FP64 pipe (16 cycles a warp instruction).  Against reversing
// sums over 5 x 5 moment matrices and their seven-entry tables (3.5 to 4.5 KB
// of local memory a thread, now 0.7 to 1.0 KB): 96,000 faces, inviscid, stage
// 1 / stage 2 5,699 / 5,659 us before, 1,918 / 1,868 now; 22,000 faces,
// viscous, 2,039 / 2,028 us before, 614 / 591 now.
//
// Energies (last entries) of sums and their adjoints are those of the doubled
// energies, as in gks_kinetic.cuh.
#pragma once

#include "gks_kinetic.cuh"

namespace gks {

// adjoints of a primitive state and what hangs on it
struct KStateAdj {
    double rho = 0.0, ir = 0.0, U = 0.0, V = 0.0, W = 0.0, h = 0.0, p = 0.0, ge = 0.0;
};

// adjoints of the moments (those of the stored multiples folded in)
template <bool HALF>
struct KMomAdj {
    double R[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, F = 0.0, Uh = 0.0, q = 0.0;
};

using KGradD = KGrad<double>;

// adjoint of kin_A<a>
template <int a, bool HALF>
__device__ __forceinline__ void adj_A(const KState<double>& s, const KMom<HALF, double>& k, const double* lo,
                                      KStateAdj& ls, KMomAdj<HALF>& lk) {
    const double Ra = k.R[a];
    lk.R[a] += lo[0] + s.V * lo[2] + s.W * lo[3] + k.q * lo[4];
    lk.R[a + 1] += lo[1];
    lk.R[a + 2] += lo[4];
    ls.V += Ra * lo[2];
    ls.W += Ra * lo[3];
    lk.q += Ra * lo[4];
}

// adjoint of kin_dA<a>: into lR, the adjoint ld of d, ldR of dR and ldq of dq
template <int a, bool HALF>
__device__ __forceinline__ void adj_dA(const KState<double>& s, const KMom<HALF, double>& k, const KGradD& d,
                                       const double* dR, double dq, const double* lo, KStateAdj& ls,
                                       KMomAdj<HALF>& lk, KGradD& ld, double* ldR, double& ldq) {
    const double Ra = k.R[a];
    ldR[a] += lo[0] + s.V * lo[2] + s.W * lo[3] + k.q * lo[4];
    ldR[a + 1] += lo[1];
    ldR[a + 2] += lo[4];
    ls.V += dR[a] * lo[2];
    ls.W += dR[a] * lo[3];
    lk.q += dR[a] * lo[4];
    ld.V += Ra * lo[2];
    ld.W += Ra * lo[3];
    ldq += Ra * lo[4];
    lk.R[a] += d.V * lo[2] + d.W * lo[3] + dq * lo[4];
}

// adjoint of kin_dB<a, YC>
template <int a, int YC, bool HALF>
__device__ __forceinline__ void adj_dB(const KState<double>& s, const KMom<HALF, double>& k, const KGradD& d,
                                       const double* dR, double dq, const double* lo, KStateAdj& ls,
                                       KMomAdj<HALF>& lk, KGradD& ld, double* ldR, double& ldq) {
    constexpr int ZC = 5 - YC;
    const double Y = YC == 2 ? s.V : s.W, dY = YC == 2 ? d.V : d.W;
    const double Z = YC == 2 ? s.W : s.V, dZ = YC == 2 ? d.W : d.V;
    const double Ra = k.R[a], Rb = k.R[a + 1], dRa = dR[a], YR = Y * Ra;
    const double X = Y * dRa + dY * Ra;
    const double q2 = k.q + 2.0 * s.h, dq2 = dq + 2.0 * d.h;
    const double loY = lo[YC], loZ = lo[ZC], l1 = lo[1], l4 = lo[4];
    const double lX = lo[0] + Y * loY + Z * loZ, lYR = dY * loY + dZ * loZ;
    const double l4Y = l4 * Y, l4dY = l4 * dY;
    // Y, dY, Z, dZ
    const double lY = X * loY + dR[a + 1] * l1 + (dR[a + 2] + q2 * dRa + dq2 * Ra) * l4 + dRa * lX + Ra * lYR;
    const double ldY = Rb * l1 + YR * loY + (k.R[a + 2] + q2 * Ra) * l4 + Ra * lX;
    (YC == 2 ? ls.V : ls.W) += lY;
    (YC == 2 ? ld.V : ld.W) += ldY;
    (YC == 2 ? ls.W : ls.V) += X * loZ;
    (YC == 2 ? ld.W : ld.V) += YR * loZ;
    // R, dR
    lk.R[a] += d.h * loY + l4dY * q2 + l4Y * dq2 + dY * lX + Y * lYR;
    lk.R[a + 1] += dY * l1;
    lk.R[a + 2] += l4dY;
    ldR[a] += s.h * loY + l4Y * q2 + Y * lX;
    ldR[a + 1] += Y * l1;
    ldR[a + 2] += l4Y;
    // q, dq, h, dh
    const double lq2 = l4dY * Ra + l4Y * dRa, ldq2 = l4Y * Ra;
    lk.q += lq2;
    ls.h += dRa * loY + 2.0 * lq2;
    ldq += ldq2;
    ld.h += Ra * loY + 2.0 * ldq2;
}

// adjoint of kin_dR<0 .. N - 1> and of dq for one direction: the adjoints ldR,
// ldq into those of the moments, the state and d
template <int N, bool HALF>
__device__ __forceinline__ void adj_dR(const KState<double>& s, const KMom<HALF, double>& k, double K2,
                                       const KGradD& d, const double* ldR, double ldq, KStateAdj& ls,
                                       KMomAdj<HALF>& lk, KGradD& ld) {
    ld.r += k.R[0] * ldR[0] + k.R[1] * ldR[1] + k.R[2] * ldR[2] + k.R[3] * ldR[3];
    ld.U += k.R[0] * ldR[1] + k.R1x2 * ldR[2] + k.R2x3 * ldR[3];
    ld.h += k.R[0] * ldR[2] + k.R1x3 * ldR[3] + K2 * ldq;
    const double h3 = 3.0 * d.h, U3 = 3.0 * d.U;
    lk.R[0] += d.r * ldR[0] + d.U * ldR[1] + d.h * ldR[2];
    lk.R[1] += d.r * ldR[1] + 2.0 * (d.U * ldR[2]) + h3 * ldR[3];
    lk.R[2] += d.r * ldR[2] + U3 * ldR[3];
    lk.R[3] += d.r * ldR[3];
    if constexpr (N == 5) {
        ld.r += k.R[4] * ldR[4];
        ld.U += k.R3x4 * ldR[4];
        ld.h += k.R2x6 * ldR[4];
        lk.R[2] += 2.0 * (h3 * ldR[4]);
        lk.R[3] += 4.0 * (d.U * ldR[4]);
        lk.R[4] += d.r * ldR[4];
    }
    if constexpr (HALF) {
        const double Fl = k.F * ldR[0];
        ld.U += Fl;
        ld.h += k.Fh * ldR[1] - k.Uh * Fl;
        lk.F += (d.U - k.Uh * d.h) * ldR[0] + 0.5 * (d.h * ldR[1]);
        lk.Uh -= d.h * Fl;
    }
    const double q2 = 2.0 * ldq;
    ld.V += s.V * q2;
    ld.W += s.W * q2;
    ls.V += d.V * q2;
    ls.W += d.W * q2;
}

// adjoint of kin_conv: ldsum (half space: adjoints of d[i]), lr1, lf1 into
// the state, the moments and the primitive gradients lg[i] (added to)
template <bool HALF>
__device__ __forceinline__ void adj_conv(const KState<double>& s, const KMom<HALF, double>& k, const KGradD* g,
                                         double K, const double (*ldsum)[5], const double* lr1, const double* lf1,
                                         KStateAdj& ls, KMomAdj<HALF>& lk, KGradD* lg) {
    const double K2 = K + 2.0;
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const KGradD& e = g[i];
        double dR[5], ldR[5] = {0.0, 0.0, 0.0, 0.0, 0.0}, ldq = 0.0;
        dR[0] = kin_dR<0>(k, e);
        dR[1] = kin_dR<1>(k, e);
        dR[2] = kin_dR<2>(k, e);
        dR[3] = kin_dR<3>(k, e);
        const double dq = 2.0 * (s.V * e.V + s.W * e.W) + K2 * e.h;
        if constexpr (HALF) adj_dA<0>(s, k, e, dR, dq, ldsum[i], ls, lk, lg[i], ldR, ldq);
        if (i == 0) {
            adj_dA<1>(s, k, e, dR, dq, lr1, ls, lk, lg[i], ldR, ldq);
            adj_dA<2>(s, k, e, dR, dq, lf1, ls, lk, lg[i], ldR, ldq);
            adj_dR<5>(s, k, K2, e, ldR, ldq, ls, lk, lg[i]);
        } else if (i == 1) {
            adj_dB<0, 2>(s, k, e, dR, dq, lr1, ls, lk, lg[i], ldR, ldq);
            adj_dB<1, 2>(s, k, e, dR, dq, lf1, ls, lk, lg[i], ldR, ldq);
            adj_dR<4>(s, k, K2, e, ldR, ldq, ls, lk, lg[i]);
        } else {
            adj_dB<0, 3>(s, k, e, dR, dq, lr1, ls, lk, lg[i], ldR, ldq);
            adj_dB<1, 3>(s, k, e, dR, dq, lf1, ls, lk, lg[i], ldR, ldq);
            adj_dR<4>(s, k, K2, e, ldR, ldq, ls, lk, lg[i]);
        }
    }
}

// adjoint of kin_time: lt into the state and the space derivatives
__device__ __forceinline__ void adj_time(const KState<double>& s, const KGradD* d, double gm1, const KGradD& lt,
                                         KStateAdj& ls, KGradD* ld) {
    const double div = d[0].U + d[1].V + d[2].W;
    const double ldiv = -lt.r - gm1 * s.h * lt.h;
    const double vel[3] = {s.U, s.V, s.W};
    double lv[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        ld[i].r -= vel[i] * lt.r;
        ld[i].U -= vel[i] * lt.U;
        ld[i].V -= vel[i] * lt.V;
        ld[i].W -= vel[i] * lt.W;
        ld[i].h -= vel[i] * lt.h;
        lv[i] = d[i].r * lt.r + d[i].U * lt.U + d[i].V * lt.V + d[i].W * lt.W + d[i].h * lt.h;
    }
    ls.U -= lv[0];
    ls.V -= lv[1];
    ls.W -= lv[2];
    ld[0].r -= s.h * lt.U;
    ld[1].r -= s.h * lt.V;
    ld[2].r -= s.h * lt.W;
    ld[0].h -= lt.U;
    ld[1].h -= lt.V;
    ld[2].h -= lt.W;
    ls.h -= d[0].r * lt.U + d[1].r * lt.V + d[2].r * lt.W + gm1 * div * lt.h;
    ld[0].U += ldiv;
    ld[1].V += ldiv;
    ld[2].W += ldiv;
}

// adjoint of the time-slope sums (kin_dA<0>, kin_dA<1> of the time
// derivative e): lr2 (half space), lf2
template <bool HALF>
__device__ __forceinline__ void adj_time_sums(const KState<double>& s, const KMom<HALF, double>& k, const KGradD* d,
                                              double K, double gm1, const double* lr2, const double* lf2,
                                              KStateAdj& ls, KMomAdj<HALF>& lk, KGradD* ld) {
    const KGradD e = kin_time(s, d, gm1);
    double dR[4], ldR[4] = {0.0, 0.0, 0.0, 0.0}, ldq = 0.0;
    dR[0] = kin_dR<0>(k, e);
    dR[1] = kin_dR<1>(k, e);
    dR[2] = kin_dR<2>(k, e);
    dR[3] = kin_dR<3>(k, e);
    const double dq = 2.0 * (s.V * e.V + s.W * e.W) + (K + 2.0) * e.h;
    KGradD le = {0.0, 0.0, 0.0, 0.0, 0.0};
    if constexpr (HALF) adj_dA<0>(s, k, e, dR, dq, lr2, ls, lk, le, ldR, ldq);
    adj_dA<1>(s, k, e, dR, dq, lf2, ls, lk, le, ldR, ldq);
    adj_dR<4>(s, k, K + 2.0, e, ldR, ldq, ls, lk, le);
    adj_time(s, d, gm1, le, ls, ld);
}

// adjoint of kin_moments
template <bool HALF>
__device__ __forceinline__ void adj_moments(const KState<double>& s, const KMom<HALF, double>& k, double K,
                                            KMomAdj<HALF>& lk, KStateAdj& ls) {
    ls.U += k.R[3] * lk.R[4];
    lk.R[3] += s.U * lk.R[4];
    ls.h += k.R2x3 * lk.R[4];
    lk.R[2] += 3.0 * (s.h * lk.R[4]);
    ls.U += k.R[2] * lk.R[3];
    lk.R[2] += s.U * lk.R[3];
    ls.h += k.R1x2 * lk.R[3];
    lk.R[1] += 2.0 * (s.h * lk.R[3]);
    ls.U += k.R[1] * lk.R[2];
    lk.R[1] += s.U * lk.R[2];
    ls.h += k.R[0] * lk.R[2];
    lk.R[0] += s.h * lk.R[2];
    ls.U += k.R[0] * lk.R[1];
    lk.R[0] += s.U * lk.R[1];
    if constexpr (HALF) {
        ls.h += k.F * lk.R[1];
        lk.F += s.h * lk.R[1];
        // d R_0 = R_0 d rho / rho + F (dU - U_h dh);  U_h = U / (2 h);
        // dF = F (d rho / rho - 2 U_h dU + (2 U_h^2 - 1 / (2 h)) dh)
        const double i2h = 0.5 / s.h;
        const double f0 = k.F * lk.R[0], f1 = k.F * lk.F;
        ls.rho += (k.R[0] * lk.R[0] + f1) * s.ir;
        ls.U += f0 - 2.0 * (k.Uh * f1) + i2h * lk.Uh;
        ls.h += -k.Uh * f0 + (2.0 * k.Uh * k.Uh - i2h) * f1 - 2.0 * (i2h * k.Uh * lk.Uh);
    } else {
        ls.rho += lk.R[0];
    }
    ls.V += 2.0 * (s.V * lk.q);
    ls.W += 2.0 * (s.W * lk.q);
    ls.h += (K + 2.0) * lk.q;
}

// adjoint of kin_grad: ld into the state and the conservative gradient, lg[5]
__device__ __forceinline__ void adj_grad(const KState<double>& s, const double* g, double gm1, const KGradD& d,
                                         KGradD ld, KStateAdj& ls, double* lg) {
    const double a = gm1 * ld.h;
    ls.ge -= d.r * ld.h;
    ld.r -= s.ge * ld.h;
    ls.U -= d.U * a;
    ls.V -= d.V * a;
    ls.W -= d.W * a;
    ld.U -= s.U * a;
    ld.V -= s.V * a;
    ld.W -= s.W * a;
    ls.U -= d.r * ld.U;
    ls.V -= d.r * ld.V;
    ls.W -= d.r * ld.W;
    ld.r -= s.U * ld.U + s.V * ld.V + s.W * ld.W;
    ls.ir += g[0] * ld.r + g[1] * ld.U + g[2] * ld.V + g[3] * ld.W + g[4] * a;
    lg[0] = s.ir * ld.r;
    lg[1] = s.ir * ld.U;
    lg[2] = s.ir * ld.V;
    lg[3] = s.ir * ld.W;
    lg[4] = s.ir * a;
}

// adjoint of kin_state: ls into lW (added to)
__device__ __forceinline__ void adj_state(const KState<double>& s, const double* W, double gm1, KStateAdj& ls,
                                          double* lW) {
    const double gge = gm1 * ls.ge;
    const double lp = ls.p + s.ir * ls.h;
    double lir = ls.ir + W[4] * gge + s.p * ls.h;
    const double gp = gm1 * lp, b = -0.5 * gp;
    lW[4] += s.ir * gge + gp;
    const double lU = ls.U + b * W[1], lV = ls.V + b * W[2], lVz = ls.W + b * W[3];
    lW[1] += b * s.U + s.ir * lU;
    lW[2] += b * s.V + s.ir * lV;
    lW[3] += b * s.W + s.ir * lVz;
    lir += W[1] * lU + W[2] * lV + W[3] * lVz;
    lW[0] += ls.rho - s.ir * s.ir * lir;
}

// A side's moments from its two transcendental ones (R0 = rho <u^0>, F)
__device__ __forceinline__ KMom<true, double> side_moments(const KState<double>& s, double K, double R0, double F) {
    KMom<true, double> k;
    k.F = F;
    k.Fh = 0.5 * F;
    k.Uh = s.U * (0.5 / s.h);
    k.q = s.V * s.V + s.W * s.W + (K + 2.0) * s.h;
    k.R[0] = R0;
    k.R[1] = s.U * R0 + s.h * F;
    k.R[2] = s.U * k.R[1] + s.h * k.R[0];
    k.R1x2 = 2.0 * k.R[1];
    k.R1x3 = 3.0 * k.R[1];
    k.R2x3 = 3.0 * k.R[2];
    k.R2x6 = 6.0 * k.R[2];
    k.R[3] = s.U * k.R[2] + s.h * k.R1x2;
    k.R3x4 = 4.0 * k.R[3];
    k.R[4] = s.U * k.R[3] + s.h * k.R2x3;
    return k;
}

// Adjoint of the point solution: output adjoints lFh, lD, lW0, ldW (face
// frame) into the input adjoints: x and lin hold [side][W (5), g[i][q] (15)].
// STAGE1: the records of the first stage; in the second only D and dW have
// adjoints.  VISC must equal ph.viscous.
template <bool VISC, bool STAGE1>
__device__ __forceinline__ void gks_point_adj(const Phys<double>& ph, const double (*x)[20], double dt,
                                              const double* lFh_out, const double* lD_out, const double* lW0_out,
                                              const double* ldW_out, double (*lin)[20]) {
    const double K = ph.K, gm1 = ph.gm1;
    const bool smooth = ph.smooth != 0;
    // ---- forward: the sums over the two sides
    KSums<double> S;
    S.init();
    double pres[2], R0[2], F[2];
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
        const double* W = x[side];
        const KState<double> s = kin_state(W, gm1);
        KGradD d[3];
#pragma unroll
        for (int i = 0; i < 3; ++i) d[i] = kin_grad(s, W + 5 + 5 * i, gm1);
        const KMom<true, double> k = kin_moments<true>(s, K, side == 0 ? +1 : -1);
        pres[side] = s.p;
        R0[side] = k.R[0];
        F[side] = k.F;
        kin_A<0>(s, k, S.w);
        kin_A<1>(s, k, S.f0);
        kin_conv<true>(s, k, d, K, S.d, S.r1, S.f1);
        if constexpr (VISC) {
            const KGradD e = kin_time(s, d, gm1);
            double dR[4];
            dR[0] = kin_dR<0>(k, e);
            dR[1] = kin_dR<1>(k, e);
            dR[2] = kin_dR<2>(k, e);
            dR[3] = kin_dR<3>(k, e);
            const double dq = 2.0 * (s.V * e.V + s.W * e.W) + (K + 2.0) * e.h;
            kin_dA<0>(s, k, e, dR, dq, S.r2);
            kin_dA<1>(s, k, e, dR, dq, S.f2);
        }
    }
    // ---- forward: the equilibrium's sums
    const double Wc[5] = {S.w[0], S.w[1], S.w[2], S.w[3], 0.5 * S.w[4]};
    const KState<double> C = kin_state(Wc, gm1);
    KGradD d[3];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        S.d[i][4] *= 0.5;
        d[i] = kin_grad(C, S.d[i], gm1);
    }
    const KMom<false, double> k = kin_moments<false>(C, K, 0);
    double f0[5] = {0, 0, 0, 0, 0}, f1[5] = {0, 0, 0, 0, 0}, f2[5] = {0, 0, 0, 0, 0}, r1[5] = {0, 0, 0, 0, 0};
    kin_A<1>(C, k, f0);
    kin_conv<false, double>(C, k, d, K, nullptr, r1, f1);
    {
        const KGradD e = kin_time(C, d, gm1);
        double dR[4];
        dR[1] = kin_dR<1>(k, e);
        dR[2] = kin_dR<2>(k, e);
        dR[3] = kin_dR<3>(k, e);
        const double dq = 2.0 * (C.V * e.V + C.W * e.W) + (K + 2.0) * e.h;
        kin_dA<1>(C, k, e, dR, dq, f2);
    }
    const TimeCoef<double> tc = time_coefs(ph, pres[0], pres[1], C.p, dt);
    const double tau = tc.tau, hd = 0.5 * dt, omE = 1.0 - tc.E;
    const double c1 = tau * tc.k0 + tc.k1, dc1 = tau * tc.dk0 + tc.dk1;

    // ---- reverse: outputs (doubled energies: half the adjoint)
    double lFh[5], lD[5], lW0[5], ldW[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        const double c = q == 4 ? 0.5 : 1.0;
        lFh[q] = STAGE1 ? c * lFh_out[q] : 0.0;
        lW0[q] = STAGE1 ? c * lW0_out[q] : 0.0;
        lD[q] = c * lD_out[q];
        ldW[q] = c * ldW_out[q];
    }
    KStateAdj lC;
    double lIWh[5] = {0, 0, 0, 0, 0}, lIWd[5] = {0, 0, 0, 0, 0};
    if constexpr (VISC) {
        if (ph.prf != 0.0) {
            // Pr fix: F_E += prf (qf - U1 qw) on Fh and D, with
            // qf = F_E - U.F_m + |U|^2/2 F_rho, qw the same of the state
            // integral IW and U = U^c
            const double U[3] = {C.U, C.V, C.W};
            const double uu = 0.5 * (U[0] * U[0] + U[1] * U[1] + U[2] * U[2]);
            const double gq[5] = {uu, -U[0], -U[1], -U[2], 1.0};  // d q / d (F or IW)
            double lU[3] = {0.0, 0.0, 0.0};
            for (int n = STAGE1 ? 0 : 1; n < 2; ++n) {
                double Fn[5], IW[5];
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    const double c = q == 4 ? 0.5 : 1.0;
                    double v, w;
                    if (smooth) {
                        v = n == 0 ? hd * f0[q] - tau * hd * f1[q] + (0.5 * hd * hd - tau * hd) * f2[q]
                                   : 0.25 * dt * dt * f2[q];
                        w = n == 0 ? hd * S.w[q] - 0.5 * hd * hd * r1[q] : -0.25 * dt * dt * r1[q];
                    } else {
                        const double e0 = S.f0[q] - f0[q], e1 = S.f1[q] - f1[q];
                        v = n == 0 ? hd * f0[q] + tc.k0 * e0 - c1 * e1 + tc.q3 * f2[q] -
                                         tau * (hd * f1[q] + tc.k0 * S.f2[q])
                                   : tc.dk0 * e0 - dc1 * e1 + tc.dq3 * f2[q] - tau * tc.dk0 * S.f2[q];
                        w = n == 0 ? hd * S.w[q] - c1 * S.r1[q] - tau * tc.k0 * S.r2[q] +
                                         (tc.k1 - 0.5 * hd * hd) * r1[q]
                                   : -dc1 * S.r1[q] - tau * tc.dk0 * S.r2[q] + (tc.dk1 - 0.25 * dt * dt) * r1[q];
                    }
                    Fn[q] = c * v;
                    IW[q] = c * w;
                }
                double* lF = n == 0 ? lFh : lD;
                double* lIW = n == 0 ? lIWh : lIWd;
                const double l = ph.prf * 2.0 * lF[4];  // of the energy itself
                const double qw = IW[4] - (U[0] * IW[1] + U[1] * IW[2] + U[2] * IW[3]) + uu * IW[0];
#pragma unroll
                for (int j = 0; j < 3; ++j)
                    lU[j] += l * (-Fn[1 + j] + U[j] * Fn[0] - (j == 0 ? qw : 0.0) -
                                  U[0] * (-IW[1 + j] + U[j] * IW[0]));
#pragma unroll
                for (int q = 0; q < 5; ++q) {
                    const double c = q == 4 ? 0.5 : 1.0;
                    lF[q] += c * l * gq[q];
                    lIW[q] = -U[0] * c * l * gq[q];
                }
            }
            lC.U += lU[0];
            lC.V += lU[1];
            lC.W += lU[2];
        }
    }
    // adjoints of the sums and of the time coefficients
    double lw[5], lf0s[5], lf1s[5], lr1s[5], lf2s[5], lr2s[5], lf0c[5], lf1c[5], lf2c[5], lr1c[5];
    double ltau = 0.0, lk0 = 0.0, lc1 = 0.0, lq3 = 0.0, ldk0 = 0.0, ldc1 = 0.0, ldq3 = 0.0, lE = 0.0, lk1 = 0.0,
           ldk1 = 0.0;
    if (smooth) {
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            lf0s[q] = lf1s[q] = lr1s[q] = lf2s[q] = lr2s[q] = 0.0;
            lf0c[q] = hd * lFh[q];
            lf1c[q] = -tau * hd * lFh[q];
            lf2c[q] = (0.5 * hd * hd - tau * hd) * lFh[q] + 0.25 * dt * dt * lD[q];
            lr1c[q] = -dt * ldW[q] - 0.5 * hd * hd * lIWh[q] - 0.25 * dt * dt * lIWd[q];
            lw[q] = lW0[q] + hd * lIWh[q];
            if constexpr (VISC) ltau -= hd * lFh[q] * (f1[q] + f2[q]);
        }
    } else {
        const double cw1 = tau - (tau + dt) * tc.E;
#pragma unroll
        for (int q = 0; q < 5; ++q) {
            const double e0 = S.f0[q] - f0[q], e1 = S.f1[q] - f1[q];
            lf0s[q] = tc.k0 * lFh[q] + tc.dk0 * lD[q];
            lf1s[q] = -c1 * lFh[q] - dc1 * lD[q];
            lf2c[q] = tc.q3 * lFh[q] + tc.dq3 * lD[q];
            lf0c[q] = hd * lFh[q] - lf0s[q];
            lf1c[q] = -lf1s[q];
            lw[q] = lW0[q];
            lr1s[q] = cw1 * ldW[q];
            lr1c[q] = -dt * omE * ldW[q];
            lf2s[q] = lr2s[q] = 0.0;
            if constexpr (STAGE1) {
                lk0 += lFh[q] * e0;
                lc1 -= lFh[q] * e1;
                if constexpr (VISC) lq3 += lFh[q] * f2[q];
            }
            ldk0 += lD[q] * e0;
            ldc1 -= lD[q] * e1;
            if constexpr (VISC) ldq3 += lD[q] * f2[q];
            lE += dt * ldW[q] * (r1[q] - S.r1[q]);
            if constexpr (VISC) {
                const double rs = S.r1[q] + S.r2[q];
                lf1c[q] -= tau * hd * lFh[q];
                lf2s[q] = -tau * (tc.k0 * lFh[q] + tc.dk0 * lD[q]);
                lr1s[q] -= tau * lW0[q];
                lr2s[q] = tau * (omE * ldW[q] - lW0[q]);
                lk0 -= tau * lFh[q] * S.f2[q];
                ldk0 -= tau * lD[q] * S.f2[q];
                lE -= tau * ldW[q] * rs;
                ltau += (omE * ldW[q] - lW0[q]) * rs - lFh[q] * (hd * f1[q] + tc.k0 * S.f2[q]) -
                        lD[q] * tc.dk0 * S.f2[q];
                // state integrals of the Pr fix
                lw[q] += hd * lIWh[q];
                lr1s[q] -= c1 * lIWh[q] + dc1 * lIWd[q];
                lr2s[q] -= tau * (tc.k0 * lIWh[q] + tc.dk0 * lIWd[q]);
                lr1c[q] += (tc.k1 - 0.5 * hd * hd) * lIWh[q] + (tc.dk1 - 0.25 * dt * dt) * lIWd[q];
                lc1 -= lIWh[q] * S.r1[q];
                ldc1 -= lIWd[q] * S.r1[q];
                lk0 -= tau * lIWh[q] * S.r2[q];
                ldk0 -= tau * lIWd[q] * S.r2[q];
                ltau -= (tc.k0 * lIWh[q] + tc.dk0 * lIWd[q]) * S.r2[q];
                lk1 += lIWh[q] * r1[q];
                ldk1 += lIWd[q] * r1[q];
            }
        }
    }
    // ---- reverse: the equilibrium
    KMomAdj<false> lk;
    KGradD lg[3] = {{0, 0, 0, 0, 0}, {0, 0, 0, 0, 0}, {0, 0, 0, 0, 0}};
    adj_A<1>(C, k, lf0c, lC, lk);
    adj_time_sums<false>(C, k, d, K, gm1, nullptr, lf2c, lC, lk, lg);
    adj_conv<false>(C, k, d, K, nullptr, lr1c, lf1c, lC, lk, lg);
    adj_moments<false>(C, k, K, lk, lC);
    double lds[3][5];
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        adj_grad(C, S.d[i], gm1, d[i], lg[i], lC, lds[i]);
        lds[i][4] *= 0.5;
    }
    // time coefficients -> tau_n, tau -> the pressures
    double lp[2] = {0.0, 0.0};
    if (!smooth) {
        // c1 = tau k0 + k1; q3 = hd^2/2 - tau hd + tau k0; dc1, dq3 alike
        lk0 += tau * (lc1 + lq3);
        lk1 += lc1;
        ldk0 += tau * (ldc1 + ldq3);
        ldk1 += ldc1;
        if constexpr (VISC) ltau += tc.k0 * (lc1 + lq3) - hd * lq3 + tc.dk0 * (ldc1 + ldq3);
        const double tn = tc.tau_n, itn = 1.0 / tn;
        const double Eh = d_exp(-hd * itn), omh = 1.0 - Eh;
        double ltn = lk0 * omh + lk1 * (2.0 * tn * omh - hd * Eh) - ldk0 * omh * omh +
                     ldk1 * omh * (dt * Eh - 2.0 * tn * omh);
        const double lomh = lk0 * tn + lk1 * tn * tn - 2.0 * ldk0 * tn * omh + ldk1 * tn * (dt * Eh - 2.0 * tn * omh);
        const double lEh = -lk1 * tn * hd + ldk1 * tn * dt * omh + 2.0 * Eh * lE - lomh;
        ltn += lEh * Eh * hd * itn * itn;
        // tn = (viscous ? tau : tau_eps dt) + tau_c |x| dt, x = (pl - pr) / (pl + pr)
        if constexpr (VISC) ltau += ltn;
        const double pl = pres[0], pr = pres[1], ips = 1.0 / (pl + pr);
        const double sx = pl > pr ? 1.0 : (pl < pr ? -1.0 : 0.0);
        const double lx = 2.0 * ltn * ph.tau_c * dt * sx * ips * ips;
        lp[0] = lx * pr;
        lp[1] = -lx * pl;
    }
    // tau = mu / p_c (viscous)
    if constexpr (VISC) lC.p -= ltau * tau / C.p;
    double lWc[5] = {0, 0, 0, 0, 0};
    adj_state(C, Wc, gm1, lC, lWc);
#pragma unroll
    for (int q = 0; q < 5; ++q) lw[q] += q == 4 ? 0.5 * lWc[q] : lWc[q];
    // ---- reverse: each side
#pragma unroll 1
    for (int side = 0; side < 2; ++side) {
        const double* W = x[side];
        const KState<double> s = kin_state(W, gm1);
        KGradD ds[3], lgs[3] = {{0, 0, 0, 0, 0}, {0, 0, 0, 0, 0}, {0, 0, 0, 0, 0}};
#pragma unroll
        for (int i = 0; i < 3; ++i) ds[i] = kin_grad(s, W + 5 + 5 * i, gm1);
        const KMom<true, double> ks = side_moments(s, K, R0[side], F[side]);
        KStateAdj ls;
        KMomAdj<true> lks;
        ls.p = lp[side];
        adj_A<0>(s, ks, lw, ls, lks);
        adj_A<1>(s, ks, lf0s, ls, lks);
        if constexpr (VISC) adj_time_sums<true>(s, ks, ds, K, gm1, lr2s, lf2s, ls, lks, lgs);
        adj_conv<true>(s, ks, ds, K, lds, lr1s, lf1s, ls, lks, lgs);
        adj_moments<true>(s, ks, K, lks, ls);
        double* l = lin[side];
#pragma unroll
        for (int i = 0; i < 3; ++i) adj_grad(s, W + 5 + 5 * i, gm1, ds[i], lgs[i], ls, l + 5 + 5 * i);
#pragma unroll
        for (int q = 0; q < 5; ++q) l[q] = 0.0;
        adj_state(s, W, gm1, ls, l);
    }
}

}  // namespace gks
