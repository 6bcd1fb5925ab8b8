// gks_device.cuh -- device-side building blocks of libgks, templated on the
// working precision T (double: FP64 path; float: FP32-bulk path).
//
//   * conversions between FP64 and FP32 off the FP64 pipe, compensated sums
//     and FP32 pairs;
//   * the time coefficients of Eq. 2nd-flux over [0, dt/2] and [0, dt];
//   * the Pr fix, the wall-independent parts of the FP32 interface deviation
//     (half-differences) and the Euler flux.
// The kinetic solution itself is in gks_kinetic.cuh.
#pragma once

#include <cstdint>

namespace gks {

// --------------------------------------------------------------- math --
__device__ __forceinline__ double d_exp(double x) { return exp(x); }
__device__ __forceinline__ float d_exp(float x) { return expf(x); }
// erfc(y) / 2, given ex = exp(-y^2).  FP64 by erfcx, which saves the second
// exponential of a pipe-bound kernel (a whole step with 49,280 faces 1,191 ->
// 1,169 us; a reverse step of 48,000 cells 5,704 -> 5,648 us).  ex carries the
// rounding of y^2, a relative error of at most y^2 half units: at most 0.2 half
// units of 1, as erfc falls faster than y^2 grows, and the same error that
// the Gaussian tail beside it has.
__device__ __forceinline__ double half_erfc(double y, double ex) {
    const double t = 0.5 * ex * erfcx(fabs(y));
    return y < 0.0 ? 1.0 - t : t;
}
__device__ __forceinline__ float half_erfc(float y, float) { return 0.5f * erfcf(y); }
__device__ __forceinline__ double d_rsqrt(double x) { return rsqrt(x); }
__device__ __forceinline__ float d_rsqrt(float x) { return rsqrtf(x); }
__device__ __forceinline__ double d_abs(double x) { return fabs(x); }
__device__ __forceinline__ float d_abs(float x) { return fabsf(x); }
__device__ __forceinline__ double d_cbrt(double x) { return cbrt(x); }
__device__ __forceinline__ float d_cbrt(float x) { return cbrtf(x); }

// |x|^(4/3) as x * cbrt(x) for x >= 0
template <typename T>
__device__ __forceinline__ T pow43(T x) { return x * d_cbrt(x); }

// FP32 <-> FP64 conversions on the integer pipe.  The FP64 unit (which also
// takes the conversion instructions) issues a warp instruction in 16 cycles,
// the integer unit in half a cycle, and the cell updates convert more than
// they add.  Same values as the conversions: widening is exact, narrowing
// rounds to nearest even; numbers outside the range the bit forms cover
// (zeros apart) take the conversion instruction.
// The conversion instructions stand in functions of their own: inlined, the
// compiler would compute both forms and select.
__device__ __noinline__ static double widen_any(float x) { return (double)x; }
__device__ __noinline__ static float narrow_any(double x) { return (float)x; }

__device__ __forceinline__ double widen(float x) {
    const uint32_t b = __float_as_uint(x), m = b & 0x7fffffffu;
    if (m - 0x00800000u >= 0x7f000000u && m != 0u) return widen_any(x);  // denormal, infinite, NaN
    const uint32_t hi = m != 0u ? (m >> 3) + (896u << 20) : 0u;
    return __hiloint2double((int)((b & 0x80000000u) | hi), (int)(m << 29));
}
__device__ __forceinline__ double widen(double x) { return x; }

// x = hi + lo + (below half an ulp of lo): hi = x and lo = x - hi, each
// rounded to nearest
__device__ __forceinline__ void split_pair(double x, float& hi, float& lo) {
    const uint64_t b = (uint64_t)__double_as_longlong(x);
    const uint32_t e = (uint32_t)(b >> 52) & 0x7ffu;
    if (e - 963u > 120u && (b << 1) != 0u) {  // not within 2^-60 .. 2^61
        hi = narrow_any(x);
        lo = narrow_any(x - widen_any(hi));
        return;
    }
    const uint64_t m = b & 0x7fffffffffffffffull;
    const uint64_t r = (m + 0x0fffffffull + ((m >> 29) & 1u)) >> 29;  // rounded to 23 fraction bits
    const uint32_t sign = (uint32_t)(b >> 32) & 0x80000000u;
    const int32_t rest = (int32_t)((uint32_t)m - (uint32_t)(r << 29));  // |rest| <= 2^28 units of 2^(e - 1075)
    const bool zero = m == 0u;
    hi = __uint_as_float(zero ? sign : sign | ((uint32_t)r - (896u << 23)));
    const float scale = __uint_as_float(sign | ((e - 948u) << 23));
    lo = zero ? 0.0f : (float)rest * scale;
}
__device__ __forceinline__ float narrow(double x) {
    const uint64_t b = (uint64_t)__double_as_longlong(x), m = b & 0x7fffffffffffffffull;
    const uint32_t e = (uint32_t)(m >> 52), sign = (uint32_t)(b >> 32) & 0x80000000u;
    if (e - 897u > 252u && m != 0u) return narrow_any(x);  // not within 2^-126 .. 2^127
    const uint64_t r = (m + 0x0fffffffull + ((m >> 29) & 1u)) >> 29;
    return __uint_as_float(m == 0u ? sign : sign | ((uint32_t)r - (896u << 23)));
}

// Error-free transformation of a sum (Knuth's TwoSum): a + b = s + e exactly.
template <typename T>
__device__ __forceinline__ void two_sum(T a, T b, T& s, T& e) {
    s = a + b;
    T bb = s - a;
    e = (a - (s - bb)) + (b - bb);
}

// Compensated accumulator: value = hi + lo.
template <typename T>
struct CSum {
    T hi, lo;
    __device__ __forceinline__ void init() { hi = T(0); lo = T(0); }
    __device__ __forceinline__ void add(T x) {
        T s, e;
        two_sum(hi, x, s, e);
        hi = s;
        lo += e;
    }
    __device__ __forceinline__ double value() const { return widen(hi) + widen(lo); }
};

// ------------------------------------------------------------ params --
template <typename T>
struct Phys {
    T gamma, gm1, K;     // K internal degrees of freedom
    T tau_eps, tau_c, mu;
    T eps_w;
    T prf;               // Pr fix: 1/Pr - 1 (0 without it)
    T twall;             // temperature p / rho of isothermal walls
    T uwall[3];          // velocity of moving walls (global frame)
    int viscous, smooth;
};

// ------------------------------------------------- time integration --
// Time coefficients of Eq. 2nd-flux over [0, dt/2] (k0, k1 for the kinetic
// factors e and t e; q2, q3 for C2, C3) and their "dt minus twice dt/2"
// differences (dk*, dq*), with E = exp(-dt/tau_n) = Eh^2.
template <typename T>
struct TimeCoef {
    T tau, tau_n, E;
    T k0, k1, q2, q3;
    T dk0, dk1, dq2, dq3;
};

template <typename T>
__device__ __forceinline__ TimeCoef<T> time_coefs(const Phys<T>& ph, T pl, T pr, T pc, T dt) {
    TimeCoef<T> c;
    c.tau = ph.viscous ? ph.mu / pc : T(0);
    const T jump = d_abs((pl - pr) / (pl + pr)) * dt;
    c.tau_n = (ph.viscous ? ph.mu / pc : ph.tau_eps * dt) + ph.tau_c * jump;
    const T hd = T(0.5) * dt;
    const T Eh = d_exp(-hd / c.tau_n);
    c.E = Eh * Eh;
    const T omh = T(1) - Eh;
    const T tn = c.tau_n, tau = c.tau;
    c.k0 = tn * omh;
    c.k1 = tn * (tn * omh - hd * Eh);
    c.q2 = c.k1 + tau * c.k0 - tau * hd;
    c.q3 = T(0.5) * hd * hd - tau * hd + tau * c.k0;
    c.dk0 = -tn * omh * omh;
    c.dk1 = -tn * tn * omh * omh + tn * dt * Eh * omh;
    c.dq2 = c.dk1 + tau * c.dk0;
    c.dq3 = T(0.25) * dt * dt + tau * c.dk0;
    return c;
}

// Pr fix of the energy flux over one time interval: F_E += (1/Pr - 1) q with
// q = int (u1 - U1) (|u - U|^2 + xi^2) / 2 f, expanded into the flux F and the
// state integral IW = int psi f over the same interval (U the interface
// equilibrium velocity, face frame):
//   q = F_E - U.F_m + |U|^2/2 F_rho - U1 (IW_E - U.IW_m + |U|^2/2 IW_rho)
template <typename T>
__device__ __forceinline__ void prandtl_fix(T prf, const T* U, const T* IW, T* F) {
    const T uu = T(0.5) * (U[0] * U[0] + U[1] * U[1] + U[2] * U[2]);
    const T qf = F[4] - (U[0] * F[1] + U[1] * F[2] + U[2] * F[3]) + uu * F[0];
    const T qw = IW[4] - (U[0] * IW[1] + U[1] * IW[2] + U[2] * IW[3]) + uu * IW[0];
    F[4] += prf * (qf - U[0] * qw);
}

// --------------------------------------------- half differences --
// A quantity known on the two sides of a face: its values l, r and, accurate
// to the rounding of itself, its half-difference h = (l - r) / 2.  The rules
// below are exact identities for finite differences (not linearisations), so
// h keeps its relative accuracy however small it is, where (l - r) / 2 formed
// from the rounded values would carry the rounding of l and r:
//   product   (l_a l_b - r_a r_b) / 2 = h_a mid_b + mid_a h_b
//   quotient  (l_a / l_b - r_a / r_b) / 2 = (h_a mid_b - mid_a h_b) / (l_b r_b)
//   root      (sqrt l - sqrt r) / 2 = h / (sqrt l + sqrt r)
// FP32 bulk uses them to form the interface state W^c (Eq. new-equ-part)
// relative to the mean of the two sides.

// What the deviation below takes of a side's half-space moments: <u^0>,
// sqrt(lambda) and e^{-s^2}, s = sqrt(lambda) U
template <typename T>
struct HalfSpace {
    T m0, rl, ex;
};

// Half-difference of psi(W) = rho <psi>_{u1>0} - rho <psi>_{u1<0} between
// the two states Wl, Wr (face frame, x1 along the normal), given the
// half-difference h of the states themselves.  With e0 = erf(s) and
// G = rho e^{-s^2} / sqrt(pi lambda), the half-space moments of Sec. 2.2 give
//   psi(W) = (rho e0, W1 e0 + G, W2 e0, W3 e0, W4 e0 + U1 G / 2),
// and W^c = rho_l <psi>_{u1>0} + rho_r <psi>_{u1<0} = (Wl + Wr) / 2 +
// (psi(Wl) - psi(Wr)) / 2, so W^c minus the mean of the two states is h_psi.
//
// (erf l - erf r) / 2 and (e^{-l^2} - e^{-r^2}) / 2 are the integrals of
// e^{-t^2} / sqrt(pi) and -t e^{-t^2} over [s_r, s_l] by one Gauss-Legendre
// rule on the same nodes: 3 points for |s_l - s_r| <= 0.1, 5 points up to 1
// (errors below 1e-9 and 2e-7 of the integrands' scale at those lengths, far
// less for shorter intervals); beyond, the differences of the tails' erfc and
// of the exponentials, which do not cancel there.
//
// The half-differences are those of U and p / rho, with the exponentials of
// the kinetic solution and of the one quadrature: carrying (l, r, h) triples
// through every product, with an expm1 and two more exponentials, took 250 of
// the stage-1 flux's instructions more (3.15 M faces: 1,108 -> 1,071 us).
__device__ __forceinline__ void psi_half_difference(const float* Wl, const float* Wr, const float* h, float gm1,
                                                    const HalfSpace<float>& hl, const HalfSpace<float>& hr,
                                                    float* out) {
    const float il = 1.0f / Wl[0], ir = 1.0f / Wr[0], ii = il * ir;
    float mid[5];
#pragma unroll
    for (int q = 0; q < 5; ++q) mid[q] = 0.5f * (Wl[q] + Wr[q]);
    // velocities and p / rho
    float U[3], hU[3];
    float hT = (h[4] * mid[0] - mid[4] * h[0]) * ii;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        U[j] = 0.5f * (Wl[1 + j] * il + Wr[1 + j] * ir);
        hU[j] = (h[1 + j] * mid[0] - mid[1 + j] * h[0]) * ii;
        hT -= U[j] * hU[j];
    }
    hT *= gm1;
    // rl = (2 T)^{-1/2} and its inverse
    const float rr = hl.rl * hr.rl, irs = 1.0f / (hl.rl + hr.rl);
    const float hir = 2.0f * (hT * rr) * irs;  // of 1 / rl
    const float hrl = -hir * rr;
    const float rm = 0.5f * (hl.rl + hr.rl), irm = rm / rr;  // mid of rl and of 1 / rl
    const float d = hU[0] * rm + U[0] * hrl;                 // of s
    const float m = 0.5f * (Wl[1] * il * hl.rl + Wr[1] * ir * hr.rl);
    // erf and e^{-s^2}
    float he, hx;
    const float ad = fabsf(d);
    if (ad <= 0.5f) {
        // nodes and weights on [-1, 1]
        const bool few = ad <= 0.05f;
        const float x1 = few ? 0.77459666924148338f : 0.53846931010568309f;
        const float w0 = few ? 0.88888888888888889f : 0.56888888888888889f;
        const float w1 = few ? 0.55555555555555556f : 0.47862867049936647f;
        const float tp = m + x1 * d, tm = m - x1 * d;
        const float g0 = w0 * expf(-m * m), gp = w1 * expf(-tp * tp), gm = w1 * expf(-tm * tm);
        float s0 = g0 + (gp + gm), s1 = m * g0 + (tp * gp + tm * gm);
        if (!few) {
            const float x2 = 0.90617984593866399f, w2 = 0.23692688505618909f;
            const float up = m + x2 * d, um = m - x2 * d;
            const float hp = w2 * expf(-up * up), hm = w2 * expf(-um * um);
            s0 += hp + hm;
            s1 += up * hp + um * hm;
        }
        he = 0.56418958354775628695f * d * s0;  // 1 / sqrt(pi)
        hx = -d * s1;
    } else {
        const float sl = Wl[1] * il * hl.rl, sr = Wr[1] * ir * hr.rl;
        he = m > 0.0f ? 0.5f * (erfcf(sr) - erfcf(sl)) : 0.5f * (erfcf(-sl) - erfcf(-sr));
        hx = 0.5f * (hl.ex - hr.ex);
    }
    // e0 on the sides from their half-space moments: 2 <u^0>_{u1>0} - 1 on
    // the left, 1 - 2 <u^0>_{u1<0} on the right
    const float e0 = hl.m0 - hr.m0;
    const float ym = 0.5f * (hl.ex / hl.rl + hr.ex / hr.rl);  // mid of e^{-s^2} / rl
    const float hy = hx * irm + 0.5f * (hl.ex + hr.ex) * hir;
    const float c = 0.56418958354775628695f;
    const float hG = c * (h[0] * ym + mid[0] * hy);
    const float Gm = 0.5f * c * (Wl[0] * (hl.ex / hl.rl) + Wr[0] * (hr.ex / hr.rl));
#pragma unroll
    for (int q = 0; q < 5; ++q) out[q] = h[q] * e0 + mid[q] * he;
    out[1] += hG;
    out[4] += 0.5f * (hU[0] * Gm + U[0] * hG);
}

// Euler flux along x1 of a face-frame state: (m1, m1 u + p, m2 u, m3 u,
// (E + p) u), u = m1 / rho.
__device__ __forceinline__ void euler_flux1(const float* W, float gm1, float* out) {
    const float u = W[1] / W[0];
    const float p = gm1 * (W[4] - 0.5f * (W[1] * W[1] + W[2] * W[2] + W[3] * W[3]) / W[0]);
    out[0] = W[1];
    out[1] = W[1] * u + p;
    out[2] = W[2] * u;
    out[3] = W[3] * u;
    out[4] = (W[4] + p) * u;
}

// F_1(Wc) - F_1(Wm) given d = Wc - Wm of the two face-frame states: exact to
// the rounding of the result itself, however close the two states.  With
// U = m / rho, U_c - U_m = (d_m - U_m d_rho) / rho_c.
__device__ __forceinline__ void flux1_difference(const float* Wc, const float* Wm, const float* d, float gm1,
                                                 float* out) {
    const float ic = 1.0f / Wc[0], im = 1.0f / Wm[0];
    float dk = 0.0f, km = 0.0f, du = 0.0f, um = 0.0f;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float U = Wm[1 + j] * im, dU = (d[1 + j] - U * d[0]) * ic;
        dk += d[1 + j] * (U + dU) + Wm[1 + j] * dU;  // of m . U
        km += Wm[1 + j] * U;
        if (j == 0) {
            um = U;
            du = dU;
        }
    }
    const float uc = um + du;
    const float dp = gm1 * (d[4] - 0.5f * dk), pm = gm1 * (Wm[4] - 0.5f * km);
    out[0] = d[1];
#pragma unroll
    for (int j = 0; j < 3; ++j) out[1 + j] = d[1 + j] * uc + Wm[1 + j] * du + (j == 0 ? dp : 0.0f);
    out[4] = (d[4] + dp) * uc + (Wm[4] + pm) * du;
}

// ------------------------------------------------- FP32 pair numbers --
// A value hi + lo carried as two FP32 numbers (|lo| <= ulp(hi) / 2): about
// 48 significant bits at FP32-pipe speed.  Sums by Knuth's TwoSum, products
// by the FMA form of Dekker's TwoProduct, quotients by one correction of an
// FP32 quotient with the exact residual.  Used where a value of O(|W|) or
// O(|F|) must stay exact to far below FP32 rounding without the FP64 unit
// (the FP32-bulk reference flux).
struct F2 {
    float hi, lo;
};

__device__ __forceinline__ F2 f2_norm(float s, float e) {
    const float h = s + e;
    return {h, e - (h - s)};
}

__device__ __forceinline__ F2 f2_add(F2 a, F2 b) {
    float s, e;
    two_sum(a.hi, b.hi, s, e);
    e += a.lo + b.lo;
    return f2_norm(s, e);
}

__device__ __forceinline__ F2 f2_mul(F2 a, F2 b) {
    const float p = a.hi * b.hi;
    float e = fmaf(a.hi, b.hi, -p);
    e += a.hi * b.lo + a.lo * b.hi;
    return f2_norm(p, e);
}

__device__ __forceinline__ F2 f2_scale(float c, F2 a) {
    const float p = c * a.hi;
    float e = fmaf(c, a.hi, -p);
    e += c * a.lo;
    return f2_norm(p, e);
}

__device__ __forceinline__ F2 f2_div(F2 a, F2 b) {
    const float q = a.hi / b.hi;
    // residual a - q b, exact to the pair's precision
    const F2 qb = f2_mul({q, 0.0f}, b);
    const F2 r = f2_add(a, {-qb.hi, -qb.lo});
    return f2_norm(q, r.hi / b.hi);
}


}  // namespace gks
