// gks_adjoint.cu -- reverse (adjoint) sweep of one two-stage step, FP64.
//
// Given the adjoint of the step's result, (lambda W^{n+1}, lambda grad
// W^{n+1}), these kernels return the adjoint of its start, (lambda W^n,
// lambda grad W^n): the transpose of the step's Jacobian applied to a vector,
// with the time step frozen.  Every part of the step but the kinetic solution
// at a Gauss point is linear in the working state (the linear-weight
// reconstruction, the evaluation of R at the Gauss points, the face frame
// rotations, the stage records of Eqs. linear-system and s2o4, the update of
// averages and of gradients by Eq. gauss-formula); those are transposed by
// hand, each as a gather so that no two threads write one location.  The
// kinetic solution (Eq. 2nd-flux with Eq. new-equ-part) is differentiated in
// reverse mode (gks_point_adj.cuh, about three point evaluations of work),
// inviscid or viscous.
//
//   k_adj_src2 / k_adj_src1  per-cell adjoints of the face-record sums
//   k_adj_point_rev<NR>      per (face, Gauss point): the point solution's
//                            adjoint in reverse mode
//   k_adj_face_back          per face: rotations and evaluation at the
//                            points transposed -> adjoints of both cells'
//                            reconstruction coefficients
//   k_adj_gather_poly        per cell: sum over its four faces
//   k_adj_recon_local        per cell: transpose of a = M2 d and of the
//                            monomial constant (linear weights)
//   k_adj_recon_weno         the same with the nonlinear WENO weights, after
//   k_adj_p1, k_adj_slopes   and the neighbours' P1 slopes those weights use
//   k_adj_recon_gather       per cell: adjoint of its working state from its
//                            own and its neighbours' stencil adjoints
//   k_adj_final              the three paths into (W^n, grad W^n)
#include <cuda_runtime.h>

#include "gks_cells.cuh"
#include "gks_device.cuh"
#include "gks_face.cuh"
#include "gks_kernels.h"
#include "gks_point_adj.cuh"
#include "gks_recon.cuh"

namespace gks {

constexpr int ADJ_IN = 40;       // inputs of the point solution: WL, gL, WR, gR (face frame)
constexpr int ADJ_THREADS = 64;  // threads per block of the face kernels

// stage 2 records: [sum w 4/3 D (5) | sum w dW n (15)]; the cell sums enter
// W^{n+1} = W^n - (S + sum s rec[0:5]) / |Omega| and
// grad W^{n+1} = (G + sum s rec[5:20]) / |Omega|
__global__ void k_adj_src2(DevMesh<double> m, const double* __restrict__ lW, const double* __restrict__ ldW,
                           double* __restrict__ src) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= m.nc) return;
    const double iv = m.inv_vol[c];
    double* o = src + c * 20;
    for (int q = 0; q < 5; ++q) o[q] = -lW[q * m.nc + c] * iv;
    for (int j = 0; j < 15; ++j) o[5 + j] = ldW[j * m.nc + c] * iv;
}

// stage 1 records: [sum w Fh | sum w (2 Fh - D/3) | sum w W* n | sum w W0 n];
// they enter W* = W^n - sum s rec[0:5] / |Omega|, S = sum s rec[5:10] (into
// W^{n+1} with -1/|Omega|), grad W* = sum s rec[10:25] / |Omega| and
// G = sum s rec[25:40] (into grad W^{n+1} with 1/|Omega|)
__global__ void k_adj_src1(DevMesh<double> m, const double* __restrict__ lW, const double* __restrict__ ldW,
                           const double* __restrict__ lXs, double* __restrict__ src) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= m.nc) return;
    const double iv = m.inv_vol[c];
    const double* xs = lXs + c * XS;
    double* o = src + c * 40;
    for (int q = 0; q < 5; ++q) {
        o[q] = -xs[q] * iv;
        o[5 + q] = -lW[q * m.nc + c] * iv;
    }
    for (int j = 0; j < 15; ++j) {
        o[10 + j] = xs[5 + j] * iv;
        o[25 + j] = ldW[j * m.nc + c] * iv;
    }
}

// adjoint of eval_poly: lc += (d val / d c)^T lv + (d g / d c)^T lg
__device__ __forceinline__ void eval_poly_adj(const double* X, const double* lv, const double (*lg)[5],
                                              double* lc) {
    const double x = X[0], y = X[1], z = X[2];
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        double* c = lc + q * 10;
        const double v = lv[q], g0 = lg[0][q], g1 = lg[1][q], g2 = lg[2][q];
        const double sx = v * x + g0, sy = v * y + g1, sz = v * z + g2;
        c[0] += v;
        c[1] += sx;
        c[2] += sy;
        c[3] += sz;
        c[4] += x * (sx + g0);
        c[5] += y * sx + x * g1;
        c[6] += z * sx + x * g2;
        c[7] += y * (sy + g1);
        c[8] += z * sy + y * g2;
        c[9] += z * (sz + g2);
    }
}

// adjoint of to_local: (lW, lg) global from (lWt, lgt) in the face frame
__device__ __forceinline__ void to_local_adj(const double (*Rm)[3], const double* lWt, const double (*lgt)[5],
                                             double* lW, double (*lg)[5]) {
    lW[0] = lWt[0];
    lW[4] = lWt[4];
    for (int i = 0; i < 3; ++i) lW[1 + i] = Rm[0][i] * lWt[1] + Rm[1][i] * lWt[2] + Rm[2][i] * lWt[3];
    double lh[3][5];
    for (int j = 0; j < 3; ++j) {
        lh[j][0] = lgt[j][0];
        lh[j][4] = lgt[j][4];
        for (int l = 0; l < 3; ++l)
            lh[j][1 + l] = Rm[0][l] * lgt[j][1] + Rm[1][l] * lgt[j][2] + Rm[2][l] * lgt[j][3];
    }
    for (int i = 0; i < 3; ++i)
        for (int q = 0; q < 5; ++q) lg[i][q] = Rm[0][i] * lh[0][q] + Rm[1][i] * lh[1][q] + Rm[2][i] * lh[2][q];
}

// the momentum block of a global vector in the face frame (the adjoint of
// to_global)
__device__ __forceinline__ void rotate_in(const double (*Rm)[3], double* v) {
    const double a = v[1], b = v[2], c = v[3];
    for (int j = 0; j < 3; ++j) v[1 + j] = Rm[j][0] * a + Rm[j][1] * b + Rm[j][2] * c;
}

// The point's inputs in the face frame (per side W, g: 20 values) from the
// stored reconstruction, with R as the plain sum of its terms where the forward
// flux takes the nested form (the same to rounding, see below), and the output
// adjoints of the point (face frame) from the record adjoints (the transposed
// record formulas of the stage).
template <int NR>
__device__ __forceinline__ void adj_point_setup(const DevMesh<double>& m, const Phys<double>& ph,
                                                const double* __restrict__ poly, const double* __restrict__ Xavg,
                                                const double* __restrict__ src, int64_t f, int k, double (*x)[20],
                                                double* lFh, double* lD, double* lW0, double* ldWt) {
    const int L = m.flr[f], R = m.flr[m.nf + f];
    const double* geo = m.fgeo + f * FGEO;
    const double n[3] = {geo[0], geo[1], geo[2]};
    const double w = geo[3];
    double Rm[3][3];
    face_frame(n, Rm);
    // record adjoints: the left cell adds the record, the right one subtracts it
    // (a boundary face has one cell)
    double lr[NR];
#pragma unroll
    for (int j = 0; j < NR; ++j)
        lr[j] = (L >= 0 ? src[(int64_t)L * NR + j] : 0.0) - (R >= 0 ? src[(int64_t)R * NR + j] : 0.0);
#pragma unroll
    for (int q = 0; q < 5; ++q) {
        double sn0 = 0.0, sn1 = 0.0;
        if (NR == 40) {
#pragma unroll
            for (int i = 0; i < 3; ++i) {
                sn0 += n[i] * lr[10 + 3 * q + i];
                sn1 += n[i] * lr[25 + 3 * q + i];
            }
            lFh[q] = w * (lr[q] + 2.0 * lr[5 + q]);
            lD[q] = -w * (1.0 / 3.0) * lr[5 + q];
            lW0[q] = w * (sn0 + sn1);
            ldWt[q] = 0.5 * w * sn0;
        } else {
#pragma unroll
            for (int i = 0; i < 3; ++i) sn0 += n[i] * lr[5 + 3 * q + i];
            lFh[q] = 0.0;
            lD[q] = w * (4.0 / 3.0) * lr[q];
            lW0[q] = 0.0;
            ldWt[q] = w * sn0;
        }
    }
    if (NR == 40) {
        rotate_in(Rm, lFh);
        rotate_in(Rm, lW0);
    }
    rotate_in(Rm, lD);
    rotate_in(Rm, ldWt);
    // R as the plain sum: where the field is uniform to rounding, the derivative
    // of |p_l - p_r| is the sign of what rounding leaves.  Nothing makes one
    // evaluation exact there, but the plain sum agrees best with the method in
    // plain FP64 arrays differentiated by autograd: gradients of the vortex
    // (48,000 cells) within 1e-11 over four seeds, two of them within 3e-14, against
    // 1e-10 to 5e-10 with the nested form and 2e-9 to 3e-9 with the derivative set
    // to zero within four ulps of a tie (either form); it takes 2 % more (5,650 ->
    // 5,790 us a reverse step).
#pragma unroll 1
    for (int side = 0; side < 2; ++side)
        side_state<double, true, true>(m, ph, Xavg, poly + side_cell(L, R, side) * POLY_STRIDE, geo, Rm, L, R, side, k,
                                 x[side], reinterpret_cast<double (*)[5]>(x[side] + 5));
}

// A forward-mode number (value and one derivative) for the Jacobian of the
// isothermal-wall ghost, the one nonlinear ghost.
struct Fwd {
    double v, d;
    __device__ Fwd() : v(0.0), d(0.0) {}
    __device__ Fwd(double x) : v(x), d(0.0) {}
    __device__ Fwd(double x, double dx) : v(x), d(dx) {}
};
__device__ __forceinline__ Fwd operator+(Fwd a, Fwd b) { return Fwd(a.v + b.v, a.d + b.d); }
__device__ __forceinline__ Fwd operator-(Fwd a, Fwd b) { return Fwd(a.v - b.v, a.d - b.d); }
__device__ __forceinline__ Fwd operator-(Fwd a) { return Fwd(-a.v, -a.d); }
__device__ __forceinline__ Fwd operator*(Fwd a, Fwd b) { return Fwd(a.v * b.v, a.d * b.v + a.v * b.d); }
__device__ __forceinline__ Fwd operator/(Fwd a, Fwd b) {
    const double q = a.v / b.v;
    return Fwd(q, (a.d - q * b.d) / b.v);
}
__device__ __forceinline__ Fwd& operator+=(Fwd& a, Fwd b) { return a = a + b; }

// li += J^T ls for a nonlinear wall ghost G (isothermal or moving wall) at
// the interior face-frame state x (W, grad W: 20 values), by one forward pass
// per input; Uw is the wall velocity in the face frame
__device__ void wall_ghost_adj(int kind, const double* x, const double* ls, double gm1, double twall,
                               const double* Uw, double* li) {
    const Fwd Uwd[3] = {Fwd(Uw[0]), Fwd(Uw[1]), Fwd(Uw[2])};
    for (int i = 0; i < 20; ++i) {
        Fwd Wd[5], gd[3][5];
        for (int q = 0; q < 5; ++q) Wd[q] = Fwd(x[q], i == q ? 1.0 : 0.0);
        for (int j = 0; j < 3; ++j)
            for (int q = 0; q < 5; ++q) gd[j][q] = Fwd(x[5 + 5 * j + q], i == 5 + 5 * j + q ? 1.0 : 0.0);
        if (kind == FLR_ISOTHERMAL_WALL)
            isothermal_wall_ghost(Wd, gd, Fwd(gm1), Fwd(twall));
        else
            moving_wall_ghost(Wd, gd, Fwd(gm1), Uwd);
        double acc = 0.0;
        for (int q = 0; q < 5; ++q) acc += ls[q] * Wd[q].d;
        for (int j = 0; j < 3; ++j)
            for (int q = 0; q < 5; ++q) acc += ls[5 + 5 * j + q] * gd[j][q].d;
        li[i] += acc;
    }
}

// One thread per (face, Gauss point): the point solution's adjoint in reverse
// mode (gks_point_adj), lx[i][f][k] for the 40 inputs i (input-major, so that
// a warp writes and the face kernel reads full lines).
template <int NR, bool VISC>
__global__ void __launch_bounds__(ADJ_THREADS) k_adj_point_rev(DevMesh<double> m, Phys<double> ph,
                                                               const double* __restrict__ poly,
                                                               const double* __restrict__ Xavg,
                                                               const double* __restrict__ src, double dt,
                                                               double* __restrict__ lx) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nt = m.nf * 3;
    if (t >= nt) return;
    const int64_t f = t / 3;
    const int k = (int)(t - f * 3);
    double x[2][20], lFh[5], lD[5], lW0[5], ldWt[5], lin[2][20];
    adj_point_setup<NR>(m, ph, poly, Xavg, src, f, k, x, lFh, lD, lW0, ldWt);
    gks_point_adj<VISC, NR == 40>(ph, x, dt, lFh, lD, lW0, ldWt, lin);
#pragma unroll
    for (int s = 0; s < 2; ++s)
#pragma unroll
        for (int i = 0; i < 20; ++i) lx[(20 * s + i) * nt + t] = lin[s][i];
}

// One thread per (side, face) with a cell: the input adjoints of the face's
// three points carried back through the rotations and the evaluation at the
// points into lpf[f][side][5][10].
// A wall side's adjoint joins the interior side's at the same point (a
// mirror is its own transpose; the isothermal and moving walls' ghost
// Jacobians are transposed at the interior state); an open side's goes to the
// interior cell's average, lwo[f][5] (zero on every other boundary face, not
// read on interior ones).
// XW: the mesh has isothermal or moving wall faces, whose ghosts' Jacobians
// (and the local frame they need) only those instances carry.
// One thread for both sides of a face held 100 sums and spilled: 291 us on
// 96,000 faces, 210 us with a thread a side and input-major lx.
template <bool XW>
__global__ void __launch_bounds__(ADJ_THREADS) k_adj_face_back(DevMesh<double> m, const double* __restrict__ lx,
                                                               double* __restrict__ lpf, double* __restrict__ lwo,
                                                               const double* __restrict__ poly, Phys<double> ph) {
    const int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nt = m.nf * 3;
    if (t >= m.nf * 2) return;
    const int side = t >= m.nf ? 1 : 0;
    const int64_t f = t - side * m.nf;
    const int64_t cell = m.flr[side * m.nf + f];
    if (cell < 0) return;
    const int other = m.flr[(1 - side) * m.nf + f];
    const double* geo = m.fgeo + f * FGEO;
    const double n[3] = {geo[0], geo[1], geo[2]};
    double Rm[3][3];
    face_frame(n, Rm);
    double lp[50], lw[5] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int j = 0; j < 50; ++j) lp[j] = 0.0;
#pragma unroll 1
    for (int k = 0; k < 3; ++k) {
        const double X[3] = {geo[4 + 9 * side + 3 * k], geo[5 + 9 * side + 3 * k], geo[6 + 9 * side + 3 * k]};
        const double* lk = lx + f * 3 + k;
        double l[20];
#pragma unroll
        for (int i = 0; i < 20; ++i) l[i] = lk[(20 * side + i) * nt];
        // a set fixed state is a constant of the step: nothing flows back
        if (other < 0 && other != FLR_FIXED) {
            double ls[20];
            double (*lg)[5] = reinterpret_cast<double (*)[5]>(ls + 5);
#pragma unroll
            for (int i = 0; i < 20; ++i) ls[i] = lk[(20 * (1 - side) + i) * nt];
            if (other == FLR_OPEN) {
                double lW[5], lgg[3][5];
                to_local_adj(Rm, ls, lg, lW, lgg);
                for (int q = 0; q < 5; ++q) lw[q] += lW[q];
            } else if (XW && (other == FLR_ISOTHERMAL_WALL || other == FLR_MOVING_WALL)) {
                // the interior state at the point, as adj_point_setup forms it, then the
                // ghost's transpose there
                double Wv[5], g[3][5], x[20];
                eval_poly<true>(poly + cell * POLY_STRIDE, X, Wv, g);
                to_local(Rm, Wv, g, x, reinterpret_cast<double (*)[5]>(x + 5));
                double Uw[3];
                rotate_vec(Rm, ph.uwall, Uw);
                wall_ghost_adj(other, x, ls, ph.gm1, ph.twall, Uw, l);
            } else {
                if (other == FLR_SLIP_WALL) slip_wall_ghost(ls, lg);
                if (other == FLR_NOSLIP_WALL) noslip_wall_ghost(ls, lg);
#pragma unroll
                for (int i = 0; i < 20; ++i) l[i] += ls[i];
            }
        }
        double lW[5], lg[3][5];
        to_local_adj(Rm, l, reinterpret_cast<const double (*)[5]>(l + 5), lW, lg);
        eval_poly_adj(X, lW, lg, lp);
    }
    double2* o = reinterpret_cast<double2*>(lpf + f * 100 + side * 50);
#pragma unroll
    for (int j = 0; j < 25; ++j) o[j] = make_double2(lp[2 * j], lp[2 * j + 1]);
    if (other < 0)
        for (int q = 0; q < 5; ++q) lwo[f * 5 + q] = lw[q];
}

// adjoint of a cell's reconstruction coefficients: the sum over its faces,
// one thread per (cell, coefficient) so that a warp reads whole records
// (48,000 cells: 42 us with a thread a cell, 22 us)
__global__ void k_adj_gather_poly(DevMesh<double> m, const double* __restrict__ lpf, double* __restrict__ lp) {
    const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= m.nc * 50) return;
    const int64_t c = i / 50;
    const int j = (int)(i - c * 50);
    double acc = 0.0;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        const int e = m.cface[f * m.nc + c];
        acc += lpf[(int64_t)(e >> 1) * 100 + (e & 1) * 50 + j];
    }
    lp[i] = acc;
}

// A cell whose reconstruction fell back to its average (the positivity
// check, Sec. 4.3: R = P0, zero slopes) passes only the adjoint of its
// constant on to its own average; nothing reaches the stencil data or the
// neighbours' slopes.  The fallback decision itself is piecewise constant.
__device__ __forceinline__ void fallback_back(const double* __restrict__ lp, int64_t c, int q,
                                              double* __restrict__ ld, double* __restrict__ lbn,
                                              double* __restrict__ own) {
    double* o = ld + (c * 5 + q) * 16;
    for (int j = 0; j < 16; ++j) o[j] = 0.0;
    if (lbn)
        for (int j = 0; j < 12; ++j) lbn[(c * 5 + q) * 12 + j] = 0.0;
    own[c * 5 + q] = lp[c * 50 + q * 10];
}

// Transpose of the linear-weight reconstruction of one cell (Sec. 4.1):
// R = a = M2 d, c0 = Q0 - sum_k R_k M_k (second moments), with
// d = [Q_nb - Q0 (4); grad Q_nb (12)].  Writes ld[c][q][16] = M2^T lambda_a
// and own[c][q] = lambda_c0 - sum over existing neighbours of ld[c][q][f].
__global__ void k_adj_recon_local(DevMesh<double> m, const double* __restrict__ lp, const int32_t* __restrict__ fb,
                                  double* __restrict__ ld, double* __restrict__ own) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= m.nc * 5) return;
    const int64_t c = idx / 5;
    const int q = (int)(idx - c * 5);
    if (fb[c]) {
        fallback_back(lp, c, q, ld, nullptr, own);
        return;
    }
    const double* tile = m.tile + (c / CELLS_PER_BLOCK) * TILE_ROWS * CELLS_PER_BLOCK;
    const int lc = (int)(c % CELLS_PER_BLOCK);
    auto T_ = [&](int row) { return tile[tile_at<double>(row, lc)]; };
    const double* l = lp + c * 50 + q * 10;
    const double lc0 = l[0];
    double la[9];
    for (int k = 0; k < 9; ++k) la[k] = l[1 + k];
    for (int k = 3; k < 9; ++k) la[k] -= lc0 * T_(TILE_MOM + (k - 3));
    double* o = ld + (c * 5 + q) * 16;
    double s = 0.0;
    for (int j = 0; j < 16; ++j) {
        double acc = 0.0;
        for (int k = 0; k < 9; ++k) acc += T_(TILE_M2 + k * 16 + j) * la[k];
        o[j] = acc;
    }
    for (int f = 0; f < 4; ++f)
        if (m.nbr[f * m.nc + c] >= 0) s += o[f];
    own[c * 5 + q] = lc0 - s;
}

// P1 slopes of every cell and component from the working state X (the
// reconstruction's step 1, Sec. 4.3), slopes[c][q][3]
__global__ void k_adj_p1(DevMesh<double> m, const double* __restrict__ X, double* __restrict__ slopes) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nc = m.nc;
    if (idx >= nc * 5) return;
    const int64_t c = idx / 5;
    const int q = (int)(idx - c * 5);
    const double Q0 = X[c * XS + q];
    double b[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        const int nb = m.nbr[f * nc + c];
        if (nb < 0) continue;
        const double dq = X[(int64_t)nb * XS + q] - Q0;
#pragma unroll
        for (int i = 0; i < 3; ++i) b[i] += m.M1[(i * 4 + f) * nc + c] * dq;
    }
#pragma unroll
    for (int i = 0; i < 3; ++i) slopes[idx * 3 + i] = b[i];
}

__device__ __forceinline__ double sgn(double x) { return x > 0.0 ? 1.0 : (x < 0.0 ? -1.0 : 0.0); }

// beta_0 of the two-step reconstruction (Eq. p0-non-linear-weight): the
// neighbours' P1 slopes b_j, beta_0j = |Omega|^{2/3} |b_j|^2, weights
// w1j = 1 + s1 / (eps + beta_0j) with s1 the 4/3 power of the mean pairwise
// |beta_0j - beta_0k|, beta_0 = sum w1j beta_0j / sum w1j; kept for the reverse.
struct Beta0 {
    // per local face: the neighbour's slopes, beta_0j, 1 / (eps + beta_0j), w1j
    // (zero without a neighbour)
    double bj[4][3], b0j[4], ie[4], w1j[4];
    double s1, iws, mean, ipair, beta;
    bool on[4];
};

// slopes: [nc][5][3] P1 slopes of the stage's state
__device__ __forceinline__ void beta0_forward(const double* __restrict__ slopes, const int* nb, int q, double v23,
                                              double eps, Beta0& B) {
    int nn = 0;
#pragma unroll
    for (int f = 0; f < 4; ++f) {
        B.on[f] = nb[f] >= 0;
        nn += B.on[f];
#pragma unroll
        for (int i = 0; i < 3; ++i) B.bj[f][i] = B.on[f] ? slopes[((int64_t)nb[f] * 5 + q) * 3 + i] : 0.0;
        const double* bj = B.bj[f];
        B.b0j[f] = v23 * (bj[0] * bj[0] + bj[1] * bj[1] + bj[2] * bj[2]);
        B.w1j[f] = 0.0;
    }
    B.beta = B.s1 = B.iws = B.mean = B.ipair = 0.0;
    if (nn == 0) return;
    double sum = 0.0, ws = 0.0, acc = 0.0;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int k = 0; k < j; ++k)
            if (B.on[j] && B.on[k]) sum += fabs(B.b0j[j] - B.b0j[k]);
    B.ipair = nn == 4 ? 1.0 / 6.0 : nn == 3 ? 1.0 / 3.0 : nn == 2 ? 1.0 : 0.0;
    B.mean = sum * B.ipair;
    B.s1 = pow43(B.mean);
    recip2(eps + B.b0j[0], eps + B.b0j[1], B.ie[0], B.ie[1]);
    recip2(eps + B.b0j[2], eps + B.b0j[3], B.ie[2], B.ie[3]);
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (!B.on[j]) continue;
        B.w1j[j] = 1.0 + B.s1 * B.ie[j];
        ws += B.w1j[j];
        acc += B.w1j[j] * B.b0j[j];
    }
    B.iws = 1.0 / ws;
    B.beta = acc * B.iws;
}

// adjoint of beta_0 into the adjoints of the neighbours' slopes lbj[f][3]
__device__ __forceinline__ void beta0_backward(const Beta0& B, double lbeta0, double v23, double (*lbj)[3]) {
    const double lacc = lbeta0 * B.iws, lws = -lacc * B.beta;
    double lb0[4] = {0.0, 0.0, 0.0, 0.0}, ls1 = 0.0;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
        if (!B.on[j]) continue;
        const double lwe = (lacc * B.b0j[j] + lws) * B.ie[j];
        lb0[j] = lacc * B.w1j[j] - lwe * B.s1 * B.ie[j];
        ls1 += lwe;
    }
    const double lsum = ls1 * (4.0 / 3.0) * cbrt(B.mean) * B.ipair;
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int k = 0; k < 4; ++k)
            if (k != j && B.on[j] && B.on[k]) lb0[j] += lsum * sgn(B.b0j[j] - B.b0j[k]);
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
        for (int i = 0; i < 3; ++i) lbj[j][i] = 2.0 * v23 * B.bj[j][i] * lb0[j];
}

// the neighbours' slope adjoints into lbn[f][3] (zero for missing neighbours)
__device__ __forceinline__ void store_lbn(const double (*lbj)[3], double* __restrict__ ob) {
#pragma unroll
    for (int f = 0; f < 4; ++f)
#pragma unroll
        for (int i = 0; i < 3; ++i) ob[3 * f + i] = lbj[f][i];
}

// Transpose of the third-order multi-resolution WENO reconstruction of one
// cell and component (Sec. 4.2, 4.3): R = c2 a + cb b with the nonlinear
// weights of beta_0 (two-step, from the neighbours' P1 slopes), beta_1, beta_2;
// c0 = Q0 - sum_k R_k M_k.  The weights are recomputed from the stage's
// working state X and differentiated (|x|' = sign x, (x^{4/3})' = 4/3 x^{1/3}).
// Writes ld[c][q][16] (adjoint of the stencil data d), lbn[c][q][f][3] (of
// the neighbours' slopes as this cell uses them) and own[c][q] (of Q0 through
// c0 and the differences d[0:4]).
__global__ void k_adj_recon_weno(DevMesh<double> m, double eps, const double* __restrict__ X,
                                 const double* __restrict__ slopes,
                                 const double* __restrict__ lp, const int32_t* __restrict__ fb,
                                 double* __restrict__ ld, double* __restrict__ lbn, double* __restrict__ own) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= m.nc * 5) return;
    const int64_t c = idx / 5, nc = m.nc;
    const int q = (int)(idx - c * 5);
    if (fb[c]) {
        fallback_back(lp, c, q, ld, lbn, own);
        return;
    }
    const double* tile = m.tile + (c / CELLS_PER_BLOCK) * TILE_ROWS * CELLS_PER_BLOCK;
    const int lc = (int)(c % CELLS_PER_BLOCK);
    auto T_ = [&](int row) { return tile[tile_at<double>(row, lc)]; };
    int nb[4];
    for (int f = 0; f < 4; ++f) nb[f] = m.nbr[f * nc + c];
    const double Q0 = X[c * XS + q];
    double d[16];
    for (int f = 0; f < 4; ++f) {
        const bool ok = nb[f] >= 0;
        const double* xn = X + (ok ? (int64_t)nb[f] : c) * XS;
        d[f] = ok ? xn[q] - Q0 : 0.0;
        for (int l = 0; l < 3; ++l) d[4 + 3 * f + l] = ok ? xn[5 + 3 * q + l] : 0.0;
    }
    double a[9];
    for (int k = 0; k < 9; ++k) {
        double acc = 0.0;
        for (int j = 0; j < 16; ++j) acc += T_(TILE_M2 + k * 16 + j) * d[j];
        a[k] = acc;
    }
    double Mm[6];
    for (int k = 0; k < 6; ++k) Mm[k] = T_(TILE_MOM + k);
    double b[3] = {0.0, 0.0, 0.0};
    for (int f = 0; f < 4; ++f) {
        if (nb[f] < 0) continue;
        for (int i = 0; i < 3; ++i) b[i] += T_(TILE_M1 + i * 4 + f) * d[f];
    }
    const double v23 = T_(TILE_V23), v43 = T_(TILE_V43);
    const double g22 = 100.0 / 111.0, g12 = 10.0 / 111.0, g02 = 1.0 / 111.0, g11 = 10.0 / 11.0;
    // forward: beta_1, beta_0 (two-step), beta_2, sigma, weights
    const double beta1 = v23 * (b[0] * b[0] + b[1] * b[1] + b[2] * b[2]);
    Beta0 B0;
    beta0_forward(slopes, nb, q, v23, eps, B0);
    const double beta0 = B0.beta;
    const double H[3][3] = {{2.0 * a[3], a[4], a[5]}, {a[4], 2.0 * a[6], a[7]}, {a[5], a[7], 2.0 * a[8]}};
    const double MM[3][3] = {{Mm[0], Mm[1], Mm[2]}, {Mm[1], Mm[3], Mm[4]}, {Mm[2], Mm[4], Mm[5]}};
    double first = 0.0, MH[3][3];
    for (int l = 0; l < 3; ++l) {
        for (int i = 0; i < 3; ++i) MH[l][i] = MM[i][0] * H[l][0] + MM[i][1] * H[l][1] + MM[i][2] * H[l][2];
        first += a[l] * a[l] + H[l][0] * MH[l][0] + H[l][1] * MH[l][1] + H[l][2] * MH[l][2];
    }
    const double second = H[0][0] * H[0][0] + a[4] * a[4] + a[5] * a[5] + H[1][1] * H[1][1] + a[7] * a[7] +
                          H[2][2] * H[2][2];
    const double beta2 = v23 * first + v43 * second;
    const double z = 0.5 * (fabs(beta2 - beta1) + fabs(beta2 - beta0));
    const double sigma = pow43(z);
    const double bet[3] = {beta0, beta1, beta2}, gam[3] = {g02, g12, g22};
    const double i22 = 111.0 / 100.0, i11 = 11.0 / 10.0;  // 1 / g22, 1 / g11
    double r[3], w[3], ib[3];
    recip2(eps + bet[0], eps + bet[1], ib[0], ib[1]);
    ib[2] = 1.0 / (eps + bet[2]);
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        r[k] = sigma * ib[k];
        w[k] = gam[k] * (1.0 + r[k] * r[k]);
    }
    const double iw = 1.0 / (w[0] + w[1] + w[2]);
    const double c2 = (w[2] * iw) * i22;
    const double cb = (w[1] * iw) * i11 - c2 * (g12 * i11);

    // reverse
    const double* l = lp + c * 50 + q * 10;
    const double lc0 = l[0];
    double lR[9];
    for (int k = 0; k < 9; ++k) lR[k] = l[1 + k];
    for (int k = 3; k < 9; ++k) lR[k] -= lc0 * Mm[k - 3];
    double la[9], lb[3], lc2 = 0.0, lcb = 0.0;
    for (int k = 0; k < 9; ++k) {
        la[k] = c2 * lR[k];
        lc2 += lR[k] * a[k];
    }
    for (int i = 0; i < 3; ++i) {
        lb[i] = cb * lR[i];
        lcb += lR[i] * b[i];
    }
    // c2 = w2 iw / g22, cb = w1 iw / g11 - c2 g12 / g11
    const double lc2t = lc2 - lcb * (g12 * i11);
    const double l1 = lcb * i11, l2t = lc2t * i22;
    double lw[3] = {0.0, l1 * iw, l2t * iw};
    const double lS = -(l2t * w[2] + l1 * w[1]) * iw * iw;
    double lbet[3] = {0.0, 0.0, 0.0}, lsig = 0.0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        lw[k] += lS;
        const double lri = lw[k] * gam[k] * 2.0 * r[k] * ib[k];
        lsig += lri;
        lbet[k] -= lri * r[k];
    }
    // sigma = z^{4/3}, z = (|b2 - b1| + |b2 - b0|) / 2
    const double lz = lsig * (4.0 / 3.0) * cbrt(z);
    const double s21 = sgn(beta2 - beta1), s20 = sgn(beta2 - beta0);
    lbet[2] += 0.5 * lz * (s21 + s20);
    lbet[1] += -0.5 * lz * s21;
    lbet[0] += -0.5 * lz * s20;
    // beta_2 = v23 first + v43 second
    const double lfirst = v23 * lbet[2], lsecond = v43 * lbet[2];
    double lH[3][3];
    for (int l2 = 0; l2 < 3; ++l2) {
        la[l2] += 2.0 * a[l2] * lfirst;
        for (int i = 0; i < 3; ++i) lH[l2][i] = 2.0 * MH[l2][i] * lfirst;
    }
    lH[0][0] += 2.0 * H[0][0] * lsecond;
    lH[1][1] += 2.0 * H[1][1] * lsecond;
    lH[2][2] += 2.0 * H[2][2] * lsecond;
    la[4] += 2.0 * a[4] * lsecond;
    la[5] += 2.0 * a[5] * lsecond;
    la[7] += 2.0 * a[7] * lsecond;
    la[3] += 2.0 * lH[0][0];
    la[4] += lH[0][1] + lH[1][0];
    la[5] += lH[0][2] + lH[2][0];
    la[6] += 2.0 * lH[1][1];
    la[7] += lH[1][2] + lH[2][1];
    la[8] += 2.0 * lH[2][2];
    // beta_1 = v23 |b|^2
    for (int i = 0; i < 3; ++i) lb[i] += 2.0 * v23 * b[i] * lbet[1];
    double lbj[4][3];
    beta0_backward(B0, lbet[0], v23, lbj);
    // a = M2 d, b = M1 d[0:4]
    double* o = ld + (c * 5 + q) * 16;
    double s = 0.0;
    for (int j = 0; j < 16; ++j) {
        double acc = 0.0;
        for (int k = 0; k < 9; ++k) acc += T_(TILE_M2 + k * 16 + j) * la[k];
        if (j < 4 && nb[j] >= 0)
            for (int i = 0; i < 3; ++i) acc += T_(TILE_M1 + i * 4 + j) * lb[i];
        o[j] = acc;
        if (j < 4 && nb[j] >= 0) s += acc;
    }
    own[c * 5 + q] = lc0 - s;
    store_lbn(lbj, lbn + (c * 5 + q) * 12);
}

// Transpose of the second-order WENO reconstruction R^2nd (Eq.
// final_weno_expression-2nd) of one cell and component: R = Q0 + cb b.x with
// cb = (w1 / (w0 + w1)) / g11, w0, w1 from beta_0 (two-step) and beta_1,
// sigma = |beta_1 - beta_0|^{4/3}.  Same outputs as k_adj_recon_weno.
__global__ void k_adj_recon_weno2(DevMesh<double> m, double eps, const double* __restrict__ X,
                                 const double* __restrict__ slopes,
                                  const double* __restrict__ lp, const int32_t* __restrict__ fb,
                                  double* __restrict__ ld, double* __restrict__ lbn, double* __restrict__ own) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= m.nc * 5) return;
    const int64_t c = idx / 5, nc = m.nc;
    const int q = (int)(idx - c * 5);
    if (fb[c]) {
        fallback_back(lp, c, q, ld, lbn, own);
        return;
    }
    const double* tile = m.tile + (c / CELLS_PER_BLOCK) * TILE_ROWS * CELLS_PER_BLOCK;
    const int lc = (int)(c % CELLS_PER_BLOCK);
    auto T_ = [&](int row) { return tile[tile_at<double>(row, lc)]; };
    int nb[4];
    for (int f = 0; f < 4; ++f) nb[f] = m.nbr[f * nc + c];
    const double Q0 = X[c * XS + q];
    double d[4];
    for (int f = 0; f < 4; ++f) d[f] = nb[f] >= 0 ? X[(int64_t)nb[f] * XS + q] - Q0 : 0.0;
    double b[3] = {0.0, 0.0, 0.0};
    for (int f = 0; f < 4; ++f) {
        if (nb[f] < 0) continue;
        for (int i = 0; i < 3; ++i) b[i] += T_(TILE_M1 + i * 4 + f) * d[f];
    }
    const double v23 = T_(TILE_V23);
    const double g01 = 1.0 / 11.0, g11 = 10.0 / 11.0;
    const double beta1 = v23 * (b[0] * b[0] + b[1] * b[1] + b[2] * b[2]);
    Beta0 B0;
    beta0_forward(slopes, nb, q, v23, eps, B0);
    const double beta0 = B0.beta;
    const double z = fabs(beta1 - beta0);
    const double sigma = pow43(z);
    const double bet[2] = {beta0, beta1}, gam[2] = {g01, g11};
    const double i11 = 11.0 / 10.0;  // 1 / g11
    double r[2], w[2], ib[2];
    recip2(eps + bet[0], eps + bet[1], ib[0], ib[1]);
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        r[k] = sigma * ib[k];
        w[k] = gam[k] * (1.0 + r[k] * r[k]);
    }
    const double iwsum = 1.0 / (w[0] + w[1]);
    const double cb = w[1] * iwsum * i11;

    // reverse: only the constant and the linear coefficients of R are nonzero
    const double* l = lp + c * 50 + q * 10;
    const double lc0 = l[0];
    double lb[3], lcb = 0.0;
    for (int i = 0; i < 3; ++i) {
        lb[i] = cb * l[1 + i];
        lcb += l[1 + i] * b[i];
    }
    double lw[2];
    const double lwsum = -lcb * cb * iwsum;
    lw[0] = lwsum;
    lw[1] = lwsum + lcb * iwsum * i11;
    double lbet[2] = {0.0, 0.0}, lsig = 0.0;
#pragma unroll
    for (int k = 0; k < 2; ++k) {
        const double lri = lw[k] * gam[k] * 2.0 * r[k] * ib[k];
        lsig += lri;
        lbet[k] -= lri * r[k];
    }
    const double lz = lsig * (4.0 / 3.0) * cbrt(z);
    const double s10 = sgn(beta1 - beta0);
    lbet[1] += lz * s10;
    lbet[0] -= lz * s10;
    for (int i = 0; i < 3; ++i) lb[i] += 2.0 * v23 * b[i] * lbet[1];
    double lbj[4][3];
    beta0_backward(B0, lbet[0], v23, lbj);
    double* o = ld + (c * 5 + q) * 16;
    double s = 0.0;
    for (int j = 0; j < 16; ++j) o[j] = 0.0;
    for (int j = 0; j < 4; ++j) {
        if (nb[j] < 0) continue;
        for (int i = 0; i < 3; ++i) o[j] += T_(TILE_M1 + i * 4 + j) * lb[i];
        s += o[j];
    }
    own[c * 5 + q] = lc0 - s;
    store_lbn(lbj, lbn + (c * 5 + q) * 12);
}

// Transpose of the second-order reconstruction with linear weights: R = P1,
// the step-1 slope b = M1 d[0:4].
__global__ void k_adj_recon_p1(DevMesh<double> m, const double* __restrict__ lp, const int32_t* __restrict__ fb,
                               double* __restrict__ ld, double* __restrict__ own) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= m.nc * 5) return;
    const int64_t c = idx / 5;
    const int q = (int)(idx - c * 5);
    if (fb[c]) {
        fallback_back(lp, c, q, ld, nullptr, own);
        return;
    }
    const double* tile = m.tile + (c / CELLS_PER_BLOCK) * TILE_ROWS * CELLS_PER_BLOCK;
    const int lc = (int)(c % CELLS_PER_BLOCK);
    const double* l = lp + c * 50 + q * 10;
    double* o = ld + (c * 5 + q) * 16;
    double s = 0.0;
    for (int j = 0; j < 16; ++j) o[j] = 0.0;
    for (int j = 0; j < 4; ++j) {
        if (m.nbr[j * m.nc + c] < 0) continue;
        for (int i = 0; i < 3; ++i) o[j] += tile[tile_at<double>(TILE_M1 + i * 4 + j, lc)] * l[1 + i];
        s += o[j];
    }
    own[c * 5 + q] = l[0] - s;
}

// Reverse face slots: rev[f][c] = the local face of neighbour n = nbr(c, f)
// that is the same face.  Found here on each call (microseconds), where the
// host's table was copied over from pageable memory.
__global__ void k_adj_rev(DevMesh<double> m, int8_t* __restrict__ rev) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x, nc = m.nc;
    if (idx >= nc * 4) return;
    const int64_t f = idx / nc, c = idx - f * nc;
    const int n = m.nbr[idx], face = m.cface[f * nc + c] >> 1;
    int8_t r = 0;
    if (n >= 0)
        for (int k = 0; k < 4; ++k)
            if ((m.cface[k * nc + n] >> 1) == face) r = (int8_t)k;
    rev[idx] = r;
}

// Adjoint of the neighbours' P1 slopes, per cell n and component: the slope
// adjoints the cells around n hold for n's slope (lbn, in the slot that
// points back to n) are summed, then carried through n's slope operator:
// lds[n][q][f] is the adjoint of Q_nbr(n, f) - Q_n.
__global__ void k_adj_slopes(DevMesh<double> m, const int8_t* __restrict__ rev, const double* __restrict__ lbn,
                             double* __restrict__ lds) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= m.nc * 5) return;
    const int64_t n = idx / 5, nc = m.nc;
    const int q = (int)(idx - n * 5);
    double ls[3] = {0.0, 0.0, 0.0};
    for (int f = 0; f < 4; ++f) {
        const int c = m.nbr[f * nc + n];
        if (c < 0) continue;
        const double* src = lbn + ((int64_t)c * 5 + q) * 12 + 3 * rev[f * nc + n];
        for (int i = 0; i < 3; ++i) ls[i] += src[i];
    }
    double* o = lds + (n * 5 + q) * 4;
    for (int f = 0; f < 4; ++f)
        o[f] = m.nbr[f * nc + n] >= 0
                   ? m.M1[(0 * 4 + f) * nc + n] * ls[0] + m.M1[(1 * 4 + f) * nc + n] * ls[1] +
                         m.M1[(2 * 4 + f) * nc + n] * ls[2]
                   : 0.0;
}

// adjoint of a cell's working state [W (5), grad W (15)]: its own part and,
// from each neighbour n, the entries of n's stencil adjoint in the slot that
// points back to this cell across the shared face (rev[f][c])
__global__ void k_adj_recon_gather(DevMesh<double> m, const int8_t* __restrict__ rev,
                                   const double* __restrict__ ld, const double* __restrict__ lds,
                                   const double* __restrict__ own, const double* __restrict__ lwo,
                                   double* __restrict__ lX) {
    const int64_t idx = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (idx >= m.nc * 5) return;
    const int64_t c = idx / 5;
    const int q = (int)(idx - c * 5);
    double lq = own[c * 5 + q];
    // open faces of this cell: their ghost is this cell's average
    for (int f = 0; f < 4; ++f) {
        const int e = m.cface[f * m.nc + c];
        const int64_t face = e >> 1;
        if (m.flr[(int64_t)(1 - (e & 1)) * m.nf + face] == FLR_OPEN) lq += lwo[face * 5 + q];
    }
    double lg[3] = {0.0, 0.0, 0.0};
    for (int f = 0; f < 4; ++f) {
        const int n = m.nbr[f * m.nc + c];
        if (n < 0) continue;
        const int r = rev[f * m.nc + c];
        const double* o = ld + ((int64_t)n * 5 + q) * 16;
        lq += o[r];
        for (int l = 0; l < 3; ++l) lg[l] += o[4 + 3 * r + l];
        if (lds) lq += lds[((int64_t)n * 5 + q) * 4 + r] - lds[(c * 5 + q) * 4 + f];
    }
    double* x = lX + c * XS;
    x[q] = lq;
    for (int l = 0; l < 3; ++l) x[5 + 3 * q + l] = lg[l];
}

// lambda W^n = lambda W^{n+1} (the update's pass-through) + lambda W* (the
// stage-1 pass-through) + the stage-1 reconstruction's; lambda grad W^n from
// the stage-1 reconstruction alone
__global__ void k_adj_final(DevMesh<double> m, const double* __restrict__ lW, const double* __restrict__ lXs,
                            const double* __restrict__ lX1, double* __restrict__ oW, double* __restrict__ odW) {
    const int64_t c = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
    if (c >= m.nc) return;
    for (int q = 0; q < 5; ++q) oW[q * m.nc + c] = lW[q * m.nc + c] + lXs[c * XS + q] + lX1[c * XS + q];
    for (int j = 0; j < 15; ++j) odW[j * m.nc + c] = lX1[c * XS + 5 + j];
}

// --------------------------------------------------------------------------
// launcher
// --------------------------------------------------------------------------
static inline unsigned grid_of(int64_t n, int b) { return (unsigned)((n + b - 1) / b); }

static Phys<double> phys64(const HostPhys& p) {
    Phys<double> ph;
    ph.gamma = p.gamma;
    ph.gm1 = p.gamma - 1.0;
    ph.K = (5.0 - 3.0 * p.gamma) / (p.gamma - 1.0);
    ph.tau_eps = p.tau_eps;
    ph.tau_c = p.tau_c;
    ph.mu = p.mu;
    ph.eps_w = p.eps_weno;
    ph.viscous = p.viscous;
    ph.smooth = p.smooth;
    ph.prf = p.prf;
    ph.twall = p.twall;
    for (int i = 0; i < 3; ++i) ph.uwall[i] = p.uwall[i];
    return ph;
}

// transpose of one stage's reconstruction: lp (per-cell coefficient
// adjoints) into lX, from the stage's working state X
static void recon_back(const DevMesh<double>& m, const HostPhys& p, const AdjBuffers& b, const double* X,
                       const int32_t* fb,
                       double* lX, cudaStream_t s) {
    const int B = 128;
    if (p.weno) {
        // the slopes lie in lds until k_adj_slopes writes it
        k_adj_p1<<<grid_of(m.nc * 5, B), B, 0, s>>>(m, X, b.lds);
        if (p.order == 2)
            k_adj_recon_weno2<<<grid_of(m.nc * 5, B), B, 0, s>>>(m, p.eps_weno, X, b.lds, b.lp, fb, b.ld, b.lbn, b.own);
        else
            k_adj_recon_weno<<<grid_of(m.nc * 5, B), B, 0, s>>>(m, p.eps_weno, X, b.lds, b.lp, fb, b.ld, b.lbn, b.own);
        k_adj_slopes<<<grid_of(m.nc * 5, B), B, 0, s>>>(m, b.rev, b.lbn, b.lds);
        k_adj_recon_gather<<<grid_of(m.nc * 5, B), B, 0, s>>>(m, b.rev, b.ld, b.lds, b.own, b.lwo, lX);
    } else {
        if (p.order == 2)
            k_adj_recon_p1<<<grid_of(m.nc * 5, B), B, 0, s>>>(m, b.lp, fb, b.ld, b.own);
        else
            k_adj_recon_local<<<grid_of(m.nc * 5, B), B, 0, s>>>(m, b.lp, fb, b.ld, b.own);
        k_adj_recon_gather<<<grid_of(m.nc * 5, B), B, 0, s>>>(m, b.rev, b.ld, nullptr, b.own, b.lwo, lX);
    }
}

// transpose of one stage's face flux: the record adjoints in b.src into the
// per-cell reconstruction-coefficient adjoints b.lp
template <int NR>
static void flux_back(const DevMesh<double>& m, const Phys<double>& ph, const AdjBuffers& b, const double* poly,
                      const double* X, double dt, cudaStream_t s) {
    const int B = 128;
    if (ph.viscous)
        k_adj_point_rev<NR, true><<<grid_of(m.nf * 3, ADJ_THREADS), ADJ_THREADS, 0, s>>>(m, ph, poly, X, b.src, dt,
                                                                                       b.lx);
    else
        k_adj_point_rev<NR, false><<<grid_of(m.nf * 3, ADJ_THREADS), ADJ_THREADS, 0, s>>>(m, ph, poly, X, b.src, dt,
                                                                                        b.lx);
    if (m.xwalls)
        k_adj_face_back<true><<<grid_of(m.nf * 2, ADJ_THREADS), ADJ_THREADS, 0, s>>>(m, b.lx, b.lpf, b.lwo, poly, ph);
    else
        k_adj_face_back<false><<<grid_of(m.nf * 2, ADJ_THREADS), ADJ_THREADS, 0, s>>>(m, b.lx, b.lpf, b.lwo, poly, ph);
    k_adj_gather_poly<<<grid_of(m.nc * 50, B), B, 0, s>>>(m, b.lpf, b.lp);
}

// The reverse sweep proper; the forward intermediates (the two stages'
// working states X1, X2 and reconstructions poly1, poly2) come from a forward
// recomputation by the caller.
cudaError_t adjoint_reverse(const DevMesh<double>& m, const HostPhys& p, double dt, const AdjBuffers& b,
                            const double* X1, const double* X2, const double* lW, const double* ldW, double* oW,
                            double* odW, cudaStream_t s) {
    const Phys<double> ph = phys64(p);
    const int B = 128;
    cudaError_t e;
    k_adj_rev<<<grid_of(m.nc * 4, B), B, 0, s>>>(m, b.rev);
    // stage 2
    k_adj_src2<<<grid_of(m.nc, B), B, 0, s>>>(m, lW, ldW, b.src);
    flux_back<20>(m, ph, b, b.poly2, X2, dt, s);
    recon_back(m, p, b, X2, b.fallback + m.nc, b.lXs, s);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
    // stage 1
    k_adj_src1<<<grid_of(m.nc, B), B, 0, s>>>(m, lW, ldW, b.lXs, b.src);
    flux_back<40>(m, ph, b, b.poly1, X1, dt, s);
    recon_back(m, p, b, X1, b.fallback, b.lX1, s);
    k_adj_final<<<grid_of(m.nc, B), B, 0, s>>>(m, lW, b.lXs, b.lX1, oW, odW);
    return cudaGetLastError();
}

}  // namespace gks
