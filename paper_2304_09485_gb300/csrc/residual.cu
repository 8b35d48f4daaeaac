// Residual R(U) of the implicit HGKS (paper Eq. (finite), Sec. 4.1), FP64.
//
// Four kernels per evaluation, all on the caller's stream:
//  1. k_coef    one thread per (cell, conservative component): polynomial
//               coefficients of Eq. (polys) = per-cell fit matrix x stencil data
//               (non-compact: Q_k - Q_i over the big stencil; compact: Q_k - Q_i
//               of the face neighbours and the cell-averaged gradients).
//  2. k_recon   one thread per (cell, local face): characteristic projection at
//               Q* (Sec. 5), smoothness indicators and nonlinear weights of
//               Eq. (weno), values and directional derivatives at the face's 3
//               Gauss points, written in characteristic variables.
//  3. k_flux    one thread per (face, Gauss point): back-projection with the
//               face's R* (shared by both sides), positivity fallback, boundary
//               state, the BGK flux of Eq. (flux) averaged over [0, dt] and, for
//               the compact scheme, the point value of Eq. (point).
//  4. k_gather  one thread per cell: R_i = -sum of its faces' fluxes (signed),
//               compact G_new_i = sum of point values * n * S / |Omega_i|
//               (Eq. (derivative)). Gather, not scatter: no atomics, and the
//               summation order is fixed (deterministic results).
// Arrays are component-major with the cell or face index fastest, so
// consecutive threads touch consecutive addresses.
#include <algorithm>
#include <cmath>
#include "hgks_internal.h"
#include "fp64.cuh"

namespace hgks {

thread_local int64_t g_launches = 0;

namespace {

constexpr int kBlock = 128;

// primitive state of a Maxwellian: il = p / rho (its variance), ir = 1 / rho
struct Prim { double rho, U, V, W, il, ir; };

// rho p of a conservative state, without a division
__device__ __forceinline__ double rho_p(const Units &u, const double *Q, double g1) {
  return u.mul(g1, fma(Q[4], Q[0], u.mul(-0.5, fma(Q[1], Q[1], fma(Q[2], Q[2], u.mul(Q[3], Q[3]))))));
}
// from Q and rp = rho p
__device__ __forceinline__ Prim to_prim(const Units &u, const double *Q, double rp) {
  Prim p;
  p.rho = Q[0];
  p.ir = rcp(Q[0], u.one);
  p.U = u.mul(Q[1], p.ir); p.V = u.mul(Q[2], p.ir); p.W = u.mul(Q[3], p.ir);
  p.il = u.mul(u.mul(rp, p.ir), p.ir);
  return p;
}

// rotate momentum into the face frame (rows of T: n, t1, t2) and back
__device__ __forceinline__ void rot_in(const Units &u, const double *T, const double *in, double *out) {
  out[0] = in[0]; out[4] = in[4];
#pragma unroll
  for (int r = 0; r < 3; r++) out[1 + r] = fma(T[3 * r], in[1], fma(T[3 * r + 1], in[2], u.mul(T[3 * r + 2], in[3])));
}
__device__ __forceinline__ void rot_out(const Units &u, const double *T, const double *in, double *out) {
  out[0] = in[0]; out[4] = in[4];
#pragma unroll
  for (int d = 0; d < 3; d++) out[1 + d] = fma(T[d], in[1], fma(T[3 + d], in[2], u.mul(T[6 + d], in[3])));
}

// Euler eigen-system along x of a face-frame state: scalars of which R (right_apply)
// and R^{-1} (k_recon's projection) are made.
struct Eig { double u, v, w, a, H, q2, ia; };
__device__ __forceinline__ Eig eig_of(const Units &u, const double *Q, double gamma, double g1) {
  Eig e;
  const double ir = rcp(Q[0], u.one);
  e.u = u.mul(Q[1], ir); e.v = u.mul(Q[2], ir); e.w = u.mul(Q[3], ir);
  e.q2 = fma(e.u, e.u, fma(e.v, e.v, u.mul(e.w, e.w)));
  const double p = u.mul(g1, fma(u.mul(-0.5, Q[0]), e.q2, Q[4]));
  const double a2 = u.mul(u.mul(gamma, p), ir);
  e.ia = rsqrt64(a2);
  e.a = u.mul(a2, e.ia);
  e.H = u.mul(u.add(Q[4], p), ir);
  return e;
}
// out = R q (characteristic -> conservative, face frame)
__device__ __forceinline__ void right_apply(const Units &u, const Eig &e, const double *q, double *out) {
  const double t = u.add(q[0], q[4]), s = u.add(t, q[1]), ad = u.mul(e.a, u.sub(q[4], q[0]));
  out[0] = s;
  out[1] = fma(e.u, s, ad);
  out[2] = fma(e.v, s, q[2]);
  out[3] = fma(e.w, s, q[3]);
  out[4] = fma(e.H, t, fma(e.u, ad, fma(u.mul(0.5, e.q2), q[1], fma(e.v, q[2], u.mul(e.w, q[3])))));
}

// ------------------------------------------------------------------------
// 1. polynomial coefficients
// ------------------------------------------------------------------------
// a real cell of a batch whose mesh still iterates (padding cells have mesh -1)
__device__ __forceinline__ bool live(const DevMesh &m, int i) {
  const int k = m.cmesh[i];
  return k >= 0 && m.mact[k];
}

// One thread per (component, cell): P0's 9 coefficients over the big stencil, then
// the four sub-stencils' 3 each over their six cells, whose differences the thread
// keeps in shared memory (its own column) from the first pass.
template <bool BATCH, class S>
__global__ void __launch_bounds__(kBlock) k_coef_weno(DevMesh m, const double *__restrict__ Q, double *__restrict__ coef) {
  constexpr int BIG = S::BIG, SUBK = S::SUBK;
  constexpr unsigned SLOTMASK = (1u << S::SLOTBITS) - 1u;
  __shared__ double sdq[BIG][kBlock];
  const int N = m.N;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int NL = BATCH ? m.NL : N;
  if (t >= 5 * NL) return;
  const int c = t / NL, i = t - c * NL;
  if (BATCH && !live(m, i)) return;
  const Units u = units();
  const double qi = Q[(size_t)c * N + i];
  double a[9];
#pragma unroll
  for (int d = 0; d < 9; d++) a[d] = 0.0;
#pragma unroll
  for (int k = 0; k < BIG; k++) {
    int j = m.sten[(size_t)k * N + i];
    if (j < 0) break;
    const double dq = u.sub(Q[(size_t)c * N + j], qi);
    sdq[k][threadIdx.x] = dq;
#pragma unroll
    for (int d = 0; d < 9; d++) a[d] = fma(m.X0[(size_t)(d * BIG + k) * N + i], dq, a[d]);
  }
#pragma unroll
  for (int d = 0; d < 9; d++) coef[(size_t)(d * 5 + c) * N + i] = a[d];
#pragma unroll
  for (int mm = 0; mm < S::NSUBW; mm++) {
    const unsigned sl = m.ssl[(size_t)mm * N + i];
    double b[3] = {0.0, 0.0, 0.0};
#pragma unroll
    for (int s = 0; s < SUBK; s++) {
      const double dq = sdq[(sl >> (S::SLOTBITS * s)) & SLOTMASK][threadIdx.x];
#pragma unroll
      for (int j = 0; j < 3; j++) b[j] = fma(m.Xs[(size_t)((mm * 3 + j) * SUBK + s) * N + i], dq, b[j]);
    }
#pragma unroll
    for (int j = 0; j < 3; j++) coef[(size_t)(kCoefA + (mm * 3 + j) * 5 + c) * N + i] = b[j];
  }
}

template <bool BATCH, class S>
__global__ void __launch_bounds__(kBlock) k_coef_hweno(DevMesh m, const double *__restrict__ Q, const double *__restrict__ G,
                                                        double *__restrict__ coef) {
  constexpr int NF = S::NF, HC = ShapeOf<S>::HCOLS;
  const int N = m.N;
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  const int NL = BATCH ? m.NL : N;
  if (t >= 5 * NL) return;
  const int c = t / NL, i = t - c * NL;
  if (BATCH && !live(m, i)) return;
  const double qi = Q[(size_t)c * N + i];
  double data[HC];
  int nb[NF];
#pragma unroll
  for (int p = 0; p < NF; p++) {
    nb[p] = m.cnb[(size_t)p * N + i];
    data[p] = nb[p] >= 0 ? Q[(size_t)c * N + nb[p]] - qi : 0.0;
  }
#pragma unroll
  for (int j = 0; j < 3; j++) data[NF + j] = G[(size_t)(3 * c + j) * N + i];
#pragma unroll
  for (int p = 0; p < NF; p++)
#pragma unroll
    for (int j = 0; j < 3; j++) data[NF + 3 + 3 * p + j] = nb[p] >= 0 ? G[(size_t)(3 * c + j) * N + nb[p]] : 0.0;
#pragma unroll
  for (int d = 0; d < 9; d++) {
    double s = 0.0;
#pragma unroll
    for (int col = 0; col < HC; col++) s = fma(m.H0[(size_t)(d * HC + col) * N + i], data[col], s);
    coef[(size_t)(d * 5 + c) * N + i] = s;
  }
#pragma unroll
  for (int mm = 0; mm < NF; mm++) {
    double dm[7] = {data[mm], data[NF], data[NF + 1], data[NF + 2], data[NF + 3 + 3 * mm], data[NF + 4 + 3 * mm],
                    data[NF + 5 + 3 * mm]};
#pragma unroll
    for (int j = 0; j < 3; j++) {
      double s = 0.0;
#pragma unroll
      for (int col = 0; col < 7; col++) s = fma(m.Hm[(size_t)((mm * 3 + j) * 7 + col) * N + i], dm[col], s);
      coef[(size_t)(kCoefA + (mm * 3 + j) * 5 + c) * N + i] = s;
    }
  }
}

// ------------------------------------------------------------------------
// 2. reconstruction at the Gauss points of one face, one side
// ------------------------------------------------------------------------
// Bound by the FP64 pipe (2 DFMA per SM and clock); all choices below save FP64 work.
// The thread first projects its cell's coefficients (9 of P0, 3 of every P_m) and average
// into characteristic variables, each vector once, and keeps them in its own column of
// shared memory; the loop over the five variables then works from there. R^{-1} q of a
// conservative vector q = (q0, m, q4) about the projection state (u, sound speed a):
//   P = (gamma - 1) / (2 a^2) (|u|^2/2 q0 - u . m + q4),   D = (n . m - u_n q0) / (2 a),
//   (P - D, q0 - 2 P, t1 . m - u_t1 q0, t2 . m - u_t2 q0, P + D): 20 operations against 25
// for five dense rows. The nonlinear weights take one division: with d_k = beta_k + eps,
// D = prod d_k, R_k = D / d_k (prefix and suffix products) and sum of the linear weights 1,
//   kap_0 = (D + tz R_0) / den,  kap_m = gm tz (R_m - R_0) / den,
//   den = D + tz (g0 R_0 + gm sum R_m).
// The projection stays in shared memory for three variables at a time, (P - D, q0 - 2 P, P + D),
// then the two shear waves: 66 doubles a thread on tetrahedra (three blocks of 128 threads an SM),
// 102 on hexahedra, 84 with the compact scheme (two; all five variables at once, 170, left four warps
// an SM and cost 12 %).
// Registers to match: 168 for 12 warps an SM, 255 for 8 (hexahedra with 168 spilled 348 bytes a
// thread: 0.843 -> 0.825 ms for 35,937, 4.07 -> 4.00 for 190,464).
// Against dense rows per variable: 28.5 -> 22.8 ms for 9.4M (cell, face) pairs (2,359,296
// tetrahedra), 1.24 -> 0.83 ms for 35,937 hexahedra (0.72 with the compact scheme's six). ncu at 648,000 tetrahedra: 1,466 FP64 instructions a
// thread, the pipe 97 % busy.
// NSUB: the scheme's sub-polynomials, one per sub-stencil or (compact) per face: on hexahedra k_coef
// writes six vectors of three for the compact scheme and eight for the other, and no more are read.
constexpr int kReconMax = 256, kReconHex = 128;
constexpr int recon_rows(int nsub) { return 3 * (10 + 3 * nsub); }
template <bool BATCH, class S, int NSUB>
__global__ void __launch_bounds__(S::NF == 4 ? 384 : 256) k_recon(DevMesh m, KParams Pv, const double *__restrict__ Q,
                                                                           const double *__restrict__ coef, double *__restrict__ wface) {
  constexpr int NF = S::NF, NG = S::NG, NV = 9 + 3 * NSUB;
  extern __shared__ double proj[];                      // [3][NV + 1][blockDim.x]: column of this thread
  const int N = m.N, F = m.F;
  const int NL = BATCH ? m.NL : N;
  // block b covers local face (b mod NF) of cell range b / NF: the blocks of a
  // range run together and read its coefficients from L2 after the first
  const int slot = blockIdx.x % NF, i = (blockIdx.x / NF) * blockDim.x + threadIdx.x;
  if (i >= NL) return;
  if (BATCH && !live(m, i)) return;                     // padding cell, or a mesh that has stopped
  const KParams &P = BATCH ? m.ptab[m.cmesh[i]] : Pv;
  const int cf = m.cface[(size_t)slot * N + i];
  const int f = cf >> 1, side = cf & 1;
  const int bd = blockDim.x;
  double *my = proj + threadIdx.x;
  const Units u = units();
  const size_t rs = (size_t)(NV + 1) * bd;              // from one kept variable to the next
  double T[9];
#pragma unroll
  for (int k = 0; k < 9; k++) T[k] = m.fT[(size_t)k * F + f];
  Eig e;
  {
    const int L = m.fl[f], R = m.fr[f];
    double Qs[5], Qsl[5];
#pragma unroll
    for (int c = 0; c < 5; c++)                          // twice Q*: only ratios are taken
      Qs[c] = R >= 0 ? u.add(Q[(size_t)c * N + L], Q[(size_t)c * N + R]) : Q[(size_t)c * N + i];
    rot_in(u, T, Qs, Qsl);
    e = eig_of(u, Qsl, P.gamma, P.g1);
  }
  // component k of vector d: a coefficient, or (d = NV) the cell average
  auto in = [&](int d, int k) { return d < NV ? coef[(size_t)(d * 5 + k) * N + i] : Q[(size_t)k * N + i]; };
  auto project = [&](int pass) {
    if (!P.characteristic) {                            // conservative variables: the coefficients themselves
#pragma unroll 1
      for (int d = 0; d <= NV; d++) {
        my[d * bd] = in(d, pass == 0 ? 0 : 2);
        my[rs + d * bd] = in(d, pass == 0 ? 1 : 3);
        if (pass == 0) my[2 * rs + d * bd] = in(d, 4);
      }
    } else if (pass == 0) {
      const double hb = u.mul(0.5 * P.g1, u.mul(e.ia, e.ia)), hi = u.mul(0.5, e.ia);
      const double minus2 = u.add(-1.0, -u.one);
      double pm[3], dm[3];                              // P = p0 q0 + pm . m + hb q4, D = d0 q0 + dm . m
      const double p0 = u.mul(u.mul(0.5, hb), e.q2), d0 = u.mul(-hi, e.u);
#pragma unroll
      for (int k = 0; k < 3; k++) {
        pm[k] = u.mul(-hb, fma(T[k], e.u, fma(T[3 + k], e.v, u.mul(T[6 + k], e.w))));
        dm[k] = u.mul(hi, T[k]);
      }
#pragma unroll
      for (int d = 0; d <= NV; d++) {
        const double q0 = in(d, 0), q1 = in(d, 1), q2 = in(d, 2), q3 = in(d, 3), q4 = in(d, 4);
        const double Pq = fma(p0, q0, fma(pm[0], q1, fma(pm[1], q2, fma(pm[2], q3, u.mul(hb, q4)))));
        const double Dq = fma(d0, q0, fma(dm[0], q1, fma(dm[1], q2, u.mul(dm[2], q3))));
        const double lo = u.sub(Pq, Dq), hi4 = u.add(Pq, Dq);
        my[d * bd] = lo;
        my[rs + d * bd] = fma(minus2, Pq, q0);
        my[2 * rs + d * bd] = hi4;
      }
    } else {
      double t[6];                                      // the tangents (T is scaled by now)
#pragma unroll
      for (int k = 0; k < 6; k++) t[k] = m.fT[(size_t)(3 + k) * F + f];
#pragma unroll
      for (int d = 0; d <= NV; d++) {
        const double q0 = in(d, 0), q1 = in(d, 1), q2 = in(d, 2), q3 = in(d, 3);
        my[d * bd] = fma(-e.v, q0, fma(t[0], q1, fma(t[1], q2, u.mul(t[2], q3))));
        my[rs + d * bd] = fma(-e.w, q0, fma(t[3], q1, fma(t[4], q2, u.mul(t[5], q3))));
      }
    }
  };
  const double ih = rcp(m.h[i], u.one), eps = u.add(P.weno_eps, u.nz);   // eps: in a register
  double m2[6], xg[3 * NG];
#pragma unroll
  for (int k = 0; k < 6; k++) m2[k] = m.m2[(size_t)k * N + i];
  // beta_0 = |a|^2 + tr(M2 H^2) + sum of squared second derivatives as a quadratic form of
  // the coefficients (xx, yy, zz, xy, xz, yz), H_xx = 2 a_xx: weights of the squares, and of
  // the products by m_xy, m_xz, m_yz without (c) and with (f) a factor from a diagonal entry
  const double w0 = fma(4.0, m2[0], 4.0), w1 = fma(4.0, m2[1], 4.0), w2 = fma(4.0, m2[2], 4.0);
  const double w3 = m2[0] + m2[1] + 1.0, w4 = m2[0] + m2[2] + 1.0, w5 = m2[1] + m2[2] + 1.0;
  const double c3 = 2.0 * m2[3], c4 = 2.0 * m2[4], c5 = 2.0 * m2[5], f3 = 2.0 * c3, f4 = 2.0 * c4, f5 = 2.0 * c5;
#pragma unroll
  for (int k = 0; k < 3 * NG; k++) xg[k] = m.xg[(size_t)(slot * 3 * NG + k) * N + i];
  // weights of the sub-stencils (compact: one per face)
  const unsigned valid = P.scheme == HGKS_WENO ? m.subvalid[i] : (1u << NF) - 1u;
  const int M = __popc(valid);
  const double gm = P.lin_weight, g0 = M ? 1.0 - gm * M : 1.0;
  const double iM = M ? rcp((double)M) : 0.0;
  project(0);
#pragma unroll
  for (int k = 0; k < 9; k++) T[k] = u.mul(T[k], ih);               // face frame rows / h: scaled derivatives
  double *out = wface + (size_t)side * NG * kFaceState * F + f;
#pragma unroll 1
  for (int v = 0; v < 5; v++) {                          // variables 0, 1, 4, then 2, 3
    if (v == 3) project(1);
    const int c = v < 2 ? v : v == 2 ? 4 : v - 1;
    const double *pc = my + (v < 3 ? v : v - 3) * rs;
    double ac[9];
#pragma unroll
    for (int d = 0; d < 9; d++) ac[d] = pc[d * bd];
    const double q0 = pc[NV * bd];
    // combined polynomial: Q = kap0 P0 + sum kap_m P_m (kap0 + sum kap_m = 1)
    double kap0 = 1.0, lin[3];
    if (P.weights == HGKS_LINEAR || M == 0) {
#pragma unroll
      for (int j = 0; j < 3; j++) lin[j] = ac[j];
    } else {
      // smoothness indicators in the scaled frame (beta_0 = avg |grad P0|^2 + sum of squared
      // second derivatives), each with weno_eps added
      const double xx = ac[3], yy = ac[4], zz = ac[5], xy = ac[6], xz = ac[7], yz = ac[8];
      double d0 = fma(ac[0], ac[0], fma(ac[1], ac[1], fma(ac[2], ac[2], eps)));
      d0 = fma(xx, fma(w0, xx, fma(f3, xy, u.mul(f4, xz))), d0);
      d0 = fma(xy, fma(w3, xy, fma(f3, yy, fma(c4, yz, u.mul(c5, xz)))), d0);
      d0 = fma(xz, fma(w4, xz, fma(f4, zz, u.mul(c3, yz))), d0);
      d0 = fma(yy, fma(w1, yy, u.mul(f5, yz)), d0);
      d0 = fma(yz, fma(w5, yz, u.mul(f5, zz)), d0);
      d0 = fma(zz, u.mul(w2, zz), d0);
      double dm[NSUB], tz = 0.0;
#pragma unroll
      for (int mm = 0; mm < NSUB; mm++) {
        const double b0 = pc[(9 + 3 * mm) * bd], b1 = pc[(10 + 3 * mm) * bd], b2 = pc[(11 + 3 * mm) * bd];
        const double de = fma(b0, b0, fma(b1, b1, fma(b2, b2, eps)));
        if (valid >> mm & 1) tz = u.add(fabs(u.sub(d0, de)), tz);
        dm[mm] = (valid >> mm & 1) ? de : 1.0;
      }
      tz = u.mul(tz, iM);
      double R[NSUB], pre = d0, R0 = 1.0, sum = 0.0;
#pragma unroll
      for (int mm = 0; mm < NSUB; mm++) {               // R[mm] = d0 dm[0] ... dm[mm - 1]
        R[mm] = pre;
        pre = u.mul(pre, dm[mm]);
      }
#pragma unroll
      for (int mm = NSUB - 1; mm >= 0; mm--) {          // times dm[mm + 1] ... dm[NSUB - 1]
        if (mm < NSUB - 1) R[mm] = u.mul(R[mm], R0);
        R0 = mm < NSUB - 1 ? u.mul(R0, dm[mm]) : dm[mm];
        if (valid >> mm & 1) sum = u.add(sum, R[mm]);
      }
      const double inv = rcp(fma(tz, fma(g0, R0, u.mul(gm, sum)), pre), u.one), h = u.mul(u.mul(gm, tz), inv);
      kap0 = u.mul(inv, fma(tz, R0, pre));
#pragma unroll
      for (int j = 0; j < 3; j++) lin[j] = u.mul(kap0, ac[j]);
#pragma unroll
      for (int mm = 0; mm < NSUB; mm++) {
        const double k = (valid >> mm & 1) ? u.mul(h, u.sub(R[mm], R0)) : 0.0;
#pragma unroll
        for (int j = 0; j < 3; j++) lin[j] = fma(k, pc[(9 + 3 * mm + j) * bd], lin[j]);
      }
    }
    double qd[6];
#pragma unroll
    for (int k = 0; k < 6; k++) qd[k] = u.mul(kap0, ac[3 + k]);
    // P(x) = q0 + lin . x + sum_k qd_k (mono_k(x) - m2_k), nested so that the value
    // and the gradient share their partial sums
    double q0m = q0;
#pragma unroll
    for (int k = 0; k < 6; k++) q0m = fma(-qd[k], m2[k], q0m);
#pragma unroll
    for (int g = 0; g < NG; g++) {
      const double x = xg[3 * g], y = xg[3 * g + 1], z = xg[3 * g + 2];
      const double ax = fma(qd[0], x, fma(qd[3], y, fma(qd[4], z, lin[0])));   // lin0 + qd0 x + qd3 y + qd4 z
      const double by = fma(qd[1], y, fma(qd[5], z, lin[1]));                  // lin1 + qd1 y + qd5 z
      const double cz = fma(qd[2], z, lin[2]);                                 // lin2 + qd2 z
      const double val = fma(x, ax, fma(y, by, fma(z, cz, q0m)));
      const double gx = fma(qd[0], x, ax);
      const double gy = fma(qd[3], x, fma(qd[1], y, by));
      const double gz = fma(qd[4], x, fma(qd[5], y, fma(qd[2], z, cz)));
      double *o = out + (size_t)g * kFaceState * F;
      o[(size_t)c * F] = val;
#pragma unroll
      for (int k = 0; k < 3; k++)
        o[(size_t)(5 + 5 * k + c) * F] = fma(T[3 * k], gx, fma(T[3 * k + 1], gy, u.mul(T[3 * k + 2], gz)));
    }
  }
}

// ------------------------------------------------------------------------
// 3. gas-kinetic flux
// ------------------------------------------------------------------------
// Moments of the normalised Maxwellian of variance il = T = p / rho about (U, V, W),
// in u over the half range (sgn = +1: u > 0, sgn = -1: u < 0) or the full one:
//   M_n = <u^n>, M_{n+1} = U M_n + n T M_{n-1} (+ T del for n = 0),
// del = sgn g(u = 0) the density at the end of the half range (0 for the full range); hd = del / 2,
// h0 = -U del / (2T).
struct Mom { double m0, m1, m2, m3, m4, hd, h0; };
__device__ __forceinline__ void mom_up(const Units &u, const Prim &p, Mom &m) {
  const double T2 = u.add(p.il, p.il);
  m.m2 = fma(p.U, m.m1, u.mul(p.il, m.m0));
  m.m3 = fma(p.U, m.m2, u.mul(T2, m.m1));
  m.m4 = fma(p.U, m.m3, u.mul(u.add(T2, p.il), m.m2));
}
__device__ __forceinline__ Mom mom_full(const Units &u, const Prim &p) {
  Mom m;
  m.m0 = 1.0; m.m1 = p.U; m.hd = 0.0; m.h0 = 0.0;
  mom_up(u, p, m);
  return m;
}
// <u^0>, <u^1> = U <u^0> + T del, del / 2 = sgn exp(-y^2) / (2 sqrt(2 pi T)) and y = U / sqrt(2T)
// over sgn u > 0; rs = 1 / sqrt(2T)
__device__ __forceinline__ void half01(const Units &u, double U, double T, double sgn, double &m0, double &m1, double &hd,
                                       double &y, double &rs) {
  const double T2 = u.add(T, T);
  rs = rsqrt64(T2);
  y = u.mul(rs, U);
  const double x = sgn > 0.0 ? -y : y, e = exp64(u.mul(-y, y));
  if (((unsigned)__double2hiint(x) & 0x7fffffffu) < kErfcRange) {
    m0 = half_erfc64(x);
  } else {
    // erfc(x) = erfcx(|x|) exp(-x^2) for x >= 0 and 2 - erfcx(|x|) exp(-x^2) below
    const double t = erfcx(fabs(x)) * e;
    m0 = 0.5 * (x >= 0.0 ? t : 2.0 - t);
  }
  hd = u.mul(sgn * 0.28209479177387814347 * e, rs);    // 1 / (2 sqrt(pi))
  m1 = fma(U, m0, u.mul(T2, hd));
}
__device__ __forceinline__ Mom mom_half(const Units &u, const Prim &p, double sgn) {
  Mom m;
  double y, rs;
  half01(u, p.U, p.il, sgn, m.m0, m.m1, m.hd, y, rs);
  m.h0 = u.mul(u.mul(-2.0 * y, rs), m.hd);
  mom_up(u, p, m);
  return m;
}

// The spatial slopes enter as derivatives of a Maxwellian along one axis, given by the
// derivatives of its own primitive variables: dg = (a . psi) g with <a . psi> = dW is the
// change of g along dW, so every moment <phi psi (a . psi)> is the derivative of <phi psi>
// along (drho, dU, dV, dW, dT), without solving for a. With r = drho, (u, v, w) =
// rho d(U, V, W), s = rho dT = dp - T r and the identities of a Gaussian of variance T
// (d/dT = (1/2) d^2/dU^2),
//   D(rho M_n) = E_n = r M_n + u dM_n/dU + s dM_n/dT,
//   dM_n/dU = n M_{n-1} (del for n = 0),
//   dM_n/dT = n (n - 1) / 2 M_{n-2} (del / 2 for n = 1, -U del / (2T) for n = 0).
// The v, w and xi moments are taken in the frame that moves with (V, W), where odd
// tangential powers vanish: v' = v - V, w' = w - W, <v'^2> = T, <v'^4> = 3 T^2,
// <xi^2> = K T. With K2 = K + 2, K4 = K + 4 and psi' = (1, u, v', w', (u^2 + v'^2 + w'^2 +
// xi^2) / 2), for derivatives (r, u, v, w, s):
//   <u^n d psi'>    = (E_n, E_{n+1}, v M_n, w M_n, (E_{n+2} + K2 (T E_n + s M_n)) / 2)
//   <u^n v' d psi'> = (v M_n, v M_{n+1}, T E_n + s M_n, 0, v (M_{n+2} + K4 T M_n) / 2)
// (w' alike). The results return to the face frame through psi = L psi',
//   psi_2 = psi'_2 + V psi'_0,   psi_3 = psi'_3 + W psi'_0,
//   psi_4 = psi'_4 + V psi'_2 + W psi'_3 + (V^2 + W^2)/2 psi'_0.
struct Dir { double r, u, v, w, p; };    // drho, rho dU, rho dV, rho dW, dp along one axis of the face frame

// out = L x, out += L x (x in the tangential frame of p, x[4] twice the component)
__device__ __forceinline__ void from_frame(const Units &u, const Prim &p, const double *x, double *out) {
  out[0] = x[0];
  out[1] = x[1];
  out[2] = fma(p.V, x[0], x[2]);
  out[3] = fma(p.W, x[0], x[3]);
  out[4] = fma(p.V, x[2], fma(p.W, x[3], 0.5 * fma(fma(p.V, p.V, u.mul(p.W, p.W)), x[0], x[4])));
}
__device__ __forceinline__ void acc_from_frame(const Units &u, const Prim &p, const double *x, double *out) {
  const double q = fma(p.V, p.V, u.mul(p.W, p.W));
  out[0] = u.add(x[0], out[0]);
  out[1] = u.add(x[1], out[1]);
  out[2] = fma(p.V, x[0], u.add(out[2], x[2]));
  out[3] = fma(p.W, x[0], u.add(out[3], x[3]));
  out[4] = fma(p.V, x[2], fma(p.W, x[3], fma(0.5, fma(q, x[0], x[4]), out[4])));
}

// What the flux and the point values of one Maxwellian share: its convective and source
// derivatives. The time derivative of the Maxwellian (<(u . grad g + dg/dt) psi> = 0 over
// the full range: the Euler equations in primitive variables) is -(conv + q),
//   conv = V d_1 + W d_2,   q = U d_0 + (rho div, dp_0, dp_1, dp_2, (gamma - 1) T rho div).
struct Slopes { double s0, s1, s2, y, cr, cu, cv, cw, cs, qr, qu, qv, qw, qs; };
__device__ __forceinline__ Slopes slopes_of(const Units &u, const Prim &p, double g1, const Dir *d) {
  Slopes k;
  k.s0 = fma(-p.il, d[0].r, d[0].p);
  k.s1 = fma(-p.il, d[1].r, d[1].p);
  k.s2 = fma(-p.il, d[2].r, d[2].p);
  k.y = u.add(d[1].v, d[2].w);
  const double div = u.add(d[0].u, k.y);
  k.cr = fma(p.V, d[1].r, u.mul(p.W, d[2].r));
  k.cu = fma(p.V, d[1].u, u.mul(p.W, d[2].u));
  k.cv = fma(p.V, d[1].v, u.mul(p.W, d[2].v));
  k.cw = fma(p.V, d[1].w, u.mul(p.W, d[2].w));
  k.cs = fma(p.V, k.s1, u.mul(p.W, k.s2));
  k.qr = fma(p.U, d[0].r, div);
  k.qu = fma(p.U, d[0].u, d[0].p);
  k.qv = fma(p.U, d[0].v, d[1].p);
  k.qw = fma(p.U, d[0].w, d[2].p);
  k.qs = fma(p.U, k.s0, u.mul(u.mul(g1, p.il), div));
  return k;
}

// The derivatives that come with one power less of the velocity, e conv + f d_t, with c rho in
// the density slot.
struct Comb { double r, u, v, w, s; };
__device__ __forceinline__ Comb combine(const Units &u, const Prim &p, const Slopes &k, double c, double e, double f) {
  const double ef = u.sub(e, f);
  return {fma(c, p.rho, fma(ef, k.cr, u.mul(-f, k.qr))), fma(ef, k.cu, u.mul(-f, k.qu)), fma(ef, k.cv, u.mul(-f, k.qv)),
          fma(ef, k.cw, u.mul(-f, k.qw)), fma(ef, k.cs, u.mul(-f, k.qs))};
}
// sums that the flux and the state moments have in common
struct Sums { double B1, B2, E2, E3, m1x2; };

// F += c rho <u psi> + e sum_d <u u_d d_d psi> + f <u d_t psi>, b = combine(c, e, f)
__device__ __forceinline__ Sums acc_flux(const Units &u, const Prim &p, const Mom &m, const Dir *d, const Slopes &k, double K2,
                                         double K4, const Comb &b, double e, double *F) {
  const double T = p.il, hd = m.hd;
  const double m1x2 = u.add(m.m1, m.m1), m1x3 = u.add(m1x2, m.m1), m2x3 = 3.0 * m.m2, m2x6 = u.add(m2x3, m2x3);
  const double m3x4 = 4.0 * m.m3;
  Sums t;
  t.m1x2 = m1x2;
  t.B1 = fma(b.r, m.m1, fma(b.u, m.m0, u.mul(b.s, hd)));
  t.B2 = fma(b.r, m.m2, fma(b.u, m1x2, u.mul(b.s, m.m0)));
  const double B3 = fma(b.r, m.m3, fma(b.u, m2x3, u.mul(b.s, m1x3)));
  t.E2 = fma(d[0].r, m.m2, fma(d[0].u, m1x2, u.mul(k.s0, m.m0)));
  t.E3 = fma(d[0].r, m.m3, fma(d[0].u, m2x3, u.mul(k.s0, m1x3)));
  const double E4 = fma(d[0].r, m.m4, fma(d[0].u, m3x4, u.mul(k.s0, m2x6)));
  const double Y1 = fma(d[1].r, m.m1, fma(d[1].u, m.m0, u.mul(k.s1, hd)));
  const double Z1 = fma(d[2].r, m.m1, fma(d[2].u, m.m0, u.mul(k.s2, hd)));
  double x[5];
  x[0] = fma(e, fma(k.y, m.m1, t.E2), t.B1);
  x[1] = fma(e, fma(k.y, m.m2, t.E3), t.B2);
  x[2] = fma(e, fma(d[0].v, m.m2, fma(T, Y1, u.mul(k.s1, m.m1))), u.mul(b.v, m.m1));
  x[3] = fma(e, fma(d[0].w, m.m2, fma(T, Z1, u.mul(k.s2, m.m1))), u.mul(b.w, m.m1));
  const double t4 = fma(K2, fma(T, t.E2, u.mul(k.s0, m.m2)), E4);
  x[4] = fma(e, fma(k.y, fma(u.mul(K4, T), m.m1, m.m3), t4), fma(K2, fma(T, t.B1, u.mul(b.s, m.m1)), B3));
  acc_from_frame(u, p, x, F);
  return t;
}

// the moments sum_d <u_d d_d psi'> without the part of conv (u d_0, v' d_1, w' d_2)
__device__ __forceinline__ void own_moments(const Units &u, const Prim &p, const Mom &m, const Dir *d, const Slopes &k,
                                            const Sums &t, double K2, double K4, double *z) {
  const double T = p.il, hd = m.hd, del = u.add(hd, hd), h0 = m.h0;
  const double E1 = fma(d[0].r, m.m1, fma(d[0].u, m.m0, u.mul(k.s0, hd)));
  const double Y0 = fma(d[1].r, m.m0, fma(d[1].u, del, u.mul(k.s1, h0)));
  const double Z0 = fma(d[2].r, m.m0, fma(d[2].u, del, u.mul(k.s2, h0)));
  z[0] = fma(k.y, m.m0, E1);
  z[1] = fma(k.y, m.m1, t.E2);
  z[2] = fma(d[0].v, m.m1, fma(T, Y0, u.mul(k.s1, m.m0)));
  z[3] = fma(d[0].w, m.m1, fma(T, Z0, u.mul(k.s2, m.m0)));
  z[4] = fma(k.y, fma(u.mul(K4, T), m.m0, m.m2), fma(K2, fma(T, E1, u.mul(k.s0, m.m1)), t.E3));   // twice the component
}
// W += c rho <psi> + e sum_d <u_d d_d psi> + f <d_t psi>: z from own_moments, b = combine(c, e, f),
// B1 and B2 the sums of b in <u d psi>
__device__ __forceinline__ void acc_state(const Units &u, const Prim &p, const Mom &m, const double *z, double K2, const Comb &b,
                                          double B1, double B2, double e, double *W) {
  const double B0 = fma(b.r, m.m0, fma(b.u, u.add(m.hd, m.hd), u.mul(b.s, m.h0)));
  double x[5];
  x[0] = fma(e, z[0], B0);
  x[1] = fma(e, z[1], B1);
  x[2] = fma(e, z[2], u.mul(b.v, m.m0));
  x[3] = fma(e, z[3], u.mul(b.w, m.m0));
  x[4] = fma(e, z[4], fma(K2, fma(p.il, B0, u.mul(b.s, m.m0)), B2));
  acc_from_frame(u, p, x, W);
}

// State outside a boundary face (face frame, x = outward normal), from the inner one: walls
// mirror it in (p, U, V, W, T = p/rho), an isothermal wall's image with the density of zero
// mass exchange; far field = free stream. M1: <u>_{u>0} of the inner state.
__device__ void image_state(const Units &un, const KParams &P, int tag, const double *T, const Prim &l, double M1, bool held, double *Wr) {
  if (tag == HGKS_BC_FARFIELD) {
    double u[3];
#pragma unroll
    for (int r = 0; r < 3; r++) u[r] = T[3 * r] * P.u_inf[0] + T[3 * r + 1] * P.u_inf[1] + T[3 * r + 2] * P.u_inf[2];
    Wr[0] = P.rho_inf;
#pragma unroll
    for (int r = 0; r < 3; r++) Wr[1 + r] = P.rho_inf * u[r];
    Wr[4] = P.p_inf * P.ig1 + 0.5 * P.rho_inf * (u[0] * u[0] + u[1] * u[1] + u[2] * u[2]);
    return;
  }
  const double u[3] = {l.U, l.V, l.W};
  const bool T_odd = tag == HGKS_BC_WALL_ISO || tag == HGKS_BC_WALL_LID;
  double ug[3];
#pragma unroll
  for (int r = 0; r < 3; r++) {
    const double uw = tag == HGKS_BC_WALL_LID ? T[3 * r] * P.lid_speed : 0.0;
    ug[r] = (r == 0 || tag != HGKS_BC_SLIP) ? 2.0 * uw - u[r] : u[r];
  }
  const double Tg = held ? 0.5 * P.wall_T : (T_odd ? 2.0 * P.wall_T - l.il : l.il);
  // isothermal wall: the image sends back as much mass as the cell sends into the
  // wall, rho_g M(U_n, T_g) = rho M(U_n, T) with M(U, T) = <u>_{u>0} of a unit-density
  // Maxwellian; otherwise the image has the cell's pressure and temperature
  double rg = l.rho;
  if (T_odd) {
    double m0, Mg, hd, y, rs;
    half01(un, l.U, Tg, 1.0, m0, Mg, hd, y, rs);
    rg = l.rho * M1 * rcp(Mg);
  }
  Wr[0] = rg;
#pragma unroll
  for (int r = 0; r < 3; r++) Wr[1 + r] = rg * ug[r];
  Wr[4] = rg * Tg * P.ig1 + 0.5 * rg * (ug[0] * ug[0] + ug[1] * ug[1] + ug[2] * ug[2]);
}
// an isothermal image colder than T_w / 2 (a cell hotter than 1.5 T_w) is held at T_w / 2, uniform
__device__ __forceinline__ bool image_held(const KParams &P, int tag, double Tl) {
  return (tag == HGKS_BC_WALL_ISO || tag == HGKS_BC_WALL_LID) && 2.0 * P.wall_T - Tl < 0.5 * P.wall_T;
}
// the image's derivatives from the inner ones, in place: quantities even under the mirror
// keep their value and flip their normal derivative, odd ones the reverse; the pressure
// gradient keeps its size relative to the pressure
__device__ __forceinline__ void image_slopes(int tag, const Prim &l, const Prim &g, bool held, Dir *d) {
  if (tag == HGKS_BC_FARFIELD) {
#pragma unroll
    for (int a = 0; a < 3; a++) d[a] = Dir{0.0, 0.0, 0.0, 0.0, 0.0};
    return;
  }
  const bool T_odd = tag == HGKS_BC_WALL_ISO || tag == HGKS_BC_WALL_LID;
  const double rr = g.rho * l.ir, ps = T_odd ? rr * g.il * rcp(l.il) : 1.0, ig = rcp(g.il);
  const double vt = tag == HGKS_BC_SLIP ? rr : -rr;
  const double tt = held ? 0.0 : (T_odd ? -rr : rr);     // rho_g dT_g from rho dT
#pragma unroll
  for (int a = 0; a < 3; a++) {
    const double sn = a == 0 ? -1.0 : 1.0;
    const double s = fma(-l.il, d[a].r, d[a].p), dp = sn * ps * d[a].p;
    d[a].r = ig * fma(-sn * tt, s, dp);
    d[a].u *= -sn * rr;
    d[a].v *= sn * vt;
    d[a].w *= sn * vt;
    d[a].p = dp;
  }
}

// Derivatives of a Maxwellian with primitive state p from the reconstruction's derivatives q
// along the three axes. In characteristic variables R* q back-projects to conservative
// derivatives, whose primitive form with respect to p follows directly: with (du, dv, dw) =
// u* - (U, V, W) and c* the sound speed of the projection state, dp = (gamma - 1)(dE - u . dm +
// |u|^2/2 drho) takes five products instead of the fourteen of R* and nine of the change of variables.
__device__ __forceinline__ void dirs_of(const Units &u, const KParams &P, const Eig &e, const double *T, const Prim &p, const double (*q)[5],
                                        Dir *d) {
  const double g1 = P.g1;
  if (P.characteristic) {
    const double du = u.sub(e.u, p.U), dv = u.sub(e.v, p.V), dw = u.sub(e.w, p.W);
    const double gu = u.mul(g1, du), gv = u.mul(g1, dv), gw = u.mul(g1, dw), a2 = u.mul(e.a, e.a);
    const double h = 0.5 * fma(gu, du, fma(gv, dv, u.mul(gw, dw)));
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const double ad = u.mul(e.a, u.sub(q[k][4], q[k][0])), t = u.add(q[k][0], q[k][4]), r = u.add(t, q[k][1]);
      d[k].r = r;
      d[k].u = fma(du, r, ad);
      d[k].v = fma(dv, r, q[k][2]);
      d[k].w = fma(dw, r, q[k][3]);
      d[k].p = fma(a2, t, fma(h, r, fma(gu, ad, fma(gv, q[k][2], u.mul(gw, q[k][3])))));
    }
  } else {
    const double h = 0.5 * fma(p.U, p.U, fma(p.V, p.V, p.W * p.W));
#pragma unroll
    for (int k = 0; k < 3; k++) {
      double x[5];
      rot_in(u, T, q[k], x);
      d[k].r = x[0];
      d[k].u = fma(-p.U, x[0], x[1]);
      d[k].v = fma(-p.V, x[0], x[2]);
      d[k].w = fma(-p.W, x[0], x[3]);
      d[k].p = g1 * (x[4] - p.U * x[1] - p.V * x[2] - p.W * x[3] + h * x[0]);
    }
  }
}
// d, derivatives with respect to a state of velocity p, with respect to Q0 (velocity p0): a
// change of the reference velocity by (du, dv, dw) adds (0, du r, dv r, dw r,
// (gamma - 1)(du . m + |du|^2 r / 2)); added to d0
__device__ __forceinline__ void add_shifted(double g1, const Prim &p, const Prim &p0, const Dir *d, double *d0, int bd) {
  const double du = p.U - p0.U, dv = p.V - p0.V, dw = p.W - p0.W, h = 0.5 * fma(du, du, fma(dv, dv, dw * dw));
#pragma unroll
  for (int a = 0; a < 3; a++) {
    double *o = d0 + 5 * a * bd;
    o[0] += d[a].r;
    o[bd] += fma(du, d[a].r, d[a].u);
    o[2 * bd] += fma(dv, d[a].r, d[a].v);
    o[3 * bd] += fma(dw, d[a].r, d[a].w);
    o[4 * bd] += fma(g1, fma(du, d[a].u, fma(dv, d[a].v, fma(dw, d[a].w, h * d[a].r))), d[a].p);
  }
}

// a state or moments in a thread's column of shared memory (rows of bd)
__device__ __forceinline__ void keep(double *c, int bd, const Prim &p) {
  c[0] = p.rho; c[bd] = p.U; c[2 * bd] = p.V; c[3 * bd] = p.W; c[4 * bd] = p.il; c[5 * bd] = p.ir;
}
__device__ __forceinline__ void keep(double *c, int bd, const Mom &m) {
  c[0] = m.m0; c[bd] = m.m1; c[2 * bd] = m.m2; c[3 * bd] = m.m3; c[4 * bd] = m.m4; c[5 * bd] = m.hd; c[6 * bd] = m.h0;
}
__device__ __forceinline__ Prim kept_prim(const double *c, int bd) {
  return {c[0], c[bd], c[2 * bd], c[3 * bd], c[4 * bd], c[5 * bd]};
}
__device__ __forceinline__ Mom kept_mom(const double *c, int bd) {
  return {c[0], c[bd], c[2 * bd], c[3 * bd], c[4 * bd], c[5 * bd], c[6 * bd]};
}
constexpr int kFluxRows = 34, kFluxMax = 256;   // doubles that a thread of k_flux keeps in shared memory, threads of a block

// Flux of Eq. (flux), averaged over [0, dt], at one Gauss point and, for the compact scheme,
// the point value of Eq. (point) at t*. Bound by the FP64 pipe (2 DFMA per SM and clock), so
// the form of the moment sums is what counts. The three Maxwellians (g_l over u > 0, g_r over
// u < 0, g_0) go through one loop body with their own moments and time coefficients, divided
// by dt throughout so that the time average needs no division of its own; the derivatives
// are read where they are used, so one side's fifteen are live at a time. Against slopes
// solved for each axis and summed with moments up to u^6: 37.5 -> 24.5 ms at 14.2M Gauss
// points (inviscid, 2,359,296 tetrahedra), 1.22 -> 0.74 ms at 295k (viscous, compact scheme);
// with the functions of fp64.cuh and the parameters' divisions on the host 19.8 and 0.63 ms;
// with g_0's derivatives from the sum of the characteristic ones 19.1 and 0.61 ms; products and
// sums as FMAs of three registers (Units) 17.9 and 0.61 ms; sums shared by flux, heat flux and
// point values 17.9 and 0.57 ms. ncu at 124,416 cells then: 743 FP64 instructions a thread
// (inviscid), the FP64 pipe 87 % busy with 8 warps an SM. What lives through the whole loop and
// is used once or twice (g_0's state and derivatives, g_r's state and moments) waits in shared
// memory instead of in spills: 7.60 -> 7.46 ms at 6.0M Gauss points (inviscid, 995,328
// tetrahedra), 0.567 -> 0.541 ms viscous and compact. The inviscid kernel then fits 168 registers, 12
// warps an SM (128 registers, 16 warps: 7.81 ms); the compact one takes 240 (168: 0.572 ms).
template <bool BATCH, class S, bool COMPACT>
__global__ void __launch_bounds__(COMPACT ? 256 : 384) k_flux(DevMesh m, KParams Pv, const double *__restrict__ Q,
                                                                      const double *__restrict__ dt, const double *__restrict__ wface,
                                                                      double *__restrict__ fflux, double *__restrict__ fpt, int *__restrict__ flags) {
  constexpr int NG = S::NG;
  const int N = m.N, F = m.F;
  const int FL = BATCH ? m.FL : F;
  // block b covers Gauss point (b mod NG) of face range b / NG: the blocks of a
  // range run together and share the face's frame and cell states in L2
  const int g = blockIdx.x % NG, f = (blockIdx.x / NG) * blockDim.x + threadIdx.x;
  if (f >= FL) return;
  if (BATCH && !m.mact[m.fmesh[f]]) return;             // a mesh of a batch that has stopped
  const KParams &P = BATCH ? m.ptab[m.fmesh[f]] : Pv;
  double T[9];
#pragma unroll
  for (int k = 0; k < 9; k++) T[k] = m.fT[(size_t)k * F + f];
  const int L = m.fl[f], R = m.fr[f];
  const bool inner = R >= 0;
  // long-lived values of the thread wait in shared memory (rows of blockDim.x): the sum of the
  // derivatives, g_r's state and moments, g_0's state
  extern __shared__ double kept[];
  const int bd = blockDim.x;
  double *const kq = kept + threadIdx.x, *const kr = kq + 15 * bd, *const k0 = kq + 28 * bd;
  const Units u = units();
  const double g1 = u.add(P.g1, u.nz), K2 = u.add(P.K2, u.nz), K4 = u.add(P.K4, u.nz);   // in registers
  Prim pk;               // state and moments of the Maxwellian at hand: g_l first
  Mom mk;
  Eig e;
  int bad = 0;            // bit s: side s fell back to its cell average with zero slopes
  bool held = false;
  double jump, pp0;       // |p_l - p_r| / (p_l + p_r), p of g_0
  {
    double QL[5], QR[5], Qs[5], Qsl[5], W[5], q[5];
#pragma unroll
    for (int c = 0; c < 5; c++) {
      QL[c] = Q[(size_t)c * N + L];
      QR[c] = inner ? Q[(size_t)c * N + R] : QL[c];
      Qs[c] = inner ? u.add(QL[c], QR[c]) : QL[c];             // twice Q*: only ratios are taken
    }
    rot_in(u, T, Qs, Qsl);
    e = eig_of(u, Qsl, P.gamma, g1);
    auto side = [&](int s, const double *Qc) {
      const double *in = wface + ((size_t)(s * NG + g) * kFaceState) * F + f;
#pragma unroll
      for (int c = 0; c < 5; c++) q[c] = in[(size_t)c * F];
      if (P.characteristic) right_apply(u, e, q, W);
      else rot_in(u, T, q, W);
      double rp = rho_p(u, W, g1);
      if (!positive(W[0]) || !positive(rp)) {
        rot_in(u, T, Qc, W);
        rp = rho_p(u, W, g1);
        bad |= 1 << s;
      }
      return rp;
    };
    double rp = side(0, QL);
    pk = to_prim(u, W, rp);
    mk = mom_half(u, pk, 1.0);
    if (inner) {
      rp = side(1, QR);
    } else {
      held = image_held(P, m.ftag[f], pk.il);
      image_state(u, P, m.ftag[f], T, pk, mk.m1, held, W);
      rp = rho_p(u, W, g1);
    }
    const Prim pr = to_prim(u, W, rp);
    const Mom mr = mom_half(u, pr, -1.0);
    // compatibility condition: Q0 = int_{u>0} psi g_l + int_{u<0} psi g_r
    double Q0[5];
    const double xl[5] = {u.mul(pk.rho, mk.m0), u.mul(pk.rho, mk.m1), 0.0, 0.0, u.mul(pk.rho, fma(u.mul(K2, pk.il), mk.m0, mk.m2))};
    const double xr[5] = {u.mul(pr.rho, mr.m0), u.mul(pr.rho, mr.m1), 0.0, 0.0, u.mul(pr.rho, fma(u.mul(K2, pr.il), mr.m0, mr.m2))};
    from_frame(u, pk, xl, Q0);
    acc_from_frame(u, pr, xr, Q0);
    const Prim p0 = to_prim(u, Q0, rho_p(u, Q0, g1));
    keep(k0, bd, p0);
    keep(kr, bd, pr);
    keep(kr + 6 * bd, bd, mr);
    const double prl = u.mul(pk.rho, pk.il), prr = u.mul(pr.rho, pr.il);
    jump = fabs(u.mul(u.sub(prl, prr), rcp(u.add(prl, prr), u.one)));
    pp0 = u.mul(p0.rho, p0.il);
  }
  double dtf;
  if (positive(P.flux_dt)) dtf = P.flux_dt;
  else dtf = (inner ? min_positive(dt[L], dt[R]) : dt[L]) * P.flux_dt_ratio;
  // collision time (Sec. 5) over dt, and the time coefficients of Eq. (flux) over dt
  const double tq = fma(P.tau_C, jump, P.viscous ? P.mu * rcp(u.mul(pp0, dtf), u.one) : P.tau_eps);   // tau / dt
  const double eta = exp64(-rcp(tq, u.one));
  const double c4 = u.mul(tq, u.sub(u.one, eta)), k4 = u.mul(tq, c4), k42 = u.add(k4, k4), tau = u.mul(tq, dtf);
  const double c1 = u.sub(u.one, c4), c2 = u.mul(dtf, fma(-tq, u.add(u.one, eta), k42)), c3 = u.mul(dtf, 0.5 - tq + k4);
  const double c5 = u.mul(dtf, fma(-tq, eta, k42));
  const bool prandtl = P.fix_prandtl;
  const double ts = P.tstar_end ? dtf : 0.0, es = P.tstar_end ? eta : 1.0;   // exp(-t* / tau)
  double Fl[5] = {0, 0, 0, 0, 0}, Wb[5] = {0, 0, 0, 0, 0}, Pt[5] = {0, 0, 0, 0, 0};
  // The derivatives of g_0 are the mean of both sides' conservative derivatives. They enter
  // linearly, so their sum is taken and the time coefficients halved. An interior face sums the
  // characteristic derivatives (which share R*) and converts the sum to Q0's primitive form;
  // other faces sum each side's primitive ones shifted to Q0's velocity.
  const bool sums = inner && P.characteristic;
  Dir d[3];
  if (!sums)
#pragma unroll
    for (int a = 0; a < 15; a++) kq[a * bd] = 0.0;
  double C = c4, Ce = -c5, Cf = u.mul(-dtf, k4);              // flux: c rho <u psi> + e sum <u u_d d_d psi> + f <u d_t psi>
  double A = es, Ae = -es * (tau + ts), Af = -es * tau; // point value
#pragma unroll 1
  for (int s = 0; s < 3; s++) {
    if (s < 2) {
      if (s == 0 || inner) {               // a boundary face's image derivatives are in d already
        const double *in = wface + ((size_t)(s * NG + g) * kFaceState + 5) * F + f;
        double q[3][5];
#pragma unroll
        for (int a = 0; a < 15; a++) q[a / 5][a % 5] = bad >> s & 1 ? 0.0 : in[(size_t)a * F];
        dirs_of(u, P, e, T, pk, q, d);
        if (sums) {
          if (s == 0) {
#pragma unroll
            for (int a = 0; a < 15; a++) kq[a * bd] = q[a / 5][a % 5];
          } else {
#pragma unroll
            for (int a = 0; a < 15; a++) kq[a * bd] = u.add(kq[a * bd], q[a / 5][a % 5]);
          }
        }
      }
      if (!sums) add_shifted(g1, pk, kept_prim(k0, bd), d, kq, bd);
    } else {
      pk = kept_prim(k0, bd);
      mk = mom_full(u, pk);
      double q[3][5];
#pragma unroll
      for (int a = 0; a < 15; a++) q[a / 5][a % 5] = kq[a * bd];
      if (sums) {
        dirs_of(u, P, e, T, pk, q, d);
      } else {
#pragma unroll
        for (int a = 0; a < 3; a++) d[a] = Dir{q[a][0], q[a][1], q[a][2], q[a][3], q[a][4]};
      }
      C = c1; Ce = 0.5 * c2; Cf = 0.5 * c3;
      A = 1.0 - es; Ae = 0.5 * fma(ts + tau, es, -tau); Af = 0.5 * (ts - tau + tau * es);
    }
    const Slopes k = slopes_of(u, pk, g1, d);
    const Comb b = combine(u, pk, k, C, Ce, Cf);
    const Sums t = acc_flux(u, pk, mk, d, k, K2, K4, b, Ce, Fl);
    if (COMPACT || prandtl) {
      double z[5];
      own_moments(u, pk, mk, d, k, t, K2, K4, z);
      if (prandtl) acc_state(u, pk, mk, z, K2, b, t.B1, t.B2, Ce, Wb);
      if (COMPACT) {
        const Comb a = combine(u, pk, k, A, Ae, Af);
        const double A1 = fma(a.r, mk.m1, fma(a.u, mk.m0, u.mul(a.s, mk.hd)));
        const double A2 = fma(a.r, mk.m2, fma(a.u, t.m1x2, u.mul(a.s, mk.m0)));
        acc_state(u, pk, mk, z, K2, a, A1, A2, Ae, Pt);
      }
    }
    if (s == 0) {
      const Prim pr = kept_prim(kr, bd);
      if (!inner) image_slopes(m.ftag[f], pk, pr, held, d);
      pk = pr;
      mk = kept_mom(kr + 6 * bd, bd);
    }
  }
  if (prandtl) {
    // heat flux of the averaged distribution about the velocity of Q0 times 1/Pr - 1
    const double U = pk.U, V = pk.V, W = pk.W, h2 = 0.5 * fma(U, U, fma(V, V, u.mul(W, W)));
    const double qf = fma(-U, Fl[1], fma(-V, Fl[2], fma(-W, Fl[3], fma(h2, Fl[0], Fl[4]))));
    const double qw = fma(-U, Wb[1], fma(-V, Wb[2], fma(-W, Wb[3], fma(h2, Wb[0], Wb[4]))));
    Fl[4] = fma(P.prandtl, fma(-U, qw, qf), Fl[4]);
  }
  // walls are impermeable: their faces carry momentum and energy, no mass
  if (!inner && m.ftag[f] >= HGKS_BC_WALL_ISO && m.ftag[f] <= HGKS_BC_NOSLIP_ADIA) Fl[0] = 0.0;
  if (bad) atomicAdd(flags, __popc(bad));
  // Gauss weight times area: 1/3 on a triangle, the area-element weight on a quadrilateral
  const double w = NG == 3 ? m.fS[f] * (1.0 / 3.0) : m.fS[f] * m.fw[(size_t)g * F + f];
  double Fg[5];
  rot_out(u, T, Fl, Fg);
#pragma unroll
  for (int c = 0; c < 5; c++) fflux[(size_t)(g * 5 + c) * F + f] = u.mul(w, Fg[c]);
  if (COMPACT) {
    rot_out(u, T, Pt, Fg);
#pragma unroll
    for (int c = 0; c < 5; c++) fpt[(size_t)(g * 5 + c) * F + f] = u.mul(w, Fg[c]);
  }
}

// ------------------------------------------------------------------------
// 4. face -> cell
// ------------------------------------------------------------------------
template <bool BATCH, class S>
__global__ void __launch_bounds__(kBlock) k_gather(DevMesh m, int compact, const double *__restrict__ fflux,
                                                    const double *__restrict__ fpt, double *__restrict__ R,
                                                    double *__restrict__ Gnew) {
  constexpr int NF = S::NF, NG = S::NG;
  const int N = m.N, F = m.F;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  if (BATCH && m.cmesh[i] < 0) {                         // padding cell of a batch
#pragma unroll
    for (int c = 0; c < 5; c++) R[(size_t)c * N + i] = 0.0;
    if (compact)
#pragma unroll
      for (int k = 0; k < 15; k++) Gnew[(size_t)k * N + i] = 0.0;
    return;
  }
  if (BATCH && !m.mact[m.cmesh[i]]) return;             // a mesh of a batch that has stopped
  double r[5] = {0, 0, 0, 0, 0}, gr[15];
#pragma unroll
  for (int k = 0; k < 15; k++) gr[k] = 0.0;
#pragma unroll
  for (int p = 0; p < NF; p++) {
    const int cf = m.cface[(size_t)p * N + i];
    const int f = cf >> 1;
    const double sg = (cf & 1) ? 1.0 : -1.0;   // the flux leaves the left cell
#pragma unroll
    for (int c = 0; c < 5; c++) {
      double s = fflux[(size_t)c * F + f];
#pragma unroll
      for (int g = 1; g < NG; g++) s += fflux[(size_t)(5 * g + c) * F + f];
      r[c] = fma(sg, s, r[c]);
    }
    if (compact) {
      double n[3];
#pragma unroll
      for (int d = 0; d < 3; d++) n[d] = -sg * m.fT[(size_t)d * F + f];   // outward normal of this cell
#pragma unroll
      for (int c = 0; c < 5; c++) {
        double s = fpt[(size_t)c * F + f];
#pragma unroll
        for (int g = 1; g < NG; g++) s += fpt[(size_t)(5 * g + c) * F + f];
#pragma unroll
        for (int d = 0; d < 3; d++) gr[3 * c + d] = fma(s, n[d], gr[3 * c + d]);
      }
    }
  }
#pragma unroll
  for (int c = 0; c < 5; c++) R[(size_t)c * N + i] = r[c];
  if (compact) {
    const double iv = m.inv_vol[i];
#pragma unroll
    for (int k = 0; k < 15; k++) Gnew[(size_t)k * N + i] = gr[k] * iv;
  }
}

template <bool BATCH, class S>
__global__ void k_local_dt(DevMesh m, KParams Pv, const double *__restrict__ Q, double *__restrict__ dt) {
  const int N = m.N, F = m.F;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  if (BATCH && m.cmesh[i] < 0) { dt[i] = 1.0; return; }   // padding cell of a batch
  if (BATCH && !m.mact[m.cmesh[i]]) return;
  const KParams &P = BATCH ? m.ptab[m.cmesh[i]] : Pv;
  double q[5];
#pragma unroll
  for (int c = 0; c < 5; c++) q[c] = Q[(size_t)c * N + i];
  const double ir = rcp(q[0]), u = q[1] * ir, v = q[2] * ir, w = q[3] * ir;
  const double p = P.g1 * (q[4] - 0.5 * q[0] * (u * u + v * v + w * w));
  const double a = sqrt64(P.gamma * p * ir);
  const double nu = P.viscous ? 2.0 * P.gamma * P.mu * rcp(P.Pr * q[0] * m.h[i]) : 0.0;
  double s = 0.0;
#pragma unroll
  for (int k = 0; k < S::NF; k++) {
    const int f = m.cface[(size_t)k * N + i] >> 1;
    const double un = u * m.fT[f] + v * m.fT[(size_t)F + f] + w * m.fT[(size_t)2 * F + f];
    s += m.fS[f] * (fabs(un) + a + nu);
  }
  dt[i] = P.cfl * m.vol[i] * rcp(s);
}

}  // namespace

// force[3] = sum over the faces tagged `tag` of the momentum part of fflux ([3][5][F],
// global frame, area included); one block, fixed summation order
__global__ void __launch_bounds__(1024) k_wall_force(DevMesh m, int tag, int ng, const double *__restrict__ fflux,
                                                     double *__restrict__ force) {
  __shared__ double sh[3][1024];
  const int F = m.F;
  double acc[3] = {0.0, 0.0, 0.0};
  for (int f = threadIdx.x; f < F; f += blockDim.x) {
    if (m.fr[f] >= 0 || m.ftag[f] != tag) continue;
    for (int g = 0; g < ng; g++)
#pragma unroll
      for (int d = 0; d < 3; d++) acc[d] += fflux[(size_t)(5 * g + 1 + d) * F + f];
  }
#pragma unroll
  for (int d = 0; d < 3; d++) sh[d][threadIdx.x] = acc[d];
  __syncthreads();
  for (int w = blockDim.x / 2; w > 0; w >>= 1) {
    if (threadIdx.x < w)
#pragma unroll
      for (int d = 0; d < 3; d++) sh[d][threadIdx.x] += sh[d][threadIdx.x + w];
    __syncthreads();
  }
  if (threadIdx.x == 0)
#pragma unroll
    for (int d = 0; d < 3; d++) force[d] = sh[d][0];
}

void launch_wall_force(const DevMesh &m, const Scratch &s, int tag, double *force_dev, cudaStream_t st) {
  HGKS_PROF_BEGIN(K_NORM, st);
  k_wall_force<<<1, 1024, 0, st>>>(m, tag, m.hex ? HexShape::NG : TetShape::NG, s.fflux, force_dev);
  HGKS_PROF_END(K_NORM, st);
}

void launch_local_dt(const DevMesh &m, const hgks_params &hp, const double *Q, double *dt, cudaStream_t st) {
  const KParams p = kernel_params(hp);
  HGKS_PROF_BEGIN(K_DT, st);
  if (m.ptab && m.hex) k_local_dt<true, HexShape><<<grid_for(m.NL, kBlock), kBlock, 0, st>>>(m, p, Q, dt);
  else if (m.ptab) k_local_dt<true, TetShape><<<grid_for(m.NL, kBlock), kBlock, 0, st>>>(m, p, Q, dt);
  else if (m.hex) k_local_dt<false, HexShape><<<grid_for(m.N, kBlock), kBlock, 0, st>>>(m, p, Q, dt);
  else k_local_dt<false, TetShape><<<grid_for(m.N, kBlock), kBlock, 0, st>>>(m, p, Q, dt);
  HGKS_PROF_END(K_DT, st);
}

int recon_block_max(const DevMesh &m) { return m.hex ? kReconHex : kReconMax; }

namespace {
// Raises a kernel's dynamic shared memory to that of its largest block. The limit is the kernel's,
// for all threads of the process: a value of the caller's own block shape would refuse the launch
// of another thread that has just set a larger one. A failure shows in the launch that follows.
template <class K>
void allow_shared(K *kernel, size_t bytes_per_thread, int max_threads) {
  cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)(bytes_per_thread * max_threads));
}
// the four residual kernels of one cell kind
template <bool BATCH, class S>
void residual_kernels(const DevMesh &m, Scratch &s, const hgks_params &hp, const double *Q, const double *G, double *R,
                      double *Gnew, cudaStream_t st) {
  const KParams p = kernel_params(hp);
  const int64_t NL = BATCH ? m.NL : m.N, FL = BATCH ? m.FL : m.F;
  HGKS_PROF_BEGIN(K_COEF, st);
  const unsigned gc = grid_for(5 * NL, kBlock);
  if (p.scheme == HGKS_WENO) k_coef_weno<BATCH, S><<<gc, kBlock, 0, st>>>(m, Q, s.coef);
  else k_coef_hweno<BATCH, S><<<gc, kBlock, 0, st>>>(m, Q, G, s.coef);
  HGKS_PROF_END(K_COEF, st);
  HGKS_PROF_BEGIN(K_RECON, st);
  const int rmax = recon_block_max(m);
  const int br = std::min(s.blk_recon, rmax);
  const bool weno = p.scheme == HGKS_WENO;
  const size_t row = sizeof(double) * recon_rows(weno ? S::NSUBW : S::NF);
  auto recon = weno ? k_recon<BATCH, S, S::NSUBW> : k_recon<BATCH, S, S::NF>;
  allow_shared(recon, row, rmax);
  recon<<<S::NF * grid_for(NL, br), br, row * br, st>>>(m, p, Q, s.coef, s.wface);
  HGKS_PROF_END(K_RECON, st);
  HGKS_PROF_BEGIN(K_FLUX, st);
  const int bf = std::min(s.blk_flux, kFluxMax);
  auto flux = p.scheme == HGKS_HWENO ? k_flux<BATCH, S, true> : k_flux<BATCH, S, false>;
  allow_shared(flux, sizeof(double) * kFluxRows, kFluxMax);
  flux<<<S::NG * grid_for(FL, bf), bf, sizeof(double) * kFluxRows * bf, st>>>(m, p, Q, s.dt, s.wface, s.fflux, s.fpt, s.flags);
  HGKS_PROF_END(K_FLUX, st);
  HGKS_PROF_BEGIN(K_GATHER, st);
  const int grad = p.scheme == HGKS_HWENO && Gnew != nullptr;   // gradients wanted
  k_gather<BATCH, S><<<grid_for(NL, kBlock), kBlock, 0, st>>>(m, grad, s.fflux, s.fpt, R, Gnew);
  HGKS_PROF_END(K_GATHER, st);
}
}  // namespace

void launch_residual(const DevMesh &m, Scratch &s, const hgks_params &p, const double *Q, const double *G, double *R,
                     double *Gnew, cudaStream_t st, bool batch, bool fresh_dt) {
  HGKS_RANGE("hgks residual");
  batch = batch || m.ptab != nullptr;
  if (fresh_dt) launch_local_dt(m, p, Q, s.dt, st);
  if (batch && m.hex) residual_kernels<true, HexShape>(m, s, p, Q, G, R, Gnew, st);
  else if (batch) residual_kernels<true, TetShape>(m, s, p, Q, G, R, Gnew, st);
  else if (m.hex) residual_kernels<false, HexShape>(m, s, p, Q, G, R, Gnew, st);
  else residual_kernels<false, TetShape>(m, s, p, Q, G, R, Gnew, st);
}

}  // namespace hgks
