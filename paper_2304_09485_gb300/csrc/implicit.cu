// Implicit part of one HGKS step (paper Sec. 4.1 - 4.3, Algorithm 1), FP64.
//
//  * A of Eq. (A-system-2) with the split Jacobians of Eq. (deri-matrix):
//      A_ii  = |Omega_i|/dt_i I + sum_p (J(Q_i) n_p + |lambda_p| I) S_p / 2
//      A_ij  = (J(Q_j) n_p - |lambda_p| I) S_p / 2
//    The Euler-Jacobian part of A_ii is J(Q_i) applied to sum_p n_p S_p, the
//    sum of a closed cell's outward area vectors, which is zero: A_ii is a
//    multiple of the identity and is stored as one number per cell. The
//    off-diagonal blocks (the per-cell "structure array" of Sec. 4.3) are kept as
//    the operands of their products (offdiag.cuh), component-major so that the
//    thread of cell i reads consecutive addresses with its warp; batches with FP64
//    vectors store them, off[(p*25 + k)][N] (p = local face of the row cell).
//  * Jacobi preconditioner of Eq. (precond), k_max sweeps (FP32: the first sweep reads
//    D^{-1} b of the neighbours on the fly).
//  * Restarted GMRES with modified Gram-Schmidt (Algorithm 1). Every inner
//    product finishes inside its launch: blocks write partial sums, the last
//    block to finish adds them in a fixed order (deterministic, no host round
//    trip); the first product (w, v_0) is fused into the last Jacobi sweep. The
//    Hessenberg least-squares problem (Givens rotations) runs on the device, so a
//    whole GMRES cycle is enqueued without synchronising the host.
#include <cmath>
#include <type_traits>
#include "hgks_internal.h"
#include "fp64.cuh"
#include "givens.cuh"
#include "offdiag.cuh"

namespace hgks {
namespace {

constexpr int kBlock = 256;
constexpr int kCellBlock = 128;
constexpr int kRedBlocks = 152 * 4;   // blocks of the vector reductions: a multiple of the SM count

// (J(Q) - lambda I) S/2 for nS = n S/2 and lS = lambda S/2, Q with primitives (vel, H), phi = (gamma - 1)|u|^2/2,
// un = u . nS: every entry from products that carry S/2 already
__device__ __forceinline__ void offdiag_block(const double *vel, double H, double phi, double g1, const double *nS,
                                              double un, double lS, double *J) {
  const double gv[3] = {g1 * vel[0], g1 * vel[1], g1 * vel[2]}, s = un - lS;
  J[0] = -lS; J[1] = nS[0]; J[2] = nS[1]; J[3] = nS[2]; J[4] = 0.0;
#pragma unroll
  for (int r = 0; r < 3; r++) {
    J[5 * (r + 1)] = fma(phi, nS[r], -vel[r] * un);
#pragma unroll
    for (int c = 0; c < 3; c++) J[5 * (r + 1) + 1 + c] = fma(vel[r], nS[c], r == c ? fma(-gv[c], nS[r], s) : -gv[c] * nS[r]);
    J[5 * (r + 1) + 4] = g1 * nS[r];
  }
  J[20] = (phi - H) * un;
#pragma unroll
  for (int c = 0; c < 3; c++) J[21 + c] = fma(H, nS[c], -gv[c] * un);
  J[24] = fma(g1, un, s);
}

// off, off_out: the blocks themselves (may be null); jv64, jv32 (may be null): the operands
// of their product form, FP32 (mixed precision) with dval32, dinv32. Bound by what it
// writes: 26 doubles a cell (jv64, tetrahedra) instead of the 100 of the blocks.
template <bool BATCH, int NF>
__global__ void __launch_bounds__(kCellBlock) k_assemble(DevMesh m, KParams Pv, const double *__restrict__ Q,
                                                         const double *__restrict__ dt, double *__restrict__ dval,
                                                         double *__restrict__ dinv, double *__restrict__ off,
                                                         double *__restrict__ diag_out, double *__restrict__ off_out,
                                                         float *__restrict__ dval32, float *__restrict__ dinv32,
                                                         float *__restrict__ jv32, double *__restrict__ jv64) {
  const int N = m.N, F = m.F;
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  if (BATCH && m.cmesh[i] < 0) {                          // padding cell of a batch: identity row
    dval[i] = 1.0;
    dinv[i] = 1.0;
    if (off)
#pragma unroll 4
      for (int k = 0; k < 25 * NF; k++) off[(size_t)k * N + i] = 0.0;
    if (jv32) {
      dval32[i] = 1.0f;
      dinv32[i] = 1.0f;
#pragma unroll 2
      for (int k = 0; k < 6 + 4 * NF; k++) jv32[(size_t)k * N + i] = 0.0f;
    }
    return;
  }
  if (BATCH && !m.mact[m.cmesh[i]]) return;             // a mesh of a batch that has stopped
  const KParams &P = BATCH ? m.ptab[m.cmesh[i]] : Pv;
  double Qi[5];
#pragma unroll
  for (int c = 0; c < 5; c++) Qi[c] = Q[(size_t)c * N + i];
  if (jv32 || jv64) {                                   // this cell's primitives, for the rows of its neighbours
    const double ir = rcp(Qi[0]), g1 = P.g1;
    const double u = Qi[1] * ir, v = Qi[2] * ir, w = Qi[3] * ir, phi = 0.5 * g1 * (u * u + v * v + w * w);
    const double pk[6] = {u, v, w, P.gamma * Qi[4] * ir - phi, phi, g1};
#pragma unroll
    for (int k = 0; k < 6; k++) {
      if (jv32) jv32[(size_t)k * N + i] = (float)pk[k];
      if (jv64) jv64[(size_t)k * N + i] = pk[k];
    }
  }
  double d = m.vol[i] * rcp(dt[i]);
#pragma unroll 1
  for (int p = 0; p < NF; p++) {
    const int cf = m.cface[(size_t)p * N + i], f = cf >> 1, side = cf & 1;
    const int j = m.cnb[(size_t)p * N + i];
    double n[3];
#pragma unroll
    for (int k = 0; k < 3; k++) {
      const double t = m.fT[(size_t)k * F + f];
      n[k] = side ? -t : t;
    }
    const double hS = 0.5 * m.fS[f];
    double Qj[5], Qf[5];                                // Qf: twice the face state (only ratios are taken)
#pragma unroll
    for (int c = 0; c < 5; c++) {
      Qj[c] = j >= 0 ? Q[(size_t)c * N + j] : Qi[c];
      Qf[c] = Qi[c] + Qj[c];
    }
    const double ir = rcp(Qf[0]);
    const double u = Qf[1] * ir, v = Qf[2] * ir, w = Qf[3] * ir;
    const double pr = P.g1 * (Qf[4] - 0.5 * Qf[0] * (u * u + v * v + w * w));
    double lam = fabs(u * n[0] + v * n[1] + w * n[2]) + sqrt64(P.gamma * pr * ir);
    if (P.viscous) lam += 4.0 * P.mu * ir * rcp(m.fdist[f]);
    const double lS = lam * hS;
    d += lS;
    if (jv32)
#pragma unroll
      for (int k = 0; k < 4; k++)
        jv32[(size_t)(6 + 4 * p + k) * N + i] = j >= 0 ? (float)(k < 3 ? hS * n[k] : lS) : 0.0f;
    if (!jv64 && !off && !off_out) continue;
    const double iq = rcp(Qj[0]), vel[3] = {Qj[1] * iq, Qj[2] * iq, Qj[3] * iq}, nS[3] = {hS * n[0], hS * n[1], hS * n[2]};
    const double un = vel[0] * nS[0] + vel[1] * nS[1] + vel[2] * nS[2];
    if (jv64) {
      const double rec[5] = {nS[0], nS[1], nS[2], un - lS, un};
#pragma unroll
      for (int k = 0; k < 5; k++) jv64[(size_t)(6 + 5 * p + k) * N + i] = j >= 0 ? rec[k] : 0.0;
    }
    if (off || off_out) {
      double J[25];
      const double phi = 0.5 * P.g1 * (vel[0] * vel[0] + vel[1] * vel[1] + vel[2] * vel[2]);
      offdiag_block(vel, P.gamma * Qj[4] * iq - phi, phi, P.g1, nS, un, lS, J);
#pragma unroll
      for (int k = 0; k < 25; k++) {
        const double o = j >= 0 ? J[k] : 0.0;
        if (off) off[(size_t)(p * 25 + k) * N + i] = o;
        if (off_out) off_out[(size_t)(p * 25 + k) * N + i] = o;
      }
    }
  }
  const double id = rcp(d);
  dval[i] = d;
  dinv[i] = id;
  if (jv32) {
    dval32[i] = (float)d;
    dinv32[i] = (float)id;
  }
  if (diag_out)
#pragma unroll
    for (int k = 0; k < 25; k++) diag_out[(size_t)k * N + i] = k % 6 == 0 ? d : 0.0;
}

// Deterministic reduction: per-block partial sums, the last block adds them in
// a fixed order (strided per thread, then a fixed tree). T is the accumulation type.
template <typename T>
__device__ __forceinline__ T block_sum(T v) {
  __shared__ T sh[32];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  T s = T(0);
  if (threadIdx.x < 32) {
    s = threadIdx.x < (blockDim.x >> 5) ? sh[threadIdx.x] : T(0);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
  }
  return s;   // valid in thread 0
}
// *out = sum of all blocks' v or its square root, stored as double
template <bool ROOT, typename T>
__device__ __forceinline__ void grid_sum(T v, T *partials, unsigned int *count, double *out) {
  __shared__ bool last;
  const T bs = block_sum(v);
  if (threadIdx.x == 0) {
    partials[blockIdx.x] = bs;
    __threadfence();
    const unsigned int prev = atomicAdd(count, 1u);
    last = (prev == gridDim.x - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
  T s = T(0);
  for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) s += ((volatile T *)partials)[b];
  s = block_sum(s);
  if (threadIdx.x == 0) {
    *out = ROOT ? (double)sqrt(s) : (double)s;
    *count = 0u;
  }
}

// 1 / h in single precision (0 for h == 0) for all threads of a block: one FP64 division instead of one per warp
__device__ __forceinline__ float block_inverse(const double *h) {
  __shared__ float ih;
  if (threadIdx.x == 0) ih = *h != 0.0 ? (float)(1.0 / *h) : 0.0f;
  __syncthreads();
  return ih;
}

// One product with the off-diagonal part of A from FP32 operands (mixed precision; FP64
// vectors: gmres64.cu). Modes:
//   kSpmv   : y = b - (d x + sum_p A_ip x_p)
//   kJacobi : y = D^{-1} (b - sum_p A_ip x_p); FirstSweep: x_p = D^{-1} b at the neighbours
//   kNeumann: y = b + D^{-1} sum_p A_ip x_p
//   kE, kNegE: y = +- D^{-1} sum_p A_ip x_p
// TV: type of b and x (and of the accumulation). Scaled: x is w, and v = w / h (0 for h == 0) is
// formed on the way: stored for the cell itself, used for its neighbours (the same rounding), so a
// new basis vector takes no launch of its own.
enum { kSpmv = 0, kJacobi = 1, kNeumann = 2, kE = 3, kNegE = 4 };

template <typename TV, int Mode, bool FirstSweep, bool Scaled, int NF>
__global__ void __launch_bounds__(kCellBlock) k_apply(DevMesh m, const float *__restrict__ jv,
                                                      const float *__restrict__ dval, const float *__restrict__ dinv,
                                                      const TV *__restrict__ b, const TV *__restrict__ x,
                                                      float *__restrict__ y, const double *__restrict__ h,
                                                      float *__restrict__ v) {
  const int N = m.N;
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  const float ih = Scaled ? block_inverse(h) : 1.0f;
  if (i >= N) return;
  if (Scaled)
#pragma unroll
    for (int r = 0; r < 5; r++) v[(size_t)r * N + i] = x[(size_t)r * N + i] * ih;
  TV acc[5];
  const TV di = Mode == kSpmv ? (TV)dval[i] : TV(0);
#pragma unroll
  for (int r = 0; r < 5; r++) acc[r] = Mode == kSpmv ? di * x[(size_t)r * N + i] : TV(0);
#pragma unroll
  for (int p = 0; p < NF; p++) {
    const int j = m.cnb[(size_t)p * N + i];
    if (j < 0) continue;
    TV xj[5];
    const TV sj = FirstSweep ? (TV)dinv[j] : TV(1);
#pragma unroll
    for (int c = 0; c < 5; c++) xj[c] = FirstSweep ? sj * b[(size_t)c * N + j] : Scaled ? x[(size_t)c * N + j] * ih : x[(size_t)c * N + j];
    offdiag_product<TV>(jv, N, i, p, j, xj, acc);
  }
#pragma unroll
  for (int r = 0; r < 5; r++) {
    const TV dd = Mode == kNegE ? -(TV)dinv[i] : (TV)dinv[i], br = Mode == kE || Mode == kNegE ? TV(0) : b[(size_t)r * N + i];
    TV o;
    if (Mode == kJacobi) o = dd * (br - acc[r]);
    else if (Mode == kE || Mode == kNegE) o = dd * acc[r];
    else if (Mode == kNeumann) o = fma(dd, acc[r], br);
    else o = br - acc[r];
    y[(size_t)r * N + i] = (float)o;
  }
}

// k_apply for the mesh's cell kind (4 or 6 off-diagonal blocks per row)
template <typename TV, int Mode, bool FirstSweep, bool Scaled = false>
void apply_launch(cudaStream_t st, const DevMesh &m, const Scratch &s, const TV *b, const TV *x, float *y,
                  const double *h = nullptr, float *v = nullptr) {
  const unsigned grid = grid_for(m.N, kCellBlock);
  if (m.hex)
    k_apply<TV, Mode, FirstSweep, Scaled, HexShape::NF><<<grid, kCellBlock, 0, st>>>(m, s.jv32, s.dval32, s.dinv32, b, x,
                                                                                     y, h, v);
  else
    k_apply<TV, Mode, FirstSweep, Scaled, TetShape::NF><<<grid, kCellBlock, 0, st>>>(m, s.jv32, s.dval32, s.dinv32, b, x,
                                                                                     y, h, v);
}

// y = x rounded to float
__global__ void k_round(int64_t n, const double *__restrict__ x, float *__restrict__ y) {
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    y[k] = (float)x[k];
}

template <typename T>
__global__ void k_diag_scale(int N, const T *__restrict__ dinv, const T *__restrict__ b, T *__restrict__ x) {
  int t = blockIdx.x * blockDim.x + threadIdx.x;
  if (t >= 5 * N) return;
  x[t] = dinv[t % N] * b[t];
}

// 16-byte vectors of T: every Krylov vector starts on a 256-byte boundary
// (vectors are padded to a multiple of 64 elements) and so do the device arrays
// the reductions read.
template <typename T> struct Vec16;
template <> struct Vec16<double> { typedef double2 type; static constexpr int n = 2; };
template <> struct Vec16<float> { typedef float4 type; static constexpr int n = 4; };

// *out = ||w||. 16 bytes per thread and step, four steps in flight; n need not be a multiple of
// the vector width.
template <typename T>
__global__ void __launch_bounds__(kBlock) k_norm(int64_t n, const T *__restrict__ w, T *partials, unsigned int *count,
                                                 double *out) {
  typedef typename Vec16<T>::type TV;
  constexpr int L = Vec16<T>::n;
  T s = T(0);
  const int64_t nv = n / L, stride = (int64_t)gridDim.x * blockDim.x;
  const TV *wv = reinterpret_cast<const TV *>(w);
#pragma unroll 4
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nv; k += stride) {
    const TV wk = wv[k];
    const T *wa = reinterpret_cast<const T *>(&wk);
#pragma unroll
    for (int l = 0; l < L; l++) s = fma(wa[l], wa[l], s);
  }
  for (int64_t k = nv * L + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += stride) s = fma(w[k], w[k], s);
  grid_sum<true>(s, partials, count, out);
}

// ---- modified Gram-Schmidt from one pass over the basis ----
// Algorithm 1 orthogonalises w against v_0..v_j one vector after the other:
// h_i = (w_i, v_i), w_{i+1} = w_i - h_i v_i. Since w_i = w - sum_{k<i} h_k v_k,
//   h_i = a_i - sum_{k<i} h_k G_ki,  a_i = (w, v_i),  G_ki = (v_k, v_i),
// so one pass over the basis (k_mdot: all a_i, and the new row of G, v_j against
// the older vectors) and a forward substitution give the same
// coefficients, and one more pass (k_mupdate) subtracts them in MGS order and
// takes ||w||: about 2 (j + 1) vector passes instead of 4 (j + 1) for step j
// (used with FP32 vectors, see gmres_t).
constexpr int kMdot = 8;              // basis vectors per k_mdot launch (register accumulators)

// block_sum of each v[q] into tot[q] with two barriers for all of them: the warps' sums, then
// eight lanes per value (the same order of additions)
template <typename T>
__device__ __forceinline__ void block_sum_all(T *v, T (*sh)[kBlock / 32], T *tot) {
  constexpr int W = kBlock / 32;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int q = 0; q < 2 * kMdot; q++) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v[q] += __shfl_down_sync(0xffffffffu, v[q], o);
    if (lane == 0) sh[q][warp] = v[q];
  }
  __syncthreads();
  if (threadIdx.x < 2 * kMdot * W) {
    T s = sh[threadIdx.x / W][threadIdx.x % W];
#pragma unroll
    for (int o = W / 2; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o, W);
    if (threadIdx.x % W == 0) tot[threadIdx.x / W] = s;
  }
  __syncthreads();
}

constexpr int kGramLd = 65;
// a[k] = (w, v_k) for k in [k0, k0 + nk), and g[k] = (v_j, v_k) for those k < j; with the last of
// them (k0 + nk > j) the MGS coefficients of step j by forward substitution: column j of H, and
// of the basis Gram matrix G (leading dimension kGramLd, G[k][i] = (v_k, v_i), k < i). The block
// that adds the partial sums does it: a launch of its own per vector took
// 9.86 instead of 9.83 ms for the mixed step of 294,912 tetrahedra, 9.18 instead of 9.06 for a batch of six.
template <typename T>
__global__ void __launch_bounds__(kBlock) k_mdot(int64_t n, const T *__restrict__ w, const T *__restrict__ V, int64_t vs,
                                                 int k0, int nk, int j, T *partials, unsigned int *count,
                                                 double *a, double *g, int mk, double *G, double *H) {
  typedef typename Vec16<T>::type TV;
  constexpr int L = Vec16<T>::n;
  T sa[kMdot], sg[kMdot];
#pragma unroll
  for (int q = 0; q < kMdot; q++) { sa[q] = T(0); sg[q] = T(0); }
  const int64_t nv = n / L, stride = (int64_t)gridDim.x * blockDim.x;
  const TV *wv = reinterpret_cast<const TV *>(w);
  const TV *jv = reinterpret_cast<const TV *>(V + (size_t)j * vs);
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nv; k += stride) {
    const TV wk = wv[k], vj = jv[k];
    const T *wa = reinterpret_cast<const T *>(&wk);
    const T *ja = reinterpret_cast<const T *>(&vj);
#pragma unroll
    for (int q = 0; q < kMdot; q++) {
      if (q < nk) {
        const TV vk = reinterpret_cast<const TV *>(V + (size_t)(k0 + q) * vs)[k];
        const T *va = reinterpret_cast<const T *>(&vk);
#pragma unroll
        for (int l = 0; l < L; l++) sa[q] = fma(wa[l], va[l], sa[q]);
        if (k0 + q < j)
#pragma unroll
          for (int l = 0; l < L; l++) sg[q] = fma(ja[l], va[l], sg[q]);
      }
    }
  }
  for (int64_t k = nv * L + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += stride) {
    const T wk = w[k], vj = V[(size_t)j * vs + k];
#pragma unroll
    for (int q = 0; q < kMdot; q++)
      if (q < nk) {
        const T vk = V[(size_t)(k0 + q) * vs + k];
        sa[q] = fma(wk, vk, sa[q]);
        if (k0 + q < j) sg[q] = fma(vj, vk, sg[q]);
      }
  }
  // per block: 2 kMdot partials; the last block adds every slot's partials in block order
  __shared__ bool last;
  __shared__ T sh[2 * kMdot][kBlock / 32], tot[2 * kMdot];
  T v[2 * kMdot];
#pragma unroll
  for (int q = 0; q < kMdot; q++) { v[q] = sa[q]; v[kMdot + q] = sg[q]; }
  block_sum_all(v, sh, tot);
  if (threadIdx.x < 2 * kMdot) {
    partials[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = tot[threadIdx.x];
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    last = (atomicAdd(count, 1u) == gridDim.x - 1);
  }
  __syncthreads();
  if (!last) return;
  __threadfence();
#pragma unroll
  for (int q = 0; q < 2 * kMdot; q++) {
    v[q] = T(0);
    for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x) v[q] += ((volatile T *)partials)[(size_t)q * gridDim.x + b];
  }
  block_sum_all(v, sh, tot);
  const int q = threadIdx.x, kk = k0 + q % kMdot;
  if (q < 2 * kMdot && q % kMdot < nk && (q < kMdot || kk < j)) (q < kMdot ? a : g)[kk] = (double)tot[q];
  if (threadIdx.x == 0) *count = 0u;
  if (k0 + nk <= j) return;
  __syncthreads();
  if (threadIdx.x < 32) mgs_coef_warp(threadIdx.x, j, mk, kGramLd, a, g, G, H);
}

// w -= sum_{k <= j} h_kj v_k in the order of k (MGS order), then h_{j+1,j} = ||w||
template <typename T>
__global__ void __launch_bounds__(kBlock) k_mupdate(int64_t n, T *__restrict__ w, const T *__restrict__ V, int64_t vs,
                                                    int j, int mk, const double *__restrict__ H, T *partials,
                                                    unsigned int *count, double *norm_out) {
  typedef typename Vec16<T>::type TV;
  constexpr int L = Vec16<T>::n;
  __shared__ T nh[kGramLd];
  for (int k = threadIdx.x; k <= j; k += blockDim.x) nh[k] = (T)(-H[k * mk + j]);
  __syncthreads();
  T s = T(0);
  const int64_t nv = n / L, stride = (int64_t)gridDim.x * blockDim.x;
  TV *wv = reinterpret_cast<TV *>(w);
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nv; k += stride) {
    TV wk = wv[k];
    T *wa = reinterpret_cast<T *>(&wk);
#pragma unroll 4
    for (int q = 0; q <= j; q++) {
      const TV vk = reinterpret_cast<const TV *>(V + (size_t)q * vs)[k];
      const T *va = reinterpret_cast<const T *>(&vk);
#pragma unroll
      for (int l = 0; l < L; l++) wa[l] = fma(nh[q], va[l], wa[l]);
    }
    wv[k] = wk;
#pragma unroll
    for (int l = 0; l < L; l++) s = fma(wa[l], wa[l], s);
  }
  for (int64_t k = nv * L + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += stride) {
    T wk = w[k];
    for (int q = 0; q <= j; q++) wk = fma(nh[q], V[(size_t)q * vs + k], wk);
    w[k] = wk;
    s = fma(wk, wk, s);
  }
  grid_sum<true>(s, partials, count, norm_out);
}

// v = w / h (v = 0 after a breakdown h == 0), 16 bytes per thread and step
template <typename T>
__global__ void k_scale(int64_t n, const T *__restrict__ w, const double *__restrict__ h, T *__restrict__ v) {
  typedef typename Vec16<T>::type TV;
  constexpr int L = Vec16<T>::n;
  const double hv = *h;
  const T ih = hv != 0.0 ? (T)rcp(hv) : T(0);
  const int64_t nv = n / L, stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nv; k += stride) {
    TV x = reinterpret_cast<const TV *>(w)[k];
    T *xa = reinterpret_cast<T *>(&x);
#pragma unroll
    for (int l = 0; l < L; l++) xa[l] *= ih;
    reinterpret_cast<TV *>(v)[k] = x;
  }
  for (int64_t k = nv * L + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += stride) v[k] = w[k] * ih;
}

// y minimises || beta e1 - H y || (Givens rotations in place on H, one thread, FP64)
__global__ void k_givens(int m, double *__restrict__ H, const double *__restrict__ beta, double *__restrict__ y,
                         double *__restrict__ res_out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  *res_out = givens_lsq(m, H, *beta, y);
}

// dx += sum_j y_j V_j (FP64 accumulation in the order of j; V of either
// precision, stride vs, read 16 bytes per vector and step)
template <typename T>
__global__ void __launch_bounds__(kBlock) k_combine(int64_t n, int64_t vs, int m, const T *__restrict__ V,
                                                    const double *__restrict__ y, double *__restrict__ dx) {
  typedef typename Vec16<T>::type TV;
  constexpr int L = Vec16<T>::n;
  __shared__ double ys[kGramLd];
  for (int j = threadIdx.x; j < m; j += blockDim.x) ys[j] = y[j];
  __syncthreads();
  const int64_t nv = n / L, stride = (int64_t)gridDim.x * blockDim.x;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nv; k += stride) {
    double acc[L];
#pragma unroll
    for (int l = 0; l < L; l++) acc[l] = dx[k * L + l];
#pragma unroll 4
    for (int j = 0; j < m; j++) {
      const TV v = reinterpret_cast<const TV *>(V + (size_t)j * vs)[k];
      const T *va = reinterpret_cast<const T *>(&v);
#pragma unroll
      for (int l = 0; l < L; l++) acc[l] = fma(ys[j], (double)va[l], acc[l]);
    }
#pragma unroll
    for (int l = 0; l < L; l++) dx[k * L + l] = acc[l];
  }
  for (int64_t k = nv * L + blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += stride) {
    double acc = dx[k];
    for (int j = 0; j < m; j++) acc = fma(ys[j], (double)V[(size_t)j * vs + k], acc);
    dx[k] = acc;
  }
}

__global__ void __launch_bounds__(kBlock) k_density_l1(int N, const double *__restrict__ R, const double *__restrict__ inv_vol,
                                                       double *partials, unsigned int *count, double *out) {
  double s = 0.0;
  for (int k = blockIdx.x * blockDim.x + threadIdx.x; k < N; k += gridDim.x * blockDim.x) s += fabs(R[k]) * inv_vol[k];
  grid_sum<false, double>(s, partials, count, out);
}

// nothing when the solve of dQ gave up (stuck): the caller's state stays the step's start
__global__ void k_update(int64_t n5, int64_t ng, double *__restrict__ Q, const double *__restrict__ dQ, double *__restrict__ G,
                         const double *__restrict__ Gnew, double relax, const int *__restrict__ stuck) {
  if (*stuck) return;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n5 + ng; k += (int64_t)gridDim.x * blockDim.x) {
    if (k < n5) Q[k] += dQ[k];
    else if (relax == 1.0) G[k - n5] = Gnew[k - n5];
    else G[k - n5] = fma(relax, Gnew[k - n5] - G[k - n5], G[k - n5]);
  }
}

// ---- matrix-free products (jv_mode 1), Eq. (frechet) ----
// Qp = Q + sigma x, sigma = sqrt(eps_mach) (1 + ||Q||) / ||x|| (0 for x = 0); nrm = {||Q||, ||x||, sigma}
template <typename TV>
__global__ void k_fd_perturb(int64_t n, const double *__restrict__ Q, const TV *__restrict__ x, double *__restrict__ nrm,
                             double *__restrict__ Qp) {
  const double nx = nrm[1];
  const double sigma = nx > 0.0 ? 0x1p-26 * (1.0 + nrm[0]) / nx : 0.0;
  if (blockIdx.x == 0 && threadIdx.x == 0) nrm[2] = sigma;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < n; k += (int64_t)gridDim.x * blockDim.x)
    Qp[k] = Q[k] + sigma * (double)x[k];
}

// y = A x or b - A x, A x = |Omega_i|/dt_i x - (L(Qp) - L(Q)) / sigma (A x = 0 when sigma = 0)
template <typename TV, typename TO>
__global__ void k_fd_combine(int N, const double *__restrict__ vol, const double *__restrict__ dt, const TV *__restrict__ x,
                             const double *__restrict__ Rp, const double *__restrict__ R0, const double *__restrict__ sig,
                             const double *__restrict__ b, TO *__restrict__ y) {
  const double sigma = *sig;
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < 5 * (int64_t)N; k += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = k % N;
    const double ax = sigma > 0.0 ? vol[i] / dt[i] * (double)x[k] - (Rp[k] - R0[k]) / sigma : 0.0;
    y[k] = (TO)(b ? b[k] - ax : ax);
  }
}

unsigned vec_grid(int64_t n) {
  int64_t g = (n + kBlock - 1) / kBlock;
  const int64_t cap = 152 * 8;
  return (unsigned)std::max<int64_t>(1, std::min(g, cap));
}

// Buffers of one precision for the Krylov part of a step.
template <typename T>
struct KBuf {
  const T *dinv;
  T *V, *w, *t, *t2, *red;
};
KBuf<double> kbuf64(Scratch &s) { return {s.dinv, s.V, s.w, s.t, s.t2, s.red}; }
KBuf<float> kbuf32(Scratch &s) { return {s.dinv32, s.V32, s.w32, s.t32, s.t232, s.red32}; }

template <typename T> T *partials(Scratch &s);
template <> double *partials<double>(Scratch &s) { return s.red; }
template <> float *partials<float>(Scratch &s) { return s.red32; }

// y = A x (b null) or b - A x with the matrix-free A of Eq. (frechet); s.R = L(Q), s.dt, ||Q|| in hs
template <typename TV, typename TO>
void fd_apply(const DevMesh &m, Scratch &s, const hgks_params &p, const double *Q, const double *G, const TV *x,
              const double *b, TO *y, cudaStream_t st) {
  const int64_t n = 5 * (int64_t)m.N;
  double *nrm = s.hs + kHsNormQ;
  HGKS_PROF_BEGIN(K_DOT, st);
  k_norm<TV><<<kRedBlocks, kBlock, 0, st>>>(n, x, partials<TV>(s), s.red_count, nrm + 1);
  HGKS_PROF_END(K_DOT, st);
  HGKS_PROF_BEGIN(K_SPMV, st);
  k_fd_perturb<TV><<<vec_grid(n), kBlock, 0, st>>>(n, Q, x, nrm, s.Qp);
  HGKS_PROF_END(K_SPMV, st);
  launch_residual(m, s, p, s.Qp, G, s.Rp, nullptr, st, false, false);
  HGKS_PROF_BEGIN(K_SPMV, st);
  k_fd_combine<TV, TO><<<vec_grid(n), kBlock, 0, st>>>(m.N, m.vol, s.dt, x, s.Rp, s.R, nrm + 2, b, y);
  HGKS_PROF_END(K_SPMV, st);
}

// x = P^{-1} b (Eq. (precond))
template <typename T>
void precondition_t(const DevMesh &m, Scratch &s, const KBuf<T> &k, int sweeps, const T *b, T *x, cudaStream_t st) {
  if (sweeps == 0) {
    HGKS_PROF_BEGIN(K_DIAG, st);
    k_diag_scale<T><<<grid_for(5 * (int64_t)m.N, kBlock), kBlock, 0, st>>>(m.N, k.dinv, b, x);
    HGKS_PROF_END(K_DIAG, st);
    return;
  }
  if constexpr (std::is_same<T, double>::value) {
    launch_sweeps_z(m, s, sweeps, b, x, st);
  } else {
    // sweep k writes to x when (sweeps - k) is even, else to t2: the last lands in x
    const float *prev = nullptr;
    for (int q = 1; q <= sweeps; q++) {
      float *dst = ((sweeps - q) % 2 == 0) ? x : k.t2;
      HGKS_PROF_BEGIN(K_JACOBI, st);
      if (q == 1) apply_launch<float, kJacobi, true>(st, m, s, b, prev, dst);
      else apply_launch<float, kJacobi, false>(st, m, s, b, prev, dst);
      HGKS_PROF_END(K_JACOBI, st);
      prev = dst;
    }
  }
}

// w = P^{-1} A v for a Krylov vector v, with the operator of precondition_t after
// the product with A. Write A = D (I + E), E = D^{-1} O (O: the off-diagonal
// blocks); the Jacobi iteration started from D^{-1} (A v) gives after k sweeps
// P^{-1} A v = v - (-E)^(k+1) v, i.e. w = v + E z with z = (-E)^k v (formed as
// E^k v with the sign in its first product): k + 1
// products with O instead of the product with A followed by k sweeps: the same
// vector up to rounding, without the diagonal terms of A and the scaling of the
// neighbours' values by D^{-1}. (FP32 vectors; FP64: launch_neumann_z.)
// With h (and sweeps > 0) v = w / h is formed on the way, otherwise it is given.
void neumann32(const DevMesh &m, Scratch &s, const KBuf<float> &k, int sweeps, const double *h, float *v, float *w,
               cudaStream_t st) {
  const float *z = h ? w : v, *none = nullptr;
  for (int q = 0; q < sweeps; q++) {
    float *dst = (q % 2 == 0) ? k.t : k.t2;
    HGKS_PROF_BEGIN(K_JACOBI, st);
    if (q == 0 && h && sweeps % 2 == 1) apply_launch<float, kNegE, false, true>(st, m, s, none, z, dst, h, v);
    else if (q == 0 && h) apply_launch<float, kE, false, true>(st, m, s, none, z, dst, h, v);
    else if (q == 0 && sweeps % 2 == 1) apply_launch<float, kNegE, false>(st, m, s, none, z, dst);
    else apply_launch<float, kE, false>(st, m, s, none, z, dst);
    HGKS_PROF_END(K_JACOBI, st);
    z = dst;
  }
  HGKS_PROF_BEGIN(K_SPMV, st);
  apply_launch<float, kNeumann, false>(st, m, s, v, z, w);
  HGKS_PROF_END(K_SPMV, st);
}

// One restarted GMRES solve in precision T; rhs and dx stay FP64.
template <typename T>
void gmres_t(const DevMesh &m, Scratch &s, const KBuf<T> &k, const hgks_params &p, const double *rhs, double *dx,
             cudaStream_t st, const double *Q, const double *G) {
  const bool fd = p.jv_mode == 1;
  const int mk = p.krylov_dim;
  const int64_t n = 5 * (int64_t)m.N, vs = s.vstride;
  double *H = s.hs, *beta = s.hs + (mk + 1) * mk, *y = beta + 1, *lres = y + mk;
  double *gram = s.gram, *ga = s.gram + kGramLd * kGramLd, *gg = ga + kGramLd;   // G, a, g of the MGS passes
  // The one-pass MGS does 3 FMAs per element and basis vector against 2 for the
  // step-by-step form, and reads about half the bytes: with FP32 vectors it is
  // bound by HBM and wins; with FP64 vectors both forms sit at GB300's FP64 rate
  // (one FP64 FMA per 8 bytes read already exceeds it), so FP64 goes by blocks
  // (gmres64.cu), 2 FMAs and 20 bytes.
  constexpr bool one_pass = std::is_same<T, float>::value;
  const unsigned vg = vec_grid(n);
  for (int it = 0; it < p.restarts; it++) {
    cudaMemsetAsync(H, 0, sizeof(double) * (mk + 1) * mk, st);
    // r0 = rhs - A dx (FP64 vectors, blocks of precision T), v1 = P^{-1} r0 / ||P^{-1} r0||
    if (fd && it > 0) {
      fd_apply<double, T>(m, s, p, Q, G, dx, rhs, k.t, st);
    } else if (fd) {                       // dx = 0: r0 = rhs (the product of a zero vector is zero)
      HGKS_PROF_BEGIN(K_SPMV, st);
      k_fd_combine<double, T><<<vec_grid(n), kBlock, 0, st>>>(m.N, m.vol, s.dt, dx, s.Rp, s.R, s.hs + kHsNormQ + 3, rhs, k.t);
      HGKS_PROF_END(K_SPMV, st);
    } else if constexpr (one_pass) {
      HGKS_PROF_BEGIN(K_SPMV, st);
      if (it > 0) apply_launch<double, kSpmv, false>(st, m, s, rhs, dx, k.t);
      else k_round<<<vec_grid(n), kBlock, 0, st>>>(n, rhs, k.t);
      HGKS_PROF_END(K_SPMV, st);
    } else if (it > 0) {
      launch_apply_A(m, s, rhs, dx, k.t, st);
    }
    const T *r0 = k.t;
    if constexpr (!one_pass)
      if (!fd && it == 0) r0 = rhs;        // dx = 0
    precondition_t<T>(m, s, k, p.jacobi_sweeps, r0, k.w, st);
    HGKS_PROF_BEGIN(K_DOT, st);
    k_norm<T><<<kRedBlocks, kBlock, 0, st>>>(n, k.w, k.red, s.red_count, beta);
    HGKS_PROF_END(K_DOT, st);
    if (it == 0) cudaMemcpyAsync(lres, beta, sizeof(double), cudaMemcpyDeviceToDevice, st);
    // v_j = w / h: FP64 with the assembled A, with the form that the products read; FP32 on the
    // way of the first product, if there is one before w is written again
    const bool on_the_way = one_pass && !fd && p.jacobi_sweeps > 0;
    auto scale = [&](const double *h, T *v) {
      if constexpr (!one_pass)
        if (!fd) return launch_scale_z(m, s, k.w, h, v, s.z[0], st);
      if (on_the_way) return;
      HGKS_PROF_BEGIN(K_SCALE, st);
      k_scale<T><<<vg, kBlock, 0, st>>>(n, k.w, h, v);
      HGKS_PROF_END(K_SCALE, st);
    };
    scale(beta, k.V);
    for (int j = 0; j < mk; j++) {
      // w = P^{-1} A v_j (FP64: with the first block's coefficients from the last product)
      T *vj = k.V + (size_t)j * vs;
      if (fd) {
        fd_apply<T, T>(m, s, p, Q, G, vj, nullptr, k.t, st);
        precondition_t<T>(m, s, k, p.jacobi_sweeps, k.t, k.w, st);
      } else if constexpr (one_pass) {
        neumann32(m, s, k, p.jacobi_sweeps, on_the_way ? (j == 0 ? beta : H + j * mk + j - 1) : nullptr, vj, k.w, st);
      } else {
        launch_neumann_z(m, s, p.jacobi_sweeps, vj, k.w, j, mk, H + j, st);
      }
      if constexpr (one_pass) {
        // modified Gram-Schmidt: the coefficients h_ij from one pass over the basis,
        // then w -= sum h_ij v_i in MGS order and h_{j+1,j} = ||w||
        for (int k0 = 0; k0 <= j; k0 += kMdot) {
          HGKS_PROF_BEGIN(K_DOT, st);
          k_mdot<T><<<kRedBlocks, kBlock, 0, st>>>(n, k.w, k.V, vs, k0, std::min(kMdot, j + 1 - k0), j, k.red,
                                                    s.red_count, ga, gg, mk, gram, H);
          HGKS_PROF_END(K_DOT, st);
        }
        HGKS_PROF_BEGIN(K_DOT, st);
        k_mupdate<T><<<kRedBlocks, kBlock, 0, st>>>(n, k.w, k.V, vs, j, mk, H, k.red, s.red_count, H + (j + 1) * mk + j);
        HGKS_PROF_END(K_DOT, st);
      } else {
        launch_mgs_blocks(s, n, k.w, j, mk, H + j, !fd, st);
      }
      if (j + 1 < mk) scale(H + (j + 1) * mk + j, k.V + (size_t)(j + 1) * vs);   // v_mk is not used
    }
    HGKS_PROF_BEGIN(K_GIVENS, st);
    k_givens<<<1, 32, 0, st>>>(mk, H, beta, y, lres + 1);
    HGKS_PROF_END(K_GIVENS, st);
    HGKS_PROF_BEGIN(K_COMBINE, st);
    k_combine<T><<<vg, kBlock, 0, st>>>(n, vs, mk, k.V, y, dx);
    HGKS_PROF_END(K_COMBINE, st);
  }
}

}  // namespace

void launch_assemble(const DevMesh &m, Scratch &s, const hgks_params &hp, const double *Q, const double *dt,
                     double *diag_out, double *off_out, cudaStream_t st, bool batch) {
  HGKS_RANGE("hgks assemble");
  const KParams p = kernel_params(hp);
  // mixed precision: the FP32 operands of the product form come out of the same pass
  const bool mixed = p.precision == HGKS_MIXED && s.jv32;
  float *dv32 = mixed ? s.dval32 : nullptr, *di32 = mixed ? s.dinv32 : nullptr, *jv = mixed ? s.jv32 : nullptr;
  HGKS_PROF_BEGIN(K_ASSEMBLE, st);
  batch = batch || m.ptab;
  // batches with FP64 vectors read the stored blocks, one mesh the operands
  double *off = batch && !mixed ? s.off : nullptr, *j64 = batch ? nullptr : s.jv64;
  if (batch && m.hex)
    k_assemble<true, HexShape::NF><<<grid_for(m.NL, kCellBlock), kCellBlock, 0, st>>>(m, p, Q, dt, s.dval, s.dinv, off,
                                                                                       diag_out, off_out, dv32, di32, jv, j64);
  else if (batch)
    k_assemble<true, TetShape::NF><<<grid_for(m.NL, kCellBlock), kCellBlock, 0, st>>>(m, p, Q, dt, s.dval, s.dinv, off,
                                                                                       diag_out, off_out, dv32, di32, jv, j64);
  else if (m.hex)
    k_assemble<false, HexShape::NF><<<grid_for(m.N, kCellBlock), kCellBlock, 0, st>>>(m, p, Q, dt, s.dval, s.dinv, off,
                                                                                       diag_out, off_out, dv32, di32, jv, j64);
  else
    k_assemble<false, TetShape::NF><<<grid_for(m.N, kCellBlock), kCellBlock, 0, st>>>(m, p, Q, dt, s.dval, s.dinv, off,
                                                                                       diag_out, off_out, dv32, di32, jv, j64);
  HGKS_PROF_END(K_ASSEMBLE, st);
}

void launch_precondition(const DevMesh &m, Scratch &s, int sweeps, const double *b, double *x, cudaStream_t st) {
  precondition_t<double>(m, s, kbuf64(s), sweeps, b, x, st);
}

void launch_norm(const DevMesh &m, Scratch &s, const double *x, double *out_dev, cudaStream_t st) {
  HGKS_PROF_BEGIN(K_DOT, st);
  k_norm<double><<<kRedBlocks, kBlock, 0, st>>>(5 * (int64_t)m.N, x, s.red, s.red_count, out_dev);
  HGKS_PROF_END(K_DOT, st);
}

void launch_apply_fd(const DevMesh &m, Scratch &s, const hgks_params &p, const double *Q, const double *G,
                     const double *x, const double *b, double *y, cudaStream_t st) {
  fd_apply<double, double>(m, s, p, Q, G, x, b, y, st);
}

void launch_density_l1(const DevMesh &m, Scratch &s, const double *R, double *out_dev, cudaStream_t st) {
  HGKS_PROF_BEGIN(K_NORM, st);
  k_density_l1<<<kRedBlocks, kBlock, 0, st>>>(m.N, R, m.inv_vol, s.red, s.red_count, out_dev);
  HGKS_PROF_END(K_NORM, st);
}

void launch_update(const DevMesh &m, const Scratch &s, double *Q, const double *dQ, double *G, const double *Gnew,
                   int ncomp_g, double relax, cudaStream_t st) {
  const int64_t n5 = 5 * (int64_t)m.N, ng = (int64_t)ncomp_g * m.N;
  HGKS_PROF_BEGIN(K_UPDATE, st);
  k_update<<<vec_grid(n5 + ng), kBlock, 0, st>>>(n5, ng, Q, dQ, G, Gnew, relax > 0.0 ? relax : 1.0,
                                                  reinterpret_cast<const int *>(s.hs + kHsStuck));
  HGKS_PROF_END(K_UPDATE, st);
}

// hs layout: H[(m+1) m] | beta | y[m] | lin residual estimates
hgks_status gmres_solve(const DevMesh &m, Scratch &s, const hgks_params &p, const double *rhs, double *dx,
                        hgks_step_info *info, cudaStream_t st, const double *Q, const double *G) {
  HGKS_RANGE("hgks gmres");
  cudaMemsetAsync(dx, 0, sizeof(double) * 5 * (size_t)m.N, st);
  if (p.jv_mode == 1) {
    if (!Q || !s.Qp) return HGKS_ERR_ARG;
    cudaMemsetAsync(s.hs + kHsNormQ + 3, 0, sizeof(double), st);
    launch_norm(m, s, Q, s.hs + kHsNormQ, st);
  }
  if (p.precision == HGKS_MIXED) gmres_t<float>(m, s, kbuf32(s), p, rhs, dx, st, Q, G);
  else if (p.jv_mode == 1 || !gmres_grid(m, s, p, rhs, dx, st)) gmres_t<double>(m, s, kbuf64(s), p, rhs, dx, st, Q, G);
  if (info) info->krylov_iters = p.restarts * p.krylov_dim;
  return HGKS_OK;
}

}  // namespace hgks
