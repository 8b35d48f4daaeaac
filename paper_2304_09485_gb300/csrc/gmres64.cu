// FP64 GMRES of one mesh with the assembled A: the Krylov products on vectors in the
// form of offdiag.cuh and modified Gram-Schmidt by blocks of basis vectors.
//
// Modified Gram-Schmidt by blocks. Algorithm 1 takes h_i = (w_i, v_i), w_{i+1} = w_i - h_i v_i
// one vector after the other. For the vectors v_c ... of a block with w_c given,
//   h_{c+q} = (w_c, v_{c+q}) - sum_{k<q} h_{c+k} (v_{c+k}, v_{c+q}),
// so one pass gives a whole block's coefficients if the inner products of its members are
// known. Those of a new v_{j+1} = w / ||w|| with the earlier members of its block come with
// ||w|| in the last pass of step j, whose subtracted vectors they are.
#include <algorithm>
#include "hgks_internal.h"
#include "fp64.cuh"
#include "offdiag.cuh"
#include "reduce.cuh"

namespace hgks {
namespace {

constexpr int kCell = 128;      // threads of the cell kernels
constexpr int kVec = 256;       // threads of the vector kernels
constexpr int kRed = 152 * 4;   // blocks of the vector kernels
constexpr int kBlk = 4;         // basis vectors of a block (separate launches)

// Reduction over the grid: the last block to arrive adds the blocks' partials in block
// order; true in that block, with the K sums in sh[0][.].
template <int K, int WARPS>
__device__ __forceinline__ bool grid_sums(double *v, double (*sh)[K], double *partials, unsigned *count) {
  __shared__ bool last;
  block_sums<K, WARPS>(v, sh);
  if (threadIdx.x < K) {
    partials[(size_t)threadIdx.x * gridDim.x + blockIdx.x] = sh[0][threadIdx.x];
    __threadfence();
  }
  __syncthreads();
  if (threadIdx.x == 0) last = atomicAdd(count, 1u) == gridDim.x - 1;
  __syncthreads();
  if (!last) return false;
  __threadfence();
  double t[K];
#pragma unroll
  for (int k = 0; k < K; k++) t[k] = 0.0;
  for (unsigned b = threadIdx.x; b < gridDim.x; b += blockDim.x)
#pragma unroll
    for (int k = 0; k < K; k++) t[k] += __ldcg(partials + (size_t)k * gridDim.x + b);
  block_sums<K, WARPS>(t, sh);
  if (threadIdx.x == 0) *count = 0u;
  return true;
}

// the coefficients of a block's vectors c, c + 1, ... from their inner products with w (one thread)
__device__ __forceinline__ void block_coef(int c, int nd, int ldg, int mk, const double *s, const double *G, double *Hj) {
  for (int q = 0; q < nd; q++) {
    double h = s[q];
    for (int k = 0; k < q; k++) h -= Hj[(c + k) * mk] * G[(c + q) * ldg + k];
    Hj[(c + q) * mk] = h;
  }
}

// The four kernels below run at the FP64 rate (2 DFMA per SM and clock) or near it. Against
// stored 5x5 blocks read with the vectors themselves, and Gram-Schmidt two vectors per pass,
// on 2,359,296 tetrahedra, per Krylov vector: products 0.41 + 0.41 + 0.47 -> 0.36 + 0.36 + 0.41 ms
// (856 -> 330 bytes a cell), scaling 0.037 -> 0.095 ms (it now forms z(v)), Gram-Schmidt of
// 60 vectors 34.6 -> 31.9 ms in 183 launches instead of 363; the step 174.0 -> 164.2 ms.

// v = w / h (v = 0 after a breakdown h == 0) and z(v)
__global__ void __launch_bounds__(kCell) k_scale_z(int N, const double *__restrict__ jv, const double *__restrict__ w,
                                                   const double *__restrict__ h, double *__restrict__ v,
                                                   double *__restrict__ zv) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const double hv = *h, ih = hv != 0.0 ? rcp(hv) : 0.0;
  double y[5], z[6];
#pragma unroll
  for (int c = 0; c < 5; c++) {
    y[c] = w[(size_t)c * N + i] * ih;
    v[(size_t)c * N + i] = y[c];
  }
  z_of(jv, N, i, y, z);
  z_store(zv, N, i, z);
}

// y = sign D^{-1} O x, both in z form
template <int NF>
__global__ void __launch_bounds__(kCell) k_zprod(int N, const int *__restrict__ cnb, const double *__restrict__ jv,
                                                 const double *__restrict__ dinv, double sign, const double *__restrict__ x,
                                                 double *__restrict__ y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  double acc[5] = {0, 0, 0, 0, 0}, z[6];
#pragma unroll
  for (int p = 0; p < NF; p++) {
    const int j = cnb[(size_t)p * N + i];
    if (j >= 0) z_product(jv, N, i, p, j, x, acc);
  }
  const double d = sign * dinv[i];
#pragma unroll
  for (int c = 0; c < 5; c++) acc[c] *= d;
  z_of(jv, N, i, acc, z);
  z_store(y, N, i, z);
}

// w = v + D^{-1} O x (x in z form), then the coefficients of the first ND basis vectors
template <int NF, int ND>
__global__ void __launch_bounds__(kCell) k_zlast(int N, const int *__restrict__ cnb, const double *__restrict__ jv,
                                                 const double *__restrict__ dinv, const double *__restrict__ x,
                                                 const double *__restrict__ v, double *__restrict__ w,
                                                 const double *__restrict__ V, int64_t vs, int mk,
                                                 const double *__restrict__ G, double *Hj, double *partials,
                                                 unsigned *count) {
  constexpr int K = ND == 3 ? 4 : ND;
  __shared__ double sh[kCell / 32][K];
  double s[K];
#pragma unroll
  for (int q = 0; q < K; q++) s[q] = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    double acc[5] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int p = 0; p < NF; p++) {
      const int j = cnb[(size_t)p * N + i];
      if (j >= 0) z_product(jv, N, i, p, j, x, acc);
    }
    const double d = dinv[i];
#pragma unroll
    for (int c = 0; c < 5; c++) {
      const size_t k = (size_t)c * N + i;
      acc[c] = fma(d, acc[c], v[k]);
      w[k] = acc[c];
#pragma unroll
      for (int q = 0; q < ND; q++) s[q] = fma(acc[c], V[(size_t)q * vs + k], s[q]);
    }
  }
  if (grid_sums<K, kCell / 32>(s, sh, partials, count) && threadIdx.x == 0) block_coef(0, ND, kBlk, mk, sh[0], G, Hj);
}

// One pass of the block Gram-Schmidt: w -= sum h_{a+q} v_{a+q} (q < NB, in order; NB = 0: the
// first block of a w that comes without its coefficients), then either the
// coefficients of the next block's ND vectors c, c + 1, ..., or (FIN) h_{j+1} = ||w|| and the
// products of v_{j+1} with the subtracted vectors when it joins their block. 16 bytes per
// vector, thread and step, every load of the step first. (2 + NB + ND) x 8 bytes and NB + ND
// FMAs per element: with NB = ND = 4 the FP64 rate (2 DFMA per SM and clock) and HBM are near balance.
template <int NB, int ND, bool FIN>
__global__ void __launch_bounds__(kVec) k_mgs_block(int64_t n, double *__restrict__ w, const double *__restrict__ V,
                                                    int64_t vs, int a, int c, int j, int mk, double *G, double *Hj,
                                                    double *partials, unsigned *count) {
  constexpr int NG = FIN ? (NB < kBlk ? NB : 0) : ND;   // products besides ||w||^2
  constexpr int NS = NG + (FIN ? 1 : 0), K = NS > 2 ? 4 : NS;
  __shared__ double sh[kVec / 32][K];
  double s[K], nh[NB > 0 ? NB : 1];
#pragma unroll
  for (int q = 0; q < K; q++) s[q] = 0.0;
#pragma unroll
  for (int q = 0; q < NB; q++) nh[q] = -Hj[(a + q) * mk];
  const int64_t nv = n / 2, stride = (int64_t)gridDim.x * blockDim.x;
  double2 *W = reinterpret_cast<double2 *>(w);
  auto vec = [&](int q) { return reinterpret_cast<const double2 *>(V + (size_t)q * vs); };
  for (int64_t k = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; k < nv; k += stride) {
    double2 wk = W[k], va[NB > 0 ? NB : 1], vc[FIN ? 1 : ND];
#pragma unroll
    for (int q = 0; q < NB; q++) va[q] = vec(a + q)[k];
    if constexpr (!FIN)
#pragma unroll
      for (int q = 0; q < ND; q++) vc[q] = vec(c + q)[k];
#pragma unroll
    for (int q = 0; q < NB; q++) {
      wk.x = fma(nh[q], va[q].x, wk.x);
      wk.y = fma(nh[q], va[q].y, wk.y);
    }
    if constexpr (FIN) s[NG] = fma(wk.x, wk.x, fma(wk.y, wk.y, s[NG]));
#pragma unroll
    for (int q = 0; q < NG; q++) {
      const double2 d = FIN ? va[q] : vc[q];
      s[q] = fma(wk.x, d.x, fma(wk.y, d.y, s[q]));
    }
    if constexpr (NB > 0) W[k] = wk;
  }
  if ((n & 1) && blockIdx.x == 0 && threadIdx.x == 0) {
    const int64_t k = n - 1;
    double wk = w[k];
#pragma unroll
    for (int q = 0; q < NB; q++) wk = fma(nh[q], V[(size_t)(a + q) * vs + k], wk);
    w[k] = wk;
    if constexpr (FIN) s[NG] = fma(wk, wk, s[NG]);
#pragma unroll
    for (int q = 0; q < NG; q++) s[q] = fma(wk, V[(size_t)((FIN ? a : c) + q) * vs + k], s[q]);
  }
  if (grid_sums<K, kVec / 32>(s, sh, partials, count) && threadIdx.x == 0) {
    if (FIN) {
      const double nrm = sqrt(sh[0][NG]);
      Hj[(j + 1) * mk] = nrm;
      for (int q = 0; q < NG; q++) G[(j + 1) * kBlk + q] = nrm > 0.0 ? sh[0][q] / nrm : 0.0;
    } else {
      block_coef(c, ND, kBlk, mk, sh[0], G, Hj);
    }
  }
}

template <int NB>
void mgs_pass(cudaStream_t st, int64_t n, double *w, const double *V, int64_t vs, int a, int c, int nd, int j, int mk,
              double *G, double *Hj, double *part, unsigned *cnt) {
#define HGKS_MGS(ND, FIN) k_mgs_block<NB, ND, FIN><<<kRed, kVec, 0, st>>>(n, w, V, vs, a, c, j, mk, G, Hj, part, cnt)
  if (nd == 0) {
    if constexpr (NB > 0) HGKS_MGS(1, true);
  } else if constexpr (NB == kBlk || NB == 0) {   // only a whole block is followed by another
    if (nd == 1) HGKS_MGS(1, false);
    else if (nd == 2) HGKS_MGS(2, false);
    else if (nd == 3) HGKS_MGS(3, false);
    else HGKS_MGS(4, false);
  }
#undef HGKS_MGS
}

template <int NF>
void zlast(cudaStream_t st, const DevMesh &m, const Scratch &s, const double *x, const double *v, double *w, int nd, int mk,
           double *Hj) {
  const unsigned g = std::min(grid_for(m.N, kCell), 152u * 8u);
#define HGKS_ZL(ND)                                                                                               \
  k_zlast<NF, ND><<<g, kCell, 0, st>>>(m.N, m.cnb, s.jv64, s.dinv, x, v, w, s.V, s.vstride, mk, s.gram, Hj, s.red, \
                                       s.red_count)
  if (nd == 1) HGKS_ZL(1);
  else if (nd == 2) HGKS_ZL(2);
  else if (nd == 3) HGKS_ZL(3);
  else HGKS_ZL(4);
#undef HGKS_ZL
}

}  // namespace

void launch_scale_z(const DevMesh &m, const Scratch &s, const double *w, const double *h, double *v, double *zv,
                    cudaStream_t st) {
  HGKS_PROF_BEGIN(K_SCALE, st);
  k_scale_z<<<grid_for(m.N, kCell), kCell, 0, st>>>(m.N, s.jv64, w, h, v, zv);
  HGKS_PROF_END(K_SCALE, st);
}

void launch_neumann_z(const DevMesh &m, const Scratch &s, int sweeps, const double *v, double *w, int j, int mk, double *Hj,
                      cudaStream_t st) {
  // s.z[0] holds z(v); E^sweeps v with the sign in its first product, then w = v + E z
  const unsigned g = grid_for(m.N, kCell);
  int src = 0;
  for (int q = 0; q < sweeps; q++, src ^= 1) {
    const double sign = q == 0 && sweeps % 2 == 1 ? -1.0 : 1.0;
    HGKS_PROF_BEGIN(K_JACOBI, st);
    if (m.hex) k_zprod<HexShape::NF><<<g, kCell, 0, st>>>(m.N, m.cnb, s.jv64, s.dinv, sign, s.z[src], s.z[src ^ 1]);
    else k_zprod<TetShape::NF><<<g, kCell, 0, st>>>(m.N, m.cnb, s.jv64, s.dinv, sign, s.z[src], s.z[src ^ 1]);
    HGKS_PROF_END(K_JACOBI, st);
  }
  const int nd = std::min(kBlk, j + 1);
  HGKS_PROF_BEGIN(K_SPMV, st);
  if (m.hex) zlast<HexShape::NF>(st, m, s, s.z[src], v, w, nd, mk, Hj);
  else zlast<TetShape::NF>(st, m, s, s.z[src], v, w, nd, mk, Hj);
  HGKS_PROF_END(K_SPMV, st);
}

// have_first: the first block's coefficients came with w
void launch_mgs_blocks(const Scratch &s, int64_t n, double *w, int j, int mk, double *Hj, bool have_first,
                       cudaStream_t st) {
  if (!have_first) {
    HGKS_PROF_BEGIN(K_DOT, st);
    mgs_pass<0>(st, n, w, s.V, s.vstride, 0, 0, std::min(kBlk, j + 1), j, mk, s.gram, Hj, s.red, s.red_count);
    HGKS_PROF_END(K_DOT, st);
  }
  // subtract a block and take the next one's coefficients
  for (int a = 0; a <= j; a += kBlk) {
    const int nb = std::min(kBlk, j + 1 - a), c = a + nb, nd = std::min(kBlk, j + 1 - c);
    HGKS_PROF_BEGIN(K_DOT, st);
    if (nb == 1) mgs_pass<1>(st, n, w, s.V, s.vstride, a, c, nd, j, mk, s.gram, Hj, s.red, s.red_count);
    else if (nb == 2) mgs_pass<2>(st, n, w, s.V, s.vstride, a, c, nd, j, mk, s.gram, Hj, s.red, s.red_count);
    else if (nb == 3) mgs_pass<3>(st, n, w, s.V, s.vstride, a, c, nd, j, mk, s.gram, Hj, s.red, s.red_count);
    else mgs_pass<4>(st, n, w, s.V, s.vstride, a, c, nd, j, mk, s.gram, Hj, s.red, s.red_count);
    HGKS_PROF_END(K_DOT, st);
  }
}

}  // namespace hgks
