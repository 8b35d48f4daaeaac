// FP64 GMRES of one mesh with the assembled A: the Krylov products on vectors in the
// form of offdiag.cuh, modified Gram-Schmidt by blocks of basis vectors, and, for
// meshes small enough, all restart cycles in one cooperative launch.
//
// Modified Gram-Schmidt by blocks. Algorithm 1 takes h_i = (w_i, v_i), w_{i+1} = w_i - h_i v_i
// one vector after the other. For the vectors v_c ... of a block with w_c given,
//   h_{c+q} = (w_c, v_{c+q}) - sum_{k<q} h_{c+k} (v_{c+k}, v_{c+q}),
// so one pass gives a whole block's coefficients if the inner products of its members are
// known. Those of a new v_{j+1} = w / ||w|| with the earlier members of its block come with
// ||w|| in the last pass of step j, whose subtracted vectors they are.
#include <algorithm>
#include <cmath>
#include "hgks_internal.h"
#include "fp64.cuh"
#include "offdiag.cuh"
#include "reduce.cuh"

namespace hgks {
namespace {

constexpr int kCell = 128;      // threads of the cell kernels
constexpr int kVec = 256;       // threads of the vector kernels
constexpr int kRed = 152 * 3;   // blocks of the vector kernels: those resident at 80 registers
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
  const Units un = units();
  const double hv = *h, ih = hv != 0.0 ? rcp(hv) : 0.0;
  double y[5], z[6];
#pragma unroll
  for (int c = 0; c < 5; c++) {
    y[c] = un.mul(w[(size_t)c * N + i], ih);
    v[(size_t)c * N + i] = y[c];
  }
  z_of(un, cell_prim(jv, N, i), y, z);
  z_store(zv, N, i, z);
}

// z(x), or z(D^{-1} x) with dinv
__global__ void __launch_bounds__(kCell) k_z(int N, const double *__restrict__ jv, const double *__restrict__ dinv,
                                             const double *__restrict__ x, double *__restrict__ zv) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const Units un = units();
  double y[5], z[6];
#pragma unroll
  for (int c = 0; c < 5; c++) y[c] = x[(size_t)c * N + i];
  if (dinv) {
    const double d = dinv[i];
#pragma unroll
    for (int c = 0; c < 5; c++) y[c] = un.mul(y[c], d);
  }
  z_of(un, cell_prim(jv, N, i), y, z);
  z_store(zv, N, i, z);
}

// One product with the off-diagonal part of A, x in z form:
//   kE      y = sign D^{-1} O x, in z form
//   kSweep  y = D^{-1} (b - O x), in z form;   kLast the same, y as it is
//   kSpmv   y = d x5 + O x, or b - that with b (x5: the vector of x)
enum { kE, kSweep, kLast, kSpmv };
template <int NF, int Mode>
__global__ void __launch_bounds__(kCell) k_zprod(int N, const int *__restrict__ cnb, const double *__restrict__ jv,
                                                 const double *__restrict__ dd, double sign, const double *__restrict__ b,
                                                 const double *__restrict__ x5, const double *__restrict__ x,
                                                 double *__restrict__ y) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= N) return;
  const Units un = units();
  double acc[5] = {0, 0, 0, 0, 0};
#pragma unroll
  for (int p = 0; p < NF; p++) {
    const int j = cnb[(size_t)p * N + i];
    if (j >= 0) z_product(un, jv, N, i, p, j, x, acc);
  }
  const double d = Mode == kE ? sign * dd[i] : dd[i];    // D^{-1}, or D for kSpmv
#pragma unroll
  for (int c = 0; c < 5; c++) {
    const size_t k = (size_t)c * N + i;
    if (Mode == kE) acc[c] = un.mul(acc[c], d);
    else if (Mode != kSpmv) acc[c] = un.mul(d, un.sub(b[k], acc[c]));
    else acc[c] = b ? b[k] - fma(d, x5[k], acc[c]) : fma(d, x5[k], acc[c]);
    if (Mode == kLast || Mode == kSpmv) y[k] = acc[c];
  }
  if (Mode == kE || Mode == kSweep) {
    double z[6];
    z_of(un, cell_prim(jv, N, i), acc, z);
    z_store(y, N, i, z);
  }
}
template <int Mode>
void zprod(cudaStream_t st, const DevMesh &m, const Scratch &s, const double *dd, double sign, const double *b,
           const double *x5, const double *x, double *y) {
  const unsigned g = grid_for(m.N, kCell);
  if (m.hex) k_zprod<HexShape::NF, Mode><<<g, kCell, 0, st>>>(m.N, m.cnb, s.jv64, dd, sign, b, x5, x, y);
  else k_zprod<TetShape::NF, Mode><<<g, kCell, 0, st>>>(m.N, m.cnb, s.jv64, dd, sign, b, x5, x, y);
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
  const Units un = units();
  double s[K];
#pragma unroll
  for (int q = 0; q < K; q++) s[q] = 0.0;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < N; i += gridDim.x * blockDim.x) {
    double acc[5] = {0, 0, 0, 0, 0};
#pragma unroll
    for (int p = 0; p < NF; p++) {
      const int j = cnb[(size_t)p * N + i];
      if (j >= 0) z_product(un, jv, N, i, p, j, x, acc);
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
__global__ void __launch_bounds__(kVec, 3) k_mgs_block(int64_t n, double *__restrict__ w, const double *__restrict__ V,
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


// ---- all restart cycles in one cooperative launch ----
// A cycle in separate launches is a chain of some 200 dependent ones, 4 to 9 microseconds each on
// a small mesh: launch gaps, block scheduling, tails of the reductions and of the FP64-bound
// kernels. Here one block per SM keeps its cells for the whole solve: w stays in registers (or
// shared memory), the basis is only touched by the thread that wrote it, and blocks meet at a
// grid barrier (1.1 us) where neighbours' vectors or sums are needed: one per product, one per
// block of kPB basis vectors, one for the norm (z(w) is written before it, unscaled, so the next
// product starts right after). Every block adds the blocks' partial sums itself, in the same
// order, so all of them hold the same H; an extra warp turns its columns into R while the others
// form the next product.
// An SM sub-partition takes 64 clocks per FP64 warp instruction, however few lanes are active and
// also when its predicate is false. So below one warp of cells per sub-partition LPC = 2 or 4
// lanes share a cell (its faces in the products, its components elsewhere), and the loops over a
// partial block of basis vectors have exact trip counts.
// Per step outside the residual, separate launches against this one: 3,072 tetrahedra 1.40 /
// 0.68 ms, 48,000 2.16 / 1.46, 124,416 (20 vectors) 8.31 / 7.36, 110,592 hexahedra 4.15 / 3.32.
constexpr int kPT = 384;        // threads with cells, three warps per SM sub-partition (and a warp for the rotations)
constexpr int kPB = 8;          // basis vectors of a block (one grid barrier each)
constexpr int kPG = 160;        // blocks at most (the sums read one partial per block)
constexpr int kPMax = 64;       // Krylov vectors at most

struct GridSolve {
  int N, C;                     // cells, cells per block
  const int *cnb;
  const double *jv, *dval, *dinv, *rhs;
  double *dx, *b, *V, *z0, *z1, *part, *lres;
  int64_t vs;
  unsigned *bar;                // arrivals, 0 at launch
  int *err;                     // set to 1 by a barrier that gave up
  unsigned want, polls;         // arrivals that open a barrier, polls before it gives up
  int mk, restarts, sweeps;
};

// shared memory of a block
struct GridShared {
  double H[(kPMax + 1) * kPMax], G[(kPMax + 1) * kPB], cs[kPMax], sn[kPMax], gv[kPMax + 1], y[kPMax];
  double sh[kPT / 32][kPB], sum[kPB], nrm, inrm;
  int used, dead;
};

// The arrival of every block at step `gen` (1, 2, ...). false: given up, the block returns.
__device__ __forceinline__ bool grid_barrier(const GridSolve &a, GridShared &S, unsigned &gen) {
  const unsigned want = ++gen * a.want;
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(a.bar) : "memory");
    unsigned seen, spin = 0;
    do {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(a.bar) : "memory");
    } while (!arrived(seen, want) && ++spin < a.polls);
    if (!arrived(seen, want)) {
      S.dead = 1;
      atomicExch(a.err, 1);
    }
  }
  __syncthreads();
  return S.dead == 0;
}

// the sums over the grid of the first `ns` of kPB values per thread, in S.sum (all threads);
// S.nrm and S.inrm: the root of sum `norm` and its reciprocal (0 for 0)
__device__ __forceinline__ bool grid_total(const GridSolve &a, GridShared &S, unsigned &gen, double *v, int ns, int nwarps,
                                           int norm) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  if (warp < nwarps) {
    const double t = warp_sums<kPB>(v);
    if (lane % (32 / kPB) == 0) S.sh[warp][lane / (32 / kPB)] = t;
  }
  __syncthreads();
  double *part = a.part + (gen & 1) * (kPB * kPG);     // two sets: a slow block may still read the last one
  if (threadIdx.x < ns) {
    double s = S.sh[0][threadIdx.x];
    for (int w = 1; w < nwarps; w++) s += S.sh[w][threadIdx.x];
    part[threadIdx.x * kPG + blockIdx.x] = s;
  }
  if (!grid_barrier(a, S, gen)) return false;
  if (warp < ns) {
    double t[5], s;
#pragma unroll
    for (int k = 0; k < 5; k++) t[k] = lane + 32 * k < gridDim.x ? __ldcg(part + warp * kPG + lane + 32 * k) : 0.0;
    s = t[0];
#pragma unroll
    for (int k = 1; k < 5; k++)
      if (32 * k < gridDim.x) s += t[k];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      S.sum[warp] = s;
      if (warp == norm) {
        const double r = sqrt64(s);
        S.nrm = r;
        S.inrm = r != 0.0 ? rcp(r) : 0.0;
      }
    }
  }
  __syncthreads();
  return true;
}

// column j of H: the earlier rotations, its own, and the right-hand side (one thread; as givens_lsq)
__device__ __forceinline__ void givens_column(GridShared &S, int mk, int j) {
  if (S.used < j) return;                               // a breakdown ended the basis before
  double h1 = S.H[j];
  for (int i = 0; i < j; i++) {
    const double h2 = S.H[(i + 1) * mk + j];
    S.H[i * mk + j] = S.cs[i] * h1 + S.sn[i] * h2;
    h1 = S.cs[i] * h2 - S.sn[i] * h1;
  }
  const double b = S.H[(j + 1) * mk + j], r = rsqrt64(h1 * h1 + b * b), c = h1 * r, s = b * r;
  S.cs[j] = c;
  S.sn[j] = s;
  S.H[j * mk + j] = c * h1 + s * b;
  const double g1 = S.gv[j];
  S.gv[j] = c * g1;
  S.gv[j + 1] = -s * g1;
  S.used = b == 0.0 ? -(j + 1) : j + 1;                 // negative: the basis ends here
}

// f(n) with the count as a constant, for n in 1..kPB: a predicated FP64 instruction costs as much as
// an executed one, so the loops over a partial block have exact trip counts
template <int n> struct Count { static constexpr int value = n; };
template <class F>
__device__ __forceinline__ void with_count(int n, F f) {
  switch (n) {
    case 1: f(Count<1>{}); break;
    case 2: f(Count<2>{}); break;
    case 3: f(Count<3>{}); break;
    case 4: f(Count<4>{}); break;
    case 5: f(Count<5>{}); break;
    case 6: f(Count<6>{}); break;
    case 7: f(Count<7>{}); break;
    case 8: f(Count<8>{}); break;
    default: break;
  }
}

// the sums over a cell's LPC lanes of acc[5], each lane keeping its components l, l + LPC, ...
template <int LPC>
__device__ __forceinline__ void lane_components(const double *acc, double *own) {
  const int l = threadIdx.x % LPC;
  auto swap = [&](bool up, double lo, double hi, int o) {   // up lanes keep hi, the others lo
    return (up ? hi : lo) + __shfl_xor_sync(0xffffffffu, up ? lo : hi, o);
  };
  if constexpr (LPC == 1) {
#pragma unroll
    for (int c = 0; c < 5; c++) own[c] = acc[c];
  } else if constexpr (LPC == 2) {
    own[0] = swap(l, acc[0], acc[1], 1);
    own[1] = swap(l, acc[2], acc[3], 1);
    own[2] = swap(l, acc[4], 0.0, 1);
  } else {
    const double t0 = swap(l >> 1, acc[0], acc[2], 2), t1 = swap(l >> 1, acc[1], acc[3], 2), t2 = swap(l >> 1, acc[4], 0.0, 2);
    own[0] = swap(l & 1, t0, t1, 1);
    own[1] = swap(l & 1, t2, 0.0, 1);
  }
}

// ONE: a thread has one cell at most (and LPC lanes share it), with what it reads of it in
// registers; otherwise its cells' w live in shared memory and it goes through them in turn.
template <int NF, int LPC, bool ONE>
__global__ void __launch_bounds__(kPT + 32, 1) k_gmres_grid(GridSolve a) {
  constexpr int CP = (5 + LPC - 1) / LPC;               // components per lane: l, l + LPC, ...
  constexpr int LF = (NF + LPC - 1) / LPC;              // faces per lane, alike
  static_assert(ONE || LPC == 1, "several cells per thread: whole cells");
  extern __shared__ __align__(16) unsigned char smem[];
  GridShared &S = *reinterpret_cast<GridShared *>(smem);
  double *ws = reinterpret_cast<double *>(smem + sizeof(GridShared));   // !ONE: [5][C]
  const int tid = threadIdx.x, mk = a.mk, l = tid % LPC;
  const Units un = units();
  const size_t N = a.N;
  const int c0 = blockIdx.x * a.C, nc = min(a.C, a.N - c0);             // this block's cells (nc <= 0: none)
  const int nwarps = min(kPT / 32, (a.C * LPC + 31) / 32);
  const bool rot = tid == kPT;                          // the thread of the rotations
  // a load after a barrier goes to L2: keep what every phase reads of the cell
  const int own_cell = tid < kPT && tid / LPC < nc ? c0 + tid / LPC : -1;
  int own_nb[LF];
  CellPrim own_prim = {0, 0, 0, 0, 0, 0};
  double own_w[CP], own_dinv = 0.0;
#pragma unroll
  for (int k = 0; k < CP; k++) own_w[k] = 0.0;
  if (ONE) {
#pragma unroll
    for (int q = 0; q < LF; q++)
      own_nb[q] = own_cell >= 0 && q * LPC + l < NF ? a.cnb[(q * LPC + l) * N + own_cell] : -1;
    if (own_cell >= 0) {
      own_prim = cell_prim(a.jv, N, own_cell);
      own_dinv = a.dinv[own_cell];
    }
  }
  // f(i, w) for every cell i of the thread and its components of w (ONE: also for none, i = -1,
  // so that all lanes of a warp reach the exchanges inside)
  auto each = [&](auto f) {
    if constexpr (ONE) {
      f(own_cell, own_w);
    } else {
      for (int r = tid; r < nc && tid < kPT; r += kPT) {
        double w[CP];
#pragma unroll
        for (int k = 0; k < CP; k++) w[k] = ws[k * a.C + r];
        f(c0 + r, w);
#pragma unroll
        for (int k = 0; k < CP; k++) ws[k * a.C + r] = w[k];
      }
    }
  };
  // component k of a lane: whether it has one, and its element
  auto mine = [&](int i, int k) { return (!ONE || i >= 0) && l + LPC * k < 5; };
  auto at = [&](int i, int k) { return (l + LPC * k) * N + i; };
  auto dinv = [&](int i) { return ONE ? own_dinv : a.dinv[i]; };
  // this lane's components of sum_p A_ip x_p
  auto off = [&](int i, const double *z, double *acc) {
    double t[5] = {0, 0, 0, 0, 0};
    int nb[LF];
#pragma unroll
    for (int q = 0; q < LF; q++) nb[q] = ONE ? own_nb[q] : a.cnb[q * N + i];
#pragma unroll
    for (int q = 0; q < LF; q++)
      if (nb[q] >= 0) z_product(un, a.jv, N, i, q * LPC + l, nb[q], z, t);
    lane_components<LPC>(t, acc);
  };
  // z form of a cell's vector from its lanes' components
  auto put_z = [&](double *z, int i, const double *x) {
    double y[5], t[6];
#pragma unroll
    for (int c = 0; c < 5; c++)
      y[c] = LPC == 1 ? x[c] : __shfl_sync(0xffffffffu, x[c / LPC], (tid & 31 & ~(LPC - 1)) | (c % LPC));
    if (ONE && i < 0) return;
    z_of(un, ONE ? own_prim : cell_prim(a.jv, N, i), y, t);
#pragma unroll
    for (int k = 0; k < 6; k++)
      if (LPC == 1 || k % LPC == l) z[k * N + i] = t[k];
  };
  unsigned gen = 0;
  if (tid == 0) S.dead = 0;
  double *zs = a.z0, *zd = a.z1;                        // the vector to multiply, and the other buffer
  auto flip = [&] { double *t = zs; zs = zd; zd = t; };
  for (int it = 0; it < a.restarts; it++) {
    // w = P^{-1} (rhs - A dx), b kept for the sweeps
    if (it > 0) {
      each([&](int i, double *) {
        double x[CP];
#pragma unroll
        for (int k = 0; k < CP; k++) x[k] = mine(i, k) ? a.dx[at(i, k)] : 0.0;
        put_z(zs, i, x);
      });
      if (!grid_barrier(a, S, gen)) return;
    }
    each([&](int i, double *w) {
      double acc[CP];
      if (it > 0) off(i, zs, acc);
#pragma unroll
      for (int k = 0; k < CP; k++)
        if (mine(i, k)) {
          double b = a.rhs[at(i, k)];
          if (it > 0) b -= fma(a.dval[i], a.dx[at(i, k)], acc[k]);
          else a.dx[at(i, k)] = 0.0;
          a.b[at(i, k)] = b;
          w[k] = dinv(i) * b;
        }
      put_z(zd, i, w);
    });
    for (int q = 0; q < a.sweeps; q++) {
      if (!grid_barrier(a, S, gen)) return;
      flip();
      each([&](int i, double *w) {
        double acc[CP];
        off(i, zs, acc);
#pragma unroll
        for (int k = 0; k < CP; k++)
          if (mine(i, k)) w[k] = dinv(i) * (a.b[at(i, k)] - acc[k]);
        put_z(zd, i, w);
      });
    }
    double s[kPB];
#pragma unroll
    for (int q = 0; q < kPB; q++) s[q] = 0.0;
    each([&](int i, double *w) {
#pragma unroll
      for (int k = 0; k < CP; k++)
        if (mine(i, k)) s[0] = fma(w[k], w[k], s[0]);
    });
    if (!grid_total(a, S, gen, s, 1, nwarps, 0)) return;
    flip();                                             // zs = z(w), unscaled
    const double beta = S.nrm;
    double ih = S.inrm;
    if (rot) {
      S.used = 0;
      S.gv[0] = beta;
      if (it == 0 && blockIdx.x == 0) a.lres[0] = beta;
    }
    for (int j = 0; j < mk; j++) {
      // v_j = w / ||w||; w = v_j + E (-E)^sweeps v_j from z(w) and the scale
      if (rot && j > 0) givens_column(S, mk, j - 1);
      each([&](int i, double *w) {
#pragma unroll
        for (int k = 0; k < CP; k++)
          if (mine(i, k)) {
            w[k] = un.mul(w[k], ih);
            a.V[(size_t)j * a.vs + at(i, k)] = w[k];
          }
      });
      double sc = ih;
      for (int q = 0; q < a.sweeps; q++) {
        if (q == 0 && a.sweeps % 2 == 1) sc = -sc;
        each([&](int i, double *) {
          double acc[CP];
          off(i, zs, acc);
          const double d = q == 0 ? sc * dinv(i) : dinv(i);
#pragma unroll
          for (int k = 0; k < CP; k++) acc[k] = un.mul(acc[k], d);
          put_z(zd, i, acc);
        });
        if (!grid_barrier(a, S, gen)) return;
        flip();
      }
      each([&](int i, double *w) {
        double acc[CP];
        off(i, zs, acc);
        const double d = a.sweeps == 0 ? sc * dinv(i) : dinv(i);
#pragma unroll
        for (int k = 0; k < CP; k++)
          if (mine(i, k)) w[k] = fma(d, acc[k], w[k]);
      });
      for (int p = 0;; p += kPB) {                      // p: the block whose coefficients are taken
        const bool fin = p > j;
        const int ns = p == 0 ? 0 : min(kPB, j + 1 - (p - kPB)), nd = fin ? 0 : min(kPB, j + 1 - p);
        const bool gram = fin && ns < kPB;              // v_{j+1} joins the last block
#pragma unroll
        for (int q = 0; q < kPB; q++) s[q] = 0.0;
        with_count(ns, [&](auto count) {                // subtract the previous block
          constexpr int n = decltype(count)::value;
          const double *h = S.H + (p - kPB) * mk + j;
          each([&](int i, double *w) {
#pragma unroll
            for (int k = 0; k < CP; k++) {
              if (!mine(i, k)) continue;
              const double *v = a.V + (int64_t)(p - kPB) * a.vs + at(i, k);
              double t[n], x = w[k];
#pragma unroll
              for (int q = 0; q < n; q++) t[q] = v[q * a.vs];
#pragma unroll
              for (int q = 0; q < n; q++) x = fma(-h[q * mk], t[q], x);
              w[k] = x;
              if constexpr (n < kPB)
                if (gram)
#pragma unroll
                  for (int q = 0; q < n; q++) s[q] = fma(x, t[q], s[q]);
            }
          });
        });
        with_count(nd, [&](auto count) {                // the next one's products
          constexpr int n = decltype(count)::value;
          each([&](int i, double *w) {
#pragma unroll
            for (int k = 0; k < CP; k++) {
              if (!mine(i, k)) continue;
              const double *v = a.V + (int64_t)p * a.vs + at(i, k);
#pragma unroll
              for (int q = 0; q < n; q++) s[q] = fma(w[k], v[q * a.vs], s[q]);
            }
          });
        });
        if (fin)
          each([&](int i, double *w) {
#pragma unroll
            for (int k = 0; k < CP; k++)
              if (mine(i, k)) s[kPB - 1] = fma(w[k], w[k], s[kPB - 1]);
            put_z(zd, i, w);
          });
        if (!grid_total(a, S, gen, s, fin ? kPB : nd, nwarps, fin ? kPB - 1 : -1)) return;
        if (fin) {
          ih = S.inrm;
          if (tid >= kPT) {                             // the warp that reads column j next
            if (rot) S.H[(j + 1) * mk + j] = S.nrm;
            if (gram && tid - kPT < ns) S.G[(j + 1) * kPB + tid - kPT] = S.sum[tid - kPT] * ih;
          }
          break;
        }
        if (tid < 32) {                                 // h by forward substitution, a lane per coefficient
          double h = tid < nd ? S.sum[tid] : 0.0;
          for (int k = 0; k < nd - 1; k++) {
            const double hk = __shfl_sync(0xffffffffu, h, k);
            if (tid > k && tid < nd) h = fma(-hk, S.G[(p + tid) * kPB + k], h);
          }
          if (tid < nd) S.H[(p + tid) * mk + j] = h;
        }
        __syncthreads();
      }
      flip();
    }
    __syncthreads();
    if (tid >= kPT) {                                   // the last column, then back substitution by the warp
      const int lane = tid - kPT;
      if (lane == 0) givens_column(S, mk, mk - 1);
      __syncwarp();
      const int used = beta == 0.0 ? 0 : abs(S.used);
      double g0 = lane < used ? S.gv[lane] : 0.0, g1 = lane + 32 < used ? S.gv[lane + 32] : 0.0;
      double y0 = 0.0, y1 = 0.0;
      for (int k = used - 1; k >= 0; k--) {
        const double yk = __shfl_sync(0xffffffffu, k < 32 ? g0 : g1, k & 31) * rcp(S.H[k * mk + k]);
        if (lane < k) g0 = fma(-S.H[lane * mk + k], yk, g0);
        if (lane + 32 < k) g1 = fma(-S.H[(lane + 32) * mk + k], yk, g1);
        if (lane == k) y0 = yk;
        if (lane + 32 == k) y1 = yk;
      }
      if (lane < mk) S.y[lane] = y0;
      if (lane + 32 < mk) S.y[lane + 32] = y1;
      if (lane == 0 && blockIdx.x == 0) a.lres[1] = beta == 0.0 ? 0.0 : fabs(S.gv[used]);
    }
    __syncthreads();
    // dx += sum_q y_q v_q
    each([&](int i, double *) {
#pragma unroll
      for (int k = 0; k < CP; k++)
        if (mine(i, k)) {
          const double *v = a.V + at(i, k);
          double x = a.dx[at(i, k)];
#pragma unroll 8
          for (int q = 0; q < mk; q++) x = fma(S.y[q], v[(size_t)q * a.vs], x);
          a.dx[at(i, k)] = x;
        }
    });
  }
}

}  // namespace

void launch_scale_z(const DevMesh &m, const Scratch &s, const double *w, const double *h, double *v, double *zv,
                    cudaStream_t st) {
  HGKS_PROF_BEGIN(K_SCALE, st);
  k_scale_z<<<grid_for(m.N, kCell), kCell, 0, st>>>(m.N, s.jv64, w, h, v, zv);
  HGKS_PROF_END(K_SCALE, st);
}

// y = A x, or b - A x
void launch_apply_A(const DevMesh &m, const Scratch &s, const double *b, const double *x, double *y, cudaStream_t st) {
  HGKS_PROF_BEGIN(K_SCALE, st);
  k_z<<<grid_for(m.N, kCell), kCell, 0, st>>>(m.N, s.jv64, nullptr, x, s.z[0]);
  HGKS_PROF_END(K_SCALE, st);
  HGKS_PROF_BEGIN(K_SPMV, st);
  zprod<kSpmv>(st, m, s, s.dval, 1.0, b, x, s.z[0], y);
  HGKS_PROF_END(K_SPMV, st);
}

// x = P^{-1} b (Eq. (precond)), at least one sweep
void launch_sweeps_z(const DevMesh &m, const Scratch &s, int sweeps, const double *b, double *x, cudaStream_t st) {
  HGKS_PROF_BEGIN(K_SCALE, st);
  k_z<<<grid_for(m.N, kCell), kCell, 0, st>>>(m.N, s.jv64, s.dinv, b, s.z[0]);
  HGKS_PROF_END(K_SCALE, st);
  for (int q = 1; q <= sweeps; q++) {
    HGKS_PROF_BEGIN(K_JACOBI, st);
    if (q < sweeps) zprod<kSweep>(st, m, s, s.dinv, 1.0, b, nullptr, s.z[(q - 1) & 1], s.z[q & 1]);
    else zprod<kLast>(st, m, s, s.dinv, 1.0, b, nullptr, s.z[(q - 1) & 1], x);
    HGKS_PROF_END(K_JACOBI, st);
  }
}

void launch_neumann_z(const DevMesh &m, const Scratch &s, int sweeps, const double *v, double *w, int j, int mk, double *Hj,
                      cudaStream_t st) {
  // s.z[0] holds z(v); E^sweeps v with the sign in its first product, then w = v + E z
  int src = 0;
  for (int q = 0; q < sweeps; q++, src ^= 1) {
    const double sign = q == 0 && sweeps % 2 == 1 ? -1.0 : 1.0;
    HGKS_PROF_BEGIN(K_JACOBI, st);
    zprod<kE>(st, m, s, s.dinv, sign, nullptr, nullptr, s.z[src], s.z[src ^ 1]);
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

namespace {
template <int NF>
const void *grid_kernel(int lpc, bool one) {
  if (lpc == 4) return (const void *)k_gmres_grid<NF, 4, true>;
  if (lpc == 2) return (const void *)k_gmres_grid<NF, 2, true>;
  return one ? (const void *)k_gmres_grid<NF, 1, true> : (const void *)k_gmres_grid<NF, 1, false>;
}
}  // namespace

// All restart cycles in one cooperative launch, for meshes small enough. false: not launched
// (mesh too large, or not on this device), which depends on the mesh and the device alone; a launch
// that fails all the same is an error like any other launch's.
bool gmres_grid(const DevMesh &m, Scratch &s, const hgks_params &p, const double *rhs, double *dx, cudaStream_t st) {
  int dev = 0, sms = 0, coop = 0, shm_max = 0;
  if (m.N > s.grid_cells || p.restarts < 1 || p.krylov_dim > kPMax || cudaGetDevice(&dev) != cudaSuccess) return false;
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  cudaDeviceGetAttribute(&coop, cudaDevAttrCooperativeLaunch, dev);
  cudaDeviceGetAttribute(&shm_max, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (!coop || sms < 1) return false;
  // Four lanes a cell and one warp per SM sub-partition are 32 cells a block; a small mesh fills its
  // SMs that far before it takes another, since a block holds its SM for the whole solve and other
  // streams' meshes wait for a free one. Steps of 1,296 cells, one stream / eight: 845 / 697 us with
  // eight cells a block, 854 / 235 with 32 (separate launches 2,352 / 641); 3,072 cells 877 / 737
  // and 882 / 647 (2,457 / 741).
  const int blocks = std::min({sms, kPG, (m.N + 31) / 32}), C = (m.N + blocks - 1) / blocks;
  const int lpc = C <= 32 ? 4 : C <= 64 ? 2 : 1;        // one warp per SM sub-partition at most
  const bool one = C <= kPT;
  const size_t shm = sizeof(GridShared) + (one ? 0 : sizeof(double) * 5 * C);
  const void *fn = m.hex ? grid_kernel<HexShape::NF>(lpc, one) : grid_kernel<TetShape::NF>(lpc, one);
  // The limit is the kernel's, for all threads of the process: always the device's largest, not this
  // mesh's, which another thread's smaller mesh would lower before the launch.
  const bool clean = cudaPeekAtLastError() == cudaSuccess;
  int fit = 0;
  if (shm > (size_t)shm_max ||
      cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, shm_max) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&fit, fn, kPT + 32, shm) != cudaSuccess || fit < 1) {
    if (clean) cudaGetLastError();                      // an error of an earlier launch stays
    return false;
  }
  cudaMemsetAsync(s.red_count + 2, 0, sizeof(unsigned), st);
  GridSolve a{m.N, C, m.cnb, s.jv64, s.dval, s.dinv, rhs, dx, s.t, s.V, s.z[0], s.z[1], s.red,
              s.hs + (p.krylov_dim + 1) * p.krylov_dim + 1 + p.krylov_dim, s.vstride, s.red_count + 2, reinterpret_cast<int *>(s.hs + kHsStuck),
              blocks + s.grid_extra, s.grid_polls, p.krylov_dim, p.restarts, p.jacobi_sweeps};
  void *args[] = {&a};
  HGKS_PROF_BEGIN(K_GMRES, st);
  cudaLaunchCooperativeKernel(fn, dim3(blocks), dim3(kPT + 32), args, shm, st);
  HGKS_PROF_END(K_GMRES, st);
  return true;
}

}  // namespace hgks
