// Product form of the off-diagonal Jacobian blocks.
#pragma once
#include <cuda_runtime.h>
#include "fp64.cuh"

namespace hgks {

// acc += 1/2 (J(Q_j) n - lambda I) S x_j, the off-diagonal block of Eq. (deri-matrix)
// applied as a product (no stored 5x5 block): J(Q_j)(n S/2) x_j from j's primitives
// (jv rows 0-5: u, v, w, H, (gamma-1)|u|^2/2, gamma-1) and the record of face p of cell i
// (rows 6 + 4p + k: n S/2, lambda S/2)
template <typename TV>
__device__ __forceinline__ void offdiag_product(const float *__restrict__ jv, int N, int i, int p, int j, const TV *x,
                                                TV *acc) {
  const TV u = jv[j], v = jv[(size_t)N + j], w = jv[2 * (size_t)N + j], H = jv[3 * (size_t)N + j];
  const TV phi = jv[4 * (size_t)N + j], g1 = jv[5 * (size_t)N + j];
  const float *f = jv + (size_t)(6 + 4 * p) * N + i;
  const TV nx = f[0], ny = f[N], nz = f[2 * (size_t)N], ls = f[3 * (size_t)N];
  const TV un = u * nx + v * ny + w * nz, nm = nx * x[1] + ny * x[2] + nz * x[3], um = u * x[1] + v * x[2] + w * x[3];
  const TV dp = g1 * (x[4] - um) + phi * x[0], t = nm - un * x[0];
  acc[0] += nm - ls * x[0];
  acc[1] += u * t + un * x[1] + nx * dp - ls * x[1];
  acc[2] += v * t + un * x[2] + ny * dp - ls * x[2];
  acc[3] += w * t + un * x[3] + nz * dp - ls * x[3];
  acc[4] += un * (x[4] + dp) + H * t - ls * x[4];
}

// The same product in FP64 with what depends on the neighbour alone taken out of the sum
// over faces (rows 6 + 5p + k of the FP64 operands: n S/2, s, t): a vector x is kept as z = (x0, a, dp, x4) per cell,
//   a = m - u x0,  dp = (gamma - 1)(x4 - u . a) - (gamma - 1)|u|^2/2 x0,
// and with s = u . n S/2 - lambda S/2 and t = u . n S/2 (stored) the block takes 17 operations
// instead of 28 (or 24 for a stored 5x5 block, whose 200 bytes per face it replaces with 40):
//   r = n . a,  r0 = r + s x0,  rows (r0, u r0 + s a + n dp, H r + s x4 + t dp).
struct CellPrim { double u, v, w, H, phi, g1; };
__device__ __forceinline__ CellPrim cell_prim(const double *__restrict__ jv, size_t N, int i) {
  return {jv[i], jv[N + i], jv[2 * N + i], jv[3 * N + i], jv[4 * N + i], jv[5 * N + i]};
}
__device__ __forceinline__ void z_of(const Units &un, const CellPrim &q, const double *y, double *z) {
  z[0] = y[0];
  z[1] = fma(-q.u, y[0], y[1]);
  z[2] = fma(-q.v, y[0], y[2]);
  z[3] = fma(-q.w, y[0], y[3]);
  z[4] = fma(q.g1, fma(-q.u, z[1], fma(-q.v, z[2], fma(-q.w, z[3], y[4]))), un.mul(-q.phi, y[0]));
  z[5] = y[4];
}
__device__ __forceinline__ void z_store(double *zv, size_t N, int i, const double *z) {
#pragma unroll
  for (int k = 0; k < 6; k++) zv[k * N + i] = z[k];
}
// zv is not const __restrict__: other blocks of the same launch may write it before a grid barrier
__device__ __forceinline__ void z_product(const Units &un, const double *__restrict__ jv, size_t N, int i, int p, int j, const double *zv,
                                          double *acc) {
  const double *f = jv + (6 + 5 * (size_t)p) * N + i;
  const double nx = f[0], ny = f[N], nz = f[2 * N], s = f[3 * N], t = f[4 * N];
  const double x0 = zv[j], a0 = zv[N + j], a1 = zv[2 * N + j], a2 = zv[3 * N + j], dp = zv[4 * N + j], x4 = zv[5 * N + j];
  const double r = fma(nx, a0, fma(ny, a1, un.mul(nz, a2))), r0 = fma(s, x0, r);
  acc[0] = un.add(r0, acc[0]);
  acc[1] = fma(jv[j], r0, fma(s, a0, fma(nx, dp, acc[1])));
  acc[2] = fma(jv[N + j], r0, fma(s, a1, fma(ny, dp, acc[2])));
  acc[3] = fma(jv[2 * N + j], r0, fma(s, a2, fma(nz, dp, acc[3])));
  acc[4] = fma(jv[3 * N + j], r, fma(s, x4, fma(t, dp, acc[4])));
}

}  // namespace hgks
