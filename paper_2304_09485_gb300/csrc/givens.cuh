// Least-squares solve of the GMRES Hessenberg system (Algorithm 1), one thread.
#pragma once
#include <cuda_runtime.h>
#include "fp64.cuh"

namespace hgks {

// y minimises || beta e1 - H y || for the (m+1) x m upper Hessenberg H
// (H[i*m + j] = h_ij), by Givens rotations applied column by column, in place:
// H's upper triangle holds R afterwards. Columns after the first zero
// subdiagonal entry (a breakdown) are left out. Returns |g_used|, the residual
// norm of the least-squares problem.
__device__ inline double givens_lsq(int m, double *__restrict__ H, double beta, double *__restrict__ y) {
  double cs[64], sn[64], gv[65];
  int used = m;
  for (int j = 0; j < m; j++)
    if (H[(j + 1) * m + j] == 0.0) { used = j + 1; break; }
  for (int j = 0; j < m; j++) y[j] = 0.0;
  if (beta == 0.0) return 0.0;
  for (int i = 0; i <= m; i++) gv[i] = 0.0;
  gv[0] = beta;
  for (int j = 0; j < used; j++) {
    double a = H[j];
    for (int i = 0; i < j; i++) {
      const double h2 = H[(i + 1) * m + j];
      H[i * m + j] = cs[i] * a + sn[i] * h2;
      a = cs[i] * h2 - sn[i] * a;
    }
    const double b = H[(j + 1) * m + j], r = rsqrt64(a * a + b * b);
    const double c = a * r, s = b * r;
    cs[j] = c;
    sn[j] = s;
    H[j * m + j] = c * a + s * b;
    H[(j + 1) * m + j] = 0.0;
    const double g1 = gv[j], g2 = gv[j + 1];
    gv[j] = c * g1 + s * g2;
    gv[j + 1] = -s * g1 + c * g2;
  }
  for (int j = used - 1; j >= 0; j--) {
    double s = gv[j];
    for (int k = j + 1; k < used; k++) s -= H[j * m + k] * y[k];
    y[j] = s * rcp(H[j * m + j]);
  }
  return fabs(gv[used]);
}

// Column j of H from a_i = (w, v_i) and the basis Gram matrix (G[k * ld + i] = (v_k, v_i), k < i),
// whose column j comes in g: h_i = a_i - sum_{k<i} h_k G_ki, by one warp, lane i (and i + 32)
// subtracting its terms in the order of k. m <= 64.
__device__ __forceinline__ void mgs_coef_warp(int lane, int j, int m, int ld, const double *a, const double *g, double *G,
                                              double *H) {
  for (int k = lane; k < j; k += 32) G[k * ld + j] = g[k];
  const int i1 = lane + 32;
  double h0 = lane <= j ? a[lane] : 0.0, h1 = i1 <= j ? a[i1] : 0.0;
  for (int k = 0; k < j; k++) {
    const double hk = __shfl_sync(0xffffffffu, k < 32 ? h0 : h1, k & 31);
    if (lane > k && lane <= j) h0 = fma(-hk, lane == j ? g[k] : G[k * ld + lane], h0);
    if (j >= 32 && i1 > k && i1 <= j) h1 = fma(-hk, i1 == j ? g[k] : G[k * ld + i1], h1);
  }
  if (lane <= j) H[lane * m + j] = h0;
  if (i1 <= j) H[i1 * m + j] = h1;
}

}  // namespace hgks
