// FP64 reciprocal, square root, exponential and half-range error function for a chip
// whose FP64 unit is the bottleneck.
//
// A GB300 SM sub-partition takes 64 clocks per FP64 warp instruction (measured with chains
// of dependent FMAs: 64.3 clocks for 1 to 8 chains a warp, for 1 to 32 active lanes), while
// its integer and FP32 units take one or two. So the seeds, range reductions and
// exponent arithmetic below run there, and FP64 instructions are left for what needs 53
// bits. FP64 instructions, here against the CUDA library's (measured in the same way):
//   rcp 2 / 5.5,  rsqrt 3 / 5.5,  sqrt 3 / 9,  exp 8 / 17,  erfc/2 11 / 70 (erfcx: 45).
// Arguments outside the normal range of each function go to the library's function.
#pragma once
#include <cuda_runtime.h>
#include "fp64_tables.h"

namespace hgks {

// An FMA of three registers takes 64 clocks; an addition, a multiplication and an FMA with a
// constant operand take 76 (measured, 4 to 32 warps a SM). So the hot kernels multiply and add by
// FMAs with -0.0 and 1.0 held in registers (the same results): loaded, or the compiler would turn
// them back.
static __device__ double kUnits[2] = {-0.0, 1.0};
struct Units {
  double nz, one;
  __device__ __forceinline__ double mul(double a, double b) const { return fma(a, b, nz); }
  __device__ __forceinline__ double add(double a, double b) const { return fma(a, one, b); }
  __device__ __forceinline__ double sub(double a, double b) const { return fma(a, one, -b); }
};
__device__ __forceinline__ Units units() {
  const volatile double *p = kUnits;
  return {p[0], p[1]};
}

__device__ __forceinline__ float frcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float frsqrt_approx(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
// The double r + c of two floats, r in [1/2, 1], |c| < 2^-21 (c <= 0 at r = 1, c >= 0 at r = 1/2):
// r's bits widened, c added to the mantissa in units of 2^-50.
__device__ __forceinline__ double join(float r, float c) {
  return __longlong_as_double(((long long)__float_as_uint(r) << 29) + (896ll << 52) +
                              ((long long)__float2int_rn(c * 0x1p50f) << 3));
}
// mantissa of x as hi (24 bits, in [1, 2)) + lo, exactly up to lo's rounding (2^-47)
__device__ __forceinline__ void mantissa(int hi, int lo, float &m1, float &m2) {
  m1 = __uint_as_float(0x3f800000u | ((unsigned)hi & 0xfffffu) << 3 | (unsigned)lo >> 29);
  m2 = __int2float_rn(lo & 0x1fffffff) * 0x1p-52f;
}

// 1 / x: a seed good to 2^-45 from two floats, one Newton step (its square is below
// rounding, so the result is the rounded reciprocal but for rare ties)
__device__ __forceinline__ double rcp(double x, double one = 1.0) {
  const int hi = __double2hiint(x), lo = __double2loint(x), e = (hi >> 20) & 0x7ff;
  if ((unsigned)(e - 2) >= 2040u) return 1.0 / x;
  float m1, m2;
  mantissa(hi, lo, m1, m2);
  const float r = fminf(fmaxf(frcp_approx(m1), 0.5f), 1.0f), t = fmaf(-m2, r, fmaf(-m1, r, 1.0f));
  const double y0 = join(r, r * t);
  const double y = __hiloint2double((__double2hiint(y0) + (1023 - e) * 0x100000) | (hi & 0x80000000), __double2loint(y0));
  return fma(y, fma(-x, y, one), y);
}

// seed of 1/sqrt(x), good to 2^-45, for a positive normal x
__device__ __forceinline__ bool rsqrt_seed(double x, double &y) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  if ((unsigned)(hi - 0x00200000) >= 0x7fc00000u) return false;
  const int e = (hi >> 20) - 1023, k = e >> 1;          // x = m 2^(2k), m in [1, 4)
  float m1, m2;
  mantissa(hi, lo, m1, m2);
  const float sc = e & 1 ? 2.0f : 1.0f;
  m1 *= sc;
  m2 *= sc;
  const float r = fminf(fmaxf(frsqrt_approx(m1), 0.5f), 1.0f), p = r * r, pl = fmaf(r, r, -p);
  const float t = fmaf(-m2, p, fmaf(-m1, pl, fmaf(-m1, p, 1.0f)));
  const double s = join(r, r * t * fmaf(0.375f, t, 0.5f));
  y = __hiloint2double(__double2hiint(s) - k * 0x100000, __double2loint(s));
  return true;
}
__device__ __forceinline__ double half(double x) {      // x / 2 for a normal x away from underflow
  return __hiloint2double(__double2hiint(x) - 0x00100000, __double2loint(x));
}
__device__ __forceinline__ double rsqrt64(double x) {
  double y;
  if (!rsqrt_seed(x, y)) return rsqrt(x);
  return fma(half(y), fma(-(x * y), y, 1.0), y);
}
__device__ __forceinline__ double sqrt64(double x) {
  double y;
  if (!rsqrt_seed(x, y)) return sqrt(x);
  const double s = x * y;
  return fma(fma(-s, s, x), half(y), s);
}

// x truncated to float, for |x| in [2^-126, 2^100]; 0 below
__device__ __forceinline__ float to_float(int hi, int lo) {
  const unsigned a = (unsigned)hi & 0x7fffffffu;
  return __uint_as_float(a < 0x38100000u ? 0u : ((unsigned)hi & 0x80000000u) | (a - 0x38000000u) << 3 | (unsigned)lo >> 29);
}
// a small integer (|n| < 2^24) held in a float, as double
__device__ __forceinline__ double to_double(float f) {
  const unsigned b = __float_as_uint(f), a = b & 0x7fffffffu;
  return __hiloint2double(a ? (int)((b & 0x80000000u) | ((a >> 3) + 0x38000000u)) : 0, a ? (int)(b << 29) : 0);
}

// exp(x) by table (P. T. P. Tang, "Table-driven implementation of the exponential function
// in IEEE floating-point arithmetic", ACM TOMS 15, 1989): x = n ln2/128 + r, |r| < 0.0029,
// exp(x) = 2^(n/128) (1 + p(r)), p the Taylor polynomial of degree 5 (error 1e-18)
__device__ __forceinline__ double exp64(double x) {
  const int hi = __double2hiint(x), lo = __double2loint(x);
  if ((unsigned)(hi & 0x7fffffff) > 0x4085e000u) return exp(x);      // |x| > 700
  const float nf = rintf(to_float(hi, lo) * 184.66496659f);           // 128 / ln 2
  const int n = (int)nf;
  const double nd = to_double(nf);
  double r = fma(nd, -0x1.62e42fefp-8, x);                            // ln2 / 128: 33 bits, and the rest
  r = fma(nd, -0x1.473de6af278edp-41, r);
  const double T = __ldg(&kExp2Tab[n & 127]), r2 = r * r;
  const double q = fma(r, fma(r, fma(r, 1.0 / 120.0, 1.0 / 24.0), 1.0 / 6.0), 0.5);
  const double y = fma(T, fma(r2, q, r), T);
  return __hiloint2double(__double2hiint(y) + (n >> 7) * 0x100000, __double2loint(y));
}

// erfc(x) / 2 for |x| < 2.25 (hi word of x below 0x40020000): Taylor polynomial of degree 9
// about the nearest k/32 (error below 1e-18 of the value), its constant term in two doubles
constexpr unsigned kErfcRange = 0x40020000u;
__device__ __forceinline__ double half_erfc64(double x) {
  const float kf = rintf(to_float(__double2hiint(x), __double2loint(x)) * 32.0f);
  const double d = fma(to_double(kf), -0.03125, x);
  const double2 *c = reinterpret_cast<const double2 *>(kErfcTab[(int)kf + 72]);
  const double2 c0 = __ldg(c), c1 = __ldg(c + 1), c3 = __ldg(c + 2), c5 = __ldg(c + 3), c7 = __ldg(c + 4), c9 = __ldg(c + 5);
  double y = fma(d, c9.x, c7.y);
  y = fma(d, fma(d, y, c7.x), c5.y);
  y = fma(d, fma(d, y, c5.x), c3.y);
  y = fma(d, fma(d, y, c3.x), c1.y);
  return c0.x + fma(d, fma(d, y, c1.x), c0.y);
}

// x > 0 (false for NaN), and min(a, b), on the integer unit: an FP64 comparison costs an FP64 instruction
__device__ __forceinline__ bool positive(double x) {
  return (unsigned long long)(__double_as_longlong(x) - 1) < 0x7ff0000000000000ull;
}
__device__ __forceinline__ double min_positive(double a, double b) {
  const long long x = __double_as_longlong(a), y = __double_as_longlong(b);
  return (x | y) >= 0 ? __longlong_as_double(x < y ? x : y) : fmin(a, b);
}

}  // namespace hgks
