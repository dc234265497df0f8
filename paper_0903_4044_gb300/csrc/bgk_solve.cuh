// bgk_solve.cuh - device helpers of the fixed-point step kernels: sums of
// integers over lanes, cheap FP64 reciprocals, and the Gaussian factors of one
// axis with their central sums.
#pragma once

#include "bgk_device.cuh"
#include "bgk_fixed.cuh"

namespace bgk {
namespace {

__device__ const unsigned long long kExp2[32] = BGK_EXP2_TABLE;

__device__ __forceinline__ fx::i96 xor_add96(fx::i96 keep, fx::i96 send, int mask) {
  const fx::i96 got = {__shfl_xor_sync(0xffffffffu, send.a0, mask), __shfl_xor_sync(0xffffffffu, send.a1, mask),
                       __shfl_xor_sync(0xffffffffu, send.a2, mask)};
  return fx::add(keep, got);
}

// An integer in the unit 2^(eref - 1081) as a double.
__device__ __forceinline__ double unit_value(fx::i96 v, int eref) {
  unsigned hi, lo;
  fx::wide_to_words(v, (unsigned)eref, hi, lo);
  return __hiloint2double((int)hi, (int)lo);
}

// 1/x and 1/sqrt(x) of positive normal x by one third-order (Householder)
// step from the FP32 approximation of relative error e0 < 2^-21: three and
// five FP64 operations, error e0^3 beside the roundings (an FP64 division or
// square root costs ten or more).
__device__ __forceinline__ float to_float_bits(double x) {  // truncated, exponent kept in range by the caller
  return __uint_as_float((((unsigned)__double2hiint(x) - 0x38000000u) << 3) | ((unsigned)__double2loint(x) >> 29));
}
__device__ __forceinline__ double to_double_bits(float y) {
  const unsigned u = __float_as_uint(y);
  return __hiloint2double((int)((u >> 3) + 0x38000000u), (int)(u << 29));
}
__device__ __forceinline__ double rcp3(double x) {
  float y;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(to_float_bits(x)));
  const double d = to_double_bits(y), e = fma(-x, d, 1.0);
  return fma(d, fma(e, e, e), d);
}
__device__ __forceinline__ double rsqrt3(double x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(to_float_bits(x)));
  const double d = to_double_bits(y), e = fma(-x * d, d, 1.0);
  return fma(d, e * fma(0.375, e, 0.5), d);
}
// Whether x is positive, finite and well inside the FP32 exponent range.
__device__ __forceinline__ bool in_range(double x) {
  const unsigned h = (unsigned)__double2hiint(x);
  return h - 0x3a000000u < 0x0c000000u;  // 2^-95 to 2^97
}
__device__ __forceinline__ unsigned abs_hi(double x) { return (unsigned)__double2hiint(x) & 0x7fffffffu; }

// 2^-t, t in units of 2^-58 below 2^63, times 2^up.
__device__ __forceinline__ double exp2_neg_fixed(unsigned long long t, unsigned up) {
  unsigned hi, lo;
  fx::gauss_words(fx::exp2_neg(t << 6, (const fx::u64*)kExp2), (unsigned)(t >> 58) - up, hi, lo);
  return __hiloint2double((int)hi, (int)lo);
}
// e^-x.  The product with log2 e is taken to 2^-57 (rounded to a double it
// cost 14 times 2^-53 of e^-x at x = 20).
__device__ __forceinline__ double exp_neg_fixed(double x) {
  const unsigned h = (unsigned)__double2hiint(x);
  if (h >= 0x40360000u) return exp(-x);  // 22 and more, negative, NaN
  const unsigned long long u = (unsigned long long)fx::to_fix58(h, (unsigned)__double2loint(x)) << 1;
  return exp2_neg_fixed(fx::mulhi(u, 0xb8aa3b295c17f0bcull), 0u);  // 2^63 log2 e
}
// x^y as 2^(y log2 x), the product as an integer: one third of pow's FP64
// operations.  Error 2^-53 of log2 x and the last rounding while the exponent's
// magnitude is below one.
__device__ __forceinline__ double pow_fixed(double x, double y) {
  const double l = log2(x);
  const unsigned hl = (unsigned)__double2hiint(l), hy = (unsigned)__double2hiint(y);
  if (max(hl & 0x7fffffffu, hy & 0x7fffffffu) >= 0x40400000u) return pow(x, y);  // 32 and more, NaN
  const long long a = fx::to_fix58(hl, (unsigned)__double2loint(l)), b = fx::to_fix58(hy, (unsigned)__double2loint(y));
  const unsigned long long ua = (unsigned long long)(a < 0 ? -a : a), ub = (unsigned long long)(b < 0 ? -b : b);
  const unsigned long long top = __umul64hi(ua, ub);
  if (top >= 1ull << 52) return pow(x, y);  // one and more
  const long long e = (long long)(top << 6 | (ua * ub) >> 58);
  return exp2_neg_fixed((unsigned long long)((1ll << 58) - ((a ^ b) < 0 ? -e : e)), 1u);
}

// One axis of a cell's Gaussians at a base point: (c_k - u) sqrt(log2 e /
// theta) = a k - c in units of 2^-58, and k0, the integer index next to u: the
// central sums are taken over k' = k - k0, where c - u = half k' + delta.
struct AxisBase {
  long long a, c;
  int k0;
};
constexpr int kMaxIndexShift = 1024;  // |k0|: keeps sum k'^2 e within 95 bits

// x sqrt(log2 e), rounded, |x| below 2^62 (a double's sqrt(log2 e) is 0.22 of
// 2^-53 too small: twice that in the width of every Gaussian, with one sign).
__device__ __forceinline__ long long times_sqrt_log2e(long long x) {
  const unsigned long long k = 0x99be610c1d827eefull;  // 2^63 sqrt(log2 e)
  const unsigned long long u = (unsigned long long)(x < 0 ? -x : x) << 1;
  const long long r = (long long)(__umul64hi(u, k) + ((u * k) >> 63));
  return x < 0 ? -r : r;
}

// The base of an axis of n velocity cells of half width `half`, centre `mid`,
// at mean u; isq = 1 / sqrt(theta).  False when a velocity lies too far out for
// the fixed-point Gaussian.
__device__ __forceinline__ bool axis_base(int n, double half, double inv_half, double mid, double u, double isq,
                                          AxisBase& B) {
  const double off = u - mid, a = half * isq, s = off * isq;
  const double r = fma(off, inv_half, 6755399441055744.0);  // 1.5 2^52: rounds to an integer
  const double reach = fma(a, (double)n, fabs(s));
  B.k0 = __double2loint(r);
  B.a = times_sqrt_log2e(fx::to_fix58((unsigned)__double2hiint(a), (unsigned)__double2loint(a)));
  B.c = times_sqrt_log2e(fx::to_fix58((unsigned)__double2hiint(s), (unsigned)__double2loint(s)));
  // |s| + a n < 26.55, times sqrt(log2 e) 31.9; |off| below kMaxIndexShift half steps (words: the exponent decides)
  return abs_hi(reach) < 0x403a8cccu && abs_hi(r) == 0x43380000u - (B.k0 < 0 ? 1u : 0u) &&
         (unsigned)(B.k0 + kMaxIndexShift) < 2u * kMaxIndexShift;
}

// sum e, sum k' e, sum k'^2 e of an axis over a group of LANES lanes (i: the
// lane's place in it); lane p < 3 of the group returns sum p.
template <int LANES>
__device__ __forceinline__ double axis_index_sums(int n, const AxisBase& B, int i) {
  fx::i96 s[3] = {{0u, 0u, 0u}, {0u, 0u, 0u}, {0u, 0u, 0u}};
#pragma unroll 1
  for (int j = i; j < n; j += LANES) {
    const int k = 2 * j + 1 - n, kk = k - B.k0;
    unsigned q2;
    const unsigned long long q = fx::gauss(B.a * k - B.c, (const fx::u64*)kExp2, q2);
    const fx::i96 e = fx::wide(q2 < 62u ? q >> (q2 + 1u) : 0);  // units of 2^-62
    s[0] = fx::add(s[0], e);
    s[1] = fx::add(s[1], fx::muls(e, kk));
    s[2] = fx::add(s[2], fx::mul(e, (unsigned)(kk * kk)));
  }
#pragma unroll
  for (int m = LANES / 2; m > 0; m >>= 1)
#pragma unroll
    for (int p = 0; p < 3; ++p) s[p] = xor_add96(s[p], s[p], m);
  return unit_value(i == 0 ? s[0] : i == 1 ? s[1] : s[2], 1081 - 62);
}

// Central sums M_m = sum (c - u)^m e from the index sums k[3].
__device__ __forceinline__ void central_sums(const double* k, int k0, double half, double mid, double u, double M[3]) {
  const double d = fma((double)k0, half, mid) - u, t1 = half * k[1];
  M[0] = k[0];
  M[1] = fma(d, k[0], t1);
  M[2] = fma(half * half, k[2], d * (t1 + M[1]));
}

}  // namespace
}  // namespace bgk
