// bgk_fixed.cuh - the donor-cell combination and the moment sums of FP64
// states on the integer pipe.
//
// sm_103 issues one FP64 warp instruction per 76 cycles and sub-partition
// (64 alone), an IMAD.WIDE in 4 to 5, a shift in 2, an add in about 1.5
// (measured), and the two pipes run side by side.  A weighted sum of three
// positive values with weights that add up to one needs no floating point:
// the significands are aligned to the largest exponent as 61-bit integers,
// multiplied with 63-bit weights, and the 60-bit result is normalised and
// rounded once.  Its error is half an ulp of the result plus about 2^-59 of
// the largest value (three FP64 operations: up to 1.5 ulp).  The sums over
// the velocities add the results as 96-bit integers in a unit 2^-75 of the
// cell's largest exponent (more on long axes): each value is rounded to that
// unit, the additions are exact, whatever the order.
//
// Everything here is plain integer arithmetic and runs on the host as well.
#pragma once

#include <stdint.h>

#ifdef __CUDACC__
#define BGK_HD __host__ __device__ __forceinline__
#else
#define BGK_HD inline
#endif

namespace bgk {
namespace fx {

typedef uint32_t u32;
typedef uint64_t u64;

// Exponent fields the fixed-point path takes: far enough from 0 for results
// and sums to stay normal, and from the top for the sums to stay finite.
constexpr u32 kExpMin = 80, kExpMax = 0x700;
constexpr int kWeightBits = 63;  // weights are integers over 2^63
// The cell's range reaches this many powers of two above its largest sampled
// value; with larger values the caller takes their exponent as the range.
constexpr u32 kHeadroom = 2;

BGK_HD int clz64(u64 x) {
#ifdef __CUDA_ARCH__
  return __clzll((long long)x);
#else
  return x ? __builtin_clzll(x) : 64;
#endif
}

BGK_HD int clz32(u32 x) {
#ifdef __CUDA_ARCH__
  return __clz((int)x);
#else
  return x ? __builtin_clz(x) : 32;
#endif
}

// x >> d for any d (0 from 64 on).
BGK_HD u64 shr64(u64 x, u32 d) {
#ifdef __CUDA_ARCH__
  u64 r;
  asm("shr.u64 %0, %1, %2;" : "=l"(r) : "l"(x), "r"(d));  // PTX clamps the amount
  return r;
#else
  return d < 64u ? x >> d : 0;
#endif
}

// x << d for any d (0 from 32 on).
BGK_HD u32 shl32(u32 x, u32 d) {
#ifdef __CUDA_ARCH__
  u32 r;
  asm("shl.b32 %0, %1, %2;" : "=r"(r) : "r"(x), "r"(d));  // clamped likewise
  return r;
#else
  return d < 32u ? x << d : 0u;
#endif
}

// 96-bit integers modulo 2^96 (two's complement for negative values).
struct i96 {
  u32 a0, a1, a2;
};
BGK_HD i96 wide(u64 x) { return {(u32)x, (u32)(x >> 32), 0u}; }
BGK_HD i96 add(i96 x, i96 y) {
#ifdef __CUDA_ARCH__
  i96 r;
  asm("add.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, %7;\n\taddc.u32 %2, %5, %8;"
      : "=r"(r.a0), "=r"(r.a1), "=r"(r.a2)
      : "r"(x.a0), "r"(x.a1), "r"(x.a2), "r"(y.a0), "r"(y.a1), "r"(y.a2));
  return r;
#else
  const u64 lo = ((u64)x.a1 << 32 | x.a0), l = lo + ((u64)y.a1 << 32 | y.a0);
  return {(u32)l, (u32)(l >> 32), x.a2 + y.a2 + (l < lo ? 1u : 0u)};
#endif
}
// x times an unsigned 32-bit integer.
BGK_HD i96 mul(i96 x, u32 k) {
  const u64 p0 = (u64)x.a0 * k, p1 = (u64)x.a1 * k + (p0 >> 32);
  return {(u32)p0, (u32)p1, x.a2 * k + (u32)(p1 >> 32)};
}
BGK_HD i96 neg(i96 x) { return add({~x.a0, ~x.a1, ~x.a2}, {1u, 0u, 0u}); }
// x times a signed 32-bit integer.
BGK_HD i96 muls(i96 x, int k) { return k < 0 ? neg(mul(x, (u32)-k)) : mul(x, (u32)k); }

// Significand of a positive normal double (words hi, lo) as a 61-bit integer
// in units of 2^(emax - 1083), emax >= its exponent field.
BGK_HD u64 align(u32 hi, u32 lo, u32 emax) {
  const u64 m = ((u64)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 8;
  return shr64(m, emax - (hi >> 20));
}

// (w0 f0 + wx fx + wy fy) / 2^64 for weights that sum to 2^63 and 61-bit
// values: below 2^60, in units of 2^(emax - 1082).  The products of the low
// words (below 3 units in all) are left out; 1 stands for their mean and
// that of the truncations.
BGK_HD u64 combine(u64 w0, u64 f0, u64 wx, u64 fx, u64 wy, u64 fy) {
  const u32 a1 = (u32)(w0 >> 32), a0 = (u32)w0, b1 = (u32)(wx >> 32), b0 = (u32)wx, c1 = (u32)(wy >> 32),
            c0 = (u32)wy;
  const u32 p1 = (u32)(f0 >> 32), p0 = (u32)f0, q1 = (u32)(fx >> 32), q0 = (u32)fx, r1 = (u32)(fy >> 32),
            r0 = (u32)fy;
  const u64 hi = (u64)a1 * p1 + (u64)b1 * q1 + (u64)c1 * r1;
  // the high words of the weights sum to at most 2^31: no carry out
  const u64 cross = (u64)a1 * p0 + (u64)b1 * q0 + (u64)c1 * r0 + (u64)a0 * p1 + (u64)b0 * q1 + (u64)c0 * r1;
  return hi + (cross >> 32) + 1u;
}

// Whether a combination keeps enough bits to be rounded to a double.
BGK_HD bool combine_ok(u64 r) { return (u32)(r >> 32) >= (1u << 22); }

// The double nearest to r in units of 2^(emax - 1082), r >= 2^54 (words).
BGK_HD void to_words(u64 r, u32 emax, u32& hi, u32& lo) {
  const u32 lz = (u32)clz32((u32)(r >> 32));
  const u64 m = ((r << ((lz - 1u) & 31u)) + 0x200u) >> 10;  // 53 bits; a carry moves into the exponent
  lo = (u32)m;
  hi = (u32)(m >> 32) + ((emax + 3u - lz) << 20);
}

// A positive double (words hi, lo) in the unit 2^(eref - 1097), truncated:
// below 2^75 for an exponent field of at most eref.
BGK_HD i96 double_to_units96(u32 hi, u32 lo, u32 eref) {
  const u64 m = ((u64)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 8;
  const u32 e = eref - (hi >> 20) + 2u;  // m 2^(16 - e)
  const u64 top = shr64(m, e + 16u);
  return {e >= 16u ? (u32)shr64(m, e - 16u) : (u32)m << ((16u - e) & 31u), (u32)top, (u32)(top >> 32)};
}

// sum + the same value rounded to the nearest.
BGK_HD i96 add_units96(i96 sum, u32 hi, u32 lo, u32 eref) {
  const u64 m = ((u64)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 8;
  const u32 e = eref - (hi >> 20) + 2u;  // m 2^(16 - e)
  const u64 top = shr64(m, e + 16u), low = shr64(m, e - 17u);  // low: 0 unless e >= 17
  const u32 v0 = (u32)(low >> 1) | shl32((u32)m, 16u - e), v1 = (u32)top, v2 = (u32)(top >> 32), half = (u32)low & 1u;
#ifdef __CUDA_ARCH__
  i96 r;  // half + (2^32 - 1) sets the carry where half is set
  asm("{\n\t.reg .u32 t;\n\tadd.cc.u32 t, %9, 0xffffffff;\n\taddc.cc.u32 %0, %3, %6;\n\taddc.cc.u32 %1, %4, %7;\n\t"
      "addc.u32 %2, %5, %8;\n\t}"
      : "=&r"(r.a0), "=&r"(r.a1), "=&r"(r.a2)
      : "r"(sum.a0), "r"(sum.a1), "r"(sum.a2), "r"(v0), "r"(v1), "r"(v2), "r"(half));
  return r;
#else
  return add(add(sum, {v0, v1, v2}), {half, 0u, 0u});
#endif
}

// The double nearest to v in units of 2^(eref - 1081), |v| < 2^95 (words).
BGK_HD void wide_to_words(i96 v, u32 eref, u32& hi, u32& lo) {
  const bool minus = v.a2 >> 31;
  if (minus) v = neg(v);
  u32 up = 32u;  // words below the top 64 bits, in bits
  if (v.a2 == 0u) {
    v = {0u, v.a0, v.a1};
    up = 0u;
  }
  u64 r = (u64)v.a2 << 32 | v.a1;  // value (r + a0 / 2^32) 2^up
  hi = lo = 0u;
  if (r) {
    const u32 lz = (u32)clz64(r);
    r = lz ? (r << lz) | ((u64)v.a0 << lz >> 32) : r;  // leading bit at 63, value r 2^(up - lz)
    const u64 n = (r >> 1) | (r & 1u);                 // the lost bit stays sticky
    const u64 m = (n + 0x1ffu + ((n >> 10) & 1u)) >> 10;  // to nearest
    lo = (u32)m;
    // value m 2^(11 + up - lz) 2^(eref - 1081); the implicit bit adds 1 to the exponent
    hi = (u32)(m >> 32) + ((eref + 4u + up - lz) << 20);
  }
  if (minus) hi |= 0x80000000u;
}

// ---- Gaussian factors -----------------------------------------------------

// a b / 2^64, at most 2 below it.
BGK_HD u64 mulhi(u64 a, u64 b) {
  const u32 a1 = (u32)(a >> 32), a0 = (u32)a, b1 = (u32)(b >> 32), b0 = (u32)b;
  return (u64)a1 * b1 + (((u64)a1 * b0) >> 32) + (((u64)a0 * b1) >> 32);
}
BGK_HD u32 mulhi32(u32 a, u32 b) { return (u32)(((u64)a * b) >> 32); }

// floor(2^(63 - i / 32) + 1/2)
#define BGK_EXP2_TABLE                                                                              \
  {0x8000000000000000ull, 0x7d41d96db915019dull, 0x7a92be8a92436616ull, 0x77f25ccdee6d7ae6ull,      \
   0x75606373ee921c97ull, 0x72dc8373be41a454ull, 0x70666f76154a7089ull, 0x6dfddbcbed791babull,      \
   0x6ba27e656b4eb57aull, 0x69540ec8f895722dull, 0x6712460a8fc24072ull, 0x64dcdec3371793d1ull,      \
   0x62b39508aa836d6full, 0x6096266533384a2bull, 0x5e8451cfac061b5full, 0x5c7dd7a3b17dcf75ull,      \
   0x5a827999fcef3242ull, 0x5891fac0e95612c8ull, 0x56ac1f752150a563ull, 0x54d0ad5a753e077cull,      \
   0x52ff6b54d8a89c75ull, 0x513821818624b40cull, 0x4f7a993048d088d7ull, 0x4dc69cdceaa72a9cull,      \
   0x4c1bf828c6dc54b8ull, 0x4a7a77d47f7b84b1ull, 0x48e1e9b9d588e19bull, 0x47521cc5a2e6a9e0ull,      \
   0x45cae0f1f545eb73ull, 0x444c0740496d4294ull, 0x42d561b3e6243d8aull, 0x4166c34c5615d0ecull}

// 2^63 2^-(f / 2^64), relative error below 2^-57: f = (i + g) / 32 of 2^64,
// 2^(-i/32) from the table and the Taylor series of 2^(-g/32) through g^7
// (coefficients (ln 2 / 32)^k / k! times 2^69, from k = 4 on times 2^58).
BGK_HD u64 exp2_neg(u64 f, const u64* table) {
  const u64 t = table[(u32)(f >> 59)];
  const u64 g = f << 5;
  const u32 gh = (u32)(g >> 32);
  u32 r = 0x0000a185u - mulhi32(gh, 0x00000080u);
  r = 0x00aec3ffu - mulhi32(gh, r);
  r = 0x9d955b7eu - mulhi32(gh, r);
  u64 s = 0x00038d611ae09417ull - mulhi(g, (u64)r << 11);
  s = 0x01ebfbdff82c58eaull - mulhi(g, s);
  s = 0xb17217f7d1cf79abull - mulhi(g, s);
  return t - (mulhi(t, mulhi(g, s)) >> 5);
}

// 2^-(w^2), w in units of 2^-58 with |w| < 2^63: returns q with
// 2^-(w^2) = q 2^-63 2^-n, q in (2^62, 2^63].
BGK_HD u64 gauss(int64_t w, const u64* table, u32& n) {
  const u64 a = (u64)(w < 0 ? -w : w);
  const u32 a1 = (u32)(a >> 32), a0 = (u32)a;
  const u64 cross = (u64)a1 * a0, low = (u64)a0 * a0;
  const u64 lo = (cross << 33) + low;
  const u64 hi = (u64)a1 * a1 + (cross >> 31) + (lo < low ? 1u : 0u);  // hi 2^64 + lo = w^2 2^116
  n = (u32)(hi >> 52);
  return exp2_neg((hi << 12) | (lo >> 52), table);
}

// q 2^-63 2^-n as a double (words), n < 1020.
BGK_HD void gauss_words(u64 q, u32 n, u32& hi, u32& lo) {
  const u64 m = (q + 0x200u) >> 10;
  lo = (u32)m;
  hi = (u32)(m >> 32) + ((1021u - n) << 20);
}

// A positive normal double (words) as m 2^(e - 1085) with m in [2^62, 2^63).
BGK_HD u64 top63(u32 hi, u32 lo) { return ((u64)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 10; }

// b f + phi for f a positive double (words), b = wb 2^(eb - 63) with wb < 2^63,
// and phi = mphi 2^(ephi - 1084), mphi < 2^62: the result in units of
// 2^(e - 1082), below 2^61, with e = max(exponent of f + eb, ephi).
BGK_HD u64 relax(u32 hi, u32 lo, u64 wb, int eb, u64 mphi, int ephi, int& e) {
  const int e1 = (int)(hi >> 20) + eb;
  e = e1 > ephi ? e1 : ephi;
  const u64 m = ((u64)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 8;
  return mulhi(shr64(m, (u32)(e - e1)), wb) + shr64(mphi, (u32)(e - ephi) + 2u) + 1u;
}

// A double (words) with |x| < 32 in units of 2^-58, rounded (0 below half of one).
BGK_HD int64_t to_fix58(u32 hi, u32 lo) {
  const u32 e = (hi >> 20) & 0x7ffu;
  const u64 m = ((u64)((hi & 0xfffffu) | 0x100000u) << 32 | lo) << 10;  // m 2^(e - 1027)
  const u32 d = 1027u - e;
  const u64 r = shr64(m, d) + ((u32)shr64(m, d - 1u) & 1u);
  return (hi >> 31) ? -(int64_t)r : (int64_t)r;
}

}  // namespace fx
}  // namespace bgk
