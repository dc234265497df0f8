// Checks csrc/bgk_fixed.cuh on the host: prints the largest relative errors.
#include "bgk_fixed.cuh"

#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>

using namespace bgk::fx;

static void words(double x, u32& hi, u32& lo) {
  u64 b;
  memcpy(&b, &x, 8);
  hi = (u32)(b >> 32);
  lo = (u32)b;
}
static double value(u32 hi, u32 lo) {
  const u64 b = (u64)hi << 32 | lo;
  double x;
  memcpy(&x, &b, 8);
  return x;
}
static const u64 kTable[32] = BGK_EXP2_TABLE;

int main() {
  std::mt19937_64 g(1);
  std::uniform_real_distribution<double> U(0, 1);
  long double worst[7] = {0, 0, 0, 0, 0, 0, 0};
  auto keep = [&](int k, long double got, long double want) {
    worst[k] = std::fmax(worst[k], std::fabs((got - want) / want));
  };
  // to_fix58 over all exponents, zeros and subnormals
  for (int t = 0; t < 100000; ++t) {
    const double edge[] = {0.0, -0.0, 0x1p-59, -0x1p-59, 0x1p-60, -0x1p-60, 0x1.8p-59, 0x1.fffffffffffffp-60, 5e-324, 1e-300, 0x1.fffffffffffffp4};
    const double x = t < 11 ? edge[t] : std::ldexp(2 * U(g) - 1, (int)(110 * U(g)) - 105);
    u32 a, b;
    words(x, a, b);
    worst[6] = std::fmax(worst[6], std::fabs(to_fix58(a, b) - std::ldexp((long double)x, 58)));
  }
  for (int t = 0; t < 300000; ++t) {
    u32 a, b, c, d, e, f, hi, lo, n;
    // donor-cell combination
    const double f0 = std::pow(10.0, -30 * U(g)) * (0.1 + U(g));
    const double fx = f0 * std::exp(4 * (U(g) - 0.5)), fy = f0 * std::exp(4 * (U(g) - 0.5));
    // every third pair of weights is spread over 60 powers of two
    const double small = t % 3 ? 1.0 : std::ldexp(1.0, -(int)(60 * U(g)));
    const u64 wx = (u64)(U(g) * 0.6 * small * 0x1p63), wy = (u64)(U(g) * 0.4 * small * 0x1p63), w0 = ((u64)1 << 63) - wx - wy;
    words(f0, a, b);
    words(fx, c, d);
    words(fy, e, f);
    const u32 em = std::max(std::max(a, c), e) >> 20;
    const u64 r = combine(w0, align(a, b, em), wx, align(c, d, em), wy, align(e, f, em));
    if (!combine_ok(r)) continue;
    to_words(r, em, hi, lo);
    keep(0, value(hi, lo), (w0 * (long double)f0 + wx * (long double)fx + wy * (long double)fy) / 0x1p63L);
    const u32 up = em + 2 + (u32)(40 * U(g));
    const i96 w96 = double_to_units96(hi, lo, up);
    const long double fine = std::ldexp(1.0L, (int)up - 1097), v96 = ((long double)w96.a2 * 0x1p32L + w96.a1) * 0x1p32L + w96.a0;
    worst[1] = std::fmax(worst[1], std::fabs(v96 - std::floor(value(hi, lo) / fine)));
    const u64 r0 = g();
    const i96 s96 = add_units96({(u32)r0, (u32)(r0 >> 32), 5u}, hi, lo, up);
    const long double whole = std::floor(value(hi, lo) / fine);
    const __int128 added = ((__int128)s96.a2 << 64 | (u64)s96.a1 << 32 | s96.a0) - ((__int128)5 << 64 | r0);
    worst[5] = std::fmax(worst[5], std::fabs((long double)(added - (__int128)whole) - (value(hi, lo) / fine - whole)));
    // Gaussian and relaxation
    const double x = 8 * (2 * U(g) - 1), y = 8 * (2 * U(g) - 1);
    words(x, a, b);
    const u64 qx = gauss(to_fix58(a, b), kTable, n);
    gauss_words(qx, n, hi, lo);
    keep(2, value(hi, lo), std::exp2(-(long double)x * x));
    const double p = std::exp2(-x * x - y * y), bw = t % 3 ? 1 - 0.3 * U(g) : std::ldexp(U(g) + 0.1, -(int)(40 * U(g)));
    const double ka = 0.1 + U(g), ft = p * std::exp(4 * (U(g) - 0.5));
    words(p, a, b);
    words(bw, c, d);
    words(ka, e, f);
    const u64 m = mulhi(top63(a, b), top63(e, f));
    int em2;
    words(ft, hi, lo);
    const u64 rr = relax(hi, lo, top63(c, d), (int)(c >> 20) - 1022, m, (int)(a >> 20) + (int)(e >> 20) - 1022, em2);
    to_words(rr, (u32)em2, hi, lo);
    keep(3, value(hi, lo), (long double)bw * ft + (long double)ka * p);
    // 96-bit sums
    const int k1 = (int)(g() % 2001) - 1000, k2 = (int)(g() % 2001) - 1000;
    const u64 v1 = g() >> 6, v2 = g() >> 6;
    const __int128 s = (__int128)v1 * k1 + (__int128)v2 * k2;
    if (s != 0) {
      wide_to_words(add(muls(wide(v1), k1), muls(wide(v2), k2)), 1000, hi, lo);
      keep(4, value(hi, lo), std::ldexp((long double)s, 1000 - 1081));
    }
  }
  for (long double w : worst) std::printf("%.6Lg\n", w);
}
