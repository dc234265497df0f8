// bgk_step.cu - the fused FP64 BGK phase-space step.
//
// A CTA owns G spatial cells; the velocities are v = jy*nvx + jx with 16-byte
// (g, h) pairs.  Per step:
//   phase 1 (each warp, its cell or its rows of one)
//     A0  diffuse-wall densities n_W of the faces the cell touches, from the
//         cell's own f^n (zero net mass flux, below Eq. bc_cavity);
//     A1  streaming: f~ = a0 f + ax f_(upwind x) + ay f_(upwind y) (2D
//         unsplit donor cell), or f~ = (1-|r|) f_(i-[C]) + |r| f_(i-[C]-sgn C)
//         (1D, Eq. upwind after the integer shift of Eq. exact); upwind
//         neighbours come from L2, boundary values from the ghost tables;
//         f~ is parked in the cell's output slots until phase 3;
//     A2  velocity sums of f~ for Eq. (macroscopic);
//   phase 2
//     A3  moments, nu = n theta^(1-omega), relaxation weights and the
//         effective Maxwellian parameters, separable factors in shared memory;
//   phase 3 (each warp, as phase 1)
//     A4  f^{n+1} = b f~ + a Phi (Eq. relaxation: b = e^{-nu dt}, a = 1 - b;
//         Euler: a = nu dt, b = 1 - a), stored to HBM.
//
// The FP64 pipe of sm_103 takes 64 to 76 cycles for a warp instruction,
// whatever the number of active lanes; an integer instruction takes 1 to 5.
// So the 2D step (step_fixed_kernel) gives half of its per-velocity work and
// nearly all of its per-cell work to the integer pipe as fixed-point
// arithmetic (bgk_fixed.cuh) that rounds less than the FP64 form: g streams
// and h relaxes on the integer pipe while h streams and g relaxes on the FP64
// pipe (3 and 2 FP64 operations per velocity), the moment sums are integers of
// 65 to 75 bits a value, and the Gaussians are evaluated directly; 5.6 FP64
// operations per velocity in all instead of 15 to 19.  Measured against the
// FP64-only form, state in and moments out included: 20 steps of 256^2 x 48^2
// 85.4 -> 49.7 ms, 100 of 64^2 x 32^2 16.9 -> 11.2 ms, 50 of 157 x 83 cells x 20
// x 28 velocities 16.3 -> 9.4 ms; error of the 20 steps against 64-bit sums
// 8.8e-16 -> 4.6e-16.  What bounds it now: 332 thread instructions per update
// (50 % of the issue slots), upwind loads and the parked f~ that L2 does not
// hold (75.5 B of DRAM traffic per update, 128^2 x 48^2).
//
// step1d_kernel is the same for 1D grids; step_f64_kernel is the FP64-only
// form, for the grids that step_f64_plan leaves to it.
#include "bgk_device.cuh"
#include "bgk_solve.cuh"

#include <algorithm>

namespace bgk {

namespace {

__device__ __forceinline__ int vi_jx(int vi) { return vi & 0xfff; }
__device__ __forceinline__ int vi_jy(int vi) { return (vi >> 12) & 0xfff; }
__device__ __forceinline__ int vi_sx(int vi) { return ((vi >> 24) & 3) - 1; }
__device__ __forceinline__ int vi_sy(int vi) { return ((vi >> 26) & 3) - 1; }

// Boundary value at velocity j (components jx, jy) for a face of the cell
// whose state starts at fc.
__device__ __forceinline__ double2 ghost_at(const Params& P, const Tables& T, int face, int j, int jx,
                                            int jy, double nw, const double2* __restrict__ fc) {
  const int kind = P.bc_kind[face];
  if (kind == BC_SPECULAR) {
    const int jr = (face == XLO || face == XHI) ? jy * P.nvx + (P.nvx - 1 - jx)
                                                : (P.nvy - 1 - jy) * P.nvx + jx;
    return fc[jr];
  }
  const double2 gv = T.ghost[face * P.nv + j];
  if (kind == BC_DIFFUSE) return make_double2(nw * gv.x, nw * gv.y);
  return gv;
}

// ---- phase 1 ---------------------------------------------------------------
// What a cell's sums (kSums doubles in shared memory) hold: the four velocity
// sums (sum g, sum c_x g, sum c_y g, sum |c|^2 g + h), or the sums over the
// integer velocity indices k = 2 j + 1 - n of the fixed-point path:
// (sum g, sum k_x g, sum k_x^2 g, sum k_y g, sum k_y^2 g, sum h).
constexpr int kSums = 6;
enum { SUMS_VELOCITY = 0, SUMS_INDEX = 1 };

// The faces the warp's cell touches and n_W of its diffuse ones.
struct CellEdge {
  bool xlo, xhi, ylo, yhi;
  double nw[4];
};

// A0: n_W for each diffuse face the cell touches (warp-uniform branch).
template <int DIM>
__device__ __forceinline__ CellEdge cell_edge(const Params& P, const Tables& T, const double2* __restrict__ fc,
                                              int ix, int iy) {
  const int lane = threadIdx.x & 31;
  CellEdge C;
  C.xlo = ix == 0;
  C.xhi = ix == P.nx - 1;
  C.ylo = DIM == 2 && iy == 0;
  C.yhi = DIM == 2 && iy == P.ny - 1;
  unsigned diff = 0;
  if (C.xlo && P.bc_kind[XLO] == BC_DIFFUSE) diff |= 1u;
  if (C.xhi && P.bc_kind[XHI] == BC_DIFFUSE) diff |= 2u;
  if (C.ylo && P.bc_kind[YLO] == BC_DIFFUSE) diff |= 4u;
  if (C.yhi && P.bc_kind[YHI] == BC_DIFFUSE) diff |= 8u;
#pragma unroll
  for (int f = 0; f < 4; ++f) C.nw[f] = 0.0;
  if (diff) {
    double inc[4] = {0.0, 0.0, 0.0, 0.0};
    for (int j = lane; j < P.nv; j += 32) {
      const int vi = T.vinfo[j];
      const double2 cxy = T.cxy[j];
      const double g = fc[j].x;
      const int sx = vi_sx(vi), sy = vi_sy(vi);
      if ((diff & 1u) && sx < 0) inc[0] = fma(-cxy.x, g, inc[0]);
      if ((diff & 2u) && sx > 0) inc[1] = fma(cxy.x, g, inc[1]);
      if ((diff & 4u) && sy < 0) inc[2] = fma(-cxy.y, g, inc[2]);
      if ((diff & 8u) && sy > 0) inc[3] = fma(cxy.y, g, inc[3]);
    }
    const double w = warp_reduce4(inc[0], inc[1], inc[2], inc[3]);
#pragma unroll
    for (int f = 0; f < 4; ++f) {
      const double tot = __shfl_sync(0xffffffffu, w, 8 * f);
      C.nw[f] = (diff >> f & 1u) ? tot * P.dv / T.emitted[f] : 0.0;
    }
  }
  return C;
}

// Sum over the warp of eight 96-bit values per lane (recursive halving as in
// warp_reduce8): lane L ends with value (L >> 2) & 7.
__device__ __forceinline__ fx::i96 shfl96(fx::i96 v, int from) {
  return {__shfl_sync(0xffffffffu, v.a0, from), __shfl_sync(0xffffffffu, v.a1, from),
          __shfl_sync(0xffffffffu, v.a2, from)};
}
__device__ __forceinline__ fx::i96 pick(bool c, fx::i96 x, fx::i96 y) {
  return {c ? x.a0 : y.a0, c ? x.a1 : y.a1, c ? x.a2 : y.a2};
}
__device__ __forceinline__ fx::i96 warp_reduce8_96(const fx::i96 (&v)[8]) {
  const int lane = threadIdx.x & 31;
  const bool b4 = lane & 16, b3 = lane & 8, b2 = lane & 4;
  fx::i96 a[4], b[2];
#pragma unroll
  for (int k = 0; k < 4; ++k) a[k] = xor_add96(pick(b4, v[k + 4], v[k]), pick(b4, v[k], v[k + 4]), 16);
#pragma unroll
  for (int k = 0; k < 2; ++k) b[k] = xor_add96(pick(b3, a[k + 2], a[k]), pick(b3, a[k], a[k + 2]), 8);
  fx::i96 x = xor_add96(pick(b2, b[1], b[0]), pick(b2, b[0], b[1]), 4);
  x = xor_add96(x, x, 2);
  return xor_add96(x, x, 1);
}

// g of f~ from its own and upwind values, in fixed point.  `ok` is false when
// the largest of them is too small or too large (a sign bit counts as large),
// or the weighted sum far below it.
__device__ __forceinline__ double combine_fast(double f0, double fxv, double fyv, unsigned long long w0,
                                               unsigned long long wx, unsigned long long wy, bool& ok) {
  const unsigned h0 = (unsigned)__double2hiint(f0), hx = (unsigned)__double2hiint(fxv),
                 hy = (unsigned)__double2hiint(fyv);
  const unsigned emax = max(max(h0, hx), hy) >> 20;
  const unsigned long long r =
      fx::combine(w0, fx::align(h0, (unsigned)__double2loint(f0), emax), wx,
                  fx::align(hx, (unsigned)__double2loint(fxv), emax), wy,
                  fx::align(hy, (unsigned)__double2loint(fyv), emax));
  ok = emax - fx::kExpMin <= fx::kExpMax - fx::kExpMin && fx::combine_ok(r);
  unsigned hi, lo;
  fx::to_words(r, emax, hi, lo);
  return __hiloint2double((int)hi, (int)lo);
}

// The same in FP64 with the FP64 weights (integers over 2^63 keep fewer than
// 53 bits of a weight below 2^-10, and beside a front that weight's error is
// the result's).  A call: inlined, it would be scheduled ahead of the branch.
__device__ __noinline__ double combine_slow(double f0, double fxv, double fyv,
                                            const double4_32a* __restrict__ coef) {
  const double4_32a co = *coef;
  return fma(co.z, fyv, fma(co.y, fxv, co.x * f0));
}

// Own and upwind values of velocity j = (jx, jy) of a cell at the edge.
__device__ __forceinline__ void load_point(const Params& P, const Tables& T, const double2* __restrict__ fc,
                                           ptrdiff_t row, const CellEdge& C, int j, int jx, int jy, int sgx, int sgy,
                                           double2& f0, double2& fxv, double2& fyv) {
  f0 = fc[j];
  fxv = fyv = f0;
  if (sgx > 0) fxv = C.xlo ? ghost_at(P, T, XLO, j, jx, jy, C.nw[XLO], fc) : fc[j - P.nv];
  else if (sgx < 0) fxv = C.xhi ? ghost_at(P, T, XHI, j, jx, jy, C.nw[XHI], fc) : fc[j + P.nv];
  if (sgy > 0) fyv = C.ylo ? ghost_at(P, T, YLO, j, jx, jy, C.nw[YLO], fc) : fc[j - row];
  else if (sgy < 0) fyv = C.yhi ? ghost_at(P, T, YHI, j, jx, jy, C.nw[YHI], fc) : fc[j + row];
}

// The velocities of a lane in the fixed-point kernels: 2^lane_bits lanes share
// a row, the rows of the cell's W warps advance together, and a lane takes its
// columns jx = l + m 2^lane_bits one after the other, each over its rows
// jy = row0 + r step.
template <int W>
struct LaneMap {
  int l, width, row0, step, rows;
  __device__ __forceinline__ LaneMap(const Params& P, int wi) {
    const int lane = threadIdx.x & 31, lb = P.lane_bits;
    width = 1 << lb;
    l = lane & (width - 1);
    row0 = wi * (32 >> lb) + (lane >> lb);
    step = W * (32 >> lb);
    rows = (P.nvy + step - 1) / step;
  }
};

// Rows ahead that a lane asks into L1: with 8 warps per sub-partition at 64
// registers the next row's values cannot wait in registers (20 steps of 256^2 x
// 48^2: 51.3 ms without, 47.1 ms with 1 to 4 rows, before the sums of 65 to 75
// bits and h's third operation).
constexpr int kAhead = 2;
__device__ __forceinline__ void prefetch_l1(const double2* p) {
  asm volatile("prefetch.global.L1 [%0];" ::"l"(p));
}

// A1 + A2 of a warp's rows of a 2D cell, g on the integer pipe and h on the
// FP64 pipe, which run side by side (20 steps of 256^2 x 48^2, before the sums
// of 65 to 75 bits and h's third operation: both on the FP64 pipe 52.7 ms, both
// on the integer pipe 58.7 ms, this 47.1 ms); a column's weights and running
// sums stay in registers.
//  g: fixed point.  The running sums of first, second and third order over a
//     column's rows give sum g, sum j_y g and sum j_y^2 g as integers, and
//     times j_x the x sums.  Their unit has to lie far below the tail of a
//     narrow distribution: weighted with the squared index its rounding is the
//     error of the energy (59 bits below the range: 3e-15 to 1.3e-14 of theta
//     on +-20 thermal speeds with a tail of 1e-9; here below 9e-16).
//  h: three FP64 operations, summed as an integer.  (Parked over the column's x
//     weight it takes two, 4 % of the time; but with the rounding of the
//     quotients and of the product back h of a uniform state drifts by 0.024 to
//     0.031 of 2^-53 a step, rms, here by 0.009 to 0.017.)
// eg, eh: largest exponents of f~ that the sums' units are cut for (of f~
// itself: a neighbour may be any number of times as large when its weight is
// small).  The sums are valid (true) when no value exceeds them; otherwise they
// return raised to the largest exponents seen.
template <int W, bool EDGE>
__device__ __forceinline__ bool stream_rows_fixed(const Params& P, const Tables& T, const double2* __restrict__ fc,
                                                  ptrdiff_t row, const CellEdge& C, int wi,
                                                  double2* __restrict__ tile, double* __restrict__ sums, int& eg,
                                                  int& eh) {
  typedef unsigned long long u64;
  const int lane = threadIdx.x & 31, nvx = P.nvx, nvy = P.nvy, eu = eg + P.sum_room;
  const LaneMap<W> L(P, wi);
  const int h = L.row0, rpw = L.step, rows = L.rows;
  int topg = 0, toph = 0;
  const fx::i96 zero = {0u, 0u, 0u};
  fx::i96 hsum = zero, n0 = zero, x1 = zero, x2 = zero, i1 = zero, i2 = zero;
#pragma unroll 1
  for (int jl = L.l; jl - L.l < nvx; jl += L.width) {
    const bool in = jl < nvx;
    const int jx = in ? jl : nvx - 1;  // a column past the row repeats its last one and is not counted
    const int sgx = vi_sx(T.vinfo[jx]);
    const int offx = EDGE ? sgx : -sgx * P.nv;  // upwind in x: ix - sgn c_x
    const u64 wx = T.wx[jx], rest = ((u64)1 << fx::kWeightBits) - wx;
    const double ax = T.awx[jx];
    fx::i96 s1 = zero, s2 = zero, s3 = zero;
#pragma unroll 1
    for (int r = 0; r < rows; ++r) {
      const int jr = h + r * rpw, jy = min(jr, nvy - 1), j = jy * nvx + jx;
      const u64 wys = T.wy[jy], wy = wys & ~((u64)1 << 63);  // top bit: c_y < 0
      const double2 co = T.a0y[j];
      double2 f0, fxv, fyv, ft;
      if (EDGE) {
        load_point(P, T, fc, row, C, j, jx, jy, offx, vi_sy(T.vinfo[jy * nvx]), f0, fxv, fyv);
      } else {
        const double2* p = fc + j;
        const ptrdiff_t offy = (long long)wys < 0 ? row : -row;  // c_y = 0: any value, its weight is 0
        f0 = p[0];
        fxv = p[offx];
        fyv = p[offy];
        if (jr + kAhead * rpw < nvy) {
          const double2* a = p + kAhead * rpw * nvx;
          prefetch_l1(a);
          prefetch_l1(a + offx);
          prefetch_l1(a + offy);
        }
      }
      bool ok;
      ft.x = combine_fast(f0.x, fxv.x, fyv.x, rest - wy, wx, wy, ok);
      ft.y = fma(co.y, fyv.y, fma(ax, fxv.y, co.x * f0.y));
      // rare: negative values, values near the smallest doubles, fronts steeper than the weights
      if (!ok) ft.x = combine_slow(f0.x, fxv.x, fyv.x, T.coef + j);
      if (in && jr < nvy) {
        const unsigned hg = (unsigned)__double2hiint(ft.x), hh = (unsigned)__double2hiint(ft.y);
        tile[j] = ft;
        s1 = fx::add_units96(s1, hg, (unsigned)__double2loint(ft.x), (unsigned)eu);
        hsum = fx::add(hsum, fx::double_to_units96(hh, (unsigned)__double2loint(ft.y), (unsigned)eh));
        topg = max(topg, (int)(hg >> 20));
        toph = max(toph, (int)(hh >> 20));
      }
      s2 = fx::add(s2, s1);
      s3 = fx::add(s3, s2);
    }
    n0 = fx::add(n0, s1);
    i1 = fx::add(i1, s2);
    i2 = fx::add(i2, s3);
    x1 = fx::add(x1, fx::mul(s1, (unsigned)jx));
    x2 = fx::add(x2, fx::mul(s1, (unsigned)(jx * jx)));
  }
  topg = __reduce_max_sync(0xffffffffu, topg);
  toph = __reduce_max_sync(0xffffffffu, toph);
  const bool valid = topg <= eg && toph <= eh;
  if (valid) {
    // j_y of row r: A - rpw (rows - r); i1 = sum (rows - r) g, i2 = sum (rows - r)(rows - r + 1) / 2 g
    const unsigned A = (unsigned)(h + rpw * rows), B = (unsigned)rpw;
    const fx::i96 b1 = fx::mul(i1, B);
    fx::i96 v[8] = {n0, x1, x2, fx::add(fx::mul(n0, A), fx::neg(b1)),
                    fx::add(fx::add(fx::mul(n0, A * A), fx::neg(fx::mul(b1, 2u * A + B))), fx::mul(i2, 2u * B * B)),
                    hsum, zero, zero};
    const fx::i96 t = warp_reduce8_96(v);
    // from j to k = 2 j + 1 - n: lane group q holds value q of (1, j_x, j_x^2, j_y, j_y^2) g sums and the h sum
    const int q = lane >> 2, n = 1 - (q <= 2 ? nvx : nvy);
    const fx::i96 first = shfl96(t, 0), prev = shfl96(t, max(lane - 4, 0));
    const bool lin = q == 1 || q == 3, quad = q == 2 || q == 4;
    const fx::i96 k = lin ? fx::add(fx::mul(t, 2u), fx::muls(first, n))
                          : quad ? fx::add(fx::add(fx::mul(t, 4u), fx::muls(prev, 4 * n)), fx::mul(first, (unsigned)(n * n)))
                                 : t;
    if ((lane & 3) == 0 && q < kSums) sums[q] = unit_value(k, (q < 5 ? eu : eh) - 16);
  }
  eg = max(eg, topg);
  eh = max(eh, toph);
  return valid;
}

// Largest exponent fields of g and h over 128 samples of the cell, spread
// over both axes by an odd stride (nv >= 128), plus the headroom.
__device__ __forceinline__ void sample_range(const double2* __restrict__ fc, int nv, int& eg, int& eh) {
  const int lane = threadIdx.x & 31;
  unsigned sg = 0, sh = 0;
  const int stride = (nv >> 7) | 1;
#pragma unroll
  for (int s = 0; s < 4; ++s) {
    const int at = (4 * lane + s) * stride;  // below 2 nv
    const double2 v = fc[at < nv ? at : at - nv];
    sg = max(sg, (unsigned)__double2hiint(v.x));
    sh = max(sh, (unsigned)__double2hiint(v.y));
  }
  eg = (int)((__reduce_max_sync(0xffffffffu, sg) >> 20) + fx::kHeadroom);
  eh = (int)((__reduce_max_sync(0xffffffffu, sh) >> 20) + fx::kHeadroom);
}

// The same rows in FP64, for any values.
template <int W>
__device__ __noinline__ void stream_rows_f64(const Params& P, const Tables& T, const double2* __restrict__ fc,
                                             ptrdiff_t row, const CellEdge& C, int wi, double2* __restrict__ tile,
                                             double* __restrict__ sums) {
  const LaneMap<W> L(P, wi);
  const int lane = threadIdx.x & 31;
  double s0 = 0.0, sx = 0.0, sy = 0.0, se = 0.0;
  for (int jx = L.l; jx < P.nvx; jx += L.width)
    for (int jy = L.row0; jy < P.nvy; jy += L.step) {
      const int j = jy * P.nvx + jx, vi = T.vinfo[j];
      const double4_32a co = T.coef[j];
      const double2 cxy = T.cxy[j];
      double2 f0, fx, fy, ft;
      load_point(P, T, fc, row, C, j, jx, jy, vi_sx(vi), vi_sy(vi), f0, fx, fy);
      ft.x = fma(co.z, fy.x, fma(co.y, fx.x, co.x * f0.x));
      ft.y = fma(co.z, fy.y, fma(co.y, fx.y, co.x * f0.y));
      tile[j] = ft;
      s0 += ft.x;
      sx = fma(cxy.x, ft.x, sx);
      sy = fma(cxy.y, ft.x, sy);
      se = fma(co.w, ft.x, se) + ft.y;
    }
  const double w = warp_reduce4(s0, sx, sy, se);
  if ((lane & 7) == 0) sums[lane >> 3] = w;
}

// A0 to A2 of a warp's rows; returns the kind of its sums.
template <int W>
__device__ __forceinline__ int stream_rows(const Params& P, const Tables& T, const double2* __restrict__ fin, int cell,
                                           int wi, double2* __restrict__ tile, double* __restrict__ sums) {
  const int ix = cell % P.nx, iy = cell / P.nx;
  const double2* __restrict__ fc = fin + (size_t)cell * P.nv;
  const ptrdiff_t row = (ptrdiff_t)P.nx * P.nv;
  const CellEdge C = cell_edge<2>(P, T, fc, ix, iy);
  int eg, eh;
  sample_range(fc, P.nv, eg, eh);
  const bool edge = C.xlo || C.xhi || C.ylo || C.yhi;
  // a second pass takes the largest exponents of the first where they exceed the sampled ones
  for (int pass = 0; pass < 2; ++pass) {
    if (min(eg, eh) < (int)fx::kExpMin || max(eg, eh) > (int)fx::kExpMax) break;
    if (edge ? stream_rows_fixed<W, true>(P, T, fc, row, C, wi, tile, sums, eg, eh)
             : stream_rows_fixed<W, false>(P, T, fc, row, C, wi, tile, sums, eg, eh))
      return SUMS_INDEX;
  }
  stream_rows_f64<W>(P, T, fc, row, C, wi, tile, sums);
  return SUMS_VELOCITY;
}

// A1 + A2 in FP64 for any grid and any values.
template <int DIM>
__device__ __forceinline__ void stream_cell_f64(const Params& P, const Tables& T, const double2* __restrict__ fin,
                                                const double2* __restrict__ fc, int ix, ptrdiff_t row,
                                                const CellEdge& C, double2* __restrict__ tile,
                                                double* __restrict__ sums) {
  const int lane = threadIdx.x & 31;
  const int nv = P.nv, nx = P.nx;
  double s0 = 0.0, sx = 0.0, sy = 0.0, se = 0.0;
  for (int j = lane; j < nv; j += 32) {
    const int vi = T.vinfo[j];
    const int sgx = vi_sx(vi);
    const double4_32a co = T.coef[j];
    const double2 cxy = T.cxy[j];
    double2 ft;
    if (DIM == 2) {
      const int jx = vi_jx(vi), jy = vi_jy(vi), sgy = vi_sy(vi);
      const double2 f0 = fc[j];
      double2 fx = f0, fy = f0;
      if (sgx > 0) fx = C.xlo ? ghost_at(P, T, XLO, j, jx, jy, C.nw[XLO], fc) : fc[j - nv];
      else if (sgx < 0) fx = C.xhi ? ghost_at(P, T, XHI, j, jx, jy, C.nw[XHI], fc) : fc[j + nv];
      if (sgy > 0) fy = C.ylo ? ghost_at(P, T, YLO, j, jx, jy, C.nw[YLO], fc) : fc[j - row];
      else if (sgy < 0) fy = C.yhi ? ghost_at(P, T, YHI, j, jx, jy, C.nw[YHI], fc) : fc[j + row];
      ft.x = fma(co.z, fy.x, fma(co.y, fx.x, co.x * f0.x));
      ft.y = fma(co.z, fy.y, fma(co.y, fx.y, co.x * f0.y));
      sy = fma(cxy.y, ft.x, sy);
    } else {
      const int i1 = ix - T.shift[j], i2 = i1 - sgx;
      double2 f1, f2;
      if (i1 < 0) f1 = ghost_at(P, T, XLO, j, j, 0, C.nw[XLO], fc);
      else if (i1 >= nx) f1 = ghost_at(P, T, XHI, j, j, 0, C.nw[XHI], fc);
      else f1 = fin[(size_t)i1 * nv + j];
      if (i2 < 0) f2 = ghost_at(P, T, XLO, j, j, 0, C.nw[XLO], fc);
      else if (i2 >= nx) f2 = ghost_at(P, T, XHI, j, j, 0, C.nw[XHI], fc);
      else f2 = fin[(size_t)i2 * nv + j];
      ft.x = fma(co.y, f2.x, co.x * f1.x);
      ft.y = fma(co.y, f2.y, co.x * f1.y);
    }
    tile[j] = ft;
    s0 += ft.x;
    sx = fma(cxy.x, ft.x, sx);
    se = fma(co.w, ft.x, se) + ft.y;
  }
  const double w = warp_reduce4(s0, sx, sy, se);
  if ((lane & 7) == 0) sums[lane >> 3] = w;
}

template <int DIM>
__device__ __forceinline__ void stream_cell(const Params& P, const Tables& T, const double2* __restrict__ fin,
                                            int cell, double2* __restrict__ tile, double* __restrict__ sums) {
  const int ix = cell % P.nx, iy = cell / P.nx;
  const double2* __restrict__ fc = fin + (size_t)cell * P.nv;
  const CellEdge C = cell_edge<DIM>(P, T, fc, ix, iy);
  stream_cell_f64<DIM>(P, T, fin, fc, ix, (ptrdiff_t)P.nx * P.nv, C, tile, sums);
}

// ---- phase 2 ---------------------------------------------------------------
// Sums of five values over the L lanes of a group (sub = 0 .. L-1, L a power
// of two >= 4), returned to every lane of the group.  Recursive halving: the
// first exchange splits the values 3 + 2 between the two halves of the
// group, the second 2 + 1 within each half, the third leaves one value per
// lane, then plain butterflies; 8 FP64 additions at L = 32 (5 at L = 4)
// instead of 5 log2 L.  The lane pattern of each value is fixed, so the
// result does not depend on the data.
template <int L>
__device__ __forceinline__ void group_sum5(double& m0, double& m1, double& m2, double& m3, double& m4,
                                           int sub) {
  static_assert(L >= 4 && (L & (L - 1)) == 0, "group of 4, 8, 16 or 32 lanes");
  constexpr unsigned kAll = 0xffffffffu;
  const int base = (threadIdx.x & 31) - sub;
  // 1: the low half keeps (m0, m1, m2), the high half (m3, m4, 0)
  const bool h1 = sub & (L / 2);
  double a0 = h1 ? m3 : m0, a1 = h1 ? m4 : m1, a2 = h1 ? 0.0 : m2;
  const double t0 = h1 ? m0 : m3, t1 = h1 ? m1 : m4, t2 = h1 ? m2 : 0.0;
  a0 += __shfl_xor_sync(kAll, t0, L / 2);
  a1 += __shfl_xor_sync(kAll, t1, L / 2);
  a2 += __shfl_xor_sync(kAll, t2, L / 2);
  // 2: of (a0, a1, a2) the low quarter keeps (a0, a1), the high one (a2, 0)
  const bool h2 = sub & (L / 4);
  double k0 = h2 ? a2 : a0, k1 = h2 ? 0.0 : a1;
  const double u0 = h2 ? a0 : a2, u1 = h2 ? a1 : 0.0;
  k0 += __shfl_xor_sync(kAll, u0, L / 4);
  k1 += __shfl_xor_sync(kAll, u1, L / 4);
  if (L == 4) {
    // lane 0: (m0, m1), lane 1: (m2, 0), lane 2: (m3, m4), lane 3: (0, 0)
    m0 = __shfl_sync(kAll, k0, base);
    m1 = __shfl_sync(kAll, k1, base);
    m2 = __shfl_sync(kAll, k0, base + 1);
    m3 = __shfl_sync(kAll, k0, base + 2);
    m4 = __shfl_sync(kAll, k1, base + 2);
    return;
  }
  // 3: one value per lane, then the remaining lane bits summed out
  const bool h3 = sub & (L / 8);
  double v = h3 ? k1 : k0;
  v += __shfl_xor_sync(kAll, h3 ? k0 : k1, L / 8);
#pragma unroll
  for (int s = L / 16; s > 0; s >>= 1) v += __shfl_xor_sync(kAll, v, s);
  // m0 at sub 0, m1 at L/8, m2 at L/4, m3 at L/2, m4 at L/2 + L/8
  m0 = __shfl_sync(kAll, v, base);
  m1 = __shfl_sync(kAll, v, base + L / 8);
  m2 = __shfl_sync(kAll, v, base + L / 4);
  m3 = __shfl_sync(kAll, v, base + L / 2);
  m4 = __shfl_sync(kAll, v, base + L / 2 + L / 8);
}

// Exponentials e_j = exp(-(c_j - u)^2 / theta) of one axis for one cell,
// lanes sub, sub + L, ... of the cell's group; stores them when `store`;
// returns the group's central sums M_m = sum d^m e, d = c_j - u, m = 0..4.
// On the uniform grid a lane's points are d_i = d_0 + i D (D = L dc), and a
// Gaussian obeys e_{i+1} = e_i r_i, r_i = exp(-(2 d_i D + D^2) / theta),
// r_{i+1} = r_i exp(-2 D^2 / theta): three exponentials per lane and two
// products per further point instead of one exponential per point (each
// product adds a rounding: after k points the relative error is about k^2
// ulp, 1e-14 at k = 8).  Lanes with fewer than four points, and where e_0
// could underflow or r_0 overflow (theta far below the grid's scale), take
// one exponential per point.
template <int L>
__device__ __forceinline__ void axis_sums(const double* __restrict__ c, int n, double dc, double u,
                                          double inv_th, int sub, bool store, double* __restrict__ out, bool want,
                                          double M[5]) {
  double m0 = 0.0, m1 = 0.0, m2 = 0.0, m3 = 0.0, m4 = 0.0;
  if (sub < n) {
    const double D = L * dc;
    const double d0 = c[sub] - u;
    const double x0 = (d0 * d0) * inv_th, y0 = (2.0 * d0 * D + D * D) * inv_th;
    const bool rec = n >= 4 * L && x0 < 600.0 && -y0 < 600.0;
    double e = exp(-x0);
    double r = rec ? exp(-y0) : 0.0;
    const double q = rec ? exp(-2.0 * D * D * inv_th) : 0.0;
    for (int j = sub;;) {
      const double d = c[j] - u;
      if (store) out[j] = e;
      if (want) {
        double t = e;
        m0 += t;
        t *= d;
        m1 += t;
        t *= d;
        m2 += t;
        t *= d;
        m3 += t;
        t *= d;
        m4 += t;
      }
      j += L;
      if (j >= n) break;
      if (rec) {
        e *= r;
        r *= q;
      } else {
        const double dn = c[j] - u;
        e = exp(-(dn * dn) * inv_th);
      }
    }
  }
  if (want) group_sum5<L>(m0, m1, m2, m3, m4, sub);
  M[0] = m0;
  M[1] = m1;
  M[2] = m2;
  M[3] = m3;
  M[4] = m4;
}

// The cell's moments from the sums of its W warps, of either kind; k -> c is
// affine on the uniform grid: c = mid + half k.
template <int W>
__device__ __forceinline__ void cell_moments(const Params& P, const VelocityGrid& V, const double (*sums)[kSums],
                                             const int* kind, double q[4]) {
  double t[4] = {0.0, 0.0, 0.0, 0.0}, u[kSums] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  bool index = false;
#pragma unroll
  for (int w = 0; w < W; ++w) {
    if (kind[w] == SUMS_VELOCITY) {
#pragma unroll
      for (int k = 0; k < 4; ++k) t[k] += sums[w][k];
    } else {
      index = true;
#pragma unroll
      for (int k = 0; k < kSums; ++k) u[k] += sums[w][k];
    }
  }
  if (index) {
    const double tx = V.half_x * u[1], ty = V.half_y * u[3];
    const double sx = fma(V.mid_x, u[0], tx), sy = fma(V.mid_y, u[0], ty);
    // sum c^2 g = mid (sum c g + half sum k g) + half^2 sum k^2 g per axis
    const double ex = fma(V.half_x * V.half_x, u[2], V.mid_x * (sx + tx));
    const double ey = fma(V.half_y * V.half_y, u[4], V.mid_y * (sy + ty));
    t[0] += u[0];
    t[1] += sx;
    t[2] += sy;
    t[3] += (ex + ey) + u[5];
  }
  moments_from_sums(t[0], t[1], t[2], t[3], P.dv, q);
}

template <int DIM, int G, int W = 1>
__device__ void maxwellian_cells(const Params& P, const Tables& T, int cell0, const double (*sums)[kSums],
                                 const int* kind,
                                 double* __restrict__ phx, double* __restrict__ phy, double* sb,
                                 double* sk, int* sok, double4_32a* __restrict__ mom,
                                 double4_32a* __restrict__ par, int* __restrict__ err) {
  constexpr int L = 32 / G;
  const int lane = threadIdx.x & 31, c = lane / L, sub = lane % L;
  const int cell = cell0 + c;
  const bool live = cell < P.nx * P.ny;
  double qm[4] = {1.0, 0.0, 0.0, 1.0};  // moments of f~ (Eq. macroscopic)
  if (live) cell_moments<W>(P, T.grid, sums + c * W, kind + c * W, qm);
  bool ok = live && moments_ok(qm);
  // a failed cell keeps its lanes busy on a harmless stand-in state
  const double q[4] = {ok ? qm[0] : 1.0, ok ? qm[1] : 0.0, ok ? qm[2] : 0.0, ok ? qm[3] : 1.0};
  double a, b;
  relax_weights(P, q, a, b);
  double* px = phx + c * P.nvx;
  double* py = phy + c * P.nvy;
  const bool cons = P.conservative != 0;
  EffState E;
  eff_init(E, q, !(cons && ok));
  double Mx[5], My[5] = {1.0, 0.0, 0.0, 0.0, 0.0};
  for (int round = 0; round <= kEffMaxIt; ++round) {
    const bool need = round == 0 || E.reeval;
    if (!__any_sync(0xffffffffu, need)) break;
    const double inv_th = E.ith;
    double Mt[5];
    axis_sums<L>(T.cx, P.nvx, P.dcx, E.base[1], inv_th, sub, need, px, cons, Mt);
    if (need)
      for (int m = 0; m < 5; ++m) Mx[m] = Mt[m];
    if (DIM == 2) {
      axis_sums<L>(T.cy, P.nvy, P.dcy, E.base[2], inv_th, sub, need, py, cons, Mt);
      if (need)
        for (int m = 0; m < 5; ++m) My[m] = Mt[m];
    }
    E.reeval = false;
    eff_iterate<DIM>(P, q, Mx, My, E);  // A3, linearised about E.base
  }
  if (E.fail) ok = false;
  const double* p = E.p;
  if (ok) {
    // A4 factors: a Phi_g = px[jx] py[jy], moved from E.base to p
    double w1x, w1y, w2;
    eff_lin(E, w1x, w1y, w2);
    const double pref = (DIM == 1) ? p[0] * rsqrt(kPi() * p[3]) : p[0] / (kPi() * p[3]);
    const double ap = a * pref;
    for (int j = sub; j < P.nvx; j += L) {
      const double d = T.cx[j] - E.base[1];
      px[j] = ap * (px[j] * fma(d, fma(d, w2, w1x), 1.0));
    }
    if (DIM == 2) {
      for (int j = sub; j < P.nvy; j += L) {
        const double d = T.cy[j] - E.base[2];
        py[j] = py[j] * fma(d, fma(d, w2, w1y), 1.0);
      }
    }
  }
  if (sub == 0) {
    sb[c] = b;
    sk[c] = (DIM == 1) ? p[3] : 0.5 * p[3];
    sok[c] = ok ? 1 : 0;
    if (live) {
      store4(mom + cell, qm[0], qm[1], qm[2], qm[3]);
      if (par) store4(par + cell, p[0], p[1], p[2], p[3]);
      if (!ok) atomicOr(err, E.fail ? ERR_EFFECTIVE : ERR_MOMENT);
    }
  }
}

// Phase 2 of a 2D CTA on two warps: the y-axis Gaussian sums and factors of
// the G cells run on warp 1 (another SM sub-partition) while warp 0 does the
// x axis and the scalar solve, so the CTA's other warps wait at the barrier
// for about one axis less.  Every value is computed by the same functions in
// the same order as in maxwellian_cells, so the results are the same bit
// for bit.  Warp 0 hands warp 1 the base point of each round and the factor
// update; warp 1 hands back the y central sums (named barrier 1, 64 threads).
template <int G>
struct SolveXchg {
  double ub[G], ith[G];  // y base velocity and 1 / theta_b of the round
  double my[G][5];       // y central sums of the round
  double w1y[G], w2[G];  // factor update (after the last round)
  int need[G], ok[G];
  int go;
};

__device__ __forceinline__ void pair_barrier() { asm volatile("bar.sync 1, 64;" ::: "memory"); }

template <int G>
__device__ void maxwellian_cells_2w(const Params& P, const Tables& T, int cell0, const double (*sums)[kSums],
                                    const int* kind,
                                    double* __restrict__ phx, double* __restrict__ phy, double* sb, double* sk,
                                    int* sok, double4_32a* __restrict__ mom, double4_32a* __restrict__ par,
                                    int* __restrict__ err, SolveXchg<G>& X) {
  constexpr int L = 32 / G;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, c = lane / L, sub = lane % L;
  const bool cons = P.conservative != 0;
  if (warp == 1) {
    double* py = phy + c * P.nvy;
    for (;;) {
      pair_barrier();  // base point of the round published
      if (!X.go) break;
      const bool need = X.need[c] != 0;
      double Mt[5];
      axis_sums<L>(T.cy, P.nvy, P.dcy, X.ub[c], X.ith[c], sub, need, py, cons, Mt);
      if (sub == 0)
        for (int m = 0; m < 5; ++m) X.my[c][m] = Mt[m];
      pair_barrier();  // sums handed over
    }
    pair_barrier();  // factor update published
    if (X.ok[c]) {
      const double ub = X.ub[c], w1y = X.w1y[c], w2 = X.w2[c];
      for (int j = sub; j < P.nvy; j += L) {
        const double d = T.cy[j] - ub;
        py[j] = py[j] * fma(d, fma(d, w2, w1y), 1.0);
      }
    }
    return;
  }
  const int cell = cell0 + c;
  const bool live = cell < P.nx * P.ny;
  double qm[4] = {1.0, 0.0, 0.0, 1.0};  // moments of f~ (Eq. macroscopic)
  if (live) cell_moments<1>(P, T.grid, sums + c, kind + c, qm);
  bool ok = live && moments_ok(qm);
  const double q[4] = {ok ? qm[0] : 1.0, ok ? qm[1] : 0.0, ok ? qm[2] : 0.0, ok ? qm[3] : 1.0};
  double* px = phx + c * P.nvx;
  EffState E;
  eff_init(E, q, !(cons && ok));
  double a = 0.0, b = 0.0;
  double Mx[5], My[5];
  // every exit from this loop goes through a published go = 0 (warp 1
  // leaves its loop on it), so the two warps pass the same barriers
  for (int round = 0;; ++round) {
    const bool need = round <= kEffMaxIt && (round == 0 || E.reeval);
    const bool go = __any_sync(0xffffffffu, need);
    if (sub == 0) {
      X.need[c] = need ? 1 : 0;
      X.ub[c] = E.base[2];
      X.ith[c] = E.ith;
    }
    if (lane == 0) X.go = go ? 1 : 0;
    pair_barrier();
    if (!go) break;
    double Mt[5];
    axis_sums<L>(T.cx, P.nvx, P.dcx, E.base[1], E.ith, sub, need, px, cons, Mt);
    if (need)
      for (int m = 0; m < 5; ++m) Mx[m] = Mt[m];
    if (round == 0) relax_weights(P, q, a, b);
    pair_barrier();
    if (need)
      for (int m = 0; m < 5; ++m) My[m] = X.my[c][m];
    E.reeval = false;
    eff_iterate<2>(P, q, Mx, My, E);  // A3, linearised about E.base
  }
  if (E.fail) ok = false;
  const double* p = E.p;
  double w1x = 0.0, w1y = 0.0, w2 = 0.0;
  if (ok) eff_lin(E, w1x, w1y, w2);
  if (sub == 0) {
    X.ok[c] = ok ? 1 : 0;
    X.ub[c] = E.base[2];
    X.w1y[c] = w1y;
    X.w2[c] = w2;
  }
  pair_barrier();
  if (ok) {
    // A4 factors: a Phi_g = px[jx] py[jy], moved from E.base to p
    const double ap = a * (p[0] / (kPi() * p[3]));
    for (int j = sub; j < P.nvx; j += L) {
      const double d = T.cx[j] - E.base[1];
      px[j] = ap * (px[j] * fma(d, fma(d, w2, w1x), 1.0));
    }
  }
  if (sub == 0) {
    sb[c] = b;
    sk[c] = 0.5 * p[3];
    sok[c] = ok ? 1 : 0;
    if (live) {
      store4(mom + cell, qm[0], qm[1], qm[2], qm[3]);
      if (par) store4(par + cell, p[0], p[1], p[2], p[3]);
      if (!ok) atomicOr(err, E.fail ? ERR_EFFECTIVE : ERR_MOMENT);
    }
  }
}

// Phase 2 of the fixed-point kernels: the Gaussians of a cell on its own warp
// and on the integer pipe, the scalar solve with cells in lanes on one warp.
template <int G>
struct CellSolve {
  AxisBase base[G][2];
  double sums[G][2][3];  // sum e, sum k' e, sum k'^2 e
  double ap[G];          // a n / (pi theta)
  int need[G];
  int go;  // 1: sums wanted, 0: factors wanted, -1: a cell is out of range (FP64 path)
};

// A cell's solve: moments q, parameters p (the base point of the Gaussians),
// ith = 1 / theta, isq = 1 / sqrt(theta) of p.
struct FixedSolve {
  double q[4], p[4];
  double ith, isq;
  double iq0, iq3, ivs;  // 1 / n, 1 / theta, 1 / sqrt(theta) of q
  int it;
  bool conv, out;  // out: parameters beyond the range of the FP32 starts, or no convergence (the FP64 path decides)
  // n / (pi theta), the same in D(p) and in Phi: a constant rounded one way in
  // one and another way in the other is a density that changes with every step
  __device__ __forceinline__ double prefactor() const {
    const double t = p[0] * ith;
    return fma(t, 0.31830988618379067, t * -1.9678676675182486e-17);  // 1 / pi
  }
};

// Publishes the base point of a cell; false when it or a velocity lies too
// far out for the fixed-point Gaussian.
template <int G>
__device__ __forceinline__ bool publish_base(const Params& P, const VelocityGrid& V, const FixedSolve& E, int c, CellSolve<G>& X) {
  AxisBase x, y;
  const bool fx = axis_base(P.nvx, V.half_x, V.inv_half_x, V.mid_x, E.p[1], E.isq, x);
  const bool fy = axis_base(P.nvy, V.half_y, V.inv_half_y, V.mid_y, E.p[2], E.isq, y);
  X.base[c][0] = x;
  X.base[c][1] = y;
  return fx && fy;
}

// nu = n theta^(1-omega) and the relaxation weights, exp(-nu dt) on the
// integer pipe where its argument allows.
__device__ __forceinline__ void relax_weights_fixed(const Params& P, const FixedSolve& E, double& a, double& b) {
  const double nu = E.q[0] * (P.omega == 0.5 ? E.q[3] * E.ivs : pow_fixed(E.q[3], 1.0 - P.omega));
  const double x = nu * P.dt;
  if (!P.relax_exact) {
    a = x;
    b = 1.0 - a;
    return;
  }
  b = exp_neg_fixed(x);
  a = 1.0 - b;
}

// One update p <- p + (q - D(p)) (A3) from the central sums M_m of both axes
// at p, with the stopping rules of eff_iterate.
__device__ __forceinline__ void eff_update(double dv, const double (&Mx)[3], const double (&My)[3],
                                           FixedSolve& E) {
  ++E.it;
  const double rxy = rcp3(Mx[0] * My[0]);
  const double rx = My[0] * rxy, ry = Mx[0] * rxy;
  const double mux = Mx[1] * rx, muy = My[1] * ry;
  double d[4];
  d[0] = E.prefactor() * dv * (Mx[0] * My[0]);
  d[1] = E.p[1] + mux;
  d[2] = E.p[2] + muy;
  const double var = fma(Mx[2], rx, -mux * mux) + fma(My[2], ry, -muy * muy);
  d[3] = (2.0 / 3.0) * fma(0.5, E.p[3], var);
  unsigned r = 0;  // high word of the largest scaled update
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const double delta = E.q[k] - d[k];
    E.p[k] += delta;
    r = max(r, abs_hi(delta * (k == 0 ? E.iq0 : k == 3 ? E.iq3 : E.ivs)));
  }
  // the high words of kEffTol = 1e-13, sqrt(kEffTol / 100) = 3.16e-8 and kEffFail = 1e-9
  if (!in_range(E.p[0]) || !in_range(E.p[3]) || r >= 0x7ff00000u) E.out = true;
  else if (r < 0x3d3c25c2u || (E.it == 1 && r < 0x3e60fa33u)) E.conv = true;
  else if (E.it >= kEffMaxIt) (r < 0x3e112e0bu ? E.conv : E.out) = true;
  E.isq = rsqrt3(E.p[3]);
  E.ith = rcp3(E.p[3]);
}

// Which axis of its cell a warp works on, with which lane of how many: half a
// warp per axis when the cell has one warp, a warp per axis when it has more
// (the others none, x = 2).
template <int W>
struct AxisMap {
  static constexpr int kLanes = W == 1 ? 16 : 32;
  int x, i;
  __device__ __forceinline__ AxisMap(int wi) {
    const int lane = threadIdx.x & 31;
    x = W == 1 ? lane >> 4 : min(wi, 2);
    i = lane & (kLanes - 1);
  }
};

// Sums of cell c's Gaussians at the base point, along the warp's axis.
template <int G, int W>
__device__ __forceinline__ void gauss_sums(const Params& P, int c, int wi, CellSolve<G>& X) {
  const AxisMap<W> A(wi);
  if (W > 2 && A.x > 1) return;  // the whole warp
  const double t = axis_index_sums<AxisMap<W>::kLanes>(A.x == 0 ? P.nvx : P.nvy, X.base[c][A.x], A.i);
  if (A.i < 3) X.sums[c][A.x][A.i] = t;
}

// Cell c's a Phi factors at the final parameters, along the warp's axis.
template <int G, int W>
__device__ __forceinline__ void gauss_factors(const Params& P, int c, int wi, const CellSolve<G>& X,
                                              double* __restrict__ px, double* __restrict__ py) {
  const AxisMap<W> A(wi);
  if (W > 2 && A.x > 1) return;
  const int n = A.x == 0 ? P.nvx : P.nvy;
  const AxisBase B = X.base[c][A.x];
  const double scale = X.ap[c];
  double* out = A.x == 0 ? px : py;
#pragma unroll 1
  for (int j = A.i; j < n; j += A.kLanes) {
    unsigned q2, hi, lo;
    const unsigned long long q = fx::gauss(B.a * (2 * j + 1 - n) - B.c, (const fx::u64*)kExp2, q2);
    fx::gauss_words(q, q2, hi, lo);
    const double e = __hiloint2double((int)hi, (int)lo);
    out[j] = A.x == 0 ? scale * e : e;
  }
}

// All threads of the CTA.  Leaves factors, weights and ok of every cell; false
// when they come from maxwellian_cells.
template <int G, int W>
__device__ __forceinline__ bool maxwellian_cells_fixed(const Params& P, const Tables& T, int cell0,
                                                       const double (*sums)[kSums], const int* kind,
                                                       double* __restrict__ phx, double* __restrict__ phy, double* sb,
                                                       double* sk, int* sok, double4_32a* __restrict__ mom,
                                                       double4_32a* __restrict__ par, int* __restrict__ err,
                                                       CellSolve<G>& X) {
  const VelocityGrid& V = T.grid;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, mine = warp / W, wi = warp % W;
  // the solving warp varies from CTA to CTA, so that the FP64 work of the
  // solves is spread over the SM's four sub-partitions
  const int solver = (int)((blockIdx.x * 0x9E3779B1u) >> 16) % (G * W);
  const bool solving = warp == solver;
  const int c = lane % G, cell = cell0 + c;
  const bool live = cell < P.nx * P.ny, wr = lane < G;
  double qm[4] = {1.0, 0.0, 0.0, 1.0}, a = 0.0, b = 0.0;
  bool ok = false;
  FixedSolve E;
  if (solving) {
    if (live) cell_moments<W>(P, T.grid, sums + c * W, kind + c * W, qm);
    ok = live && moments_ok(qm);
    bool fit = !ok || (in_range(qm[0]) && in_range(qm[3]));
#pragma unroll
    for (int k = 0; k < 4; ++k) E.q[k] = E.p[k] = ok && fit ? qm[k] : (k == 0 || k == 3) ? 1.0 : 0.0;
    E.ivs = E.isq = rsqrt3(E.q[3]);
    E.iq3 = E.ith = rcp3(E.q[3]);
    E.iq0 = rcp3(E.q[0]);
    E.it = 0;
    E.conv = P.conservative == 0 || !ok;
    E.out = false;
    if (wr) {
      const bool reach = publish_base(P, V, E, c, X);
      fit = fit && (reach || !ok);
      X.need[c] = !E.conv;
    }
    const bool all = __all_sync(0xffffffffu, fit);
    const bool any = __any_sync(0xffffffffu, wr && !E.conv);
    if (lane == 0) X.go = !all ? -1 : any ? 1 : 0;
  }
  __syncthreads();
  bool weighted = false;
  while (X.go > 0) {
    if (solving && !weighted) {
      relax_weights_fixed(P, E, a, b);
      weighted = true;
    }
    if (X.need[mine]) gauss_sums<G, W>(P, mine, wi, X);
    __syncthreads();
    if (solving) {
      bool fit = true;
      if (!E.conv) {
        double M[2][3];
        central_sums(X.sums[c][0], X.base[c][0].k0, V.half_x, V.mid_x, E.p[1], M[0]);
        central_sums(X.sums[c][1], X.base[c][1].k0, V.half_y, V.mid_y, E.p[2], M[1]);
        eff_update(P.dv, M[0], M[1], E);
        if (wr) fit = !E.out && publish_base(P, V, E, c, X);
      }
      if (wr) X.need[c] = !E.conv;
      const bool all = __all_sync(0xffffffffu, fit);
      const bool any = __any_sync(0xffffffffu, wr && !E.conv);
      if (lane == 0) X.go = !all ? -1 : any ? 1 : 0;
    }
    __syncthreads();
  }
  if (X.go < 0) {
    if (warp == 0) maxwellian_cells<2, G, W>(P, T, cell0, sums, kind, phx, phy, sb, sk, sok, mom, par, err);
    __syncthreads();
    return false;
  }
  if (solving) {
    if (!weighted) relax_weights_fixed(P, E, a, b);
    if (wr) {
      X.ap[c] = a * E.prefactor();
      sb[c] = b;
      sk[c] = 0.5 * E.p[3];
      sok[c] = ok ? 1 : 0;
      if (live) {
        store4(mom + cell, qm[0], qm[1], qm[2], qm[3]);
        if (par) store4(par + cell, E.p[0], E.p[1], E.p[2], E.p[3]);
        if (!ok) atomicOr(err, ERR_MOMENT);
      }
    }
  }
  __syncthreads();
  if (sok[mine]) gauss_factors<G, W>(P, mine, wi, X, phx + mine * P.nvx, phy + mine * P.nvy);
  if (W == 1) __syncwarp();
  else __syncthreads();
  return true;
}

// ---- phase 3 ---------------------------------------------------------------
// A4 for the warp's cell: f^{n+1} = b f~ + a Phi from the f~ parked in the
// cell's output slots, a Phi_g = px[jx] py[jy], a Phi_h = kappa a Phi_g.
template <int DIM>
__device__ __forceinline__ void relax_cell(const Params& P, const Tables& T, double2* __restrict__ fo,
                                           const double* __restrict__ px, const double* __restrict__ py, double b,
                                           double kappa) {
  const int lane = threadIdx.x & 31;
#pragma unroll 4
  for (int j = lane; j < P.nv; j += 32) {
    const double2 ft = fo[j];
    double aphi;
    if (DIM == 2) {
      const int vi = T.vinfo[j];
      aphi = px[vi_jx(vi)] * py[vi_jy(vi)];
    } else {
      aphi = px[j];
    }
    fo[j] = make_double2(fma(b, ft.x, aphi), fma(b, ft.y, kappa * aphi));
  }
}

// h of one value in FP64 (a call, see combine_slow).
__device__ __noinline__ double relax_slow(double h, double aphi, double b, double kappa) {
  return fma(b, h, kappa * aphi);
}

// The same for a cell streamed by stream_rows_fixed (rows and columns of a
// lane as there): g in two FP64 operations, h on the integer pipe beside them, as two products of 63-bit
// significands aligned, added and rounded once (error half an ulp plus about
// 2^-58).  Values that are not positive normals well inside the range take
// FP64.
template <int W>
__device__ __forceinline__ void relax_rows_fixed(const Params& P, int wi, double2* __restrict__ fo,
                                                 const double* __restrict__ px, const double* __restrict__ py,
                                                 double b, double kappa) {
  typedef unsigned long long u64;
  constexpr int kRows = 4;
  const LaneMap<W> L(P, wi);
  const int rpw = L.step, nvx = P.nvx, nvy = P.nvy;
  const unsigned hk = (unsigned)__double2hiint(kappa);
  const u64 wk = fx::top63(hk, (unsigned)__double2loint(kappa));
  const int ek = (int)(hk >> 20) - 1022;
  // weights as 63-bit significands and exponents; a or b not positive (Euler
  // form, steps beyond the collision time): every value takes FP64
  const unsigned hb = (unsigned)__double2hiint(b);
  const bool fit = min(hb, hk) >= (400u << 20) && max(hb, hk) < (1600u << 20);
  const u64 wb = fx::top63(hb, (unsigned)__double2loint(b));
  const int eb = (int)(hb >> 20) - 1022;
#pragma unroll 1
  for (int jx = L.l; jx < nvx; jx += L.width) {
    const double xv = px[jx];
#pragma unroll 1
    for (int j0 = L.row0; j0 < nvy; j0 += kRows * rpw) {
      double2 ft[kRows];
      double2* __restrict__ p = fo + j0 * nvx + jx;
#pragma unroll
      for (int u = 0; u < kRows; ++u) ft[u] = j0 + u * rpw < nvy ? p[u * rpw * nvx] : make_double2(1.0, 1.0);
#pragma unroll
      for (int u = 0; u < kRows; ++u) {
        if (j0 + u * rpw < nvy) {
          const double aphi = xv * py[j0 + u * rpw];
          const unsigned ha = (unsigned)__double2hiint(aphi);
          int e;
          const u64 m = fx::mulhi(fx::top63(ha, (unsigned)__double2loint(aphi)), wk);
          const u64 r = fx::relax((unsigned)__double2hiint(ft[u].y), (unsigned)__double2loint(ft[u].y), wb, eb, m,
                                  (int)(ha >> 20) + ek, e);
          unsigned hi, lo;
          fx::to_words(r, (unsigned)e, hi, lo);
          double2 o = make_double2(fma(b, ft[u].x, aphi), __hiloint2double((int)hi, (int)lo));
          if (!fit || e < (int)fx::kExpMin || e > (int)fx::kExpMax) o.y = relax_slow(ft[u].y, aphi, b, kappa);
          p[u * rpw * nvx] = o;
        }
      }
    }
  }
}

// A4 of a warp's rows in FP64.
template <int W>
__device__ __noinline__ void relax_rows_f64(const Params& P, int wi, double2* __restrict__ fo,
                                            const double* __restrict__ px, const double* __restrict__ py, double b,
                                            double kappa) {
  const LaneMap<W> L(P, wi);
  for (int jx = L.l; jx < P.nvx; jx += L.width)
    for (int jy = L.row0; jy < P.nvy; jy += L.step) {
      double2* p = fo + jy * P.nvx + jx;
      const double2 ft = *p;
      const double aphi = px[jx] * py[jy];
      *p = make_double2(fma(b, ft.x, aphi), fma(b, ft.y, kappa * aphi));
    }
}

}  // namespace

// Resident CTAs per SM that the register budget is cut for (FP64 kernel).
__host__ __device__ constexpr int step_min_ctas(int G) { return G == 4 ? 8 : (G == 8 ? 4 : 1); }

template <int DIM, int G>
__global__ void __launch_bounds__(32 * G, step_min_ctas(G))
    step_f64_kernel(const double2* __restrict__ fin, double2* __restrict__ fout,
                    double4_32a* __restrict__ mom, double4_32a* __restrict__ par, const Params P,
                    const Tables T, int* __restrict__ err) {
  extern __shared__ double4_32a smem4[];
  double* phx = reinterpret_cast<double*>(smem4);
  double* phy = phx + G * P.nvx;
  __shared__ double s_sum[G][kSums];
  __shared__ int s_kind[G];
  __shared__ double s_b[G], s_k[G];
  __shared__ int s_ok[G];

  const int warp = threadIdx.x >> 5;
  const int cell = blockIdx.x * G + warp;
  const bool live = cell < P.nx * P.ny;
  // f~ of the warp's cell is parked in the cell's own output slots between
  // the passes (the values come back from L2): staging it in shared memory
  // (16 B per velocity) held an SM to 3 CTAs, measured 21 % (64^2 x 32^2) and
  // 40 % (256^2 x 48^2) slower
  double2* tile = fout + (size_t)cell * P.nv;

  if (live) stream_cell<DIM>(P, T, fin, cell, tile, s_sum[warp]);
  if ((threadIdx.x & 31) == 0) s_kind[warp] = SUMS_VELOCITY;
  __syncthreads();
  if constexpr (DIM == 2 && G >= 2) {
    __shared__ SolveXchg<G> s_x;
    if (warp < 2)
      maxwellian_cells_2w<G>(P, T, blockIdx.x * G, s_sum, s_kind, phx, phy, s_b, s_k, s_ok, mom, par, err, s_x);
  } else if (warp == 0) {
    maxwellian_cells<DIM, G>(P, T, blockIdx.x * G, s_sum, s_kind, phx, phy, s_b, s_k, s_ok, mom, par, err);
  }
  __syncthreads();
  // a failed cell keeps f^{n+1} = f~ (flagged)
  if (live && s_ok[warp])
    relax_cell<DIM>(P, T, tile, phx + warp * P.nvx, phy + warp * P.nvy, s_b[warp], s_k[warp]);
}

// The 2D step with the work split over the integer and the FP64 pipe: 8
// warps, G cells of W = 8 / G warps each.
template <int G>
__global__ void __launch_bounds__(256, 4)
    step_fixed_kernel(const double2* __restrict__ fin, double2* __restrict__ fout, double4_32a* __restrict__ mom,
                      double4_32a* __restrict__ par, const Params P, const Tables T, int* __restrict__ err) {
  constexpr int W = 8 / G;
  extern __shared__ double4_32a smem4[];
  double* phx = reinterpret_cast<double*>(smem4);
  double* phy = phx + G * P.nvx;
  __shared__ double s_sum[8][kSums];
  __shared__ int s_kind[8];
  __shared__ double s_b[G], s_k[G];
  __shared__ int s_ok[G];
  __shared__ CellSolve<G> s_x;

  const int warp = threadIdx.x >> 5, mine = warp / W, wi = warp % W;
  const int cell = blockIdx.x * G + mine;
  const bool live = cell < P.nx * P.ny;
  double2* tile = fout + (size_t)cell * P.nv;  // f~ is parked in the output slots
  int kind = SUMS_VELOCITY;
  if (live) kind = stream_rows<W>(P, T, fin, cell, wi, tile, s_sum[warp]);
  if ((threadIdx.x & 31) == 0) s_kind[warp] = kind;
  __syncthreads();
  const bool fixed =
      maxwellian_cells_fixed<G, W>(P, T, blockIdx.x * G, s_sum, s_kind, phx, phy, s_b, s_k, s_ok, mom, par, err, s_x);
  if (!live) return;
  const double *px = phx + mine * P.nvx, *py = phy + mine * P.nvy;
  if (!s_ok[mine]) return;  // a failed cell keeps f^{n+1} = f~ (flagged)
  if (kind == SUMS_INDEX && fixed) relax_rows_fixed<W>(P, wi, tile, px, py, s_b[mine], s_k[mine]);
  else relax_rows_f64<W>(P, wi, tile, px, py, s_b[mine], s_k[mine]);
}

namespace {

// ---- 1D, inflow ends, at most 160 velocities ----------------------------------
// One warp per cell and no barrier: f~ stays in registers (KV velocities per
// lane), the moment sums are integers in a unit 2^-72 of the cell's largest
// exponent, and the Gaussians and the relaxation weight come from the integer pipe, as
// in the 2D fixed-point kernels.  A cell's step is one chain of operations
// (12 800 points give an SM one or two warps), so what counts is their number:
// about 90 FP64 operations of 64 cycles where the FP64 form has 340.  Mach 2
// shock, 200 cells x 64 velocities, 200 steps with state in and moments out:
// 2396 -> 1445 us.

// Sum over the warp of four 96-bit values per lane: lane L ends with value
// (L >> 3) & 3 (recursive halving, as warp_reduce4).
__device__ __forceinline__ fx::i96 warp_reduce4_96(fx::i96 v0, fx::i96 v1, fx::i96 v2, fx::i96 v3) {
  const int lane = threadIdx.x & 31;
  const bool b4 = lane & 16, b3 = lane & 8;
  const fx::i96 a = xor_add96(pick(b4, v2, v0), pick(b4, v0, v2), 16);
  const fx::i96 b = xor_add96(pick(b4, v3, v1), pick(b4, v1, v3), 16);
  fx::i96 x = xor_add96(pick(b3, b, a), pick(b3, a, b), 8);
  x = xor_add96(x, x, 4);
  x = xor_add96(x, x, 2);
  return xor_add96(x, x, 1);
}

// The cell's step in FP64, for any values (one warp; sm: nvx + 1 doubles).
__device__ __noinline__ void cell1d_f64(const Params& P, const Tables& T, const double2* __restrict__ fin,
                                        double2* __restrict__ fo, double4_32a* __restrict__ mom,
                                        double4_32a* __restrict__ par, int* __restrict__ err, int cell, double* sm,
                                        double (*sums)[kSums], double* sbk, int* sok) {
  const int kind = SUMS_VELOCITY;
  stream_cell<1>(P, T, fin, cell, fo, sums[0]);
  __syncwarp();
  maxwellian_cells<1, 1>(P, T, cell, sums, &kind, sm, sm + P.nvx, sbk, sbk + 1, sok, mom, par, err);
  __syncwarp();
  if (*sok) relax_cell<1>(P, T, fo, sm, sm + P.nvx, sbk[0], sbk[1]);
}

template <int KV>
__global__ void __launch_bounds__(256) step1d_kernel(const double2* __restrict__ fin, double2* __restrict__ fout,
                                                     double4_32a* __restrict__ mom, double4_32a* __restrict__ par,
                                                     const Params P, const Tables T, int* __restrict__ err) {
  extern __shared__ double4_32a smem4[];
  __shared__ double s_sum[8][1][kSums], s_bk[8][2];
  __shared__ int s_ok[8];
  constexpr unsigned kAll = 0xffffffffu;
  const VelocityGrid& V = T.grid;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nv = P.nvx;
  const int cell = blockIdx.x * (blockDim.x >> 5) + warp;
  if (cell >= P.nx) return;
  double2* fo = fout + (size_t)cell * nv;
  // A1
  double2 ft[KV];
  unsigned tg = 0, th = 0;
#pragma unroll
  for (int k = 0; k < KV; ++k) {
    const int j = min(lane + 32 * k, nv - 1);  // a velocity past the last repeats it and is not counted
    const int i1 = cell - T.shift[j], i2 = i1 - vi_sx(T.vinfo[j]);
    const double2 f1 = *(i1 < 0 ? T.ghost + j : i1 >= P.nx ? T.ghost + nv + j : fin + (size_t)i1 * nv + j);
    const double2 f2 = *(i2 < 0 ? T.ghost + j : i2 >= P.nx ? T.ghost + nv + j : fin + (size_t)i2 * nv + j);
    const double4_32a co = T.coef[j];
    ft[k].x = fma(co.y, f2.x, co.x * f1.x);
    ft[k].y = fma(co.y, f2.y, co.x * f1.y);
    tg = max(tg, (unsigned)__double2hiint(ft[k].x));
    th = max(th, (unsigned)__double2hiint(ft[k].y));
  }
  const unsigned eg = __reduce_max_sync(kAll, tg) >> 20, eh = __reduce_max_sync(kAll, th) >> 20;
  bool fit = min(eg, eh) >= fx::kExpMin && max(eg, eh) <= fx::kExpMax;
  // A2: sums over (1, k, k^2, h), k = 2 j + 1 - nv: 160 values of 72 bits times
  // 159^2 stay within 95 (59 bits left 9e-16 of theta on +-20 thermal speeds
  // with a tail of 1e-9)
  constexpr int kRoom = 3;
  const fx::i96 zero = {0u, 0u, 0u};
  fx::i96 v0 = zero, v1 = zero, v2 = zero, v3 = zero;
#pragma unroll
  for (int k = 0; k < KV; ++k) {
    const int j = lane + 32 * k, kk = 2 * j + 1 - nv;
    if (j < nv) {
      const fx::i96 g = fx::double_to_units96((unsigned)__double2hiint(ft[k].x), (unsigned)__double2loint(ft[k].x),
                                              eg + kRoom);
      v0 = fx::add(v0, g);
      v1 = fx::add(v1, fx::muls(g, kk));
      v2 = fx::add(v2, fx::mul(g, (unsigned)(kk * kk)));
      v3 = fx::add(v3, fx::double_to_units96((unsigned)__double2hiint(ft[k].y), (unsigned)__double2loint(ft[k].y),
                                             eh + kRoom));
    }
  }
  const double t = unit_value(warp_reduce4_96(v0, v1, v2, v3), (int)(lane < 24 ? eg : eh) + kRoom - 16);
  const double s0 = __shfl_sync(kAll, t, 0), s1 = __shfl_sync(kAll, t, 8), s2 = __shfl_sync(kAll, t, 16),
               sh = __shfl_sync(kAll, t, 24);
  // A3, every lane alike: moments about the box centre
  fit = fit && in_range(s0);
  const double in = rcp3(fit ? s0 : 1.0), m1 = V.half_x * s1 * in;
  double q[3], p[3];  // n, u, theta
  q[0] = s0 * P.dv;
  q[1] = V.mid_x + m1;
  q[2] = (2.0 / 3.0) * (fma(V.half_x * V.half_x, s2 * in, -m1 * m1) + sh * in);
  fit = fit && in_range(q[0]) && in_range(q[2]);
  AxisBase B;
  double isq = 1.0;
  if (fit) {
    isq = rsqrt3(q[2]);
    fit = axis_base(nv, V.half_x, V.inv_half_x, V.mid_x, q[1], isq, B);
  }
  double a = 0.0, b = 0.0;
  if (fit) {
#pragma unroll
    for (int k = 0; k < 3; ++k) p[k] = q[k];
    const double x = q[0] * (P.omega == 0.5 ? q[2] * isq : pow_fixed(q[2], 1.0 - P.omega)) * P.dt;  // nu dt
    b = P.relax_exact ? exp_neg_fixed(x) : 1.0 - x;
    a = P.relax_exact ? 1.0 - b : x;
    if (P.conservative) {
      const double ivs = isq, iq2 = isq * isq, iq0 = in * (1.0 / P.dv);
      for (int it = 1;; ++it) {
        v0 = v1 = v2 = zero;
#pragma unroll
        for (int k = 0; k < KV; ++k) {
          const int j = lane + 32 * k, kk = 2 * j + 1 - nv - B.k0;
          if (j < nv) {
            unsigned n2;
            const unsigned long long g = fx::gauss(B.a * (2 * j + 1 - nv) - B.c, (const fx::u64*)kExp2, n2);
            const fx::i96 e = fx::wide(n2 < 62u ? g >> (n2 + 1u) : 0);  // units of 2^-62
            v0 = fx::add(v0, e);
            v1 = fx::add(v1, fx::muls(e, kk));
            v2 = fx::add(v2, fx::mul(e, (unsigned)(kk * kk)));
          }
        }
        const double u = unit_value(warp_reduce4_96(v0, v1, v2, zero), 1081 - 62);
        const double ks[3] = {__shfl_sync(kAll, u, 0), __shfl_sync(kAll, u, 8), __shfl_sync(kAll, u, 16)};
        double M[3];
        central_sums(ks, B.k0, V.half_x, V.mid_x, p[1], M);
        const double r0 = rcp3(M[0]), mu = M[1] * r0;
        const double d0 = p[0] * isq * 0.5641895835477563 * P.dv * M[0];  // 1 / sqrt(pi); prefactor as in A4
        const double d2 = (2.0 / 3.0) * (fma(M[2], r0, -mu * mu) + p[2]);
        const double e0 = q[0] - d0, e1 = q[1] - (p[1] + mu), e2 = q[2] - d2;
        p[0] += e0;
        p[1] += e1;
        p[2] += e2;
        const unsigned r = max(max(abs_hi(e0 * iq0), abs_hi(e1 * ivs)), abs_hi(e2 * iq2));
        // the high words of kEffTol = 1e-13, sqrt(kEffTol / 100) = 3.16e-8 and kEffFail = 1e-9
        const bool conv = r < 0x3d3c25c2u || (it == 1 && r < 0x3e60fa33u) || (it >= kEffMaxIt && r < 0x3e112e0bu);
        // beyond the range of the FP32 starts, or no convergence: the FP64 path decides
        fit = in_range(p[0]) && in_range(p[2]) && r < 0x7ff00000u && (conv || it < kEffMaxIt);
        if (!fit) break;
        isq = rsqrt3(p[2]);
        fit = axis_base(nv, V.half_x, V.inv_half_x, V.mid_x, p[1], isq, B);
        if (conv || !fit) break;
      }
    }
  }
  if (!fit) {  // uniform over the warp
    double* sm = reinterpret_cast<double*>(smem4) + warp * (nv + 1);
    cell1d_f64(P, T, fin, fo, mom, par, err, cell, sm, s_sum[warp], s_bk[warp], &s_ok[warp]);
    return;
  }
  if (lane == 0) {
    store4(mom + cell, q[0], q[1], 0.0, q[2]);
    if (par) store4(par + cell, p[0], p[1], 0.0, p[2]);
  }
  // A4
  const double ap = a * (p[0] * isq * 0.5641895835477563);
#pragma unroll
  for (int k = 0; k < KV; ++k) {
    const int j = lane + 32 * k;
    if (j < nv) {
      unsigned n2, hi, lo;
      const unsigned long long g = fx::gauss(B.a * (2 * j + 1 - nv) - B.c, (const fx::u64*)kExp2, n2);
      fx::gauss_words(g, n2, hi, lo);
      const double aphi = ap * __hiloint2double((int)hi, (int)lo);
      fo[j] = make_double2(fma(b, ft[k].x, aphi), fma(b, ft[k].y, p[2] * aphi));
    }
  }
}

size_t step_smem(const Params& P, int G) {
  return sizeof(double) * (size_t)G * (P.nvx + P.nvy);
}

typedef void (*StepKernel)(const double2*, double2*, double4_32a*, double4_32a*, const Params, const Tables, int*);

// The problem's kernel and its threads per CTA; null for an unknown tile.
StepKernel step_kernel(const Params& P, unsigned* threads) {
  *threads = 32u * (unsigned)P.tile;
  if (P.dim == 1 && P.lane_bits && P.tile <= 8) switch ((P.nvx + 31) / 32) {
      case 1: return step1d_kernel<1>;
      case 2: return step1d_kernel<2>;
      case 3: return step1d_kernel<3>;
      case 4: return step1d_kernel<4>;
      default: return step1d_kernel<5>;
    }
  if (P.dim == 1) switch (P.tile) {
      case 1: return step_f64_kernel<1, 1>;
      case 2: return step_f64_kernel<1, 2>;
      case 4: return step_f64_kernel<1, 4>;
      case 8: return step_f64_kernel<1, 8>;
      default: return nullptr;
    }
  if (P.lane_bits == 0) switch (P.tile) {
      case 1: return step_f64_kernel<2, 1>;
      case 2: return step_f64_kernel<2, 2>;
      case 4: return step_f64_kernel<2, 4>;
      case 8: return step_f64_kernel<2, 8>;
      default: return nullptr;
    }
  *threads = 256u;
  switch (P.tile) {
    case 1: return step_fixed_kernel<1>;
    case 2: return step_fixed_kernel<2>;
    case 4: return step_fixed_kernel<4>;
    case 8: return step_fixed_kernel<8>;
    default: return nullptr;
  }
}

}  // namespace

size_t step_f64_smem_bytes(const Params& P, int tile) { return step_smem(P, tile); }

// Lanes per velocity row of the fixed-point kernels: the 4, 8, 16 or 32 that
// leave the fewest lanes idle (more lanes on a tie, for wider accesses).  They
// need weights that sum to one (Courant number at most 1), y weights below one
// (their top bit is the sign of c_y; the margin covers host and device
// rounding: with it the x part is at most 2^-40 of one), 128 velocities to
// sample, and sums fine enough (at most 512 velocities per axis): the sum of
// squared indices times nv values of 75 - sum_room bits stays within 95 bits
// (32^2: 75 bits a value, 48^2 and 64^2: 71, 8 x 512: 65).  In 1D any non-zero
// value selects step1d_kernel.
void step_f64_plan(Params& P, double max_courant, double max_courant_y) {
  P.lane_bits = P.sum_room = 0;
  if (P.dim == 1 && P.nvx >= 8 && P.nvx <= 160 && P.bc_kind[XLO] == BC_INFLOW && P.bc_kind[XHI] == BC_INFLOW)
    P.lane_bits = 5;
  if (P.dim != 2 || P.nv < 128 || P.nvx > 512 || P.nvy > 512 || max_courant > 1.0 + 4e-15 ||
      max_courant_y > 1.0 - 0x1p-40)
    return;
  const auto bits = [](int n) {
    int b = 0;
    while (1 << b < n) ++b;
    return b;
  };
  P.sum_room = std::max(0, bits(P.nv) + 2 * bits(std::max(P.nvx, P.nvy)) - 20);
  double best = 0.0;
  for (int lb = 5; lb >= 2; --lb) {
    const int lw = 1 << lb, rpw = 32 >> lb;
    const int width = (P.nvx + lw - 1) / lw * lw, rows = (P.nvy + rpw - 1) / rpw * rpw;
    const double use = (double)P.nv / ((double)width * rows);
    if (use > best + 1e-9) {
      best = use;
      P.lane_bits = lb;
    }
  }
}

// The attribute belongs to the kernel, not to a solver: set it to the
// largest dynamic shared memory any solver may request (what the device
// allows a CTA beside the kernel's static shared memory) so that solvers
// with different grids sharing an instantiation never shrink it.
cudaError_t prepare_step_f64(const Params& P) {
  unsigned threads = 0;
  const StepKernel k = step_kernel(P, &threads);
  if (!k) return cudaErrorInvalidValue;
  int dev = 0, optin = 0;
  cudaFuncAttributes fa;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e == cudaSuccess) e = cudaFuncGetAttributes(&fa, k);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, optin - (int)fa.sharedSizeBytes);
}

cudaError_t launch_step_f64(const Params& P, const Tables& T, const double2* fin, double2* fout,
                            double4_32a* mom, int* err, cudaStream_t stream, double4_32a* par) {
  unsigned threads = 0;
  const StepKernel k = step_kernel(P, &threads);
  if (!k) return cudaErrorInvalidValue;
  const unsigned grid = (unsigned)((P.nx * P.ny + P.tile - 1) / P.tile);
  k<<<grid, threads, step_smem(P, P.tile), stream>>>(fin, fout, mom, par, P, T, err);
  return cudaGetLastError();
}

}  // namespace bgk
