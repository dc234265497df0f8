// bgk_step3v.cu - the FP64 BGK step on a full three-dimensional velocity
// grid with one spatial dimension: the normal shock of Sec. 4.1 as the paper
// computed it (the Chu reduction is not made; f lives on N_vx x N_vy x N_vz
// velocity cells per spatial cell; Delta t = 0.05 puts the fast velocities
// several cells per step, so streaming is the integer shift of Eq. (exact)
// followed by the upwind remainder of Eq. (upwind)).
//
// One CTA of 256 threads per spatial cell (4 096 to 27 000 velocities):
//   pass 1  f~ = (1 - r) f_{i-[C]} + r f_{i-[C]-sgn C} per velocity (inflow
//           Maxwellians beyond the ends) and the five sums of Eq.
//           (macroscopic) (n, n U, E), reduced over the CTA;
//   cell    nu = n theta^(1-omega), the relaxation weights, and the
//           effective parameters p (Sec. 2.1 remark) by p <- p + (q - D(p))
//           with the Gaussian factored per axis: warp a of the first three
//           evaluates axis a's 1D factor and its sums, the three warps
//           synchronise on a named barrier;
//   pass 2  f^{n+1} = b f~ + a Phi, Phi = px[jx] py[jy] pz[jz], on the f~
//           values pass 1 parked in the cell's output slots (each thread
//           rereads its own writes, from L2).
#include "bgk_solve.cuh"

namespace bgk {

namespace {

constexpr int kT = 256;  // threads per CTA
constexpr int kW = kT / 32;

struct Idx3 {
  int jx, jy, jz;
};
__device__ __forceinline__ Idx3 split3(const Params3v& P, int j) {
  const int jyz = j / P.nvx;
  const int jz = jyz / P.nvy;
  return {j - jyz * P.nvx, jyz - jz * P.nvy, jz};
}

// f~ at velocity j of cell i: Eq. (exact) shift by [C], Eq. (upwind) with
// the remainder |C - [C]| toward the upwind side.
__device__ __forceinline__ double stream3(const Params3v& P, const Tables3v& T, const double* __restrict__ fin,
                                          int i, int j, int jx) {
  const int i1 = i - T.shift[jx];
  const int i2 = i1 - T.upwind[jx];
  const double f1 = i1 < 0 ? T.ghost[j] : i1 >= P.nx ? T.ghost[P.nv + j] : fin[(size_t)i1 * P.nv + j];
  const double f2 = i2 < 0 ? T.ghost[j] : i2 >= P.nx ? T.ghost[P.nv + j] : fin[(size_t)i2 * P.nv + j];
  return fma(T.rem[jx], f2 - f1, f1);
}

// Sums of N values over the CTA in a fixed order, totals in out (all threads).
__device__ __forceinline__ void cta_sum8(const double (&v)[8], double* red, double* out) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const double x = warp_reduce8(v);  // lane 4k + r holds total k
  if ((lane & 3) == 0) red[warp * 8 + (lane >> 2)] = x;
  __syncthreads();
  if (threadIdx.x < 8) {
    double t = 0.0;
    for (int w = 0; w < kW; ++w) t += red[w * 8 + threadIdx.x];
    out[threadIdx.x] = t;
  }
  __syncthreads();
}

__device__ __forceinline__ int axis_n(const Params3v& P, int a) { return a == 0 ? P.nvx : a == 1 ? P.nvy : P.nvz; }

// The three warps' barrier (warps 0..2, 96 threads).
__device__ __forceinline__ void bar_axes() { asm volatile("bar.sync 1, 96;" ::: "memory"); }

// Warp `a` (0..2): 1D Gaussian e_j = exp(-(c_j - u)^2 / theta) of its axis
// at p; returns the warp totals (sum e, sum d e, sum d^2 e) in every lane and
// leaves e_j in fac (when not null).
__device__ __forceinline__ void axis_sums3v(const Params3v& P, const Tables3v& T, int a, double u, double inv_th,
                                          double* fac, double (&s)[3]) {
  const int lane = threadIdx.x & 31;
  s[0] = s[1] = s[2] = 0.0;
  for (int j = lane; j < axis_n(P, a); j += 32) {
    const double d = T.c[a][j] - u;
    const double e = exp(-(d * d) * inv_th);
    if (fac) fac[j] = e;
    s[0] += e;
    s[1] = fma(d, e, s[1]);
    s[2] = fma(d * d, e, s[2]);
  }
  for (int k = 0; k < 3; ++k)
    for (int m = 16; m > 0; m >>= 1) s[k] += __shfl_xor_sync(0xffffffffu, s[k], m);
}

// Scratch of a CTA.
struct Shared3v {
  double red[kW * 8], tot[8];
  double ax[3][3];  // per axis: sum e, sum d e, sum d^2 e (fixed point: index sums)
  double ab[2];     // relaxation weights a (on Phi; fixed point: its factor), b (on f~)
  AxisBase base[3];
  int ok, go, valid[kW];
};

// The step of cell i in FP64, for any grid and any values (all threads).
__device__ __noinline__ void cell3v_f64(const Params3v& P, const Tables3v& T, const double* __restrict__ fin,
                                        double* __restrict__ fout, double* __restrict__ mom, int* __restrict__ err,
                                        int i, double* fac, Shared3v& S) {
  double *red = S.red, *tot = S.tot, (*s_ax)[3] = S.ax, *s_ab = S.ab;
  int& s_ok = S.ok;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // pass 1: stream (f~ parked in the cell's output slots) and the five sums
  // of Eq. (macroscopic)
  double* fo = fout + (size_t)i * P.nv;
  double acc[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int j = threadIdx.x; j < P.nv; j += kT) {
    const Idx3 k = split3(P, j);
    const double ft = stream3(P, T, fin, i, j, k.jx);
    fo[j] = ft;
    acc[0] += ft;
    acc[1] = fma(T.c[0][k.jx], ft, acc[1]);
    acc[2] = fma(T.c[1][k.jy], ft, acc[2]);
    acc[3] = fma(T.c[2][k.jz], ft, acc[3]);
    acc[4] = fma(T.c2[j], ft, acc[4]);
  }
  cta_sum8(acc, red, tot);

  // per-cell parameters, warps 0..2 (warp a works on axis a)
  if (warp < 3) {
    const double n = tot[0] * P.dv;
    const double q[5] = {n, tot[1] / tot[0], tot[2] / tot[0], tot[3] / tot[0],
                         (2.0 / 3.0) * (tot[4] / tot[0] -
                                        ((tot[1] / tot[0]) * (tot[1] / tot[0]) + (tot[2] / tot[0]) * (tot[2] / tot[0]) +
                                         (tot[3] / tot[0]) * (tot[3] / tot[0])))};
    bool ok = q[0] > 0.0 && q[4] > 0.0 && isfinite(q[0]) && isfinite(q[1]) && isfinite(q[2]) && isfinite(q[3]) &&
              isfinite(q[4]);
    double p[5] = {q[0], q[1], q[2], q[3], q[4]};
    if (!ok) {
      p[0] = 1.0;
      p[1] = p[2] = p[3] = 0.0;
      p[4] = 1.0;
    }
    bool fail_eff = false;
    if (ok && P.conservative) {
      const double vs = sqrt(q[4]);
      for (int it = 1; it <= kEffMaxIt; ++it) {
        double s[3];
        axis_sums3v(P, T, warp, p[1 + warp], 1.0 / p[4], nullptr, s);
        if (lane == 0)
          for (int m = 0; m < 3; ++m) s_ax[warp][m] = s[m];
        bar_axes();
        double d[5];
        const double S0 = s_ax[0][0] * s_ax[1][0] * s_ax[2][0];
        d[0] = p[0] / (kPi() * p[4] * sqrt(kPi() * p[4])) * P.dv * S0;
        double th = 0.0;
        for (int a = 0; a < 3; ++a) {
          const double mu = s_ax[a][1] / s_ax[a][0];
          d[1 + a] = p[1 + a] + mu;
          th += s_ax[a][2] / s_ax[a][0] - mu * mu;
        }
        d[4] = (2.0 / 3.0) * th;
        bar_axes();  // s_ax is rewritten by the next iteration
        double r = 0.0;
        for (int m = 0; m < 5; ++m) {
          const double delta = q[m] - d[m];
          p[m] += delta;
          r = fmax(r, fabs(delta) / (m == 0 ? q[0] : m == 4 ? q[4] : vs));
        }
        if (!(p[0] > 0.0) || !(p[4] > 0.0) || !isfinite(r)) {
          fail_eff = true;
          break;
        }
        if (r < kEffTol) break;
        if (it == kEffMaxIt && r >= kEffFail) fail_eff = true;
      }
    }
    if (fail_eff) ok = false;
    // factors at the final p: px carries a n (pi theta)^(-3/2)
    const double nu = q[0] * pow(q[4], 1.0 - P.omega);
    const double a = !ok ? 0.0 : P.relax_exact ? 1.0 - exp(-nu * P.dt) : nu * P.dt;
    const double b = !ok ? 1.0 : P.relax_exact ? exp(-nu * P.dt) : 1.0 - a;
    double* fw = fac + (warp == 0 ? 0 : warp == 1 ? P.nvx : P.nvx + P.nvy);
    double s[3];
    axis_sums3v(P, T, warp, p[1 + warp], 1.0 / p[4], fw, s);
    if (warp == 0) {
      __syncwarp();
      const double scale = a * p[0] / (kPi() * p[4] * sqrt(kPi() * p[4]));
      for (int j = lane; j < P.nvx; j += 32) fw[j] *= scale;
      if (lane == 0) {
        s_ab[0] = a;
        s_ab[1] = b;
        s_ok = ok ? 1 : 0;
        mom[(size_t)i * 5 + 0] = q[0];
        mom[(size_t)i * 5 + 1] = q[1];
        mom[(size_t)i * 5 + 2] = q[2];
        mom[(size_t)i * 5 + 3] = q[3];
        mom[(size_t)i * 5 + 4] = q[4];
        if (!ok) atomicOr(err, fail_eff ? ERR_EFFECTIVE : ERR_MOMENT);
      }
    }
  }
  __syncthreads();

  // pass 2: f^{n+1} = b f~ + a Phi, each thread on the f~ values it parked
  const double b = s_ab[1];
  const double* px = fac;
  const double* py = fac + P.nvx;
  const double* pz = py + P.nvy;
  if (s_ok == 0) return;  // f^{n+1} = f~ (flagged)
  for (int j = threadIdx.x; j < P.nv; j += kT) {
    const Idx3 k = split3(P, j);
    fo[j] = fma(b, fo[j], px[k.jx] * py[k.jy] * pz[k.jz]);
  }
}

}  // namespace

__global__ void __launch_bounds__(kT) step3v_kernel(const Params3v P, const Tables3v T,
                                                    const double* __restrict__ fin, double* __restrict__ fout,
                                                    double* __restrict__ mom, int* __restrict__ err) {
  extern __shared__ double fac[];  // px[nvx], py[nvy], pz[nvz]
  __shared__ Shared3v S;
  cell3v_f64(P, T, fin, fout, mom, err, blockIdx.x, fac, S);
}

namespace {

// ---- fixed-point kernel -------------------------------------------------------
// The FP64 pipe takes 64 to 76 cycles per warp instruction and bounded the
// step (12.1 operations per velocity).  Here four remain, two to stream and
// two to relax; the moment sums are integers of 75 bits a value, the Gaussians
// and the relaxation weight come from the integer pipe.  With state in and
// moments out: 10 steps of 2048 x 30^3 13.2 -> 7.3 ms, 20 of 512 x 16^3 2.61 ->
// 1.06 ms.  What bounds it now: the FP64 pipe at 97 % of its measured rate on
// 608 x 30^3 (5.0 operations issued per velocity, idle lanes and solve
// included); in pass 1 each lane's column comes from another cell (8 of each 32
// bytes are used); the solve of a 16^3 cell takes as long as its passes.
//
// 2^lane_bits lanes share a velocity row (fixed jy, jz); the 8 warps split z
// 2^zw_bits ways and y the rest.  A lane takes its columns jx one after the
// other over its rows, y inside z.
struct Map3v {
  int l, width, y0, ystep, yrows, z0, zstep, zrows;
  __device__ __forceinline__ explicit Map3v(const Params3v& P) {
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, lb = P.lane_bits, zb = P.zw_bits;
    width = 1 << lb;
    l = lane & (width - 1);
    z0 = warp & ((1 << zb) - 1);
    zstep = 1 << zb;
    ystep = (kW >> zb) * (32 >> lb);
    y0 = (warp >> zb) * (32 >> lb) + (lane >> lb);
    yrows = (P.nvy + ystep - 1) / ystep;
    zrows = (P.nvz + zstep - 1) / zstep;
  }
};

// Sources of a column of cell i: the shifted cell and its upwind neighbour,
// or the inflow Maxwellian beyond an end.
__device__ __forceinline__ const double* column_source(const Params3v& P, const Tables3v& T,
                                                       const double* __restrict__ fin, int i) {
  return i < 0 ? T.ghost : i >= P.nx ? T.ghost + P.nv : fin + (size_t)i * P.nv;
}

// Integer sums of weight (first + step k) along an axis of `rows` rows from
// the running sums r0 = sum g, r1 = sum (rows - k) g, r2 = sum (rows - k)
// (rows - k + 1) / 2 g: sum w g and sum w^2 g with w = 2 j + 1 - n.
__device__ __forceinline__ void axis_weights(fx::i96 r0, fx::i96 r1, fx::i96 r2, int first, int step, int rows, int n,
                                             fx::i96& w1, fx::i96& w2) {
  const int A = 2 * (first + step * rows) + 1 - n, B = 2 * step;
  const fx::i96 b1 = fx::mul(r1, (unsigned)B);
  w1 = fx::add(fx::muls(r0, A), fx::neg(b1));
  w2 = fx::add(fx::add(fx::mul(r0, (unsigned)(A * A)), fx::neg(fx::muls(b1, 2 * A + B))),
               fx::mul(r2, (unsigned)(2 * B * B)));
}

// Rows whose values are loaded together (2048 x 30^3, a step, at the time the
// line was drawn: 0.77 ms with 4, 0.71 with 8; 0.65 since).
constexpr int kAhead3 = 8;

// Pass 1 of the warp's rows: f~ into fo, the sums of (1, k_x, k_x^2,
// k_y, k_y^2, k_z, k_z^2) f~ into sums.  eg: largest exponent the units are
// cut for; on return the largest seen.  False when the sums are not valid.
__device__ __forceinline__ bool stream3v_fixed(const Params3v& P, const Tables3v& T, const double* __restrict__ fin,
                                               double* __restrict__ fo, int i, int& eg, double* sums) {
  const Map3v L(P);
  const int nvx = P.nvx, nvy = P.nvy, nvz = P.nvz;
  const fx::i96 zero = {0u, 0u, 0u};
  double v[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  int top = 0;
  unsigned over = 0;
#pragma unroll 1
  for (int jl = L.l; jl - L.l < nvx; jl += L.width) {
    const bool in = jl < nvx;
    const int jx = in ? jl : nvx - 1;  // a column past the row repeats its last one and is not counted
    const int i1 = i - T.shift[jx];
    const double* p1 = column_source(P, T, fin, i1);
    const double* p2 = column_source(P, T, fin, i1 - T.upwind[jx]);
    const double rem = T.rem[jx];
    fx::i96 n0 = zero, y1 = zero, y2 = zero, z1 = zero, z2 = zero;
#pragma unroll 1
    for (int kz = 0; kz < L.zrows; ++kz) {
      const int jz = L.z0 + kz * L.zstep;
      const bool zin = in && jz < nvz;
      const int jb = min(jz, nvz - 1) * nvy * nvx + jx;
      fx::i96 t1 = zero, t2 = zero, t3 = zero;
#pragma unroll 1
      for (int k0 = 0; k0 < L.yrows; k0 += kAhead3) {
        double f1[kAhead3], f2[kAhead3];
#pragma unroll
        for (int u = 0; u < kAhead3; ++u) {
          if (k0 + u >= L.yrows) break;  // the same for every lane
          const int j = jb + min(L.y0 + (k0 + u) * L.ystep, nvy - 1) * nvx;
          f1[u] = p1[j];
          f2[u] = p2[j];
        }
#pragma unroll
        for (int u = 0; u < kAhead3; ++u) {
          if (k0 + u >= L.yrows) break;
          const int jy = L.y0 + (k0 + u) * L.ystep;
          const double ft = fma(rem, f2[u] - f1[u], f1[u]);
          if (zin && jy < nvy) {
            const unsigned hi = (unsigned)__double2hiint(ft);
            fo[jb + jy * nvx] = ft;
            top = max(top, (int)(hi >> 20));
            t1 = fx::add(t1, fx::double_to_units96(hi, (unsigned)__double2loint(ft), (unsigned)eg));
          }
          t2 = fx::add(t2, t1);
          t3 = fx::add(t3, t2);
        }
      }
      n0 = fx::add(n0, t1);
      y1 = fx::add(y1, t2);
      y2 = fx::add(y2, t3);
      z1 = fx::add(z1, n0);
      z2 = fx::add(z2, z1);
    }
    over |= n0.a2 >> 16;  // 2^12 rows of 2^75 do not wrap; below 2^80 the squared indices fit too
    fx::i96 a1, a2, b1, b2;
    axis_weights(n0, y1, y2, L.y0, L.ystep, L.yrows, nvy, a1, a2);
    axis_weights(n0, z1, z2, L.z0, L.zstep, L.zrows, nvz, b1, b2);
    const double sn = unit_value(n0, eg - 16), kx = (double)(2 * jx + 1 - nvx), kn = kx * sn;
    v[0] += sn;
    v[1] += kn;
    v[2] = fma(kx, kn, v[2]);
    v[3] += unit_value(a1, eg - 16);
    v[4] += unit_value(a2, eg - 16);
    v[5] += unit_value(b1, eg - 16);
    v[6] += unit_value(b2, eg - 16);
  }
  top = __reduce_max_sync(0xffffffffu, top);
  const bool valid = top <= eg && !__any_sync(0xffffffffu, over != 0);
  const int lane = threadIdx.x & 31;
  const double t = warp_reduce8(v);  // lane 4 k + r holds total k
  if ((lane & 3) == 0) sums[lane >> 2] = t;
  eg = top;
  return valid;
}

// Largest exponent of the cell's own state along the x lines through the
// middle of the (y, z) box, plus the headroom: the peak of a flow along x
// with little transverse motion lies there.
__device__ __forceinline__ int sample3v(const Params3v& P, const double* __restrict__ f) {
  const int lane = threadIdx.x & 31;
  unsigned m = 0;
  for (int jx = lane; jx < P.nvx; jx += 32) {
    const int j = ((P.nvz >> 1) * P.nvy + (P.nvy >> 1)) * P.nvx + jx;
    const int k = ((max(P.nvz - 1, 0) >> 1) * P.nvy + (max(P.nvy - 1, 0) >> 1)) * P.nvx + jx;
    m = max(m, max((unsigned)__double2hiint(f[j]), (unsigned)__double2hiint(f[k])));
  }
  return (int)((__reduce_max_sync(0xffffffffu, m) >> 20) + fx::kHeadroom);
}

constexpr double kPi15 = 0.17958712212516656;  // pi^(-3/2); the prefactor is the same in D(p) and in Phi

// Warps 0 to 2 (an axis each) and 3 (the relaxation weight).
__device__ __forceinline__ void bar_solve() { asm volatile("bar.sync 2, 128;" ::: "memory"); }

// The cell's parameters on warps 0 to 3, from the totals in S.tot.  Leaves
// S.go = 0, S.ab and the factors in fac, or S.go = -1 when the cell needs FP64.
__device__ __forceinline__ void solve3v_fixed(const Params3v& P, int i, Shared3v& S, double* fac,
                                              double* __restrict__ mom, int* __restrict__ err) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int n3[3] = {P.nvx, P.nvy, P.nvz};
  double half[3], mid[3];
#pragma unroll
  for (int a = 0; a < 3; ++a) {
    half[a] = P.half[a];
    mid[a] = P.mid[a];
  }
  double q[5], p[5], ith = 1.0, isq = 1.0, iq0 = 1.0, iq4 = 1.0, ivs = 1.0;
  bool conv = true;
  if (warp == 0) {  // all lanes alike
    const double* t = S.tot;
    bool fit = in_range(t[0]);
    const double in = rcp3(fit ? t[0] : 1.0);
    q[0] = t[0] * P.dv;
    double e = 0.0, uu = 0.0;
#pragma unroll
    for (int a = 0; a < 3; ++a) {
      const double m1 = half[a] * t[1 + 2 * a] * in;  // mean of c - mid
      const double u = mid[a] + m1;
      q[1 + a] = u;
      // mean of c^2 less u^2, both about mid
      e += fma(half[a] * half[a], t[2 + 2 * a] * in, -m1 * m1);
      uu += u;
    }
    q[4] = (2.0 / 3.0) * e;
    const bool ok = q[0] > 0.0 && q[4] > 0.0 && isfinite(q[0]) && isfinite(q[4]) && isfinite(uu);
    fit = fit && ok && in_range(q[0]) && in_range(q[4]);
    if (fit) {
      ivs = isq = rsqrt3(q[4]);
      iq4 = ith = rcp3(q[4]);
      iq0 = rcp3(q[0]);
    }
#pragma unroll
    for (int k = 0; k < 5; ++k) p[k] = fit ? q[k] : (k == 0 || k == 4) ? 1.0 : 0.0;
    if (fit) {
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        AxisBase B;
        fit = axis_base(n3[a], half[a], P.inv_half[a], mid[a], p[1 + a], isq, B) && fit;
        if (lane == 0) S.base[a] = B;
      }
    }
    conv = P.conservative == 0;
    if (lane == 0) {
      S.go = !fit ? -1 : conv ? 0 : 1;
      S.tot[7] = q[4];
    }
  }
  bar_solve();
  if (S.go < 0) return;
  if (warp == 3) {  // nu = n theta^(1 - omega), the weights
    const double x = S.tot[0] * P.dv * pow_fixed(S.tot[7], 1.0 - P.omega) * P.dt;  // nu dt
    const double b = P.relax_exact ? exp_neg_fixed(x) : 1.0 - x;
    if (lane == 0) {
      S.ab[0] = P.relax_exact ? 1.0 - b : x;
      S.ab[1] = b;
    }
  }
  int it = 0;
  while (S.go > 0) {
    if (warp < 3) {
      const double t = axis_index_sums<32>(n3[warp], S.base[warp], lane);
      if (lane < 3) S.ax[warp][lane] = t;
    }
    bar_solve();
    if (warp == 0) {
      ++it;
      double M[3][3], d[5];
#pragma unroll
      for (int a = 0; a < 3; ++a) central_sums(S.ax[a], S.base[a].k0, half[a], mid[a], p[1 + a], M[a]);
      d[0] = p[0] * (ith * isq) * kPi15 * P.dv * (M[0][0] * M[1][0] * M[2][0]);
      double var = 0.0;
#pragma unroll
      for (int a = 0; a < 3; ++a) {
        const double r = rcp3(M[a][0]), mu = M[a][1] * r;
        d[1 + a] = p[1 + a] + mu;
        var += fma(M[a][2], r, -mu * mu);
      }
      d[4] = (2.0 / 3.0) * var;
      unsigned r = 0;  // high word of the largest scaled update
#pragma unroll
      for (int k = 0; k < 5; ++k) {
        const double delta = q[k] - d[k];
        p[k] += delta;
        r = max(r, abs_hi(delta * (k == 0 ? iq0 : k == 4 ? iq4 : ivs)));
      }
      // the high words of kEffTol = 1e-13 and kEffFail = 1e-9 (no early stop: on
      // coarse grids, 16^3 on the paper's box, the contraction is 20 times the
      // first update, and the skipped one would show at 1e-14)
      conv = r < 0x3d3c25c2u || (it >= kEffMaxIt && r < 0x3e112e0bu);
      // beyond the range of the FP32 starts, or no convergence: the FP64 path decides
      bool fit = in_range(p[0]) && in_range(p[4]) && r < 0x7ff00000u && (conv || it < kEffMaxIt);
      if (fit) {
        isq = rsqrt3(p[4]);
        ith = rcp3(p[4]);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
          AxisBase B;
          fit = axis_base(n3[a], half[a], P.inv_half[a], mid[a], p[1 + a], isq, B) && fit;
          if (lane == 0) S.base[a] = B;
        }
      }
      if (lane == 0) S.go = !fit ? -1 : conv ? 0 : 1;
    }
    bar_solve();
  }
  if (S.go < 0) return;
  bar_solve();  // the weights of warp 3, when there was no round
  if (warp == 0) {
    if (lane == 0) {
      S.tot[6] = S.ab[0] * (p[0] * (ith * isq) * kPi15);
      for (int k = 0; k < 5; ++k) mom[(size_t)i * 5 + k] = q[k];
    }
  }
  bar_solve();
  if (warp < 3) {
    const AxisBase B = S.base[warp];
    const double scale = warp == 0 ? S.tot[6] : 1.0;
    double* fw = fac + (warp == 0 ? 0 : warp == 1 ? P.nvx : P.nvx + P.nvy);
    for (int j = lane; j < n3[warp]; j += 32) {
      unsigned q2, hi, lo;
      const unsigned long long g = fx::gauss(B.a * (2 * j + 1 - n3[warp]) - B.c, (const fx::u64*)kExp2, q2);
      fx::gauss_words(g, q2, hi, lo);
      fw[j] = scale * __hiloint2double((int)hi, (int)lo);
    }
  }
}

}  // namespace

__global__ void __launch_bounds__(kT, 4) step3v_fixed_kernel(const Params3v P, const Tables3v T,
                                                             const double* __restrict__ fin, double* __restrict__ fout,
                                                             double* __restrict__ mom, int* __restrict__ err) {
  extern __shared__ double fac[];  // px[nvx], py[nvy], pz[nvz]
  __shared__ Shared3v S;
  const int i = blockIdx.x, warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double* fo = fout + (size_t)i * P.nv;
  bool valid = false;
  int eg = sample3v(P, fin + (size_t)i * P.nv);
  // a second pass takes the largest exponent of the first as its range
  for (int pass = 0; pass < 2 && !valid; ++pass) {
    if (eg < (int)fx::kExpMin || eg > (int)fx::kExpMax) break;
    valid = stream3v_fixed(P, T, fin, fo, i, eg, S.red + warp * 8);
  }
  if (lane == 0) S.valid[warp] = valid ? 1 : 0;
  __syncthreads();
  bool all = true;
  for (int w = 0; w < kW; ++w) all = all && S.valid[w];
  if (all) {
    if (warp == 0) {
      double t = 0.0;
      if (lane < 7)
        for (int w = 0; w < kW; ++w) t += S.red[w * 8 + lane];
      if (lane < 7) S.tot[lane] = t;
      __syncwarp();
    }
    if (warp < 4) solve3v_fixed(P, i, S, fac, mom, err);
    __syncthreads();
    all = S.go >= 0;
  }
  if (!all) {
    __syncthreads();
    cell3v_f64(P, T, fin, fout, mom, err, i, fac, S);
    return;
  }
  // pass 2: f^{n+1} = b f~ + a Phi on the rows of pass 1
  const Map3v L(P);
  const int nvx = P.nvx, nvy = P.nvy, ys = L.ystep * nvx;
  const double b = S.ab[1];
  const double *py = fac + nvx, *pz = py + nvy;
#pragma unroll 1
  for (int jx = L.l; jx < nvx; jx += L.width) {
    const double x = fac[jx];
#pragma unroll 1
    for (int jz = L.z0; jz < P.nvz; jz += L.zstep) {
      const double xz = x * pz[jz];
      double* p = fo + (jz * nvy + L.y0) * nvx + jx;
#pragma unroll 1
      for (int jy = L.y0; jy < nvy; jy += kAhead3 * L.ystep, p += kAhead3 * ys) {
        double ft[kAhead3];
#pragma unroll
        for (int u = 0; u < kAhead3; ++u) ft[u] = jy + u * L.ystep < nvy ? p[u * ys] : 0.0;
#pragma unroll
        for (int u = 0; u < kAhead3; ++u)
          if (jy + u * L.ystep < nvy) p[u * ys] = fma(b, ft[u], xz * py[jy + u * L.ystep]);
      }
    }
  }
}

// Moments (n, ux, uy, uz, theta) of a state, one CTA per cell.
__global__ void __launch_bounds__(kT) moments3v_kernel(const Params3v P, const Tables3v T,
                                                       const double* __restrict__ f, double* __restrict__ mom) {
  __shared__ double red[kW * 8], tot[8];
  const int i = blockIdx.x;
  double acc[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
  for (int j = threadIdx.x; j < P.nv; j += kT) {
    const Idx3 k = split3(P, j);
    const double v = f[(size_t)i * P.nv + j];
    acc[0] += v;
    acc[1] = fma(T.c[0][k.jx], v, acc[1]);
    acc[2] = fma(T.c[1][k.jy], v, acc[2]);
    acc[3] = fma(T.c[2][k.jz], v, acc[3]);
    acc[4] = fma(T.c2[j], v, acc[4]);
  }
  cta_sum8(acc, red, tot);
  if (threadIdx.x == 0) {
    const double ux = tot[1] / tot[0], uy = tot[2] / tot[0], uz = tot[3] / tot[0];
    mom[(size_t)i * 5 + 0] = tot[0] * P.dv;
    mom[(size_t)i * 5 + 1] = ux;
    mom[(size_t)i * 5 + 2] = uy;
    mom[(size_t)i * 5 + 3] = uz;
    mom[(size_t)i * 5 + 4] = (2.0 / 3.0) * (tot[4] / tot[0] - (ux * ux + uy * uy + uz * uz));
  }
}

// 3D Maxwellian n (pi theta)^(-3/2) exp(-|c - U|^2 / theta) at velocity j.
__device__ __forceinline__ double maxwell3(const Params3v& P, const double* c0, const double* c1, const double* c2,
                                           const double s[5], int j) {
  const Idx3 k = split3(P, j);
  const double dx = c0[k.jx] - s[1], dy = c1[k.jy] - s[2], dz = c2[k.jz] - s[3];
  return s[0] / (kPi() * s[4] * sqrt(kPi() * s[4])) * exp(-(dx * dx + dy * dy + dz * dz) / s[4]);
}

// Per-velocity tables: cell centres, |c|^2, Courant shift and remainder,
// inflow Maxwellians of both ends.
__global__ void tables3v_kernel(const Params3v P, double* c0, double* c1, double* c2, double* cc, int* shift,
                                int* upwind, double* rem, double* ghost, Inflow3v inflow) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j < P.nvx) {
    const double cx = P.vmin[0] + (j + 0.5) * P.dc[0];
    c0[j] = cx;
    const double C = cx * P.dt / P.dx;
    const int s = (int)C;
    shift[j] = s;
    upwind[j] = C > 0.0 ? 1 : -1;
    rem[j] = fabs(C - s);
  }
  if (j < P.nvy) c1[j] = P.vmin[1] + (j + 0.5) * P.dc[1];
  if (j < P.nvz) c2[j] = P.vmin[2] + (j + 0.5) * P.dc[2];
  if (j < P.nv) {
    const Idx3 k = split3(P, j);
    const double cx = P.vmin[0] + (k.jx + 0.5) * P.dc[0];
    const double cy = P.vmin[1] + (k.jy + 0.5) * P.dc[1];
    const double cz = P.vmin[2] + (k.jz + 0.5) * P.dc[2];
    cc[j] = cx * cx + cy * cy + cz * cz;
  }
}

// Inflow Maxwellians (after the axis tables exist).
__global__ void ghost3v_kernel(const Params3v P, const double* c0, const double* c1, const double* c2,
                               double* ghost, Inflow3v inflow) {
  const int j = blockIdx.x * blockDim.x + threadIdx.x;
  if (j >= P.nv) return;
  ghost[j] = maxwell3(P, c0, c1, c2, inflow.s[0], j);
  ghost[P.nv + j] = maxwell3(P, c0, c1, c2, inflow.s[1], j);
}

__global__ void init3v_kernel(const Params3v P, const Tables3v T, double x_split, Inflow3v lr, double* f) {
  const size_t idx = (size_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (idx >= (size_t)P.nx * P.nv) return;
  const int i = (int)(idx / P.nv), j = (int)(idx % P.nv);
  const double x = P.x0 + (i + 0.5) * P.dx;
  f[idx] = maxwell3(P, T.c[0], T.c[1], T.c[2], lr.s[x < x_split ? 0 : 1], j);
}

cudaError_t launch_tables3v(const Params3v& P, double* c0, double* c1, double* c2, double* cc, int* shift,
                            int* upwind, double* rem, double* ghost, const Inflow3v& inflow, cudaStream_t stream) {
  const int n = P.nv > P.nvx ? P.nv : P.nvx;
  tables3v_kernel<<<(n + 255) / 256, 256, 0, stream>>>(P, c0, c1, c2, cc, shift, upwind, rem, ghost, inflow);
  ghost3v_kernel<<<(P.nv + 255) / 256, 256, 0, stream>>>(P, c0, c1, c2, ghost, inflow);
  return cudaGetLastError();
}

cudaError_t launch_init3v(const Params3v& P, const Tables3v& T, double x_split, const Inflow3v& lr, double* f,
                          cudaStream_t stream) {
  const size_t total = (size_t)P.nx * P.nv;
  init3v_kernel<<<(unsigned)((total + 255) / 256), 256, 0, stream>>>(P, T, x_split, lr, f);
  return cudaGetLastError();
}

// Lanes per row and warps along z with the least work per lane: its rows, two
// rows' time for the wait of each batch of kAhead3 loads, and a tenth more for
// each further column, which reads the same sectors again (11 x 21 x 23
// velocities, 1400 cells: 346 us a step with three columns at 77 % use of the
// lanes, 291 with one at 63 %; 18 x 26 x 11, 600 cells: 162 and 115).  By the
// lanes' use alone, 22 x 31 x 19 took three columns with one row a batch: 126 us
// a step on 100 cells and 342 on 600, 58 and 121 with one column of 16 rows.  More
// lanes per row, then more warps along z, unless the gain is above 3 %.  The
// fixed-point kernel takes at most 64 velocities per axis (its squared indices
// and sums then stay within 95 bits), and no plan that leaves more than 70 % of
// the lanes idle: a few dozen velocities or an axis just past a power of two.  On
// 600 cells, us a step fixed / FP64: 3 x 20 x 1 (23 % in use) 38 / 29, 9 x 17 x 1
// (30 %) 33 / 22, 33 x 3 x 3 (29 %) 38 / 37, 5^3 (24 %) 33 / 34, 4^3 (25 %) 24 / 33,
// 9^3 (28 %) 29 / 41; above the line 5 x 33 x 1 (32 %) 35 / 35, 34 x 5 x 5 (33 %) 43
// / 39, 10^3 (39 %) 30 / 43, 6^3 (42 %) 23 / 35, 8^3 25 / 37.
void plan3v(Params3v& P) {
  const int n3[3] = {P.nvx, P.nvy, P.nvz};
  for (int a = 0; a < 3; ++a) {
    P.half[a] = 0.5 * P.dc[a];
    P.inv_half[a] = 1.0 / P.half[a];
    P.mid[a] = std::fma((double)n3[a], P.half[a], P.vmin[a]);  // see velocity_grid
  }
  P.lane_bits = P.zw_bits = 0;
  if (P.nvx > 64 || P.nvy > 64 || P.nvz > 64) return;
  double best = 0.0;
  for (int lb = 5; lb >= 2; --lb)
    for (int zb = 3; zb >= 0; --zb) {
      const int lw = 1 << lb, ys = (kW >> zb) * (32 >> lb), zs = 1 << zb;
      const int cols = (P.nvx + lw - 1) / lw, rows = (P.nvy + ys - 1) / ys, z = (P.nvz + zs - 1) / zs;
      const double work = cols * z * (rows + 2.0 * ((rows + kAhead3 - 1) / kAhead3)) * (1.0 + 0.1 * (cols - 1));
      if (best == 0.0 || work < 0.97 * best) {
        best = work;
        P.lane_bits = lb;
        P.zw_bits = zb;
      }
    }
  const int lw = 1 << P.lane_bits, ys = (kW >> P.zw_bits) * (32 >> P.lane_bits), zs = 1 << P.zw_bits;
  const double lanes = (double)((P.nvx + lw - 1) / lw * lw) * ((P.nvy + ys - 1) / ys * ys) * ((P.nvz + zs - 1) / zs * zs);
  if (P.nv < 0.3 * lanes) P.lane_bits = 0;
}

cudaError_t launch_step3v(const Params3v& P, const Tables3v& T, const double* fin, double* fout, double* mom,
                          int* err, cudaStream_t stream) {
  const size_t smem = sizeof(double) * (size_t)(P.nvx + P.nvy + P.nvz);
  if (P.lane_bits) step3v_fixed_kernel<<<P.nx, kT, smem, stream>>>(P, T, fin, fout, mom, err);
  else step3v_kernel<<<P.nx, kT, smem, stream>>>(P, T, fin, fout, mom, err);
  return cudaGetLastError();
}

cudaError_t launch_moments3v(const Params3v& P, const Tables3v& T, const double* f, double* mom,
                             cudaStream_t stream) {
  moments3v_kernel<<<P.nx, kT, 0, stream>>>(P, T, f, mom);
  return cudaGetLastError();
}

}  // namespace bgk
