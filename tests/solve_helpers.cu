// Checks the device helpers of csrc/bgk_solve.cuh: prints the largest relative
// error of each over its range, in units of 2^-53.
#include "bgk_solve.cuh"

#include <cmath>
#include <cstdio>
#include <random>
#include <vector>

enum { RCP, RSQRT, EXP, POW, KINDS };

__global__ void eval(int kind, int n, const double* x, const double* y, double* out) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[i] = kind == RCP     ? bgk::rcp3(x[i])
           : kind == RSQRT ? bgk::rsqrt3(x[i])
           : kind == EXP   ? bgk::exp_neg_fixed(x[i])
                           : bgk::pow_fixed(x[i], y[i]);
}

int main() {
  const int n = 1 << 17;
  std::mt19937_64 g(1);
  std::uniform_real_distribution<double> U(0, 1);
  std::vector<double> x(n), y(n), r(n);
  double *dx, *dy, *dr;
  bool ok = cudaMalloc(&dx, n * 8) == cudaSuccess && cudaMalloc(&dy, n * 8) == cudaSuccess && cudaMalloc(&dr, n * 8) == cudaSuccess;
  for (int kind = 0; ok && kind < KINDS; ++kind) {
    for (int i = 0; i < n; ++i) {
      // the whole range of the FP32 starts; e^-x to 22 (below 32 log2 units); theta^(1 - omega) of moderate theta
      x[i] = kind == RCP || kind == RSQRT ? std::ldexp(1 + U(g), (int)(190 * U(g)) - 95) : kind == EXP ? 22 * U(g) * (i % 2 ? 1 : U(g)) : std::exp2(2 * U(g) - 1);
      y[i] = 2 * U(g) - 1;
    }
    ok = cudaMemcpy(dx, x.data(), n * 8, cudaMemcpyHostToDevice) == cudaSuccess &&
         cudaMemcpy(dy, y.data(), n * 8, cudaMemcpyHostToDevice) == cudaSuccess;
    if (!ok) break;
    eval<<<n / 128, 128>>>(kind, n, dx, dy, dr);
    ok = cudaMemcpy(r.data(), dr, n * 8, cudaMemcpyDeviceToHost) == cudaSuccess;
    long double worst = 0;
    for (int i = 0; i < n; ++i) {
      const long double v = x[i], want = kind == RCP     ? 1 / v
                                         : kind == RSQRT ? 1 / std::sqrt(v)
                                         : kind == EXP   ? std::exp(-v)
                                                         : std::pow(v, (long double)y[i]);
      worst = std::fmax(worst, std::fabs(r[i] / want - 1));
    }
    std::printf("%.4Lf\n", worst * 0x1p53L);
  }
  return ok ? 0 : 1;
}
