// Accuracy of the fixed-point exponential (exp_fixed.cuh) against the host's
// long-double expl: the largest error in units of the last place over random
// s for several a2, its exact cases and its range test. Exits non-zero when an
// error is above 0.85 ulp (0.5 from the one rounding, below 0.3 from the
// truncated products and the table, which hold at least 2^-55).
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
#include <cuda_runtime.h>
#include "exp_fixed.cuh"
using namespace hpac;

__global__ void values(const double *s, double *y, int *ok, int n, ExpFixed ex) {
  __shared__ uint64_t ta[32], tb[64];
  if (threadIdx.x < 32) ta[threadIdx.x] = ex.a[threadIdx.x];
  if (threadIdx.x < 64) tb[threadIdx.x] = ex.b[threadIdx.x];
  __syncthreads();
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  ok[i] = exp_fixed_in_range(s[i], ex.limit) ? 1 : 0;
  y[i] = ok[i] ? exp_fixed(s[i], ta, tb, ex.c, ex.ex) : -1.0;
}

int main() {
  const int n = 1 << 18;
  double *ds, *dy;
  int *dok, fails = 0;
  cudaMalloc(&ds, n * sizeof(double));
  cudaMalloc(&dy, n * sizeof(double));
  cudaMalloc(&dok, n * sizeof(int));
  std::vector<double> s(n), y(n);
  std::vector<int> ok(n);
  std::mt19937_64 g(2308);
  for (double a2 : {0.5, 0.0, 1e-9, 0.3, 7.25, 4000.0, 1e12}) {
    const ExpFixed ex = exp_fixed_constants(a2);
    std::uniform_real_distribution<double> near(0.0, 4.0), all(0.0, a2 > 0 ? 720.0 / a2 : 1e300), mag(-300.0, 3.0);
    for (int i = 0; i < n; ++i) s[i] = i % 3 == 0 ? near(g) : i % 3 == 1 ? all(g) : std::pow(10.0, mag(g));
    const double special[] = {0.0, 5e-324, 1e-310, 2.2250738585072014e-308, INFINITY, NAN, -1.0, 1.7e308};
    for (int i = 0; i < 8; ++i) s[i] = special[i];
    cudaMemcpy(ds, s.data(), n * sizeof(double), cudaMemcpyHostToDevice);
    values<<<(n + 255) / 256, 256>>>(ds, dy, dok, n, ex);
    if (cudaDeviceSynchronize() != cudaSuccess) return 2;
    cudaMemcpy(y.data(), dy, n * sizeof(double), cudaMemcpyDeviceToHost);
    cudaMemcpy(ok.data(), dok, n * sizeof(int), cudaMemcpyDeviceToHost);
    double worst = 0.0;
    int taken = 0, wrong = 0;
    for (int i = 0; i < n; ++i) {
      const bool must = s[i] >= 0.0 && std::isfinite(s[i]) && a2 * s[i] < 690.0;
      const bool may = s[i] >= 0.0 && std::isfinite(s[i]) && a2 * s[i] <= 700.0;
      wrong += (must && !ok[i]) || (ok[i] && !may);
      if (!ok[i]) continue;
      ++taken;
      const long double r = expl(-(long double)a2 * s[i]);
      const double ulp = std::nextafter((double)r, 2.0) - (double)r;
      const double e = (double)(fabsl(y[i] - r) / ulp);
      if (e > worst) worst = e;
    }
    const bool exact = y[0] == 1.0 && y[1] == 1.0 && y[2] == 1.0;
    printf("a2 %g: %d values, worst %.3f ulp, exact cases %d, range test mismatches %d\n", a2, taken, worst, exact, wrong);
    fails += worst > 0.85 || !exact || wrong;
  }
  return fails;
}
