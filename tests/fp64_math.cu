// Harness of test_gpu_fp64_math.py: the float64 exponential by table and the distance with
// its reciprocal on the GPU against the host's long double.  Prints the largest errors in
// units in the last place, "<exp> <r> <1/r>", then one line per special case that is not
// what CUDA's exp, sqrt and division give.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "device_common.cuh"

using namespace apip;

__global__ void run(const double2* tab, const double* x, const double* r2, double* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  out[6 * i] = exp_tab(tab, x[i]);
  out[6 * i + 1] = exp(x[i]);
  len_inv(r2[i], &out[6 * i + 2], &out[6 * i + 3]);
  out[6 * i + 4] = sqrt(r2[i]);
  out[6 * i + 5] = 1.0 / sqrt(r2[i]);
}

static double ulps(double got, long double want) {
  int e;
  std::frexp((double)want, &e);
  return (double)(std::fabs((long double)got - want) / std::ldexp(1.0L, e - 53));
}

int main() {
  const double inf = INFINITY;
  std::vector<double> x = {0.0, -0.0, 1e-300, -1e-20, 689.9999, -689.9999, 690.0, -690.0, 709.7, -745.0, -800.0, 800.0, inf, -inf, NAN, 1e-3};
  std::vector<double> r2 = {0.0, 4.9e-324, 1e-310, 2.3e-308, 1.7e308, inf, NAN, 1.0, 4.0, 0.25, 2.0, 3.0, 1e-30, 25.0, 19.36, 30.25};
  const int special = (int)x.size(), n = special + (1 << 20);
  std::mt19937_64 gen(7);
  std::uniform_real_distribution<double> u(-1, 1);
  for (int i = special; i < n; ++i) {
    x.push_back(i % 2 ? 20 * u(gen) : 690 * u(gen));
    r2.push_back(i % 2 ? 15 + 15 * u(gen) : std::exp(690 * u(gen)));
  }
  std::vector<double2> h(kExpTab);
  exp_table_fill(h.data());
  double2* tab;
  double *dx, *dr, *d;
  std::vector<double> out(6 * (size_t)n);
  if (cudaMalloc(&tab, sizeof(double2) * kExpTab) || cudaMalloc(&dx, 8 * n) || cudaMalloc(&dr, 8 * n) || cudaMalloc(&d, 48 * (size_t)n)) return 1;
  cudaMemcpy(tab, h.data(), sizeof(double2) * kExpTab, cudaMemcpyHostToDevice);
  cudaMemcpy(dx, x.data(), 8 * n, cudaMemcpyHostToDevice);
  cudaMemcpy(dr, r2.data(), 8 * n, cudaMemcpyHostToDevice);
  run<<<(n + 255) / 256, 256>>>(tab, dx, dr, d, n);
  if (cudaMemcpy(out.data(), d, 48 * (size_t)n, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  double worst[3] = {0, 0, 0};
  for (int i = special; i < n; ++i) {
    const double* o = out.data() + 6 * (size_t)i;
    const long double s = sqrtl((long double)r2[i]);
    worst[0] = std::fmax(worst[0], ulps(o[0], expl((long double)x[i])));
    worst[1] = std::fmax(worst[1], ulps(o[2], s));
    worst[2] = std::fmax(worst[2], ulps(o[3], 1.0L / s));
  }
  std::printf("%.4f %.4f %.4f\n", worst[0], worst[1], worst[2]);
  auto near = [](double a, double b) { return (std::isnan(a) && std::isnan(b)) || a == b || std::fabs(a - b) <= 5e-16 * std::fabs(b); };
  for (int i = 0; i < special; ++i) {
    const double* o = out.data() + 6 * (size_t)i;
    if (!near(o[0], o[1])) std::printf("exp(%g) = %g, not %g\n", x[i], o[0], o[1]);
    if (!near(o[2], o[4]) || !near(o[3], o[5])) std::printf("r^2 = %g: %g %g, not %g %g\n", r2[i], o[2], o[3], o[4], o[5]);
  }
  return 0;
}
