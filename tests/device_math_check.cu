// exp_fixed and recip_fixed (fixexp.h) as the device computes them, elementwise:
// prints how many of the exponentials differ from the host's integer code, how
// many reciprocals from the division, and the number of each.
#include "fixexp.h"

#include <cstdio>
#include <random>
#include <vector>

__global__ void eval(int n, const double* x, const double* d, double* e, double* r) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  e[i] = bd::exp_fixed(x[i]);
  r[i] = bd::recip_fixed(d[i]);
}

int main() {
  const int n = 1 << 20;
  std::mt19937_64 g(11);
  std::uniform_real_distribution<double> u(-1.0, 1.0);
  std::vector<double> x(n), d(n), e(n), r(n);
  for (int i = 0; i < n; ++i) {
    x[i] = i % 3 == 0 ? 64 * u(g) : i % 3 == 1 ? std::ldexp(u(g), 6 - int(g() % 70)) : 64 - std::ldexp(std::fabs(u(g)), -int(g() % 46));
    if (!(std::fabs(x[i]) < 64)) x[i] = 0.0;
    uint64_t m = g() & 0xfffffffffffffull;
    if (i % 4 == 1) m &= 0x3fffff;
    if (i % 4 == 2) m |= 0xfffffffc00000ull;
    if (i % 4 == 3) m = (m & 0xfffffe0000000ull) | (i % 8 == 3 ? 0x1fffffffull : 0);
    const uint64_t b = (g() & 1) << 63 | (1 + g() % 2043) << 52 | m;
    std::memcpy(&d[i], &b, 8);
  }
  const double edge[] = {0.0, -0.0, 5e-324, 1e-310, 1.7e308, -1.7e308, INFINITY, -INFINITY, 1.0, -2.0};
  for (int i = 0; i < 10; ++i) d[i] = edge[i];
  double* p[4];
  for (double*& q : p)
    if (cudaMalloc(&q, n * 8) != cudaSuccess) return 1;
  cudaMemcpy(p[0], x.data(), n * 8, cudaMemcpyHostToDevice);
  cudaMemcpy(p[1], d.data(), n * 8, cudaMemcpyHostToDevice);
  eval<<<n / 256, 256>>>(n, p[0], p[1], p[2], p[3]);
  if (cudaMemcpy(e.data(), p[2], n * 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  if (cudaMemcpy(r.data(), p[3], n * 8, cudaMemcpyDeviceToHost) != cudaSuccess) return 1;
  long be = 0, br = 0;
  for (int i = 0; i < n; ++i) {
    const double he = bd::exp_fixed(x[i]), hr = 1.0 / d[i];
    be += std::memcmp(&he, &e[i], 8) != 0;
    br += std::memcmp(&hr, &r[i], 8) != 0;
  }
  std::printf("%ld %ld %d\n", be, br, n);
  return 0;
}
