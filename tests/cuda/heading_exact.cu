// atan2_table against the host's long double atan2: built and run by
// tests/test_heading_exact.py with the library's flags.  Vectors of every
// direction and of lengths 1e-28 .. 1e28.  Output: "points=... worst=..." in
// thousandths of 2^-52, modulo a turn.
#include <cmath>
#include <cstdio>
#include <vector>

#include "rvh_device.cuh"

using namespace rvh;

__global__ void k_angles(const double2* trig, int n, double* x, double* y, double* t) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint4 u = philox4x32_10(make_uint4((uint32_t)i, 9u, 0u, 0u), make_uint2(4u, 0u));
  const double a = (double)u.x * (6.283185307179586 / 4294967296.0);
  const double r = exp(((double)u.y / 4294967296.0 - 0.5) * ((i & 1) ? 128.0 : 8.0));
  x[i] = r * cos(a);
  y[i] = (i & 15) == 0 ? 1e-9 * r * sin(a) : r * sin(a);  // headings near 0 and pi too
  t[i] = atan2_table(trig, y[i], x[i]);
}

int main() {
  std::vector<double2> tab(kTrigSize);
  for (int k = -kTrigHalf; k <= kTrigHalf; ++k)
    tab[k + kTrigHalf] = make_double2(std::cos(k / 128.0), std::sin(k / 128.0));
  const int n = 1 << 20;
  double2* trig = nullptr;
  double* d = nullptr;
  if (cudaMalloc(&trig, sizeof(double2) * kTrigSize) != cudaSuccess) return 2;
  if (cudaMalloc(&d, sizeof(double) * 3 * n) != cudaSuccess) return 2;
  cudaMemcpy(trig, tab.data(), sizeof(double2) * kTrigSize, cudaMemcpyHostToDevice);
  k_angles<<<n / 256, 256>>>(trig, n, d, d + n, d + 2 * n);
  std::vector<double> h(3 * (size_t)n);
  if (cudaMemcpy(h.data(), d, sizeof(double) * 3 * n, cudaMemcpyDeviceToHost) != cudaSuccess) return 2;
  const long double turn = 2.0L * std::acos(-1.0L);
  long double worst = 0.0L;
  for (int i = 0; i < n; ++i) {
    const long double e = std::fabs((long double)h[2 * (size_t)n + i] - std::atan2((long double)h[n + (size_t)i], (long double)h[i]));
    const long double w = std::fmin(e, std::fabs(e - turn));
    if (!(w <= worst)) worst = w;
  }
  std::printf("points=%d worst=%lld\n", n, (long long)(worst * 0x1p52L * 1000.0L));
  cudaFree(trig);
  cudaFree(d);
  return 0;
}
