// atan2_table against the library's atan2: built and run by
// tests/test_heading.py with the library's flags.  Vectors of every direction
// and of lengths 1e-28 .. 1e28, the axes with both signs of zero, and the
// arguments left to the library.  Output: "points=... worst=... diff=..." --
// the largest difference in units of 2^-52 (modulo a turn), and how many of the
// special arguments give another result than the library.
#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "rvh_device.cuh"

using namespace rvh;

__device__ unsigned long long g_worst, g_n, g_diff;

__global__ void k_check(const double2* trig, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint4 u = philox4x32_10(make_uint4((uint32_t)i, 5u, 0u, 0u), make_uint2(3u, 0u));
  const double t = (double)u.x * (6.283185307179586 / 4294967296.0);
  const double r = exp(((double)u.y / 4294967296.0 - 0.5) * ((i & 1) ? 128.0 : 8.0));
  double x = r * cos(t), y = r * sin(t);
  if ((i & 1023) < 8) {  // axes
    const double z = (i & 1) ? -0.0 : 0.0;
    if (i & 4) x = z; else y = z;
    if (i & 2) { x = -x; y = -y; }
  }
  const double d = fabs(atan2_table(trig, y, x) - atan2(y, x));
  const double e = fmin(d, fabs(d - 6.283185307179586));
  atomicMax(&g_worst, (unsigned long long)(e * 0x1p52 * 1000.0));
  atomicAdd(&g_n, 1ull);
  if (i == 0) {
    const double inf = __longlong_as_double(0x7ff0000000000000LL), nan = __longlong_as_double(0x7ff8000000000000LL);
    const double v[10] = {0.0, -0.0, 1.0, -1.0, inf, -inf, 1e-40, -1e300, nan, 5e-324};
    for (int p = 0; p < 10; ++p)
      for (int q = 0; q < 10; ++q) {
        const double m = fmax(fabs(v[p]), fabs(v[q]));
        if (m >= 1e-30 && m <= 1e30) continue;
        const double a = atan2_table(trig, v[p], v[q]), b = atan2(v[p], v[q]);
        if (__double_as_longlong(a) != __double_as_longlong(b) && !(a != a && b != b)) atomicAdd(&g_diff, 1ull);
      }
  }
}

int main() {
  std::vector<double2> tab(kTrigSize);
  for (int k = -kTrigHalf; k <= kTrigHalf; ++k)
    tab[k + kTrigHalf] = make_double2(std::cos(k / 128.0), std::sin(k / 128.0));
  double2* trig = nullptr;
  if (cudaMalloc(&trig, sizeof(double2) * kTrigSize) != cudaSuccess) return 2;
  cudaMemcpy(trig, tab.data(), sizeof(double2) * kTrigSize, cudaMemcpyHostToDevice);
  const int n = 1 << 24;
  k_check<<<n / 256, 256>>>(trig, n);
  unsigned long long worst = 0, cnt = 0, diff = 0;
  cudaMemcpyFromSymbol(&worst, g_worst, 8);
  cudaMemcpyFromSymbol(&cnt, g_n, 8);
  cudaMemcpyFromSymbol(&diff, g_diff, 8);
  const cudaError_t e = cudaDeviceSynchronize();
  printf("points=%llu worst=%.3f diff=%llu\n", cnt, worst * 1e-3, diff);
  cudaFree(trig);
  return e == cudaSuccess ? 0 : 2;
}
