// The 3D refinement's seed residuals from FP32 rows and their low parts,
// against FP64: built and run by tests/test_low_residual.py with the library's
// flags.  Points of several azimuth / elevation ranges, velocities that nearly
// solve the point (as a trial's do), are unrelated to it, or are very large.
// Output: "points=... bad=... worst=..." -- points whose difference from FP64
// exceeds the bound the function returns (must be 0), and the largest
// difference in units of that bound.
#include <cmath>
#include <cstdio>
#include <vector>

#include "rvh_device.cuh"

using namespace rvh;

__device__ unsigned long long g_bad, g_n, g_worst;

__device__ float unit(uint32_t x) { return (float)(x >> 8) * 0x1p-24f; }

__global__ void k_check(const double2* trig, int n, double4_32a* pre) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint4 u = philox4x32_10(make_uint4((uint32_t)i, 1u, 0u, 0u), make_uint2(9u, 0u));
  const uint4 v = philox4x32_10(make_uint4((uint32_t)i, 2u, 0u, 0u), make_uint2(9u, 0u));
  const float span = (i & 3) == 0 ? 3.1415925f : ((i & 3) == 1 ? 1.05f : ((i & 3) == 2 ? 1e-3f : 3.2f));
  const float az = (2.0f * unit(u.x) - 1.0f) * span;
  const float el = (2.0f * unit(u.y) - 1.0f) * ((i & 4) ? 0.26f : 1.5f);
  const float scale = (i & 8) ? 40.0f : ((i & 16) ? 4000.0f : 0.5f);
  const float X[3] = {(2.0f * unit(u.z) - 1.0f) * scale, (2.0f * unit(u.w) - 1.0f) * scale,
                      (2.0f * unit(v.x) - 1.0f) * scale};
  double a64[3];
  row_f64<3>(trig, az, el, a64);
  // Doppler: next to the model's, or anywhere
  const double model = a64[0] * X[0] + a64[1] * X[1] + a64[2] * X[2];
  const float w = (i & 32) ? (2.0f * unit(v.y) - 1.0f) * scale : (float)(model + (unit(v.y) - 0.5f) * 1e-4);
  const float4 row = row_f32<3>(az, el, w);
  pre[i] = make_double4_32a(a64[0], a64[1], a64[2],
                            pack_low(low_part(a64[0], row.x), low_part(a64[1], row.y), low_part(a64[2], row.z)));
  const LowSeeds seeds = {pre, {i, i, i}};
  const float sx = fabsf(X[0]) + fabsf(X[1]) + fabsf(X[2]);
  float err;
  const float rf = seed_residual<3>(seeds, 0, row, w, X, sx, &err);
  const double r64 = (double)w - fma((double)X[0], a64[0], fma((double)X[1], a64[1], (double)X[2] * a64[2]));
  // FP64's own rounding of the reference
  const double slack = 0x1p-51 * ((double)fabsf(w) + (double)sx);
  const double d = fabs((double)rf - r64);
  atomicAdd(&g_n, 1ull);
  if (!(d <= (double)err + slack)) atomicAdd(&g_bad, 1ull);
  atomicMax(&g_worst, (unsigned long long)(1e6 * d / ((double)err + slack)));
}

int main() {
  std::vector<double2> tab(kTrigSize);
  for (int k = -kTrigHalf; k <= kTrigHalf; ++k)
    tab[k + kTrigHalf] = make_double2(std::cos(k / 128.0), std::sin(k / 128.0));
  const int n = 1 << 22;
  double2* trig = nullptr;
  double4_32a* pre = nullptr;
  if (cudaMalloc(&trig, sizeof(double2) * kTrigSize) != cudaSuccess ||
      cudaMalloc(&pre, sizeof(double4_32a) * (size_t)n) != cudaSuccess)
    return 2;
  cudaMemcpy(trig, tab.data(), sizeof(double2) * kTrigSize, cudaMemcpyHostToDevice);
  k_check<<<(n + 255) / 256, 256>>>(trig, n, pre);
  unsigned long long bad = 0, cnt = 0, worst = 0;
  cudaMemcpyFromSymbol(&bad, g_bad, 8);
  cudaMemcpyFromSymbol(&cnt, g_n, 8);
  cudaMemcpyFromSymbol(&worst, g_worst, 8);
  const cudaError_t e = cudaDeviceSynchronize();
  printf("points=%llu bad=%llu worst=%.6f\n", cnt, bad, worst * 1e-6);
  cudaFree(trig);
  cudaFree(pre);
  return e == cudaSuccess ? 0 : 2;
}
