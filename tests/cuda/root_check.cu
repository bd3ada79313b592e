// sqrt_t(double) and rcp_t(double) of fr_arith.cuh against CUDA's correctly rounded operations on 2^20
// inputs each (counter-based splitmix64), over all normal exponents of sqrt_t's fast path and below it,
// and on special values.  Prints the worst error in ulps and the special values that differ.
#include <cstdint>
#include <cstdio>
#include <cuda_runtime.h>

#include "fr_arith.cuh"

using namespace frg;

__device__ uint64_t splitmix64(uint64_t i) {
  uint64_t z = i * 0x9E3779B97F4A7C15ull + 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

__global__ void k_check(int64_t n, unsigned long long* worst) {
  const int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const uint64_t r = splitmix64(uint64_t(i));
  const int e = (i & 1) ? 1 + int((r >> 52) % 2046u) : 1023 - 8 + int((r >> 52) % 16u);
  const double x = __longlong_as_double((long long)((uint64_t(e) << 52) | (r & 0xFFFFFFFFFFFFFull)));
  long long d = __double_as_longlong(sqrt_t(x)) - __double_as_longlong(sqrt(x));
  atomicMax(&worst[0], (unsigned long long)(d < 0 ? -d : d));
  if (e > 100 && e < 1940) {
    d = __double_as_longlong(rcp_t(x)) - __double_as_longlong(1.0 / x);
    atomicMax(&worst[1], (unsigned long long)(d < 0 ? -d : d));
  }
  if (i == 0) {
    const double inf = __longlong_as_double(0x7FF0000000000000ll);
    const double sp[6] = {0.0, -0.0, inf, 4.9e-324, 2.3e-308, 1.0};
    for (int k = 0; k < 6; ++k)
      if (__double_as_longlong(sqrt_t(sp[k])) != __double_as_longlong(sqrt(sp[k]))) atomicAdd(&worst[2], 1ull);
    if (sqrt_t(-1.0) == sqrt_t(-1.0)) atomicAdd(&worst[2], 1ull);
    if (sqrt_t(sqrt(-1.0)) == sqrt_t(sqrt(-1.0))) atomicAdd(&worst[2], 1ull);
  }
}

int main() {
  const int64_t n = int64_t(1) << 20;
  unsigned long long* d = nullptr;
  if (cudaMalloc(&d, 3 * sizeof(unsigned long long)) != cudaSuccess) return 2;
  cudaMemset(d, 0, 3 * sizeof(unsigned long long));
  k_check<<<unsigned((n + 255) / 256), 256>>>(n, d);
  unsigned long long h[3];
  if (cudaMemcpy(h, d, sizeof(h), cudaMemcpyDeviceToHost) != cudaSuccess) return 3;
  cudaFree(d);
  printf("sqrt %llu\nrcp %llu\nspecial %llu\n", h[0], h[1], h[2]);
  return 0;
}
