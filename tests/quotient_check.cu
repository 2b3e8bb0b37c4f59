// Compares csrc/quotient.cuh with the division, for test_gpu_quotient.py.
#include <stdint.h>

#include "quotient.cuh"

namespace {

// The distance of two floats of one sign in units in the last place (0 and -0
// are the same).
__device__ uint32_t ulps(float a, float b) {
  if (a == b) return 0;
  const uint32_t x = __float_as_uint(a), y = __float_as_uint(b);
  return x > y ? x - y : y - x;
}

__device__ void note(uint32_t far, unsigned long long* differ, uint32_t* most) {
  if (far == 0) return;
  atomicAdd(differ, 1ull);
  atomicMax(most, far);
}

// silu_mid against silu for every float that it takes, and how many there are.
__global__ void silu_kernel(unsigned long long* taken, unsigned long long* differ, uint32_t* most) {
  const uint64_t n = (uint64_t)gridDim.x * blockDim.x;
  unsigned long long mine = 0;
  for (uint64_t u = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; u < (1ull << 32); u += n) {
    const float x = __uint_as_float((uint32_t)u);
    if (!as2d::silu_mid_takes(x)) continue;
    ++mine;
    note(ulps(as2d::silu_mid(x), as2d::silu(x)), differ, most);
  }
  atomicAdd(taken, mine);
}

__device__ uint64_t mix(uint64_t z) {  // splitmix64
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// quotient against the division for n sums of weights d in [1, 65536] (every
// row's largest weight is 1) and numerators x of both signs, 2^-60 to 2^60.
__global__ void quotient_kernel(uint64_t n, unsigned long long* differ, uint32_t* most) {
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (uint64_t)gridDim.x * blockDim.x) {
    const uint64_t a = mix(i);
    const float d = __uint_as_float(0x3F800000u + (uint32_t)(a >> 32) % 0x08000000u);
    const float x = __uint_as_float(((uint32_t)a & 0x80000000u) | (0x21800000u + ((uint32_t)a & 0x7FFFFFFFu) % 0x3C000000u));
    note(ulps(as2d::quotient(x, d, 1.f / d), x / d), differ, most);
  }
}

}  // namespace

// out: [0] values taken, [1] silu results that differ, [2] their largest
// distance, [3] quotients that differ of n, [4] their largest distance.
extern "C" int quotient_check(uint64_t n, uint64_t* out) {
  unsigned long long* d = nullptr;
  if (cudaMalloc(&d, 40) != cudaSuccess) return 1;
  cudaMemset(d, 0, 40);
  silu_kernel<<<152 * 8, 256>>>(d, d + 1, (uint32_t*)(d + 2));
  quotient_kernel<<<152 * 8, 256>>>(n, d + 3, (uint32_t*)(d + 4));
  const cudaError_t e = cudaMemcpy(out, d, 40, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e == cudaSuccess ? 0 : 2;
}
