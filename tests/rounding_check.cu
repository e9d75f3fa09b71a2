// Compares the branch-free square root, reciprocal and quotient of the
// particle kernel's kick with CUDA's IEEE ones: the first two on every float
// of [2^-100, 2^100] (the reciprocal up to 2^100 so that its residual stays
// normal), the quotient on 2^32 mantissa and exponent pairs.  Prints the
// number of differences of each.
#include <cstdio>
#include <cstdint>

#include "device_common.cuh"

using namespace slpic;

__device__ unsigned long long g_bad[3];

__global__ void k_unary(uint32_t lo, uint32_t hi) {
  for (uint64_t i = lo + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < hi;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const float x = __uint_as_float((uint32_t)i);
    if (__float_as_uint(sqrt_mid(x)) != __float_as_uint(__fsqrt_rn(x))) atomicAdd(&g_bad[0], 1ull);
    if (__float_as_uint(rcp_mid(x)) != __float_as_uint(__frcp_rn(x))) atomicAdd(&g_bad[1], 1ull);
  }
}

__global__ void k_pairs(uint64_t n) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    uint64_t z = (i + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    const uint32_t ea = 127 - 40 + (uint32_t)((z >> 32) % 80);
    const uint32_t eb = 127 - 40 + (uint32_t)((z >> 48) % 80);
    const float a = __uint_as_float((uint32_t)(z >> 63) << 31 | ea << 23 | ((uint32_t)z & 0x7FFFFF));
    const float b = __uint_as_float(eb << 23 | ((uint32_t)i & 0x7FFFFF));
    if (__float_as_uint(div_mid(a, b)) != __float_as_uint(__fdiv_rn(a, b)))
      atomicAdd(&g_bad[2], 1ull);
  }
}

int main() {
  k_unary<<<1216, 256>>>((127u - 100) << 23, (127u + 100) << 23);
  k_pairs<<<1216, 256>>>(1ull << 32);
  unsigned long long bad[3];
  const cudaError_t e = cudaMemcpyFromSymbol(bad, g_bad, sizeof bad);
  std::printf("%llu %llu %llu %s\n", bad[0], bad[1], bad[2], cudaGetErrorString(e));
  return e != cudaSuccess;
}
