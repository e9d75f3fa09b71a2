// The branch-free square root, reciprocal and quotient of the particle kernel's
// kick against CUDA's IEEE ones at the ends of the range they are stated for:
// the first two on every float of [2^100, 2^126], the quotient on 2^32 pairs of
// mantissas and of exponents from 2^-100 to 2^126 whose quotient lies there too.
// Prints the number of differences of each.
#include <cstdint>
#include <cstdio>

#include "device_common.cuh"

using namespace slpic;

__device__ unsigned long long g_bad[4];  // (the last counts the pairs)

__global__ void k_unary(uint32_t lo, uint32_t hi) {
  for (uint64_t i = lo + blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i <= hi;
       i += (uint64_t)gridDim.x * blockDim.x) {
    const float x = __uint_as_float((uint32_t)i);
    if (__float_as_uint(sqrt_mid(x)) != __float_as_uint(__fsqrt_rn(x))) atomicAdd(&g_bad[0], 1ull);
    if (__float_as_uint(rcp_mid(x)) != __float_as_uint(__frcp_rn(x))) atomicAdd(&g_bad[1], 1ull);
  }
}

__global__ void k_pairs(uint64_t n) {
  unsigned long long bad = 0, seen = 0;
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    uint64_t z = (i + 77) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    z ^= z >> 31;
    const uint32_t eb = 27u + (uint32_t)(z >> 40) % 226u;  // 2^-100 .. 2^126
    // the quotient's exponent from -99 to 125, as far as a stays in its range
    const int lo = max(-99, 27 - (int)eb), hi = min(125, 252 - (int)eb);
    const uint32_t ea = (uint32_t)((int)eb + lo + (int)((uint32_t)(z >> 47) % (uint32_t)(hi - lo + 1)));
    const float a = __uint_as_float((uint32_t)(z >> 63) << 31 | ea << 23 | ((uint32_t)z & 0x7FFFFF));
    const float b = __uint_as_float(eb << 23 | ((uint32_t)i & 0x7FFFFF));
    ++seen;
    if (__float_as_uint(div_mid(a, b)) != __float_as_uint(__fdiv_rn(a, b))) ++bad;
  }
  atomicAdd(&g_bad[2], bad);
  atomicAdd(&g_bad[3], seen);
}

int main() {
  k_unary<<<1216, 256>>>((127u + 100) << 23, (127u + 126) << 23);
  k_pairs<<<1216, 256>>>(1ull << 32);
  unsigned long long bad[4];
  const cudaError_t e = cudaMemcpyFromSymbol(bad, g_bad, sizeof bad);
  std::printf("%llu %llu %llu of %llu %s\n", bad[0], bad[1], bad[2], bad[3],
              cudaGetErrorString(e));
  return e != cudaSuccess;
}
