// Compares the branch-free square root, reciprocal and quotient of the
// particle kernel's kick with CUDA's IEEE ones: the first two on every float
// of [2^-100, 2^100] (the reciprocal up to 2^100 so that its residual stays
// normal), the quotient on 2^32 mantissa and exponent pairs; and what the
// collision kernel builds on them with its forms in IEEE operations: the
// elastic scattering (directions along and near the axes, components down to
// nothing, speeds and energies beyond its range among them) and beta (speeds
// and limits of all sizes).  Prints the number of differences of each.
#include <cstdio>
#include <cstdint>

#include "device_common.cuh"
#include "step_ops.cuh"

using namespace slpic;

__device__ unsigned long long g_bad[5];

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

__device__ __forceinline__ uint32_t next(uint64_t& z) {
  z = z * 6364136223846793005ull + 1442695040888963407ull;
  return (uint32_t)(z >> 33);
}
__device__ __forceinline__ float u01(uint64_t& z) { return ((next(z) >> 8) + 0.5f) * 1.1920929e-07f; }

__global__ void k_scatter(uint64_t n, StepConsts<float> K) {
  for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < n;
       i += (uint64_t)gridDim.x * blockDim.x) {
    uint64_t z = i * 0x9E3779B97F4A7C15ull + 12345u;
    float v[3];
    const float size = exp2f(-12.0f + 44.0f * u01(z));
    const uint32_t kind = next(z) % 4u;
    for (int k = 0; k < 3; ++k) {
      const float c = kind == 0u ? 2.0f * u01(z) - 1.0f : exp2f(-40.0f * u01(z));
      v[k] = next(z) % 16u == 0u ? 0.0f : size * (next(z) & 1u ? c : -c);
    }
    if (kind == 3u) v[next(z) % 3u] = size;
    const float eps = exp2f(-34.0f + 68.0f * u01(z)), u2 = u01(z), u3 = u01(z), kv = 3.5e11f;
    const float v2 = v[0] * v[0] + v[1] * v[1] + v[2] * v[2];
    const Velocity<float> a = scatter_elastic_any(K, kv, v[0], v[1], v[2], eps, u2, u3);
    const Velocity<float> b =
        scatter_elastic<float>(K, kv, v[0], v[1], v[2], sqrtf(v2), eps, u2, u3);
    if (__float_as_uint(a.vx) != __float_as_uint(b.vx) ||
        __float_as_uint(a.vy) != __float_as_uint(b.vy) ||
        __float_as_uint(a.vz) != __float_as_uint(b.vz))
      if (v2 > 0.0f) atomicAdd(&g_bad[3], 1ull);
    const float w2 = next(z) % 64u == 0u ? 0.0f : exp2f(-140.0f + 268.0f * u01(z));
    const float L = next(z) % 8u == 0u ? INFINITY : exp2f(-100.0f + 200.0f * u01(z));
    if (__float_as_uint(beta_any(w2, L)) != __float_as_uint(beta_of(sqrtf(w2), L)))
      atomicAdd(&g_bad[4], 1ull);
  }
}

int main() {
  k_unary<<<1216, 256>>>((127u - 100) << 23, (127u + 100) << 23);
  k_pairs<<<1216, 256>>>(1ull << 32);
  StepConsts<float> K = {};
  K.two_pi = 6.2831855f;
  K.R2 = 2.7464e-5f;
  k_scatter<<<1216, 256>>>(1ull << 28, K);
  unsigned long long bad[5];
  const cudaError_t e = cudaMemcpyFromSymbol(bad, g_bad, sizeof bad);
  std::printf("%llu %llu %llu %llu %llu %s\n", bad[0], bad[1], bad[2], bad[3], bad[4],
              cudaGetErrorString(e));
  return e != cudaSuccess;
}
