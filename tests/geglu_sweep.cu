// Device sweep for test_gpu_geglu_pair.py: the packed GeGLU against the recipe, fp32 bit for bit, on a
// contiguous range of gate bit patterns.  counts: {gates in range, mismatches, a mismatching gate's bits}.
#include "../paper_2608_28003_gb300/csrc/common.cuh"

using namespace w8a8;

__global__ void sweep_kernel(uint32_t first, unsigned long long n, float u, unsigned long long* counts) {
  const f32x2 nz = f2_neg_zero();
  unsigned long long taken = 0, wrong = 0;
  uint32_t at = 0;
  const unsigned long long step = 2ull * gridDim.x * blockDim.x;
  for (unsigned long long i = 2ull * (blockIdx.x * blockDim.x + threadIdx.x); i + 1 < n; i += step) {
    const float g0 = __uint_as_float(first + (uint32_t)i), g1 = __uint_as_float(first + (uint32_t)i + 1);
    float h0, h1;
    geglu_pair(g0, g1, u, u, nz, h0, h1);
    if (!geglu_in_range(g0) || !geglu_in_range(g1)) continue;
    taken += 2;
    if (__float_as_uint(h0) != __float_as_uint(geglu_recipe(g0, u))) {
      ++wrong;
      at = __float_as_uint(g0);
    }
    if (__float_as_uint(h1) != __float_as_uint(geglu_recipe(g1, u))) {
      ++wrong;
      at = __float_as_uint(g1);
    }
  }
  atomicAdd(counts, taken);
  if (wrong) {
    atomicAdd(counts + 1, wrong);
    atomicExch(counts + 2, (unsigned long long)at);
  }
}

extern "C" int geglu_sweep(uint32_t first, unsigned long long n, float u, unsigned long long* counts) {
  sweep_kernel<<<1216, 256>>>(first, n, u, counts);
  return (int)cudaDeviceSynchronize();
}
