// math_check.cu — the branch-free elementary functions of the block forward (fwd_block.cuh) against
// the ones that define the bits (devmath.cuh), input by input.
#include <cstdint>

#include "fwd_block.cuh"
#include "kernels.h"

namespace simx {

namespace {
// which 0: tanh on every fp32 pattern; 1: exp on those that are not above zero (and NaN).  Counts
// the inputs whose results differ; two NaNs count as the same.
__global__ void __launch_bounds__(256) k_math_check(int which, unsigned long long* count) {
  unsigned long long bad = 0ull;
  const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
  for (uint64_t i = (uint64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (1ull << 32); i += stride) {
    const float x = __uint_as_float((uint32_t)i);
    if (which == 1 && x > 0.0f) continue;
    const float a = which == 0 ? det_tanh(x) : det_exp(x);
    const float b = which == 0 ? fwd::tanh_flat(x) : fwd::exp_flat(x);
    if (__float_as_uint(a) != __float_as_uint(b) && !(a != a && b != b)) ++bad;
  }
  if (bad) atomicAdd(count, bad);
}
}  // namespace

cudaError_t launch_math_check(int which, unsigned long long* count, cudaStream_t s) {
  const cudaError_t e = cudaMemsetAsync(count, 0, sizeof(*count), s);
  if (e != cudaSuccess) return e;
  k_math_check<<<sm_count() * 8, 256, 0, s>>>(which, count);
  count_launches(1);
  return cudaGetLastError();
}

}  // namespace simx
