// pipe_phase.h — phases of a ring of stages, plain arithmetic for the device and the host.
#pragma once
#include <cstdint>

#ifdef __CUDACC__
#define SIMX_HD __host__ __device__ __forceinline__
#else
#define SIMX_HD inline
#endif

namespace simx {

// Chunk g of a sequence lands in stage g mod S and completes phase g / S of that stage's barrier.
// The parity of the phase that the last chunk issued into stage st completes, `issued` chunks having
// been issued in order; -1: none went there.  A wait for it ends when no copy into the stage is in
// flight: a chunk is issued into a stage only after the one before it has landed.
SIMX_HD int last_parity(uint32_t issued, uint32_t S, uint32_t st) {
  return st < issued ? (int)((issued - 1u - st) / S & 1u) : -1;
}

}  // namespace simx
