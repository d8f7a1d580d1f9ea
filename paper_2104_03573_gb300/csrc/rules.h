// Rules the launches and kernels follow that are plain arithmetic on sizes:
// C++ without CUDA headers, so that the host compiler builds them too.
#pragma once

#include <cstddef>
#include <cstdint>

#ifdef __CUDACC__
#define MCBTE_RULE __host__ __device__ __forceinline__
#else
#define MCBTE_RULE inline
#endif

namespace mcbte {

// Last event of a tail round that begins after event e and covers `span`
// events: never past the run's last one, so that it lies beyond e (the round
// makes progress) until e + 1 = max_events ends the particle.  e + span alone
// wraps within `span` of 2^32.
MCBTE_RULE uint32_t round_end(uint32_t e, uint32_t span, uint32_t max_events) {
  const uint32_t left = max_events - 1u - e;
  return e + (span < left ? span : left);
}

}  // namespace mcbte
