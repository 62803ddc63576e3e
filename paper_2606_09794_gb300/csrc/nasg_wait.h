// Time that a bounded wait on the GPU has spent waiting. Plain arithmetic, shared by the kernels
// and a host-side check.
#pragma once

#include <stdint.h>

#if defined(__CUDACC__)
#define NASG_WAIT_HD __host__ __device__ __forceinline__
#else
#define NASG_WAIT_HD inline
#endif

namespace nasg {

// The clock goes on while another process has the GPU (time slicing, a debugger), and then the
// block that is waited for did not run either. So a step between two looks at the clock, some
// 0.2 ms of polling, counts for kStepNs at most.
struct WaitClock {
  static constexpr uint64_t kStepNs = 1000000ull;
  uint64_t last, waited;

  NASG_WAIT_HD explicit WaitClock(uint64_t now) : last(now), waited(0) {}
  // Whether more than `limit` ns have been spent waiting by `now`.
  NASG_WAIT_HD bool over(uint64_t now, uint64_t limit) {
    const uint64_t step = now - last;
    last = now;
    waited += step < kStepNs ? step : kStepNs;
    return waited > limit;
  }
};

}  // namespace nasg
