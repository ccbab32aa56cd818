// svv_team.cuh -- a team of co-resident CTAs that runs one query phase.
//
// A single query uses the whole cooperative grid as one team; the batch kernel
// splits its grid into several teams that each run whole queries.  A team has
// its own barrier state and error flag (`bar`) and reports errors of the
// query it runs in `qerr`.
#pragma once

#include "svv_device.cuh"

namespace svv {

struct Team {
  TeamCtl* bar;
  uint32_t* qerr;
  unsigned nblocks, rank;
  unsigned long long spin_ns;
  TeamBar* tb;  // this CTA's barrier state, in shared memory (thread 0's)
  // start of the kernel: no barrier of this launch has been passed
  __device__ __forceinline__ void begin() const {
    if (threadIdx.x == 0) *tb = TeamBar{{0ull, 0ull}, 0u};
  }
  __device__ __forceinline__ unsigned nthreads() const { return nblocks * blockDim.x; }
  __device__ __forceinline__ unsigned tid() const { return rank * blockDim.x + threadIdx.x; }
  __device__ __forceinline__ bool sync() const {
    uint32_t none;
    return team_sync(bar, qerr, tb, nblocks, spin_ns, 0u, none);
  }
  // the barrier, and the sum over the team's CTAs of `add` (thread 0's)
  __device__ __forceinline__ bool sync(uint32_t add, uint32_t& sum) const {
    return team_sync(bar, qerr, tb, nblocks, spin_ns, add, sum);
  }
};

}  // namespace svv
