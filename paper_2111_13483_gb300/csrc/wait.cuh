// Bounded device-side waits shared by the sweeps: the handle's error word block and the clock.
#pragma once
#include "hm_internal.h"

namespace hm {

// err[ERR_CODE] is set by a failing wait, err[ERR_HOLD] names a block row the sweeps leave out (a
// test hook: -1 = none; every wait on that row then runs out), err[ERR_BOUND..+1] holds the bound
// on any single wait in ns (2 s unless a test sets it).
__device__ __forceinline__ unsigned long long wait_bound(const int *err)
{
    return __ldcg((const unsigned long long *)(err + ERR_BOUND));
}
__device__ __forceinline__ bool held_back(const int *err, int blk) { return __ldcg(err + ERR_HOLD) == blk; }

__device__ __forceinline__ unsigned long long gtimer()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

}  // namespace hm
