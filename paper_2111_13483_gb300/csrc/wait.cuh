// Bounded device-side waits shared by the sweeps: the handle's error word block, the clock, and the
// words in which one CTA hands results to another.
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

// A hand-over word has 64 bits, the low half first.  Of a vector access only each element is a
// single access: with 32-bit elements a reader could meet a word of which one half is written.
// So the elements are the words.
__device__ __forceinline__ uint2 word_halves(unsigned long long w) { return make_uint2((unsigned)w, (unsigned)(w >> 32)); }
__device__ __forceinline__ unsigned long long word_of(unsigned lo, unsigned hi)
{
    return (unsigned long long)hi << 32 | lo;
}
__device__ __forceinline__ uint2 ld_word(const void *p)
{
    unsigned long long a;
    asm volatile("ld.volatile.global.u64 %0, [%1];" : "=l"(a) : "l"(p));
    return word_halves(a);
}
__device__ __forceinline__ uint4 ld_words2(const void *p)   // two words, p on 16 bytes
{
    unsigned long long a, b;
    asm volatile("ld.volatile.global.v2.u64 {%0, %1}, [%2];" : "=l"(a), "=l"(b) : "l"(p));
    const uint2 u = word_halves(a), v = word_halves(b);
    return make_uint4(u.x, u.y, v.x, v.y);
}
__device__ __forceinline__ void st_word(void *p, uint2 v)
{
    asm volatile("st.volatile.global.u64 [%0], %1;" ::"l"(p), "l"(word_of(v.x, v.y)) : "memory");
}
__device__ __forceinline__ void st_words2(void *p, uint4 v)
{
    asm volatile("st.volatile.global.v2.u64 [%0], {%1, %2};" ::"l"(p), "l"(word_of(v.x, v.y)), "l"(word_of(v.z, v.w))
                 : "memory");
}

}  // namespace hm
