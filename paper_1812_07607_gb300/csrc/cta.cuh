// cta.cuh -- counting over a CTA, for the selections that find a k-th value bit by bit.
#pragma once

namespace dl {

// Sum of v over the CTA, the same in every thread. s_cnt: two shared words, zeroed before the first
// call and used in turn (turn counts the calls).
__device__ __forceinline__ unsigned cta_count(unsigned v, unsigned *s_cnt, int turn)
{
    v = __reduce_add_sync(0xffffffffu, v);
    if (threadIdx.x == 0) s_cnt[(turn + 1) & 1] = 0u;
    if ((threadIdx.x & 31) == 0 && v) atomicAdd(&s_cnt[turn & 1], v);
    __syncthreads();
    const unsigned r = s_cnt[turn & 1];
    __syncthreads();
    return r;
}

}  // namespace dl
