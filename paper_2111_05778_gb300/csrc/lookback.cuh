// One-pass scans over tiles (decoupled look-back, Merrill and Garland 2016):
// blocks take tiles in order by a ticket, publish a tile's sum in a status
// word, and the block of the next tile adds up its predecessors' words until
// it meets one that already holds the whole sum before it.  A tile waits only
// for tiles taken earlier, whose blocks are running, so every wait ends; it is
// bounded all the same (2 s of %globaltimer, then the timeout flag is set).
// A status word is call number << 34 | state << 32 | value, so words of
// earlier calls read as not written and nothing has to be cleared.
#pragma once

#include <stdint.h>

#include "gh_internal.cuh"

namespace gh {
namespace {

constexpr unsigned long long LB_SUM = 1ull << 32, LB_PREFIX = 2ull << 32;

// The sum of the tiles before `tile`; the first warp of the block calls it.
// expire: give up at once, as if the wait had run out (its caller's test device).
__device__ __forceinline__ uint32_t lb_prefix(unsigned long long *words, unsigned long long call, long long tile,
                                              uint32_t sum, Counters *ctr, bool expire) {
    const int lane = threadIdx.x & 31;
    volatile unsigned long long *w = words;
    const unsigned long long tag = call << 34;
    uint32_t before = 0;
    if (tile > 0 && expire) {
        if (lane == 0) atomicOr(&ctr->flags, FLAG_TIMEOUT);
    } else if (tile > 0) {
        if (lane == 0) w[tile] = tag | LB_SUM | sum;
        for (long long last = tile - 1; last >= 0; last -= 32) {
            const long long t = last - lane;
            unsigned long long v = t >= 0 ? w[t] : tag | LB_PREFIX;  // before the first tile: 0
            unsigned long long t0 = 0;
            while ((v >> 34) != call || (v & (LB_SUM | LB_PREFIX)) == 0ull) {
                unsigned long long now;
                asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(now));
                if (t0 == 0) t0 = now;
                else if (now - t0 > 2000000000ull) {
                    atomicOr(&ctr->flags, FLAG_TIMEOUT);
                    v = tag | LB_PREFIX;
                    break;
                }
                v = w[t];
            }
            __syncwarp();
            const unsigned done = __ballot_sync(0xFFFFFFFFu, (v & LB_PREFIX) != 0ull);
            const int stop = done ? __ffs(done) - 1 : 31;
            uint32_t x = lane <= stop ? (uint32_t)v : 0u;
            for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xFFFFFFFFu, x, o);
            before += x;
            if (done) break;
        }
    }
    if (lane == 0) w[tile] = tag | LB_PREFIX | (uint32_t)(before + sum);
    return before;
}

}  // namespace
}  // namespace gh
