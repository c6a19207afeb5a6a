// pool.h -- the counter that hands out the weight table's pool of lines (frozen_table.cuh).
#pragma once

#ifdef __CUDACC__
#define ADE_POOL_FN __device__ __forceinline__
#else
#define ADE_POOL_FN inline
#endif

namespace ade {

constexpr unsigned kNoRoom = 0xffffffffu;

// Takes `used` of the pool's `cap` lines (cap < 2^31) and returns the first, or kNoRoom when fewer are left.
// cur: the counter as last seen; cas(seen, next): its compare-and-swap, returning what it held.  Only
// a claim that fits moves the counter, so it stays at or below cap however many lines are asked for
// in all (a counter that every demand were added to would pass 2^32 on a set that outgrows the table
// far enough, and hand out lines that others hold).
template <class Cas>
ADE_POOL_FN unsigned claim_lines(unsigned cur, unsigned cap, unsigned used, Cas cas)
{
    while (used <= cap && cur <= cap - used) {
        const unsigned seen = cas(cur, cur + used);
        if (seen == cur) return cur;
        cur = seen;
    }
    return kNoRoom;
}

// Lines of a chunk so far and those of one more row, held below 2^32 (a row has fewer than 2^31).
ADE_POOL_FN unsigned add_lines(unsigned used, unsigned row) { return (used < 0x80000000u ? used : 0x80000000u) + row; }

}  // namespace ade
