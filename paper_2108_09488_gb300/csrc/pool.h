// pool.h -- the arithmetic of the counter that hands out the weight table's pool of lines (frozen_table.cuh).
#pragma once

#ifdef __CUDACC__
#define ADE_POOL_FN __device__ __forceinline__
#else
#define ADE_POOL_FN inline
#endif

namespace ade {

constexpr unsigned kNoRoom = 0xffffffffu;

// First of the `used` lines claimed from a pool of `cap` lines (cap < 2^31), or kNoRoom when fewer are left.
// before: what the counter held when `used` was added to it.  The counter has 64 bits: every demand is
// added, room or no room, and the demands of one call (fewer than 2^24 chunks of fewer than 2^32 lines) cannot wrap
// it, where 32 bits would hand out lines that others hold.  (A compare-and-swap that only moves the
// counter for claims that fit takes its turns one by one: 2,500 claims 1.2 ms.)
ADE_POOL_FN unsigned claim_lines(unsigned long long before, unsigned cap, unsigned used)
{
    return before <= cap && cap - before >= used ? (unsigned)before : kNoRoom;
}

// Lines of a chunk so far and those of one more row, held below 2^32 (a row has fewer than 2^31).
ADE_POOL_FN unsigned add_lines(unsigned used, unsigned row) { return (used < 0x80000000u ? used : 0x80000000u) + row; }

}  // namespace ade
