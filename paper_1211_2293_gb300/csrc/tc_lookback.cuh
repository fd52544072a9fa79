// tc_lookback.cuh -- decoupled look-back (Merrill & Garland's single-pass
// prefix scan): a tile publishes its own sum, adds up the sums of the tiles
// before it back to the nearest published prefix, and publishes its own
// prefix.  Tiles take their index from an atomic counter in launch order, so
// a tile only ever waits for tiles that have already started and publish
// before they look back themselves.  Every wait is bounded.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

namespace tc {

namespace {

constexpr unsigned long long kFlagAgg = 1ull << 62;
constexpr unsigned long long kFlagPrefix = 2ull << 62;
constexpr unsigned kLookbackMaxPolls = 1u << 22;  // about a second of polling

// One warp: the sum of the tiles before `tile`, whose own sum is agg; 32
// predecessors a round.  st: one word per tile, zero before the launch.
// *ok = false where a wait ran out.
__device__ __forceinline__ uint32_t tile_prefix(volatile unsigned long long* st, int64_t tile, uint32_t agg, bool* ok)
{
    const int lane = threadIdx.x & 31;
    *ok = true;
    uint32_t excl = 0;
    if (tile > 0) {
        if (lane == 0) st[tile] = kFlagAgg | agg;
        unsigned polls = 0;
        for (int64_t k = tile - 1;;) {
            const int64_t j = k - lane;
            unsigned long long v = kFlagPrefix;  // before tile 0: a prefix of zero
            if (j >= 0) v = st[j];
            const unsigned f = (unsigned)(v >> 62);
            if (__any_sync(0xffffffffu, f == 0)) {
                if (++polls > kLookbackMaxPolls) {
                    *ok = false;
                    break;
                }
                if (polls > 64) __nanosleep(32);
                continue;
            }
            const unsigned pm = __ballot_sync(0xffffffffu, f == 2);
            const int last = pm ? __ffs(pm) - 1 : 31;
            excl += __reduce_add_sync(0xffffffffu, lane <= last ? (unsigned)v : 0u);
            if (pm) break;
            k -= 32;
        }
    }
    if (lane == 0) st[tile] = kFlagPrefix | (uint32_t)(excl + agg);
    return excl;
}

}  // namespace

}  // namespace tc
