// Exclusive sums in one pass: a CTA takes the next tile from a ticket counter, publishes
// the tile's sum, and adds up the sums of the tiles before it that are already there until
// it meets one that knows its own prefix (decoupled look-back: D. Merrill and M. Garland,
// "Single-pass parallel prefix scan with decoupled look-back", NVIDIA Technical Report
// NVR-2016-002).  The input is read once, and producers or consumers of the sums can share
// the launch: the passes around a scan are a few microseconds each here, so launches
// count for more than bytes.
//
// State: word 0 is the ticket, word 1 + t tile t's (value << 2 | kind); zeroed before the
// launch.  A tile's ticket orders it after every tile it waits for, and those have begun,
// so the waits end; they are bounded all the same (EMB_ERR_TIMEOUT).
#pragma once

#include "emb_internal.cuh"

#define SCAN_PART 1ull    // the tile's own sum
#define SCAN_PREFIX 2ull  // the sum up to and including the tile
#define SCAN_POLLS (1 << 20)

static inline int64_t scan_state_words(int64_t tiles) { return tiles + 1; }

// The CTA's tile (every thread of the CTA calls; shared memory word `s_tile`).
__device__ __forceinline__ uint32_t scan_ticket(uint64_t *state, uint32_t *s_tile)
{
    if (threadIdx.x == 0) *s_tile = atomicAdd((unsigned int *)state, 1u);
    __syncthreads();
    return *s_tile;
}

// Sum of the tiles before `tile`, whose own sum is `sum`: called by one whole warp.
__device__ __forceinline__ uint64_t scan_lookback(uint64_t *state, uint32_t tile, uint64_t sum, int *st)
{
    volatile uint64_t *w = state + 1;
    const int lane = threadIdx.x & 31;
    if (tile == 0) {
        if (lane == 0) w[0] = sum << 2 | SCAN_PREFIX;
        return 0;
    }
    if (lane == 0) w[tile] = sum << 2 | SCAN_PART;
    uint64_t before = 0;
    int64_t top = (int64_t)tile - 1;  // lane l looks at tile top - l
    for (int polls = 0;; ) {
        const int64_t i = top - lane;
        const uint64_t v = i >= 0 ? w[i] : SCAN_PREFIX;
        const unsigned ready = __ballot_sync(0xffffffffu, (v & 3u) != 0);
        const unsigned pre = __ballot_sync(0xffffffffu, (v & 3u) == SCAN_PREFIX);
        // the lanes up to the nearest prefix (or all of them) are needed
        const int last = pre ? __ffs(pre) - 1 : 31;
        const unsigned need = 0xffffffffu >> (31 - last);
        if ((ready & need) != need) {
            if (++polls > SCAN_POLLS) {
                if (lane == 0) emb_set_status(st, EMB_ERR_TIMEOUT);
                return 0;
            }
            __nanosleep(20);
            continue;
        }
        uint64_t part = lane <= last ? v >> 2 : 0ull;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
        before += part;
        if (pre) break;
        top -= 32;
    }
    if (lane == 0) w[tile] = (before + sum) << 2 | SCAN_PREFIX;
    return before;
}
