// rows.cuh - a warp over 32 consecutive rows (vertices) of a structure of lists.  Most lists are
// short, and a warp per list leaves its lanes idle and waits for one list's loads at a time; here
// the warp reads the 32 rows' bounds together, and then takes as many consecutive rows of at most
// 32 entries as fit its lanes at once, or one longer row alone.
#pragma once

#include <stdint.h>

namespace tc {

// A lane's entry in a pack of rows: its row (lane index of the 32), the lane its row starts at and
// the row's lanes; valid if the lane holds an entry.
struct PackedEntry {
    uint32_t row, first, lanes;
    bool valid;
};

// Calls, in order of the rows: pack(PackedEntry) for packs of rows of 1 to 32 entries (entry lane -
// first of row), and one(row) for a row of more.  len: this lane's row's entries (0 past the last
// row).  at: 32 bytes of shared scratch of this warp.  Every lane takes part in every call.
template <typename Pack, typename One>
__device__ __forceinline__ void for_rows(uint32_t len, volatile uint8_t* at, Pack pack, One one) {
    const uint32_t lane = threadIdx.x & 31u;
    const uint32_t small = len <= 32u ? len : 0u;
    uint32_t incl = small;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= (uint32_t)o) incl += y;
    }
    const uint32_t excl = incl - small;
    const uint32_t longs = __ballot_sync(0xffffffffu, len > 32u);
    uint32_t rest = __ballot_sync(0xffffffffu, len != 0u);   // rows still to do
    while (rest) {
        const uint32_t r = __ffs(rest) - 1u;
        if ((longs >> r) & 1u) {
            one(r);
            rest &= rest - 1u;
            continue;
        }
        // the rows from r up to the first long one, as long as they fit 32 lanes
        const uint32_t base = __shfl_sync(0xffffffffu, excl, r);
        const uint32_t over = __ballot_sync(0xffffffffu, lane >= r && (len > 32u || incl - base > 32u));
        const uint32_t end = over ? __ffs(over) - 1u : 32u;
        const uint32_t mine = end == 32u ? 0xffffffffu : (1u << end) - 1u;
        const bool in = lane >= r && lane < end && len != 0u;
        if (in) at[excl - base] = (uint8_t)lane;
        const uint32_t starts = __reduce_or_sync(0xffffffffu, in ? 1u << (excl - base) : 0u);
        __syncwarp();
        PackedEntry p;
        p.first = 31u - __clz(starts & ((2u << lane) - 1u));   // bit 0 is set: row r starts there
        p.row = at[p.first];
        p.lanes = __shfl_sync(0xffffffffu, len, p.row);
        p.valid = lane - p.first < p.lanes;
        const uint32_t ones = p.lanes == 32u ? 0xffffffffu : (1u << p.lanes) - 1u;
        p.lanes = ones << p.first;
        pack(p);
        __syncwarp();
        rest &= ~mine;
    }
}

}  // namespace tc
