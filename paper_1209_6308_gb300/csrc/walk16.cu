// walk16.cu - the triangle walk of large single graphs whose walked prefixes are long (triangles.cu
// describes the walk and its general kernel), in three launches over the plan's items, which
// ascend by vertex b and so descend by degree:
//   k_walk16     b < kTableFrom: the prefixes from the 16-bit lower lists (GraphDev::blk16) against a
//                byte map of L(b) in shared memory;
//   k_walk_table the other vertices of degree above kHubDeg: the prefixes as stored, against a
//                table of L(b) with one 16-bit slot per id modulo its size;
//   k_walk_warp  the items of smaller vertices and the one-warp vertices, a warp each, against a
//                hash of L(b), without a barrier.
//
// The 16-bit walk: a pair's entries of N[c] below b are prefixes of c's class lists, so within a
// segment (pair, window, class) the triangle's tricode depends only on dir(b, a).  The map answers
// an id with the shift of that class's 8-bit field, and a lane adds 1 << shift for the eight ids of
// a 16-byte block with no test, branch or atomic per entry.  A CTA takes one item at a time, a
// thread per pair (and window): each computes its segments from the pair tables, a CTA-wide scan
// places them in one flattened range of blocks, and the warps take rounds of 32 blocks of that
// range, so long and short prefixes share the lanes evenly and only the range's end is ragged.
//
// Census of R-MAT scale 20 / 26 (edge factor 16): 2.20 -> 1.60 ms / 391.6 -> 275.1 ms against the walk
// of 32-bit entries alone.  At scale 20 no unit is full under k_walk16 (1.12 ms): the load/store data
// pipe is 74% busy, 57% with shared memory (32 lookups at random ids cost 3.0 wavefronts), the issue slots
// 53%, the L2 15%; per issue 4.2 warps wait for the L2 or DRAM, 3.3 for shared memory, 2.2 at a barrier, of
// eight per scheduler, which registers and shared memory both limit.  A denser map (two bits per
// id: 2.6 wavefronts) and a plain-shift map for window 0 (fewer instructions) each left the time as it
// was: latency at this occupancy more than any pipe.  CTAs of 128 or 512 threads, maps of 2^14 and 2^16 ids and 4 to 6 rounds in
// flight (spills) were slower.
#include <cstring>

#include "graph.cuh"
#include "rows.cuh"
#include "triangles.cuh"

namespace tc {
namespace {

constexpr int kT16 = 256;                       // threads of a CTA = pairs of a batch
constexpr int kW16 = kT16 / 32;
constexpr int kCtas16 = 4;                      // resident CTAs per SM (shared memory, 64 registers)
constexpr int kCtasWarp = 8;                    // of k_walk_warp (scale 20 / 24 / 26 at 6: 1.623 / 48.6 / 279.2 ms, at 8: 1.636 / 48.0 / 277.8)
// rounds of a warp in flight (scale 26, k_walk16 at 2 / 3 / 4: 282 / 279 / 330 ms, 4 spills)
constexpr int kRing = 3, kRingTable = 2;
constexpr uint32_t kWindow = 8192;              // blocks of the flattened range per window
constexpr uint32_t kAccBlocks = 255 / 8;        // blocks an 8-bit field of a lane's counter holds
constexpr uint32_t kTable = 16384;              // slots of the table walk's table of L(b): 16-bit entries
constexpr uint32_t kTableMaxN = (1u << 28) - kTable;   // ids whose tag (id / kTable) fits 14 bits, all ones unused
constexpr uint32_t kSpill = 512;                // slots of the exact hash of entries whose table slot is shared
constexpr uint32_t kStage = 2048;               // entries of L(b) staged per pass of the table walk
constexpr uint32_t kWarpSlots16 = 2 * kHubDeg;  // slots of a k_walk_warp hash

// The flattened range of a batch and the counters, common to both CTA kernels.
struct Flat {
    uint32_t acc[kW16][9][32];                  // a lane's counts per (class, dir(b, c)), 8 bits per dir_ba
    uint2 seg[3 * kT16];                        // (first block - its place in the range, index of acc | rotation << 8)
    uint32_t start[kWindow / 32];               // bit per block of the window that starts a segment
    uint16_t at[kWindow / 32];                  // the segment of each 32nd block of the window
    uint32_t hist[kW16][64];                    // the warps' tricodes
    uint8_t lanes[kW16][32];                    // walk_pairs' scratch
    uint32_t nblk[kW16], nseg[kW16];
    Item item;                                  // the next item and its vertex's list: offset, table index,
    uint64_t base, table;                       // lower entries
    uint32_t lower, next;
};

struct Shared16 {
    uint8_t map[kWin16 + 16];                   // per id mod kWin16: see k_walk16; kPad16 is always a miss
    Flat f;
};

struct SharedTable {
    uint16_t tab[kTable];
    Flat f;
    uint32_t spill[kSpill], spilled;
};

// ------------------------------------------------------------------ the 16-bit lists
// Entries of a list L of h below id `limit` (L ascends).
__device__ __forceinline__ uint32_t entries_below(const uint32_t* __restrict__ L, uint32_t h, uint32_t limit) {
    uint32_t lo = 0;
    while (lo < h) {
        const uint32_t mid = (lo + h) >> 1;
        if ((L[mid] >> 2) < limit) lo = mid + 1;
        else h = mid;
    }
    return lo;
}

// Entries of x's 16-bit lower list, and a bound on its blocks: 12 segments of h entries in all take
// at most min(h, (h + 84) / 8) blocks.
__global__ void k_count16(const uint64_t* __restrict__ off, const uint32_t* __restrict__ adj,
                          const uint32_t* __restrict__ up, uint32_t n, uint32_t* n16, uint32_t* blocks) {
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < n; x += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t h = x > kIds16 ? entries_below(adj + off[x], up[x], kIds16) : up[x];
        const uint32_t segs = x > kWin16 ? 12u : 3u;
        n16[x] = h;
        blocks[x] = min(h, (h + 7u * segs) / 8u);
    }
}

// The 16-bit lower lists of the vertices that have entries in them (only those are ever a walked
// pair's c).  The n_wide vertices of more than 32 neighbours go a warp each, in two passes per window,
// one that counts the classes and one (from the caches) that places each entry behind the earlier
// ones of its class; for the others a warp takes 32 vertices (rows.cuh) whose lists share its lanes,
// an entry's place counted by one ballot per segment (one with entries past the windows goes alone).
__global__ void __launch_bounds__(256) k_lists16(GraphDev g, uint32_t n, uint32_t n_wide, const uint32_t* __restrict__ n16,
                                                 const uint32_t* __restrict__ first, uint4* rec, uint4* rec2, uint16_t* ids) {
    __shared__ uint8_t s_at[8][32];
    const uint32_t lane = threadIdx.x & 31, lt = (1u << lane) - 1u;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    // classes 1 and 2 of the upper entries of x: the first one, and those after it from its pair's table
    auto upper = [&](uint64_t x, uint64_t base, uint32_t low, uint32_t deg) {
        if (low >= deg) return make_uint2(0u, 0u);
        const uint2 after = g.us[g.ub[x]];
        const uint32_t d = g.adj[base + low] & 3u;
        return make_uint2(after.x + (d == 1u), after.y + (d == 2u));
    };
    // one list by the whole warp
    auto long_list = [&](uint64_t x, uint64_t base, uint32_t h, uint32_t f, uint32_t low, uint32_t v1, uint32_t v2) {
        const uint32_t* __restrict__ L = g.adj + base;
        uint16_t* lens = reinterpret_cast<uint16_t*>(rec2 + 2 * x);
        // classes 1 and 2 of all of N[x]: the lower entries past the lists here, those of the lists below
        uint32_t t1 = 0, t2 = 0;
        for (uint32_t k = h + lane; k < low; k += 32) {
            const uint32_t e = L[k];
            t1 += (e & 3u) == 1u;
            t2 += (e & 3u) == 2u;
        }
        t1 = __reduce_add_sync(0xffffffffu, t1) + v1;
        t2 = __reduce_add_sync(0xffffffffu, t2) + v2;
        uint64_t at = 8ull * f;
        uint32_t k1 = 0;
        for (uint32_t w = 0; w < 4u; ++w) {
            const uint32_t k0 = k1;
            k1 = x <= kWin16 ? h : k0 < h ? entries_below(L, h, (w + 1u) * kWin16) : h;
            uint32_t a1 = 0, a2 = 0;
#pragma unroll 4
            for (uint32_t k = k0 + lane; k < k1; k += 32) {
                const uint32_t e = L[k];
                a1 += (e & 3u) == 1u;
                a2 += (e & 3u) == 2u;
            }
            a1 = __reduce_add_sync(0xffffffffu, a1);
            a2 = __reduce_add_sync(0xffffffffu, a2);
            const uint32_t a3 = k1 - k0 - a1 - a2;
            t1 += a1;
            t2 += a2;
            if (lane == 0) {
                if (w == 0) {
                    rec[x].x = f;
                    rec[x].y = a1 | (a2 << 16);
                    if (x >= kWin16) lens[0] = (uint16_t)a3;
                } else {
                    lens[3 * w - 2] = (uint16_t)a1;
                    lens[3 * w - 1] = (uint16_t)a2;
                    lens[3 * w] = (uint16_t)a3;
                }
            }
            uint64_t p1 = at, p2 = p1 + ((a1 + 7u) & ~7u), p3 = p2 + ((a2 + 7u) & ~7u);
            at = p3 + ((a3 + 7u) & ~7u);
            for (uint32_t kb = k0; kb < k1; kb += 32) {
                const uint32_t k = kb + lane, e = k < k1 ? L[k] : 0u, d = e & 3u;
                const uint32_t b1 = __ballot_sync(0xffffffffu, d == 1u), b2 = __ballot_sync(0xffffffffu, d == 2u);
                const uint32_t b3 = __ballot_sync(0xffffffffu, d == 3u);
                const uint64_t p = d == 1u ? p1 + __popc(b1 & lt)
                                           : d == 2u ? p2 + __popc(b2 & lt) : p3 + __popc(b3 & lt);
                if (d) ids[p] = (uint16_t)((e >> 2) & (kWin16 - 1u));
                p1 += __popc(b1);
                p2 += __popc(b2);
                p3 += __popc(b3);
            }
            if (lane < 7u) {
                if (p1 + lane < ((p1 + 7u) & ~7ull)) ids[p1 + lane] = (uint16_t)kPad16;
                if (p2 + lane < ((p2 + 7u) & ~7ull)) ids[p2 + lane] = (uint16_t)kPad16;
                if (p3 + lane < ((p3 + 7u) & ~7ull)) ids[p3 + lane] = (uint16_t)kPad16;
            }
            if (x < kWin16) break;
            if (k1 == h) {   // nothing in the windows after this one
                if (lane >= 3 * w && lane < 9u) lens[lane + 1u] = 0u;
                break;
            }
        }
        if (lane == 0) {
            rec[x].z = t1;
            rec[x].w = t2;
        }
    };
    for (uint64_t x = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5; x < n_wide; x += stride >> 5) {
        const uint64_t base = g.off[x];
        const uint32_t h = n16[x], low = g.up[x];
        if (!h) continue;
        const uint2 v = upper(x, base, low, (uint32_t)(g.off[x + 1] - base));
        long_list(x, base, h, first[x], low, v.x, v.y);
    }
    for (uint64_t x0 = n_wide + blockIdx.x * (uint64_t)blockDim.x + (threadIdx.x & ~31u); x0 < n; x0 += stride) {
        const bool ok = x0 + lane < n;
        const uint64_t vbase = ok ? g.off[x0 + lane] : 0ull;
        const uint32_t vdeg = ok ? (uint32_t)(g.off[x0 + lane + 1] - vbase) : 0u, vlow = ok ? g.up[x0 + lane] : 0u;
        const uint32_t vh = ok ? n16[x0 + lane] : 0u, vf = ok ? first[x0 + lane] : 0u;
        const uint2 vu = vh ? upper(x0 + lane, vbase, vlow, vdeg) : make_uint2(0u, 0u);
        const uint32_t v1 = vu.x, v2 = vu.y;
        for_rows(vlow != vh ? 33u : vh, s_at[threadIdx.x >> 5],
            [&](const PackedEntry& p) {
                const uint64_t base = __shfl_sync(0xffffffffu, vbase, p.row), x = x0 + p.row;
                const uint32_t f = __shfl_sync(0xffffffffu, vf, p.row);
                uint32_t t1 = __shfl_sync(0xffffffffu, v1, p.row), t2 = __shfl_sync(0xffffffffu, v2, p.row);
                const uint32_t e = p.valid ? g.adj[base + (lane - p.first)] : 0u, d = e & 3u, w = e >> 17;
                const uint32_t last = __reduce_max_sync(0xffffffffu, w);   // windows the pack's entries lie in
                const bool head = p.valid && lane == p.first;
                uint16_t* lens = reinterpret_cast<uint16_t*>(rec2 + 2 * x);   // from window 0's class 3 on
                uint32_t blocks = 0, at = 0, cls1 = 0;   // of the row's segments so far; this entry's place
                uint32_t pads = 0;
                for (uint32_t v = 0; v <= last; ++v)
#pragma unroll
                    for (uint32_t q = 1; q <= 3; ++q) {
                        const uint32_t m = __ballot_sync(0xffffffffu, d == q && w == v) & p.lanes, cnt = __popc(m);
                        if (d == q && w == v) {
                            at = 8u * blocks + __popc(m & lt);
                            pads = (m & lt) ? 0u : (0u - cnt) & 7u;   // the segment's first entry pads it
                            if (pads) pads |= (8u * blocks + cnt) << 8;
                        }
                        blocks += (cnt + 7u) >> 3;
                        t1 += q == 1u ? cnt : 0u;
                        t2 += q == 2u ? cnt : 0u;
                        if (head) {
                            if (v == 0u && q == 1u) cls1 = cnt;
                            else if (v == 0u && q == 2u) rec[x] = make_uint4(f, cls1 | (cnt << 16), 0u, 0u);
                            else if (x >= kWin16) lens[v == 0u ? 0u : 3u * v - 3u + q] = (uint16_t)cnt;
                        }
                    }
                if (p.valid) {
                    ids[8ull * f + at] = (uint16_t)((e >> 2) & (kWin16 - 1u));
                    for (uint32_t k = 0; k < (pads & 255u); ++k) ids[8ull * f + (pads >> 8) + k] = (uint16_t)kPad16;
                }
                if (head) {
                    if (x >= kWin16)
                        for (uint32_t k = 3u * last + 1u; k < 10u; ++k) lens[k] = 0u;
                    rec[x].z = t1;
                    rec[x].w = t2;
                }
            },
            [&](uint32_t row) {
                long_list(x0 + row, __shfl_sync(0xffffffffu, vbase, row), __shfl_sync(0xffffffffu, vh, row),
                          __shfl_sync(0xffffffffu, vf, row), __shfl_sync(0xffffffffu, vlow, row),
                          __shfl_sync(0xffffffffu, v1, row), __shfl_sync(0xffffffffu, v2, row));
            });
    }
}

// ------------------------------------------------------------------ the walks
// Eight ids against the map: the two bits of the segment's window, rotated to bits 3-4, are the
// shift of the id's 8-bit field (dir(b, a) - 1; misses run off the top).
__device__ __forceinline__ uint32_t block_sum(const uint8_t* __restrict__ map, uint4 x, uint32_t rot) {
    auto one = [&](uint32_t id) {
        const uint32_t v = map[id];
        return 1u << (__funnelshift_r(v, v, rot) & 24u);
    };
    return one(x.x & 0xffffu) + one(x.x >> 16) + one(x.y & 0xffffu) + one(x.y >> 16) + one(x.z & 0xffffu) +
           one(x.z >> 16) + one(x.w & 0xffffu) + one(x.w >> 16);
}

// Add a warp's lane counters to its tricode bins and clear them.
__device__ __forceinline__ void flush_acc(Flat& S, int warp, int lane) {
    __syncwarp();
#pragma unroll
    for (int i = 0; i < 9; ++i) {
        const uint32_t v = S.acc[warp][i][lane];
        S.acc[warp][i][lane] = 0u;
        const uint32_t s13 = __reduce_add_sync(0xffffffffu, v & 0x00ff00ffu);   // 32 x 255 fits 16 bits
        const uint32_t s2 = __reduce_add_sync(0xffffffffu, (v >> 8) & 255u);
        const int q = i / 3, r = i % 3;         // class of a in N[c], dir(b, c) - 1
        const uint32_t t = ((uint32_t)(r + 1) << 2) | (q == 0 ? 32u : q == 1 ? 16u : 48u);
        if (lane < 3) S.hist[warp][t + 1u + lane] += lane == 0 ? s13 & 0xffffu : lane == 1 ? s2 : s13 >> 16;
    }
    __syncwarp();
}


// What both CTA kernels do around an item's walk.
struct Runner {
    const TriParams& P;
    Flat& F;
    const int tid, warp, lane;
    uint32_t rounds = 0, walked = 0;   // of this warp: since the counters / the bins were flushed
    Item ahead1, ahead2;               // thread 0 runs ahead: the next item, the one after it,
    uint32_t ahead3;                   // and the index of a third, so no item waits for that chain
    uint64_t nbase = 0, ntable = 0;
    uint32_t nlower = 0;
    static constexpr uint32_t kNone = 0xffffffffu;

    __device__ Runner(const TriParams& p, Flat& f)
        : P(p), F(f), tid(threadIdx.x), warp(threadIdx.x >> 5), lane(threadIdx.x & 31) {
        for (uint32_t k = tid; k < kW16 * 9 * 32; k += kT16) (&F.acc[0][0][0])[k] = 0u;
        for (uint32_t k = tid; k < kW16 * 64; k += kT16) (&F.hist[0][0])[k] = 0u;
        for (uint32_t k = tid; k < kWindow / 32; k += kT16) F.start[k] = 0u;
        ahead1 = ahead2 = Item{kNone, 0u, 0u, 0u};
        ahead3 = P.n_items;
        if (tid == 0) {
            ahead1 = take(atomicAdd(P.ctr, 1u));
            look();
            publish();
            ahead1 = take(atomicAdd(P.ctr, 1u));
            ahead3 = atomicAdd(P.ctr, 1u);
        }
    }
    __device__ Item take(uint32_t i) const { return i < P.n_items ? P.items[i] : Item{kNone, 0u, 0u, 0u}; }
    __device__ void look() {   // thread 0: the list of ahead1's vertex
        if (ahead1.u == kNone) return;
        nbase = P.g.off[ahead1.u];
        nlower = P.g.up[ahead1.u];
        ntable = P.g.ub[ahead1.u];
    }
    __device__ void publish() {   // thread 0
        F.item = ahead1;
        F.base = nbase;
        F.lower = nlower;
        F.table = ntable - nlower;
    }
    __device__ void run_ahead() {
        if (tid) return;
        look();
        ahead2 = take(ahead3);
        ahead3 = ahead3 < P.n_items ? atomicAdd(P.ctr, 1u) : P.n_items;
    }
    __device__ void next_item(bool had_barrier) {   // a barrier must follow the item's reads
        if (!had_barrier) __syncthreads();
        if (tid) return;
        publish();
        ahead1 = ahead2;
    }
    __device__ void flush_all() {
        flush_acc(F, warp, lane);
        rounds = 0;
        flush_warp_hist(F.hist[warp], P.hist, lane);
        walked = 0;
    }
    // Exclusive scan over the CTA of m (a thread's blocks) and n (its warp's segments): the place of
    // the thread's first block and of its warp's first segment in the batch, and the total blocks.
    __device__ uint32_t scan(uint32_t m, uint32_t n, uint32_t& first, uint32_t& seg) {
        uint32_t incl = m;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        if (lane == 31) {
            F.nblk[warp] = incl;
            F.nseg[warp] = n;
        }
        __syncthreads();
        uint32_t total = 0;
        first = incl - m;
        seg = 0;
#pragma unroll
        for (int k = 0; k < kW16; ++k) {
            const uint32_t y = F.nblk[k];
            if (k < warp) {
                first += y;
                seg += F.nseg[k];
            }
            total += y;
        }
        if (total == 0u) __syncthreads();   // the sums are read before the next batch writes its own
        return total;
    }
    // Segment g = [s, e) of the range in the window [w0, w0 + wn): its start bit, and the 32nd blocks
    // it holds.
    __device__ void mark(uint32_t s, uint32_t e, uint32_t g, uint32_t w0, uint32_t wn) {
        if (e <= w0 || s >= w0 + wn || s == e) return;
        if (s >= w0) atomicOr(&F.start[(s - w0) >> 5], 1u << ((s - w0) & 31u));
        for (uint32_t k = s > w0 ? (s - w0 + 31u) >> 5 : 0u; 32u * k < wn && w0 + 32u * k < e; ++k) F.at[k] = (uint16_t)g;
    }
    // The segment of this lane's block in round k of the window: the last one to start at or before it.
    __device__ uint32_t segment(uint32_t k) const {
        return F.at[k] + __popc(F.start[k] & ((2u << lane) - 1u) & ~1u);
    }
    // Walk the window's rounds: a warp takes every kW16-th, `ring` of them in flight (fetch(k, i)
    // starts round k into ring place i, use(i) counts it).
    template <int RING, typename Fetch, typename Use>
    __device__ void walk(uint32_t wn, uint32_t entries, Fetch fetch, Use use) {
        const uint32_t n_rounds = (wn + 31u) >> 5;
#pragma unroll
        for (int i = 0; i < RING; ++i) fetch(warp + i * kW16, i);
        for (uint32_t k = warp; k < n_rounds; k += RING * kW16) {
            if (rounds + RING > kAccBlocks) {
                flush_acc(F, warp, lane);
                rounds = 0;
            }
            rounds += RING;
            walked += entries * RING;
#pragma unroll
            for (int i = 0; i < RING; ++i) {
                use(i);
                fetch(k + (RING + i) * kW16, i);
            }
        }
        if (walked >= kFlushElems) flush_all();
        __syncthreads();
        for (uint32_t k = tid; k < n_rounds; k += kT16) F.start[k] = 0u;
    }
    // The general walk of an item's pairs [j0, j1): L(b)[c0, c1) in a hash, at most `room` bytes of it
    // per pass, in the place of a table whose idle state is all ones.
    __device__ void hash_walk(void* at, uint32_t room, uint64_t bbase, uint64_t pb, uint32_t j0, uint32_t j1, uint32_t c0,
                              uint32_t c1) {
        uint32_t dirty = 0;
        uint32_t* sH = static_cast<uint32_t*>(at);
        const uint32_t chunk = min(P.chunk, room / 8u);   // two slots per entry
        for (; c0 < c1; c0 += chunk) {
            const uint32_t LA = min(chunk, c1 - c0);
            int hb = 6;
            while ((1u << hb) < 2u * LA) ++hb;
            const uint32_t H = 1u << hb, hmask = H - 1u;
            dirty = max(dirty, H);
            __syncthreads();
            for (uint32_t k = tid; k < H; k += kT16) sH[k] = 0u;
            if (tid == 0) F.next = j0;
            __syncthreads();
            for (uint32_t k = tid; k < LA; k += kT16) {
                const uint32_t e = P.g.adj[bbase + c0 + k];
                uint32_t h = tri_hash(e >> 2, hb);
                while (atomicCAS(&sH[h], 0u, e) != 0u) h = (h + 1u) & hmask;
            }
            __syncthreads();
            for (;;) {
                uint32_t jb, g;
                grab_pairs(&F.next, j1, lane, jb, g);
                if (jb >= j1) break;
                walked += walk_pairs<false, false, true>(P, P.g, bbase, pb, jb, min(jb + g, j1), sH, nullptr, hb,
                                                               hmask, 0u, nullptr, F.hist[warp], F.lanes[warp], lane);
                if (walked >= kFlushElems) flush_all();
            }
        }
        if (!dirty) return;
        __syncthreads();
        for (uint32_t k = tid; k < dirty; k += kT16) sH[k] = ~0u;
    }
};

// Which of tc_census_profile's times this launch writes.
struct Stamps {
    uint32_t start, items;
};

// The map's byte holds, for each of the four windows, two bits of the id there: dir(b, a) - 1, or 3
// for an id that is not in L(b).  All of L(b) is in the lists' id range:
static_assert(kTableFrom <= kIds16, "k_walk16's vertices have their lower neighbours in the 16-bit lists");
__global__ void __launch_bounds__(kT16, kCtas16) k_walk16(TriParams P, Stamps T) {
    extern __shared__ __align__(16) unsigned char smem[];
    Shared16& S = *reinterpret_cast<Shared16*>(smem);
    const GraphDev& G = P.g;
    if (P.phase && T.start) tri_stamp(P, 0, tri_clock_ns());
    Flat& F = S.f;
    Runner R(P, F);
    const int tid = R.tid, warp = R.warp, lane = R.lane;
    const uint32_t lt_mask = (1u << lane) - 1u;
    for (uint32_t k = tid; k < sizeof(S.map) / 4u; k += kT16) reinterpret_cast<uint32_t*>(S.map)[k] = ~0u;
    for (;;) {
        __syncthreads();
        const Item w = F.item;
        if (w.u == Runner::kNone) break;
        const long long t0 = clock64();
        const uint32_t b = w.u;
        const uint64_t bbase = F.base, pb = F.table;   // table index of the pair (b, N[b][j]) is pb + j
        const uint32_t lb = F.lower;
        R.run_ahead();
        for (uint32_t k = tid; k < lb; k += kT16) {
            const uint32_t e = G.adj[bbase + k], a = (e >> 2) & (kWin16 - 1u);
            // 3 -> dir - 1 in the two bits of the id's window
            const uint32_t clear = (4u - (e & 3u)) << (8u * (a & 3u) + 2u * (e >> 17));
            atomicAnd(reinterpret_cast<uint32_t*>(S.map) + (a >> 2), ~clear);
        }
        // threads per pair: one for each window of 16-bit ids below b (1, 2 or 4)
        const uint32_t wb = b >> 15;
        const uint32_t ws = wb == 0u ? 0u : wb == 1u ? 1u : 2u;
        for (uint32_t jb = w.j0; lb && jb < w.j1; jb += kT16 >> ws) {
            // this thread's segments (its pair's in its window): their lengths and first blocks
            const uint32_t j = jb + (tid >> ws), win = tid & ((1u << ws) - 1u);
            uint32_t m1 = 0, m2 = 0, m3 = 0, f1 = 0, f2 = 0, f3 = 0, tag = 0;
            if (j < w.j1 && win <= wb) {
                const uint32_t e = __ldg(G.adj + bbase + j), c = e >> 2, r = e & 3u;
                const uint4 rec = __ldg(G.rec + c);
                uint32_t l1 = rec.y & 0xffffu, l2 = rec.y >> 16, l3 = 0, p1 = 0, p2 = 0, p3 = 0;
                f1 = rec.x;
                if (ws) {
                    const uint4 x = __ldg(G.rec2 + 2ull * c), y = __ldg(G.rec2 + 2ull * c + 1ull);
                    l3 = x.x & 0xffffu;
                    // over the windows before this one: blocks (f1) and lengths per class (p1..p3)
#pragma unroll
                    for (uint32_t v = 1; v < 4; ++v)
                        if (v <= win) {
                            f1 += ((l1 + 7u) >> 3) + ((l2 + 7u) >> 3) + ((l3 + 7u) >> 3);
                            p1 += l1;
                            p2 += l2;
                            p3 += l3;
                            l1 = v == 1 ? x.x >> 16 : v == 2 ? x.z & 0xffffu : x.w >> 16;
                            l2 = v == 1 ? x.y & 0xffffu : v == 2 ? x.z >> 16 : y.x & 0xffffu;
                            l3 = v == 1 ? x.y >> 16 : v == 2 ? x.w & 0xffffu : y.x >> 16;
                        }
                }
                m1 = l1;
                m2 = l2;
                m3 = l3;
                if (win == wb) {
                    // b's own window: the class's entries of N[c], less those after b and b itself (whose
                    // class seen from c mirrors r) and those of the windows before
                    const uint2 vs = __ldg(G.vs + pb + j);
                    const uint32_t q1 = rec.z - vs.x - (r == 2u), q2 = rec.w - vs.y - (r == 1u);
                    m1 = q1 - p1;
                    m2 = q2 - p2;
                    m3 = __ldg(G.rp + pb + j) - q1 - q2 - p3;
                }
                m1 = (m1 + 7u) >> 3;
                m2 = (m2 + 7u) >> 3;
                m3 = (m3 + 7u) >> 3;
                f2 = f1 + ((l1 + 7u) >> 3);
                f3 = f2 + ((l2 + 7u) >> 3);
                tag = (r - 1u) | (((2u * win + 29u) & 31u) << 8);
            }
            const uint32_t z1 = __ballot_sync(0xffffffffu, m1 != 0u), z2 = __ballot_sync(0xffffffffu, m2 != 0u);
            const uint32_t z3 = __ballot_sync(0xffffffffu, m3 != 0u);
            const uint32_t m = m1 + m2 + m3;
            uint32_t s1, seg;
            const uint32_t total = R.scan(m, __popc(z1) + __popc(z2) + __popc(z3), s1, seg);
            const uint32_t s2 = s1 + m1, s3 = s2 + m2, s4 = s3 + m3;
            const uint32_t g1 = seg + __popc(z1 & lt_mask) + __popc(z2 & lt_mask) + __popc(z3 & lt_mask);
            const uint32_t g2 = g1 + (m1 != 0u), g3 = g2 + (m2 != 0u);
            if (m1) F.seg[g1] = make_uint2(f1 - s1, tag);
            if (m2) F.seg[g2] = make_uint2(f2 - s2, tag + 3u);
            if (m3) F.seg[g3] = make_uint2(f3 - s3, tag + 6u);
            for (uint32_t w0 = 0; w0 < total; w0 += kWindow) {
                const uint32_t wn = min(kWindow, total - w0);
                if (w0) __syncthreads();
                R.mark(s1, s2, g1, w0, wn);
                R.mark(s2, s3, g2, w0, wn);
                R.mark(s3, s4, g3, w0, wn);
                __syncthreads();
                uint4 x[kRing];
                uint32_t ai[kRing];   // index of acc | rotation << 8, or none
                R.walk<kRing>(wn, 256u,
                    [&](uint32_t k, int i) {
                        const uint32_t at = 32u * k + lane;
                        ai[i] = ~0u;
                        if (at < wn) {
                            const uint2 sg = F.seg[R.segment(k)];
                            ai[i] = sg.y;
                            x[i] = __ldg(G.blk16 + (sg.x + w0 + at));
                        }
                    },
                    [&](int i) {
                        if (ai[i] != ~0u) F.acc[warp][ai[i] & 255u][lane] += block_sum(S.map, x[i], ai[i] >> 8);
                    });
            }
        }
        for (uint32_t k = tid; k < lb; k += kT16) S.map[(G.adj[bbase + k] >> 2) & (kWin16 - 1u)] = 0xffu;
        if (P.vcost && tid == 0) atomicAdd(&P.vcost[b], (unsigned long long)(clock64() - t0));
        R.next_item(lb != 0u);
    }
    R.flush_all();
    if (P.phase && T.items) tri_stamp(P, 1, tri_clock_ns());
}

// The table walk: the pairs' whole prefixes as stored, 32-bit entries in aligned blocks of four,
// against a table of L(b) with one 16-bit entry (tag << 2 | dir) per slot a mod kTable: one lookup
// and one subtraction answer an id, no probing.  Entries of L(b) that share a slot go to a small
// exact hash (the slot then reads 0); should that overflow, the general walk does the pass.
__global__ void __launch_bounds__(kT16, kCtas16) k_walk_table(TriParams P, Stamps T) {
    extern __shared__ __align__(16) unsigned char smem[];
    SharedTable& S = *reinterpret_cast<SharedTable*>(smem);
    const GraphDev& G = P.g;
    if (P.phase && T.start) tri_stamp(P, 0, tri_clock_ns());
    Flat& F = S.f;
    Runner R(P, F);
    const int tid = R.tid, warp = R.warp, lane = R.lane;
    const uint32_t lt_mask = (1u << lane) - 1u;
    uint4* seg = reinterpret_cast<uint4*>(F.seg);   // (first block - place, place, lead entries, length | dir(b, c) << 30)
    for (uint32_t k = tid; k < kTable / 2u; k += kT16) reinterpret_cast<uint32_t*>(S.tab)[k] = ~0u;
    auto slot = [&](uint32_t e) { return reinterpret_cast<unsigned short*>(&S.tab[(e >> 2) & (kTable - 1u)]); };
    auto spill = [&](uint32_t e) {
        if (atomicAdd(&S.spilled, 1u) >= kSpill / 2u) return;
        uint32_t h = tri_hash(e >> 2, 9);
        while (atomicCAS(&S.spill[h], 0u, e) != 0u) h = (h + 1u) & (kSpill - 1u);
    };
    for (;;) {
        __syncthreads();
        const Item w = F.item;
        if (w.u == Runner::kNone) break;
        const long long t0 = clock64();
        const uint32_t b = w.u;
        const uint64_t bbase = F.base, pb = F.table;
        const uint32_t lb = F.lower;
        R.run_ahead();
        for (uint32_t c0 = 0; c0 < lb; c0 += kStage) {
            const uint32_t c1 = min(lb, c0 + kStage);
            for (uint32_t k = tid; k < kSpill; k += kT16) S.spill[k] = 0u;
            if (tid == 0) S.spilled = 0u;
            __syncthreads();
            for (uint32_t k = c0 + tid; k < c1; k += kT16) {
                const uint32_t e = G.adj[bbase + k];
                const unsigned short v = (unsigned short)((e >> 16) << 2 | (e & 3u));
                if (atomicCAS(slot(e), (unsigned short)0xffffu, v) != 0xffffu) spill(e);
            }
            __syncthreads();
            const bool shared_slots = S.spilled != 0u;
            if (shared_slots) {
                // the first entry of a shared slot joins the others in the hash
                uint32_t mine[kSpill / kT16];
#pragma unroll
                for (int i = 0; i < (int)(kSpill / kT16); ++i) mine[i] = S.spill[tid + i * kT16];
                __syncthreads();
#pragma unroll
                for (int i = 0; i < (int)(kSpill / kT16); ++i)
                    if (mine[i]) {
                        const unsigned short t = *(volatile unsigned short*)slot(mine[i]);
                        if (t && atomicCAS(slot(mine[i]), t, (unsigned short)0u) == t)
                            spill(((uint32_t)(t >> 2) << 16) | (mine[i] & (4u * kTable - 4u)) | (t & 3u));
                    }
                __syncthreads();
            }
            const bool fits = S.spilled <= kSpill / 2u;
            for (uint32_t jb = w.j0; fits && jb < w.j1; jb += kT16) {
                const uint32_t j = jb + tid;
                uint32_t m = 0, len = 0, lead = 0, r = 0;
                uint64_t first = 0;
                if (j < w.j1) {
                    const uint32_t e = __ldg(G.adj + bbase + j);
                    r = e & 3u;
                    first = __ldg(G.off + (e >> 2));
                    len = __ldg(G.rp + pb + j);
                    lead = (uint32_t)first & 3u;
                    m = len ? (lead + len + 3u) >> 2 : 0u;
                }
                const uint32_t z = __ballot_sync(0xffffffffu, m != 0u);
                uint32_t s0, g;
                const uint32_t total = R.scan(m, __popc(z), s0, g);
                g += __popc(z & lt_mask);
                if (m) seg[g] = make_uint4((uint32_t)(first >> 2) - s0, s0, lead, len | (r << 30));
                for (uint32_t w0 = 0; w0 < total; w0 += kWindow) {
                    const uint32_t wn = min(kWindow, total - w0);
                    if (w0) __syncthreads();
                    R.mark(s0, s0 + m, g, w0, wn);
                    __syncthreads();
                    uint4 x[kRingTable];
                    uint32_t valid[kRingTable];   // bit i: entry i is one of the pair's; bits 4-5: dir(b, c)
                    R.walk<kRingTable>(wn, 128u,
                        [&](uint32_t k, int i) {
                            const uint32_t at = 32u * k + lane;
                            valid[i] = 0u;
                            if (at < wn) {
                                const uint4 sg = seg[R.segment(k)];
                                x[i] = __ldg(reinterpret_cast<const uint4*>(G.adj) + (sg.x + w0 + at));
                                // the block's first entry in the pair's prefix, and those left from it on
                                const int p = (int)(4u * (w0 + at - sg.y)) - (int)sg.z;
                                const int left = (int)(sg.w & 0x3fffffffu) - p;
                                valid[i] = ((15u << (p < 0 ? -p : 0)) & (left < 4 ? (1u << left) - 1u : 15u)) | ((sg.w >> 30) << 4);
                            }
                        },
                        [&](int i) {
                            if (!valid[i]) return;
                            uint32_t* acc = &F.acc[warp][(valid[i] >> 4) - 1u][lane];
                            auto count = [&](uint32_t e, bool ok) {
                                const uint32_t t = *slot(e);
                                uint32_t d = t - ((e >> 16) << 2);
                                if (shared_slots && t == 0u) {
                                    uint32_t h = tri_hash(e >> 2, 9), y;
                                    while ((y = S.spill[h]) != 0u && (y >> 2) != (e >> 2)) h = (h + 1u) & (kSpill - 1u);
                                    d = y & 3u;
                                }
                                if (ok && d - 1u < 3u) atomicAdd(acc + 96u * ((e & 3u) - 1u), 1u << (8u * (d - 1u)));
                            };
                            count(x[i].x, valid[i] & 1u);
                            count(x[i].y, valid[i] & 2u);
                            count(x[i].z, valid[i] & 4u);
                            count(x[i].w, valid[i] & 8u);
                        });
                }
            }
            for (uint32_t k = c0 + tid; k < c1; k += kT16) *slot(G.adj[bbase + k]) = 0xffffu;
            if (!fits) R.hash_walk(S.tab, sizeof(S.tab), bbase, pb, w.j0, w.j1, c0, c1);
            __syncthreads();
        }
        if (P.vcost && tid == 0) atomicAdd(&P.vcost[b], (unsigned long long)(clock64() - t0));
        R.next_item(lb != 0u);
    }
    R.flush_all();
    if (P.phase && T.items) tri_stamp(P, 1, tri_clock_ns());
}

// The small vertices' items and the one-warp vertices, a warp each.
__global__ void __launch_bounds__(kT16, kCtasWarp) k_walk_warp(TriParams P, Stamps T) {
    __shared__ uint32_t s_hash[kW16][kWarpSlots16], s_hist[kW16][64];
    __shared__ uint8_t s_at[kW16][32];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const GraphDev& G = P.g;
    if (P.phase && T.start) tri_stamp(P, 0, tri_clock_ns());
    for (int k = lane; k < 64; k += 32) s_hist[warp][k] = 0u;
    __syncwarp();
    uint32_t* wH = s_hash[warp];
    uint32_t walked = 0;
    // the pairs [j0, j1) of b against a hash of L(b)
    auto walk = [&](uint32_t b, uint32_t j0, uint32_t j1) {
        const uint64_t bbase = G.off[b];
        const uint32_t lb = G.up[b];
        if (lb == 0u || j0 >= j1) return;   // no triangle has b in the middle
        int hb = 6;
        while ((1u << hb) < 2u * lb) ++hb;
        const uint32_t hmask = (1u << hb) - 1u;
        __syncwarp();
        for (uint32_t k = lane; k < (1u << hb); k += 32) wH[k] = 0u;
        __syncwarp();
        for (uint32_t k = lane; k < lb; k += 32) {
            const uint32_t e = G.adj[bbase + k];
            uint32_t h = tri_hash(e >> 2, hb);
            while (atomicCAS(&wH[h], 0u, e) != 0u) h = (h + 1u) & hmask;
        }
        __syncwarp();
        walked += walk_pairs<false, false, false>(P, G, bbase, G.ub[b] - lb, j0, j1, wH, nullptr, hb, hmask, 0u, nullptr,
                                                 s_hist[warp], s_at[warp], lane);
        if (walked >= kFlushElems) {
            flush_warp_hist(s_hist[warp], P.hist, lane);
            walked = 0;
        }
    };
    for (;;) {
        uint32_t it = 0;
        if (lane == 0) it = atomicAdd(P.ctr, 1u);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= P.n_items) break;
        const Item w = P.items[it];
        const long long t0 = clock64();
        walk(w.u, w.j0, w.j1);
        // a CTA's cycles, as the other kernels count them
        if (P.vcost && lane == 0) atomicAdd(&P.vcost[w.u], (unsigned long long)(clock64() - t0) / kW16 + 1ull);
    }
    if (P.phase && T.items) {
        __syncthreads();
        tri_stamp(P, 1, tri_clock_ns());
    }
    for (;;) {
        uint32_t vb = 0;
        if (lane == 0) vb = atomicAdd(P.ctr + 1, 1u << P.wshift);
        vb = __shfl_sync(0xffffffffu, vb, 0);
        if (vb >= P.warp_end - P.warp_begin) break;
        const uint32_t b0 = P.warp_begin + vb, b1 = min(b0 + (1u << P.wshift), P.warp_end);
        walked += walk_rows(P, G, b0, b1, wH, s_hist[warp], s_at[warp], lane);
        if (walked >= kFlushElems) {
            flush_warp_hist(s_hist[warp], P.hist, lane);
            walked = 0;
        }
    }
    flush_warp_hist(s_hist[warp], P.hist, lane);
    if (P.phase) {
        __syncthreads();
        tri_stamp(P, 2, tri_clock_ns());
    }
}

}  // namespace

// Against the general kernel (triangles.cu), a graph's first census, which makes the lists, and a later
// one, in ms, this / that.  Taken: R-MAT 19 edge factor 16 (500 M entries walked, 65 per pair) 1.18 /
// 1.39, later 0.80 / 1.16; R-MAT 20 e.f. 16 (1.2 G, 78) 2.29 / 2.54, 1.62 / 2.22; R-MAT 24 e.f. 16
// (42 G, 160) 56.5 / 73.4, 47.5 / 70.1; G(2400, 0.5) (1.3 G, 594) 1.11 / 1.45, 0.87 / 1.31.  Not taken,
// as the first census would lose (this side with k_lists16 on fewer warps than long lists, so G(1600, 0.5)
// may have come to gain since): R-MAT 22 e.f. 8 (2.0 G, 60) 4.94 / 4.80, 3.34 / 4.28; R-MAT 18 e.f. 16
// (204 M, 54) 0.84 / 0.76, 0.53 / 0.57; Chung-Lu 9 M x 16 (3.8 G, 31) 17.4 / 13.4, 10.5 / 12.0; G(1600,
// 0.5) (378 M, 394) 0.71 / 0.62, 0.33 / 0.48.
bool walk16_takes(const GraphStore& g) {
    return g.n <= kTableMaxN && g.sum_tri_walk >= (7ull << 26) && g.sum_tri_walk >= 64ull * g.e_sym;
}

tc_status lists16_build(GraphStore& g, cudaStream_t st) {
    DevBuf n16, blocks, first, total;
    const uint32_t n = g.n_active;   // the others have no list
    TC_TRY(g.rec.alloc_persistent(3ull * sizeof(uint4) * n));   // rec and rec2
    TC_TRY(n16.alloc(sizeof(uint32_t) * n, st));
    TC_TRY(blocks.alloc(sizeof(uint32_t) * n, st));
    TC_TRY(first.alloc(sizeof(uint32_t) * n, st));
    const GraphDev gd = g.dev();
    TC_TRY(total.alloc(sizeof(uint32_t), st));
    k_count16<<<grid_for(n, 256, 1u << 16), 256, 0, st>>>(gd.off, gd.adj, gd.up, n, n16.as<uint32_t>(),
                                                          blocks.as<uint32_t>());
    TC_LAUNCH("k_count16");
    TC_TRY(scan_u32(blocks.as<uint32_t>(), first.as<uint32_t>(), n, total.as<uint32_t>(), st));
    uint32_t n_blocks = 0;
    TC_CUDA(cudaMemcpyAsync(&n_blocks, total.p, sizeof(n_blocks), cudaMemcpyDeviceToHost, st));
    TC_CUDA(cudaStreamSynchronize(st));
    DevBuf blk;
    TC_TRY(blk.alloc_persistent(sizeof(uint4) * (n_blocks ? n_blocks : 1u)));
    k_lists16<<<grid_lists(n, g.n_wide), 256, 0, st>>>(gd, n, g.n_wide, n16.as<uint32_t>(), first.as<uint32_t>(), g.rec.as<uint4>(),
                                                          g.rec.as<uint4>() + n, blk.as<uint16_t>());
    TC_LAUNCH("k_lists16");
    TC_CUDA(cudaStreamSynchronize(st));   // later censuses may come on other streams
    std::swap(g.blk16.p, blk.p);          // held only once the lists are made: a failed call starts afresh
    std::swap(g.blk16.bytes, blk.bytes);
    std::swap(g.blk16.st, blk.st);
    std::swap(g.blk16.async, blk.async);
    return TC_OK;
}

tc_status walk16_launch(const TriParams& P0, const uint32_t split[2], uint32_t grid, uint32_t* ctr, cudaStream_t st) {
    const unsigned sms = (unsigned)sm_count();
    const unsigned ctas = grid < sms * kCtas16 ? grid : sms * kCtas16;
    const uint32_t s1 = split[0], s2 = split[1];
    Stamps T = {1u, s2 == s1};
    TriParams P = P0;
    if (s1) {
        P.ctr = ctr;
        P.n_items = s1;
        TC_CUDA(cudaFuncSetAttribute((const void*)k_walk16, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(Shared16)));
        k_walk16<<<ctas, kT16, sizeof(Shared16), st>>>(P, T);
        TC_LAUNCH("k_walk16");
        T.start = 0u;
    }
    if (s2 > s1) {
        P.ctr = ctr + 1;
        P.items = P0.items + s1;
        P.n_items = s2 - s1;
        T.items = 1u;
        TC_CUDA(cudaFuncSetAttribute((const void*)k_walk_table, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SharedTable)));
        k_walk_table<<<ctas, kT16, sizeof(SharedTable), st>>>(P, T);
        TC_LAUNCH("k_walk_table");
        T.start = 0u;
    }
    P.ctr = ctr + 2;
    P.items = P0.items + s2;
    P.n_items = P0.n_items - s2;
    T.items = s2 == 0u;
    const unsigned wide = grid < sms * kCtasWarp ? grid : sms * kCtasWarp;
    k_walk_warp<<<wide, kT16, 0, st>>>(P, T);
    TC_LAUNCH("k_walk_warp");
    return TC_OK;
}

}  // namespace tc
