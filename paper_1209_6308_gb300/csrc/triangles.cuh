// triangles.cuh - the parts the triangle walk's kernels share (triangles.cu describes the walk):
// its parameters, the walk of 32-bit entries, and the warps' tricode bins.
#pragma once

#include "graph.cuh"

namespace tc {

struct TriParams {
    GraphDev g;
    const Item* items;
    uint32_t n_items;
    uint32_t warp_begin, warp_end;
    uint32_t wshift;              // warp tier: 2^wshift consecutive vertices per grab
    uint32_t chunk;               // entries of L(b) staged per pass of a CTA item (hash: 2 x chunk slots)
    uint32_t* ctr;                // [0] next item, [1] next warp-tier vertex
    const uint32_t* old;          // OLD: the caller's id of each vertex
    const uint8_t* perm_state;    // OLD: [9][64] state of a tricode under the rank pattern 3 ra + rb
    unsigned long long* hist;     // 64 bins (triangle tricodes, or states with OLD); batched: graph g's at
                                  // hist + kBatchStride g
    unsigned long long* vcost;    // optional [n]: SM cycles per CTA-tier vertex b
    unsigned long long* phase;    // optional [3 * stamps]: globaltimer at start, end of items, end per CTA of
    uint32_t stamps;              // the option's grid; a smaller launch's CTAs fill several entries
    uint32_t marks;               // k_triangles: which of the times this launch writes (bits 0, 1, 2)
    // batched launch: item.pad is the graph index, warp-tier blocks are (u0, u1, graph)
    const GraphDev* graphs;
    const uint4* wblocks;
    uint32_t n_wblocks;
    // serving wave: n_items / n_wblocks are the wave's totals over its request slices
    const WaveReq* reqs;
    uint32_t n_reqs;
};

namespace {

constexpr int kThreads = 256;
constexpr int kWarps = kThreads / 32;
// Prefixes of at least kLongPrefix entries are walked one pair at a time by the whole warp
// (walk_pairs<..., LONGW = true>), kLongRounds loads of 32 entries in flight per lane; shorter
// ones share flattened ranges.
// (Swept at scales 20 and 26: thresholds 64-512, 2-8 rounds.)
constexpr uint32_t kLongPrefix = 128;
constexpr int kLongRounds = 8;
constexpr uint32_t kWarpSlots = 256;     // per-warp hash slots: |L(b)| <= warp_max_deg <= 128
constexpr uint32_t kFlushElems = 1u << 30;

__device__ __forceinline__ unsigned long long tri_clock_ns() {
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// Per-CTA times (tc_census_profile): slot 0, 1 or 2 of this CTA's entries.
__device__ __forceinline__ void tri_stamp(const TriParams& P, uint32_t slot, unsigned long long t) {
    for (uint32_t k = blockIdx.x + gridDim.x * threadIdx.x; k < P.stamps; k += gridDim.x * blockDim.x) P.phase[3 * k + slot] = t;
}

__device__ __forceinline__ uint32_t tri_hash(uint32_t x, int hb) { return (x * 2654435761u) >> (32 - hb); }

// Tricode of the triangle (a, b, c) from the direction bits of three stored entries: a in N[b]
// (seen from b: 1 b->a, 2 a->b), c in N[b] (1 b->c, 2 c->b) and a in N[c] (1 c->a, 2 a->c).
// Tricode bits: 1 b->a, 2 a->b, 4 b->c, 8 c->b, 16 a->c, 32 c->a.  The walk keeps the second
// term pre-shifted per pair (bc_bits = (dir(b,c)) << 2) and maps the third through a four-entry
// byte table: dir(c,a) 1 -> 32, 2 -> 16, 3 -> 48.
__device__ __forceinline__ uint32_t tri_code(uint32_t dir_ba, uint32_t bc_bits, uint32_t e_ca) {
    return dir_ba | bc_bits | __byte_perm(0x30102000u, 0u, e_ca & 3u);
}


// batched triangle form: per graph 96 uint64 of scratch, the 21 bulk sums at [0, 21) and the 64
// triangle tricodes at [32, 96); a serving wave's requests have the same scratch at WaveReq.out
constexpr uint32_t kBatchStride = 96;

// launch modes: one graph; a batch of graphs (items tagged with the graph, blocks (u0, u1, g));
// a serving wave (slices of several requests, descriptors in global memory)
// (kTriItems: one graph's CTA items alone)
enum { kTriSingle = 0, kTriBatch = 1, kTriWave = 2, kTriItems = 3 };

// index r of the last request whose prefix is <= i (prefixes ascend from 0)
template <typename F>
__device__ __forceinline__ uint32_t find_req(uint32_t count, uint32_t i, F pre) {
    uint32_t lo = 0, hi = count;
    while (hi - lo > 1) {
        const uint32_t mid = (lo + hi) >> 1;
        if (pre(mid) <= i) lo = mid; else hi = mid;
    }
    return lo;
}

// The lane that holds the lane-th set bit of mask (lanes past the last one get any lane), `mine` =
// this lane's bit; at: 32 bytes of shared scratch of this warp.  (__fns searches bit by bit: 1024
// batched graphs 5.70 -> 5.54 ms, the 64-state census of scale 20 6.56 -> 6.32 without it.)
__device__ __forceinline__ uint32_t nth_set(uint32_t mask, bool mine, volatile uint8_t* at, int lane) {
    if (mine) at[__popc(mask & ((1u << lane) - 1u))] = (uint8_t)lane;
    __syncwarp();
    const uint32_t src = at[lane] & 31u;
    __syncwarp();
    return src;
}

// Walk, for the pairs (b, c = N[b][j]), j in [j0, j1), 32 pairs per batch, the entries of N[c]
// below b (rp = b's position in N[c], from the pair tables; pb + j indexes the pair) and count
// each a found in the staged L(b).  MAP: L(b) is a direct map of two direction bits per id (every
// a < b is in its range); else a hash.  One warp: a batch's pairs with long prefixes are walked
// one after another by all lanes, and the lanes share the flattened (pair, position) range of
// the others.  Returns the entries walked (warp-uniform).
template <bool OLD, bool MAP, bool LONGW>
__device__ __forceinline__ uint32_t walk_pairs(const TriParams& P, const GraphDev& G, uint64_t bbase, uint64_t pb,
                                               uint32_t j0, uint32_t j1, const uint32_t* sH, const uint32_t* sO,
                                               int hb, uint32_t hmask, uint32_t ob, const uint8_t* sPerm,
                                               uint32_t* myHist, volatile uint8_t* at, int lane) {
    const uint64_t* __restrict__ off = G.off;
    const uint32_t* __restrict__ adj = G.adj;
    const uint32_t* __restrict__ rp = G.rp;
    const uint32_t le_mask = (2u << lane) - 1u;
    uint32_t walked = 0;
    // one walked entry e_ca = a in N[c] of the pair whose b-c tricode bits are bcb (and whose c has
    // the caller id oc2): look a up in L(b), count the triangle's tricode (or state) if found
    auto count = [&](uint32_t e_ca, uint32_t bcb, uint32_t oc2) {
        if (!e_ca) return;
        const uint32_t a = e_ca >> 2;
        uint32_t dir, oa = 0;
        if (MAP) {   // word a / 16, bits 2 (a mod 16), read straight from the entry
            dir = (sH[e_ca >> 6] >> ((e_ca >> 1) & 30u)) & 3u;
            if (OLD && dir) oa = P.old[a];
        } else {
            uint32_t h = tri_hash(a, hb);
            uint32_t e = sH[h];
            while (e != 0u && (e >> 2) != a) {
                h = (h + 1u) & hmask;
                e = sH[h];
            }
            dir = e & 3u;
            if (OLD && e) oa = sO[h];
        }
        if (dir != 0u) {
            uint32_t t = tri_code(dir, bcb, e_ca);
            if (OLD) {
                const uint32_t ra = (oa > ob) + (oa > oc2), rb = (ob > oa) + (ob > oc2);
                t = sPerm[(3u * ra + rb) * 64u + t];
            }
            atomicAdd(&myHist[t], 1u);
        }
    };
    for (uint32_t jb = j0; jb < j1; jb += 32) {
        const uint32_t j = jb + lane;
        const bool ok = j < j1;
        uint32_t e_bc = ok ? adj[bbase + j] : 0u;
        const uint32_t c = e_bc >> 2;
        uint64_t cb = ok ? off[c] : 0ull;
        uint32_t len = ok ? rp[pb + j] : 0u;
        uint32_t oc = (OLD && ok) ? P.old[c] : 0u;
        if (LONGW) {
            // pairs with long prefixes, one at a time over the whole warp: consecutive entries,
            // no search for the pair that holds an entry
            uint32_t lm = __ballot_sync(0xffffffffu, len >= kLongPrefix);
            while (lm) {
                const int q = __ffs(lm) - 1;
                lm &= lm - 1u;
                const uint64_t B = __shfl_sync(0xffffffffu, cb, q);
                const uint32_t L = __shfl_sync(0xffffffffu, len, q);
                const uint32_t bcb = (__shfl_sync(0xffffffffu, e_bc, q) & 3u) << 2;
                const uint32_t oq = OLD ? __shfl_sync(0xffffffffu, oc, q) : 0u;
                walked += L;
                for (uint32_t i = lane; i < L; i += 32u * kLongRounds) {
                    uint32_t x[kLongRounds];
#pragma unroll
                    for (int r = 0; r < kLongRounds; ++r)
                        x[r] = i + 32u * r < L ? __ldg(adj + (B + i + 32u * r)) : 0u;
#pragma unroll
                    for (int r = 0; r < kLongRounds; ++r) count(x[r], bcb, oq);
                }
            }
            if (len >= kLongPrefix) len = 0u;
        }
        // compact the pairs with a non-empty L(c) into lanes 0 .. cnt-1
        const uint32_t nz = __ballot_sync(0xffffffffu, len != 0u);
        if (!nz) continue;
        const uint32_t cnt = __popc(nz);
        const uint32_t src = nth_set(nz, len != 0u, at, lane);
        e_bc = __shfl_sync(0xffffffffu, e_bc, src);
        cb = __shfl_sync(0xffffffffu, cb, src);
        len = __shfl_sync(0xffffffffu, len, src);
        if (OLD) oc = __shfl_sync(0xffffffffu, oc, src);
        if ((uint32_t)lane >= cnt) len = 0u;
        uint32_t incl = len;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t excl = incl - len;
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        walked += total;
        // entry i of the flattened range lies at adj[cbx + i] for the pair that holds it (modular
        // arithmetic: i >= excl), and its tricode's b-c bits are bcb
        const uint64_t cbx = cb - excl;
        const uint32_t bcb = (e_bc & 3u) << 2;
        int seg_prev = -1;
        // two rounds of 32 entries per iteration, so each lane has two loads in flight
        for (uint32_t base = 0; base < total; base += 64) {
            // the pairs whose range starts in a round mark their start; lane i's pair is the
            // last one started at or before the round's entry i
            const bool stA = (uint32_t)lane < cnt && excl >= base && excl < base + 32u;
            const bool stB = (uint32_t)lane < cnt && excl >= base + 32u && excl < base + 64u;
            const uint32_t MA = __reduce_or_sync(0xffffffffu, stA ? (1u << (excl - base)) : 0u);
            const uint32_t MB = __reduce_or_sync(0xffffffffu, stB ? (1u << (excl - base - 32u)) : 0u);
            // (lane 31's count covers the whole round: the last pair of a round needs no shuffle)
            const int segA = seg_prev + __popc(MA & le_mask);
            const int lastA = seg_prev + __popc(MA);
            const int segB = lastA + __popc(MB & le_mask);
            seg_prev = lastA + __popc(MB);
            const uint32_t sa = (uint32_t)segA & 31u, sb = (uint32_t)segB & 31u;
            const uint64_t BA = __shfl_sync(0xffffffffu, cbx, sa), BB = __shfl_sync(0xffffffffu, cbx, sb);
            const uint32_t EA = __shfl_sync(0xffffffffu, bcb, sa), EB = __shfl_sync(0xffffffffu, bcb, sb);
            uint32_t OA = 0, OB = 0;
            if (OLD) {
                OA = __shfl_sync(0xffffffffu, oc, sa);
                OB = __shfl_sync(0xffffffffu, oc, sb);
            }
            const uint32_t iA = base + lane, iB = base + 32u + lane;
            const uint32_t xA = iA < total ? __ldg(adj + (BA + iA)) : 0u;
            const uint32_t xB = iB < total ? __ldg(adj + (BB + iB)) : 0u;
            count(xA, EA, OA);
            count(xB, EB, OB);
        }
    }
    return walked;
}

// Walk the entries adj[cb, cb + len) of each lane's pair as one flattened range: count(e, tag) for each
// entry e, with its pair's tag (e = 0 past the end).  Returns the entries (warp-uniform).
template <typename Count>
__device__ __forceinline__ uint32_t walk_flat(const uint32_t* __restrict__ adj, uint64_t cb, uint32_t len, uint32_t tag,
                                              volatile uint8_t* at, int lane, Count count) {
    const uint32_t le_mask = (2u << lane) - 1u;
    const uint32_t nz = __ballot_sync(0xffffffffu, len != 0u);
    if (!nz) return 0u;
    const uint32_t cnt = __popc(nz), src = nth_set(nz, len != 0u, at, lane);
    cb = __shfl_sync(0xffffffffu, cb, src);
    len = __shfl_sync(0xffffffffu, len, src);
    tag = __shfl_sync(0xffffffffu, tag, src);
    if ((uint32_t)lane >= cnt) len = 0u;
    uint32_t incl = len;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const uint32_t excl = incl - len, total = __shfl_sync(0xffffffffu, incl, 31);
    const uint64_t cbx = cb - excl;   // entry i of the range is adj[cbx + i] for the pair that holds it
    int before = -1;
    // two rounds of 32 entries at a time: lane i's pair is the last one started at or before its entry
    for (uint32_t base = 0; base < total; base += 64) {
        const bool st = (uint32_t)lane < cnt;
        const uint32_t ra = excl - base, rb = ra - 32u;
        const uint32_t MA = __reduce_or_sync(0xffffffffu, st && ra < 32u ? 1u << ra : 0u);
        const uint32_t MB = __reduce_or_sync(0xffffffffu, st && rb < 32u ? 1u << rb : 0u);
        const uint32_t sa = (uint32_t)(before + __popc(MA & le_mask)) & 31u;
        before += __popc(MA);
        const uint32_t sb = (uint32_t)(before + __popc(MB & le_mask)) & 31u;
        before += __popc(MB);
        const uint64_t BA = __shfl_sync(0xffffffffu, cbx, sa), BB = __shfl_sync(0xffffffffu, cbx, sb);
        const uint32_t TA = __shfl_sync(0xffffffffu, tag, sa), TB = __shfl_sync(0xffffffffu, tag, sb);
        const uint32_t iA = base + lane, iB = iA + 32u;
        const uint32_t xA = iA < total ? __ldg(adj + (BA + iA)) : 0u;
        const uint32_t xB = iB < total ? __ldg(adj + (BB + iB)) : 0u;
        count(xA, TA);
        count(xB, TB);
    }
    return total;
}

// The one-warp vertices b in [b0, b1), at most 32 consecutive ones.  Most have a handful of pairs, so
// one at a time leaves the lanes idle and waits for each one's loads in turn: here as many as fit
// (32 upper pairs, kPackLower lower entries, 2^rb rows) are walked together, a lane per pair,
// against one hash of all their lower neighbours, keyed by (a, row): (a << rb | row) << 2 | dir fits
// a 32-bit slot, rb = the bits an id leaves over, at most 5.  A vertex with more than 32 upper pairs
// goes alone.  1024 batched Chung-Lu graphs (mean degree 8): 5.54 -> 4.53 ms.  Returns the entries walked.
constexpr uint32_t kPackLower = kWarpSlots / 2;
__device__ __forceinline__ uint32_t walk_rows(const TriParams& P, const GraphDev& G, uint32_t b0, uint32_t b1, uint32_t* wH,
                                              uint32_t* myHist, volatile uint8_t* at, int lane) {
    const uint32_t* __restrict__ adj = G.adj;
    const uint32_t rb = min(5u, 30u - (32u - __clz(G.n - 1u | 1u)));
    const uint32_t x = b0 + lane;
    const bool ok = x < b1;
    const uint64_t base = ok ? G.off[x] : 0ull, pb = ok ? G.ub[x] : 0ull;
    uint32_t low = ok ? G.up[x] : 0u;
    uint32_t pairs = ok ? (uint32_t)(G.off[x + 1] - base) - low : 0u;
    // no lower or no upper neighbour: no triangle has b in the middle
    if (!low || !pairs) low = pairs = 0u;
    const bool alone = pairs > 32u;
    // both counts' prefixes in one scan (at most 32 x 128 and 32 x 32)
    uint32_t incl = alone ? 0u : low << 16 | pairs;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
        if (lane >= o) incl += y;
    }
    const uint32_t excl = incl - (alone ? 0u : low << 16 | pairs);
    uint32_t rest = __ballot_sync(0xffffffffu, pairs != 0u), walked = 0;
    while (rest) {
        const uint32_t r = __ffs(rest) - 1u;
        if (__shfl_sync(0xffffffffu, alone, r)) {
            rest &= rest - 1u;
            const uint64_t bb = __shfl_sync(0xffffffffu, base, r), pr = __shfl_sync(0xffffffffu, pb, r);
            const uint32_t lb = __shfl_sync(0xffffffffu, low, r), cnt = __shfl_sync(0xffffffffu, pairs, r);
            int hb = 6;
            while ((1u << hb) < 2u * lb) ++hb;
            const uint32_t hmask = (1u << hb) - 1u;
            __syncwarp();
            for (uint32_t k = lane; k < (1u << hb); k += 32) wH[k] = 0u;
            __syncwarp();
            for (uint32_t k = lane; k < lb; k += 32) {
                const uint32_t e = adj[bb + k];
                uint32_t h = tri_hash(e >> 2, hb);
                while (atomicCAS(&wH[h], 0u, e) != 0u) h = (h + 1u) & hmask;
            }
            __syncwarp();
            walked += walk_pairs<false, false, false>(P, G, bb, pr - lb, lb, lb + cnt, wH, nullptr, hb, hmask, 0u, nullptr,
                                                      myHist, at, lane);
            continue;
        }
        const uint32_t from = __shfl_sync(0xffffffffu, excl, r);
        const uint32_t mine = incl - from;   // rows r .. lane: lower entries << 16 | pairs
        const uint32_t over = __ballot_sync(0xffffffffu, (uint32_t)lane >= r && (alone || (mine & 0xffffu) > 32u ||
                                                                               (mine >> 16) > kPackLower || lane - r >= 1u << rb));
        const uint32_t end = over ? __ffs(over) - 1u : 32u;
        rest &= end == 32u ? 0u : ~((1u << end) - 1u);
        const uint32_t sum = __shfl_sync(0xffffffffu, mine, end - 1u), n_low = sum >> 16, n_pairs = sum & 0xffffu;
        // the row of the pack's i-th lower entry (sh = 16) or pair (sh = 0): the first one whose prefix passes i
        auto row_of = [&](uint32_t i, uint32_t sh) {
            uint32_t lo = r, hi = end - 1u;
#pragma unroll
            for (int s = 0; s < 5; ++s) {
                const uint32_t mid = (lo + hi) >> 1;
                const uint32_t v = __shfl_sync(0xffffffffu, mine, mid) >> sh & 0xffffu;
                if (lo < hi) {
                    if (v > i) hi = mid;
                    else lo = mid + 1u;
                }
            }
            return lo;
        };
        int hb = 6;
        while ((1u << hb) < 2u * n_low) ++hb;
        const uint32_t hmask = (1u << hb) - 1u;
        __syncwarp();
        for (uint32_t k = lane; k < (1u << hb); k += 32) wH[k] = 0u;
        // this lane's pair, its loads on their way while the hash is filled
        uint32_t row = row_of(lane, 0u);
        const uint32_t my = lane - ((__shfl_sync(0xffffffffu, excl, row) - from) & 0xffffu);
        const uint64_t rbase = __shfl_sync(0xffffffffu, base, row), rpb = __shfl_sync(0xffffffffu, pb, row);
        const uint32_t rlow = __shfl_sync(0xffffffffu, low, row);
        const bool valid = (uint32_t)lane < n_pairs;
        const uint32_t e_bc = valid ? __ldg(adj + rbase + rlow + my) : 0u;
        const uint32_t len = valid ? __ldg(G.rp + rpb + my) : 0u;
        __syncwarp();
        for (uint32_t i0 = 0; i0 < n_low; i0 += 32) {
            const uint32_t i = i0 + lane, q = row_of(i, 16u);
            const uint64_t qb = __shfl_sync(0xffffffffu, base, q);
            const uint32_t first = (__shfl_sync(0xffffffffu, excl, q) - from) >> 16;
            if (i < n_low) {
                const uint32_t e = __ldg(adj + qb + (i - first)), key = ((e >> 2) << rb | (q - r)) << 2 | (e & 3u);
                uint32_t h = tri_hash(key >> 2, hb);
                while (atomicCAS(&wH[h], 0u, key) != 0u) h = (h + 1u) & hmask;
            }
        }
        const uint64_t cb = len ? G.off[e_bc >> 2] : 0ull;
        __syncwarp();
        walked += walk_flat(adj, cb, len, (row - r) << 8 | (e_bc & 3u) << 2, at, lane, [&](uint32_t e_ca, uint32_t tag) {
            if (!e_ca) return;
            const uint32_t key = (e_ca >> 2) << rb | tag >> 8;
            uint32_t h = tri_hash(key, hb), e = wH[h];
            while (e != 0u && (e >> 2) != key) {
                h = (h + 1u) & hmask;
                e = wH[h];
            }
            if (e) atomicAdd(&myHist[tri_code(e & 3u, tag & 255u, e_ca)], 1u);
        });
    }
    return walked;
}

// A warp's next pairs of the CTA's item: guided sizes, 32 pairs while many remain, then fewer
// (down to 4) as the item runs out, so that the warps reach the item's end barrier together.
__device__ __forceinline__ void grab_pairs(uint32_t* s_next, uint32_t j1, int lane, uint32_t& jb, uint32_t& g) {
    jb = 0;
    g = 32;
    if (lane == 0) {
        const uint32_t cur = *(volatile uint32_t*)s_next;
        const uint32_t rem = cur < j1 ? j1 - cur : 0u;
        g = max(4u, min(32u, rem / (2u * kWarps)));
        jb = atomicAdd(s_next, g);
    }
    jb = __shfl_sync(0xffffffffu, jb, 0);
    g = __shfl_sync(0xffffffffu, g, 0);
}

// Add a warp's 64 bins to the graph's histogram and clear them (one warp).
__device__ __forceinline__ void flush_warp_hist(uint32_t* myHist, unsigned long long* hist, int lane) {
    __syncwarp();
    for (int t = lane; t < 64; t += 32) {
        const uint32_t v = myHist[t];
        if (v) atomicAdd(&hist[t], (unsigned long long)v);
        myHist[t] = 0u;
    }
    __syncwarp();
}

}  // namespace
}  // namespace tc
