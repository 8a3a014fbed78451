// triangles.cu - the census with the common neighbours enumerated once per triangle.
//
// For a connected pair (u, v), u < v (Fig. 5 step 2.1), every third vertex w of
// S = N[u] u N[v] \ {u, v} that only one endpoint reaches has a class fixed by two direction
// bits (dir(u,v) and the link of w to that endpoint), so those triads are counted in bulk
// from the per upper pair tables' direction-class suffix counts; only the common neighbours
// need their full tricode (the union-free rewrite of step 2.1.4).  The suffix kernel finds
// each pair's common neighbours by walking N[v] past u.  Here each common neighbour is found
// once, as a triangle: with ids in descending degree, L(x) = the neighbours of x with smaller
// ids (a prefix of N[x]) is short for every x, and the triangle a < b < c is met exactly
// once, when the walk of the entries of N[c] below b (a prefix of L(c), its length the pair
// table's position of b in N[c]) for the pair (b, c) finds a in L(b), staged in shared memory
// (a hash, or a direct map of two direction bits per id when b's id is small).
// Its tricode (roles (a, b, c)) then gives every correction it makes to the pairs' bulk
// counts (Fig. 5 steps 2.1.2 - 2.1.4):
//   + the triad itself, counted once at the pair (a, b) with w = c > b (step 2.1.4's rule);
//   - c among the u-only third vertices of (a, b) and among its v-only ones, b among the
//     v-only ones of (a, c): common neighbours, not one-sided;
//   + one common neighbour in the dyadic count n - |S| - 2 of each of its three pairs.
// So the kernel only histograms the 64 tricodes of the triangles; a small fold kernel turns
// them and the bulk sums into the 16 classes on the device.
//
// The same walk in the caller's id order (the triangle's state with its actors ordered by
// their original ids) serves the 64-state census (census64.cu).
//
// Work: a vertex b with degree above the warp tier becomes CTA items (b, range of its upper
// pairs (b, c)), cut by the plan (plan.cuh) with pair work |L(c)|; the CTA stages L(b) in a
// shared-memory hash, and its warps walk the lists L(c) of 32 pairs at a time as one
// flattened range, so short and long lists share the lanes.  The other vertices run one warp
// each, with L(b) in the warp's own hash.
#include <algorithm>
#include <atomic>
#include <cstring>

#include "graph.cuh"
#include "triangles.cuh"

namespace tc {

tc_status walk16_launch(const TriParams& P, const uint32_t split[2], uint32_t grid, uint32_t* ctr, cudaStream_t st);   // walk16.cu

namespace {

// A warp's copy of its graph's record.  No lane still reads the last one.
__device__ __forceinline__ void load_graph(GraphDev& to, const GraphDev* from, int lane) {
    static_assert(sizeof(GraphDev) % 8 == 0 && sizeof(GraphDev) <= 256, "a lane per word");
    __syncwarp();
    if (lane < (int)(sizeof(GraphDev) / 8)) reinterpret_cast<uint64_t*>(&to)[lane] = reinterpret_cast<const uint64_t*>(from)[lane];
    __syncwarp();
}

// Resident CTAs per SM; a single graph's launch has no more.  (CTAs beyond them start when others end and
// find the counters run out, so their times say nothing of the walk's balance.)  The packed one-warp
// vertices need the registers of six; the items alone run at eight (32 registers, no spills), which hide
// more of the latency of short lists, but are a launch more.  A graph takes the two from kItemsApart items
// on, where that pays; one launch / two, ms: random graphs, 2^16 vertices of degree 60 (18 k items)
// 0.276 / 0.282, 2^15 of 80 (31 k) 0.247 / 0.247, 2^16 of 100 (65 k) 0.532 / 0.510, 2^18 of 100 (258 k) 2.79 /
// 2.45, 2^20 of 128 (1 M) 16.3 / 13.9; R-MAT 18 e.f. 16 (21 k) 0.537 / 0.533, R-MAT 20 e.f. 8 (52 k) 0.993 /
// 0.950, R-MAT 22 e.f. 8 (131 k) 4.24 / 3.96; Chung-Lu 1 M x 16 (54 k) 1.079 / 1.034.
constexpr int kCtasTri = 6, kCtasOld = 5, kCtasItems = 8;
constexpr uint32_t kItemsApart = 1u << 15;

template <bool OLD, int MODE>
// 1024 batched graphs at 8 / 6 / 5 resident CTAs: 4.67 / 4.53 / 4.66 ms (8 spill 500 bytes).  The
// 64-state census of scale 20 with 4 CTAs and 2048-entry chunks / 5 and 1024 / 8 and 512: 5.94 / 5.49 /
// 5.46 ms (at the 32 registers of 8 CTAs, 4 resident: 6.32).
__global__ void __launch_bounds__(kThreads, OLD ? kCtasOld : MODE == kTriItems ? kCtasItems : kCtasTri) k_triangles(TriParams P) {
    extern __shared__ __align__(16) unsigned char smem[];
    const uint32_t slots = 2u * P.chunk;
    uint32_t* sH = reinterpret_cast<uint32_t*>(smem);                 // [slots] CTA hash of L(b)
    uint32_t* sO = sH + slots;                                         // [slots] OLD: caller ids
    uint32_t* sWH = sO + (OLD ? slots : 0u);                           // [kWarps][kWarpSlots]
    uint32_t* sWO = sWH + kWarps * kWarpSlots;                         // [kWarps][kWarpSlots] OLD
    uint32_t* sHist = sWO + (OLD ? kWarps * kWarpSlots : 0u);         // [kWarps][64]
    uint8_t* sPerm = reinterpret_cast<uint8_t*>(sHist + kWarps * 64);  // [9][64] OLD
    __shared__ uint32_t s_item, s_next;
    __shared__ uint8_t s_at[kWarps][32];   // walk_pairs' scratch
    constexpr bool kOne = MODE == kTriSingle || MODE == kTriItems;
    __shared__ GraphDev s_g[kOne ? 1 : kWarps];

    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    // the whole-warp walk of long prefixes, except in a batch of graphs (small graphs, short
    // prefixes: the path would only cost the kernel registers); the one-warp tier's prefixes
    // are below its degree bound, never long
    constexpr bool kLongWalk = MODE != kTriBatch;
    if (P.marks & 1u) tri_stamp(P, 0, tri_clock_ns());
    for (int k = tid; k < kWarps * 64; k += kThreads) sHist[k] = 0u;
    if (OLD)
        for (int k = tid; k < 9 * 64; k += kThreads) sPerm[k] = P.perm_state[k];
    __syncthreads();
    uint32_t* myHist = sHist + warp * 64;
    const GraphDev& G = kOne ? P.g : s_g[warp];   // several graphs: the warp's
    unsigned long long* ghist = P.hist;
    uint32_t cur_graph = 0xffffffffu;   // batched: the graph whose counts the warp's bins hold
    // batched: move to graph gi, flushing this warp's bins to the graph they belong to
    auto use_graph = [&](uint32_t gi) {
        if (cur_graph != 0xffffffffu) flush_warp_hist(myHist, ghist, lane);
        cur_graph = gi;
        load_graph(s_g[warp], MODE == kTriWave ? &P.reqs[gi].g : &P.graphs[gi], lane);
        ghist = MODE == kTriWave ? P.reqs[gi].out + 32 : P.hist + (uint64_t)kBatchStride * gi;
    };
    uint32_t since_flush = 0;   // warp-uniform: entries walked since this warp's bins were flushed
    // the hash region (2 x chunk words) holds a direct map of 32 x chunk ids at two bits each
    const uint32_t map_ids = 32u * P.chunk;

    // ---------------------------------------------------------------- CTA items
    for (;;) {
        if (tid == 0) s_item = atomicAdd(&P.ctr[0], 1u);
        __syncthreads();
        const uint32_t it = s_item;
        if (it >= P.n_items) break;
        Item w;
        if (MODE == kTriWave) {
            const uint32_t r = find_req(P.n_reqs, it, [&](uint32_t q) { return P.reqs[q].item_pre; });
            w = P.reqs[r].items[it - P.reqs[r].item_pre];
            if (r != cur_graph) use_graph(r);
        } else {
            w = P.items[it];
            if (MODE == kTriBatch && w.pad != cur_graph) use_graph(w.pad);
        }
        const long long t0 = clock64();
        const uint32_t b = w.u;
        const uint64_t bbase = G.off[b];
        const uint32_t lb = G.up[b];
        const uint32_t ob = OLD ? P.old[b] : 0u;
        const uint64_t pb = G.ub[b] - lb;   // table index of the pair (b, N[b][j]) is pb + j
        if (b <= map_ids) {
            // L(b) as a direct map of two direction bits per id below b: one pass, no probing
            for (uint32_t k = tid; k < map_ids / 16u; k += kThreads) sH[k] = 0u;
            if (tid == 0) s_next = w.j0;
            __syncthreads();
            for (uint32_t k = tid; k < lb; k += kThreads) {
                const uint32_t e = G.adj[bbase + k], a = e >> 2;
                atomicOr(&sH[a >> 4], (e & 3u) << ((a & 15u) << 1));
            }
            __syncthreads();
            for (;;) {
                uint32_t jb, g;
                grab_pairs(&s_next, w.j1, lane, jb, g);
                if (jb >= w.j1) break;
                since_flush += walk_pairs<OLD, true, kLongWalk>(P, G, bbase, pb, jb, min(jb + g, w.j1), sH, nullptr, 0, 0u, ob,
                                                     sPerm, myHist, s_at[warp], lane);
                if (since_flush >= kFlushElems) {
                    flush_warp_hist(myHist, ghist, lane);
                    since_flush = 0;
                }
            }
            __syncthreads();
        }
        // L(b) = N[b][0, lb), staged `chunk` entries per pass in a hash; every pass walks the item's pairs
        for (uint32_t c0 = 0; b > map_ids && c0 < lb; c0 += P.chunk) {
            const uint32_t LA = min(P.chunk, lb - c0);
            int hb = 6;
            while ((1u << hb) < 2u * LA) ++hb;
            const uint32_t H = 1u << hb, hmask = H - 1u;
            for (uint32_t k = tid; k < H; k += kThreads) sH[k] = 0u;
            if (tid == 0) s_next = w.j0;
            __syncthreads();
            for (uint32_t k = tid; k < LA; k += kThreads) {
                const uint32_t e = G.adj[bbase + c0 + k];
                uint32_t h = tri_hash(e >> 2, hb);
                while (atomicCAS(&sH[h], 0u, e) != 0u) h = (h + 1u) & hmask;
                if (OLD) sO[h] = P.old[e >> 2];
            }
            __syncthreads();
            for (;;) {
                uint32_t jb, g;
                grab_pairs(&s_next, w.j1, lane, jb, g);
                if (jb >= w.j1) break;
                since_flush += walk_pairs<OLD, false, kLongWalk>(P, G, bbase, pb, jb, min(jb + g, w.j1), sH, sO, hb, hmask, ob,
                                                      sPerm, myHist, s_at[warp], lane);
                if (since_flush >= kFlushElems) {
                    flush_warp_hist(myHist, ghist, lane);
                    since_flush = 0;
                }
            }
            __syncthreads();   // every warp is done with this pass before the hash is replaced
        }
        if (P.vcost && tid == 0) atomicAdd(&P.vcost[b], (unsigned long long)(clock64() - t0));
        __syncthreads();   // every thread has read s_item before thread 0 takes the next item
    }

    if (P.marks & 2u) tri_stamp(P, 1, tri_clock_ns());
    if (MODE == kTriItems) {
        flush_warp_hist(myHist, ghist, lane);
        return;
    }

    // ---------------------------------------------------------------- one warp per vertex
    uint32_t* wH = sWH + warp * kWarpSlots;
    uint32_t* wO = sWO + (OLD ? warp * kWarpSlots : 0u);
    for (;;) {
        uint32_t b0, b1;
        if (MODE == kTriWave) {
            uint32_t bk = 0;
            if (lane == 0) bk = atomicAdd(&P.ctr[1], 1u);
            bk = __shfl_sync(0xffffffffu, bk, 0);
            if (bk >= P.n_wblocks) break;
            const uint32_t r = find_req(P.n_reqs, bk, [&](uint32_t q) { return P.reqs[q].block_pre; });
            if (r != cur_graph) use_graph(r);
            const WaveReq& q = P.reqs[r];
            b0 = q.warp_begin + ((bk - q.block_pre) << q.pad);
            b1 = min(b0 + (1u << q.pad), q.warp_end);
        } else if (MODE == kTriBatch) {
            uint32_t bk = 0;
            if (lane == 0) bk = atomicAdd(&P.ctr[1], 1u);
            bk = __shfl_sync(0xffffffffu, bk, 0);
            if (bk >= P.n_wblocks) break;
            const uint4 wb = P.wblocks[bk];
            if (wb.z != cur_graph) use_graph(wb.z);
            b0 = wb.x;
            b1 = wb.y;
        } else {
            uint32_t vb = 0;
            if (lane == 0) vb = atomicAdd(&P.ctr[1], 1u << P.wshift);
            vb = __shfl_sync(0xffffffffu, vb, 0);
            if (vb >= P.warp_end - P.warp_begin) break;
            b0 = P.warp_begin + vb;
            b1 = min(b0 + (1u << P.wshift), P.warp_end);
        }
        if (!OLD) {
            since_flush += walk_rows(P, G, b0, b1, wH, myHist, s_at[warp], lane);
            if (since_flush >= kFlushElems) {
                flush_warp_hist(myHist, ghist, lane);
                since_flush = 0;
            }
            continue;
        }
        for (uint32_t b = b0; b < b1; ++b) {
            const uint64_t bbase = G.off[b];
            const uint32_t db = (uint32_t)(G.off[b + 1] - bbase), lb = G.up[b];
            if (lb == 0u || lb >= db) continue;   // no lower or no upper neighbour: no triangle has b in the middle
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
                if (OLD) wO[h] = P.old[e >> 2];
            }
            __syncwarp();
            since_flush += walk_pairs<OLD, false, false>(P, G, bbase, G.ub[b] - lb, lb, db, wH, wO, hb, hmask,
                                                  OLD ? P.old[b] : 0u, sPerm, myHist, s_at[warp], lane);
            if (since_flush >= kFlushElems) {
                flush_warp_hist(myHist, ghist, lane);
                since_flush = 0;
            }
        }
    }
    if (MODE == kTriSingle || cur_graph != 0xffffffffu) flush_warp_hist(myHist, ghist, lane);
    if (P.marks & 4u) {   // uniform over the CTA
        __syncthreads();
        tri_stamp(P, 2, tri_clock_ns());
    }
}

// One pair's bulk sums into acc (see k_pair_bulk): u of degree du, the pair's entry e = N[u][j]
// and its table index p.
__device__ __forceinline__ void bulk_pair(const GraphDev& g, uint32_t du, uint32_t j, uint32_t e, uint64_t p, int (&acc)[21]) {
    const uint32_t v = e >> 2, duv = e & 3u;
    const uint32_t cuv = ((duv & 1u) << 1) | (duv >> 1);
    const uint2 vs = g.vs[p], us = g.us[p];
    const uint32_t rpv = g.rp[p];
    const uint32_t dv = (uint32_t)(g.off[v + 1] - g.off[v]);
    const uint32_t vlen = dv - 1u - rpv, ulen = du - 1u - j;
    const uint32_t val[7] = {vs.x, vs.y, vlen - vs.x - vs.y, us.x, us.y, ulen - us.x - us.y, g.n - du - dv};
#pragma unroll
    for (int c = 0; c < 3; ++c)
        if (cuv == (uint32_t)(c + 1))
#pragma unroll
            for (int k = 0; k < 7; ++k) acc[7 * c + k] += (int)val[k];
}

// The warp's sum of acc[k] in lane k < 21 (0 in the others); acc is left zero.  Low and high halves
// are reduced apart, so 32 lanes cannot overflow.
__device__ __forceinline__ long long bulk_reduce(int (&acc)[21], int lane) {
    long long mine = 0;
#pragma unroll
    for (int k = 0; k < 21; ++k) {
        const int lo = __reduce_add_sync(0xffffffffu, acc[k] & 0xffff), hi = __reduce_add_sync(0xffffffffu, acc[k] >> 16);
        if (lane == k) mine = lo + hi * 65536ll;
        acc[k] = 0;
    }
    return mine;
}

// Bulk counts of the census's pairs: per dir(u,v) code c (tricode bits 1|2, 1..3),
// raw[7(c-1) + d - 1] += the entries of N[v] past u with direction class d (v-only third
// vertices before the common ones come off), raw[7(c-1) + 3 + d - 1] += those of N[u] past v
// (u-only), raw[7(c-1) + 6] += the dyadic base n - d_u - d_v (steps 2.1.2 - 2.1.3 before the
// common neighbours).  The pairs are the plan's: its CTA items (at most kMaxItemPairs pairs of
// one vertex each, a warp per item), then the one-warp vertices in blocks of 32 consecutive
// ones, whose upper pairs are consecutive in the table order and are walked as one flattened
// range.  Work comes from the counters ctr[2] (items) and ctr[3] (blocks), zeroed by the caller.
// Batched: item.pad and the blocks' third field name the graph (graphs[g], sums at raw +
// kBatchStride g); serving wave: request slices as in the census kernel's wave mode (sums at
// the request's scratch, WaveReq.out).
struct BulkParams {
    GraphDev g;
    const Item* items;
    uint32_t n_items;
    uint32_t wb, we;              // single graph: the one-warp vertices
    const GraphDev* graphs;       // batched
    const uint4* wblocks;
    uint32_t n_wblocks;
    const WaveReq* reqs;          // serving wave (n_items, n_wblocks: the wave's totals)
    uint32_t n_reqs;
    uint32_t* ctr;
    unsigned long long* raw;
};

// Blocks of one-warp vertices a warp takes per grab of a serving wave: the blocks follow the
// requests, so a warp that takes single ones meets another request, hence a reduction of its sums, at
// nearly every block (256 requests to 16 graphs: 3.53 -> 3.39 ms).  A batch of small graphs takes
// single blocks all the same (1024 graphs: 3.82 ms, in runs 4.08): all warps are then in the same few
// graphs, whose offsets and lists stay in the caches.
__device__ __forceinline__ uint32_t block_run(uint32_t blocks, uint32_t warps) {
    return min(16u, max(1u, blocks / (4u * warps)));
}

template <int MODE>
__global__ void __launch_bounds__(256, 4) k_pair_bulk(BulkParams P) {
    __shared__ uint8_t s_at[kWarps][32];
    __shared__ GraphDev s_g[MODE == kTriSingle ? 1 : kWarps];
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t le_mask = (2u << lane) - 1u;
    int acc[21];
#pragma unroll
    for (int k = 0; k < 21; ++k) acc[k] = 0;
    // A pair's values are at most n in size, so a lane's 32-bit sums hold `limit` rounds; then (and
    // at the end of a graph) the warp's go to 64 bits, the k-th sum in lane k.  64-bit sums in every
    // lane took 42 of the 64 registers, and with the graph's record per lane a tenth of the
    // instructions were spills (1024 batched graphs 4.50 -> 3.82 ms, 256 served requests 4.11 -> 3.39
    // ms, a census of scale 20 1.627 -> 1.602 ms; at five CTAs per SM, spilling again, slower).
    long long sum = 0;
    uint32_t rounds = 0, limit = MODE == kTriSingle ? 0x7fffffffu / P.g.n : 0u;
    auto round_done = [&] {
        if (++rounds < limit) return;
        sum += bulk_reduce(acc, lane);
        rounds = 0;
    };
    // several graphs: the warp's graph lies in shared memory (as a copy of each lane it was in local
    // memory, and its pointers' reloads missed L1)
    const GraphDev& G = MODE == kTriSingle ? P.g : s_g[threadIdx.x >> 5];
    unsigned long long* raw = P.raw;
    uint32_t cur_graph = 0xffffffffu;
    auto flush = [&] {
        sum += bulk_reduce(acc, lane);
        if (sum) atomicAdd(&raw[lane], (unsigned long long)sum);
        sum = 0;
        rounds = 0;
    };
    auto use_graph = [&](uint32_t gi) {
        if (cur_graph != 0xffffffffu) flush();
        cur_graph = gi;
        load_graph(s_g[threadIdx.x >> 5], MODE == kTriWave ? &P.reqs[gi].g : &P.graphs[gi], lane);
        raw = MODE == kTriWave ? P.reqs[gi].out : P.raw + (uint64_t)kBatchStride * gi;
        limit = 0x7fffffffu / G.n;
    };
    // the CTA items, a warp each
    for (;;) {
        uint32_t it = 0;
        if (lane == 0) it = atomicAdd(&P.ctr[2], 1u);
        it = __shfl_sync(0xffffffffu, it, 0);
        if (it >= P.n_items) break;
        Item w;
        if (MODE == kTriWave) {
            const uint32_t r = find_req(P.n_reqs, it, [&](uint32_t q) { return P.reqs[q].item_pre; });
            w = P.reqs[r].items[it - P.reqs[r].item_pre];
            if (r != cur_graph) use_graph(r);
        } else {
            w = P.items[it];
            if (MODE == kTriBatch && w.pad != cur_graph) use_graph(w.pad);
        }
        const uint64_t ubase = G.off[w.u];
        const uint32_t du = (uint32_t)(G.off[w.u + 1] - ubase);
        const uint64_t pb = G.ub[w.u] - G.up[w.u];
        for (uint32_t j0 = w.j0; j0 < w.j1; j0 += 32) {
            const uint32_t j = j0 + lane;
            if (j < w.j1) bulk_pair(G, du, j, G.adj[ubase + j], pb + j, acc);
            round_done();
        }
    }
    // the one-warp vertices, blocks of 32 consecutive ones
    const uint32_t run = MODE != kTriWave ? 1u : block_run(P.n_wblocks, gridDim.x * kWarps);
    for (uint32_t blk = 0, last = 0;; ++blk) {
        if (blk == last) {
            if (lane == 0) blk = atomicAdd(&P.ctr[3], run);
            blk = __shfl_sync(0xffffffffu, blk, 0);
            last = blk + run;
        }
        uint64_t base, end;
        if (MODE == kTriWave) {
            if (blk >= P.n_wblocks) break;
            const uint32_t r = find_req(P.n_reqs, blk, [&](uint32_t q) { return P.reqs[q].block_pre; });
            if (r != cur_graph) use_graph(r);
            const WaveReq& q = P.reqs[r];
            base = q.warp_begin + ((uint64_t)(blk - q.block_pre) << q.pad);
            end = base + (1u << q.pad) < q.warp_end ? base + (1u << q.pad) : q.warp_end;
        } else if (MODE == kTriBatch) {
            if (blk >= P.n_wblocks) break;
            const uint4 wbk = P.wblocks[blk];
            if (wbk.z != cur_graph) use_graph(wbk.z);
            base = wbk.x;
            end = wbk.y;
        } else {
            base = (uint64_t)P.wb + 32ull * blk;
            if (base >= P.we) break;
            end = base + 32u < P.we ? base + 32u : P.we;
        }
        const uint64_t u = base + lane;
        const bool ok = u < end;
        uint64_t ubase = ok ? G.off[u] : 0ull;
        uint32_t du = ok ? (uint32_t)(G.off[u + 1] - ubase) : 0u;
        uint32_t upu = ok ? G.up[u] : 0u;
        uint32_t cnt = du - upu;                  // upper pairs of u (0 past the block)
        const uint64_t pstart = G.ub[base];       // table index of the block's first pair
        // compact the vertices with upper pairs into lanes 0 .. nv-1, keeping their order
        const uint32_t nz = __ballot_sync(0xffffffffu, cnt != 0u);
        if (!nz) continue;
        const uint32_t nv = __popc(nz);
        const uint32_t src = nth_set(nz, cnt != 0u, s_at[threadIdx.x >> 5], (int)lane);
        ubase = __shfl_sync(0xffffffffu, ubase, src);
        du = __shfl_sync(0xffffffffu, du, src);
        upu = __shfl_sync(0xffffffffu, upu, src);
        cnt = __shfl_sync(0xffffffffu, cnt, src);
        if ((uint32_t)lane >= nv) cnt = 0u;
        uint32_t incl = cnt;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
            const uint32_t y = __shfl_up_sync(0xffffffffu, incl, o);
            if (lane >= o) incl += y;
        }
        const uint32_t excl = incl - cnt;
        const uint32_t total = __shfl_sync(0xffffffffu, incl, 31);
        int seg_prev = -1;
        for (uint32_t r0 = 0; r0 < total; r0 += 32) {
            const bool st = (uint32_t)lane < nv && excl >= r0 && excl < r0 + 32u;
            const uint32_t M = __reduce_or_sync(0xffffffffu, st ? (1u << (excl - r0)) : 0u);
            const int seg = seg_prev + __popc(M & le_mask);
            seg_prev = __shfl_sync(0xffffffffu, seg, 31);
            const uint32_t sg = (uint32_t)seg & 31u;
            const uint32_t sP = __shfl_sync(0xffffffffu, excl, sg);
            const uint64_t sB = __shfl_sync(0xffffffffu, ubase, sg);
            const uint32_t sD = __shfl_sync(0xffffffffu, du, sg), sU = __shfl_sync(0xffffffffu, upu, sg);
            const uint32_t i = r0 + lane;
            if (i < total) {
                const uint32_t j = sU + (i - sP);         // the pair's position in N[u]
                bulk_pair(G, sD, j, G.adj[sB + j], pstart + i, acc);
            }
            round_done();
        }
    }
    if (MODE == kTriSingle) {
        // one graph: the warps' sums meet in shared memory, so a CTA adds 21 counters once (a small
        // census waited for its warps' atomics on them)
        __shared__ long long s_sum[kWarps][32];
        s_sum[threadIdx.x >> 5][lane] = sum + bulk_reduce(acc, lane);
        __syncthreads();
        if (threadIdx.x < 21) {
            long long s = 0;
#pragma unroll
            for (int w = 0; w < kWarps; ++w) s += s_sum[w][threadIdx.x];
            if (s) atomicAdd(&raw[threadIdx.x], (unsigned long long)s);
        }
    } else if (cur_graph != 0xffffffffu) {
        flush();
    }
}

struct Table64 {
    uint8_t t[64];
};

// 16 classes from the bulk sums and the triangle tricodes (see the file comment) into out16 (index
// 0 gets 0).  One block of 64 threads.  Batched: block g folds raw + kBatchStride g and hist + kBatchStride g into out16 + 16 g.
__global__ void k_tri_fold(const unsigned long long* __restrict__ raw, const unsigned long long* __restrict__ hist,
                           Table64 T, unsigned long long* out16) {
    __shared__ unsigned long long s[16];
    const uint32_t t = threadIdx.x;
    raw += (uint64_t)kBatchStride * blockIdx.x;
    hist += (uint64_t)kBatchStride * blockIdx.x;
    out16 += 16ull * blockIdx.x;
    if (t < 16) s[t] = 0ull;
    __syncthreads();
    if (t < 21) {
        const uint32_t c = t / 7 + 1, k = t % 7;
        const unsigned long long v = raw[t];
        uint32_t cls;
        if (k < 3) cls = T.t[c | ((k + 1) << 2)];          // v-only: dir(v,w) = k + 1
        else if (k < 6) cls = T.t[c | ((k - 2) << 4)];     // u-only: dir(u,w) = k - 2
        else cls = c == 3u ? 2u : 1u;                       // dyadic base: 102 if mutual, else 012
        if (v) atomicAdd(&s[cls], v);
    }
    const unsigned long long h = hist[t];
    if (h) {
        const uint32_t cab = t & 3u;                                   // tricode bits of the pair (a, b)
        const uint32_t dac = (t >> 4) & 3u;                            // dir(a,c) seen from a
        const uint32_t dbc = (t >> 2) & 3u;                            // dir(b,c) seen from b
        const uint32_t dcb = ((dbc & 1u) << 1) | (dbc >> 1);           // dir(c,b) seen from c
        const uint32_t cac = ((dac & 1u) << 1) | (dac >> 1);           // tricode bits of the pair (a, c)
        const unsigned long long m = 0ull - h;
        atomicAdd(&s[T.t[t]], h);                                      // the triad, at (a, b) with w = c
        atomicAdd(&s[T.t[cab | (dac << 4)]], m);                       // c is no u-only vertex of (a, b)
        atomicAdd(&s[T.t[cab | (dbc << 2)]], m);                       // nor a v-only one
        atomicAdd(&s[T.t[cac | (dcb << 2)]], m);                       // b is no v-only vertex of (a, c)
        atomicAdd(&s[cab == 3u ? 2u : 1u], h);                         // a common neighbour of each pair
        atomicAdd(&s[dac == 3u ? 2u : 1u], h);
        atomicAdd(&s[dbc == 3u ? 2u : 1u], h);
    }
    __syncthreads();
    if (t < 16) out16[t] = t ? s[t] : 0ull;
}

// Serving: fold each finished request's scratch (block r) into its 16 counts in mapped host
// memory (dst + 16 r, index 0 = 0) and zero the scratch for the slot's next request.
struct TriCollect {
    unsigned long long* src[kMaxWave];
    unsigned long long* dst;
    uint32_t n;
};

__global__ void k_tri_collect(TriCollect a, Table64 T) {
    __shared__ unsigned long long out[16];
    const uint32_t r = blockIdx.x, t = threadIdx.x;
    if (r >= a.n) return;
    if (t < 16) out[t] = 0ull;
    __syncthreads();
    unsigned long long* sc = a.src[r];
    // the same fold as k_tri_fold, into shared memory
    if (t < 21) {
        const uint32_t c = t / 7 + 1, k = t % 7;
        const unsigned long long v = sc[t];
        const uint32_t cls = k < 3 ? T.t[c | ((k + 1) << 2)] : (k < 6 ? T.t[c | ((k - 2) << 4)] : (c == 3u ? 2u : 1u));
        if (v) atomicAdd(&out[cls], v);
    }
    const unsigned long long h = sc[32 + t];
    if (h) {
        const uint32_t cab = t & 3u, dac = (t >> 4) & 3u, dbc = (t >> 2) & 3u;
        const uint32_t dcb = ((dbc & 1u) << 1) | (dbc >> 1), cac = ((dac & 1u) << 1) | (dac >> 1);
        const unsigned long long m = 0ull - h;
        atomicAdd(&out[T.t[t]], h);
        atomicAdd(&out[T.t[cab | (dac << 4)]], m);
        atomicAdd(&out[T.t[cab | (dbc << 2)]], m);
        atomicAdd(&out[T.t[cac | (dcb << 2)]], m);
        atomicAdd(&out[cab == 3u ? 2u : 1u], h);
        atomicAdd(&out[dac == 3u ? 2u : 1u], h);
        atomicAdd(&out[dbc == 3u ? 2u : 1u], h);
    }
    __syncthreads();
    if (t < 16) a.dst[16 * r + t] = t ? out[t] : 0ull;
    for (uint32_t k = t; k < kBatchStride; k += blockDim.x) sc[k] = 0ull;
}

std::atomic<int> g_tri_limit[5][64] = {};   // dynamic shared memory the form's kernel was set to, per device

size_t tri_smem(uint32_t chunk, bool old) {
    const size_t slots = 2ull * chunk;
    return sizeof(uint32_t) * (slots * (old ? 2 : 1) + (size_t)kWarps * kWarpSlots * (old ? 2 : 1) + kWarps * 64) +
           (old ? 9 * 64 : 0);
}

// form: 0 single graph, 1 caller-id states (64-state census), 2 batched, 3 serving wave, 4 a single graph's items
tc_status tri_prepare(int form, size_t smem) {
    int dev = 0;
    TC_CUDA(cudaGetDevice(&dev));
    std::atomic<int>& limit = g_tri_limit[form][dev & 63];
    int lim = limit.load();
    if (!lim) {
        const void* fns[5] = {(const void*)k_triangles<false, kTriSingle>, (const void*)k_triangles<true, kTriSingle>,
                              (const void*)k_triangles<false, kTriBatch>, (const void*)k_triangles<false, kTriWave>,
                              (const void*)k_triangles<false, kTriItems>};
        int optin = 0;
        TC_CUDA(cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev));
        cudaFuncAttributes fa;
        TC_CUDA(cudaFuncGetAttributes(&fa, fns[form]));
        lim = optin - (int)fa.sharedSizeBytes;
        TC_CUDA(cudaFuncSetAttribute(fns[form], cudaFuncAttributeMaxDynamicSharedMemorySize, lim));
        limit.store(lim);
    }
    if ((int)smem > lim) return fail(TC_ERR_ARG, "chunk_entries too large for this GPU's shared memory");
    return TC_OK;
}

tc_status fold_table(Table64* T) {
    const uint8_t* ht = host_tricode_table();
    if (!ht) return fail(TC_ERR_ARG, "tricode table derivation failed");
    std::memcpy(T->t, ht, 64);
    return TC_OK;
}

}  // namespace

tc_status triangles_launch(const GraphDev& gd, const Opts& o, const Item* items, uint32_t n_items, uint32_t warp_begin,
                           uint32_t warp_end, uint32_t* ctr, const uint32_t* old, const uint8_t* d_perm_state,
                           unsigned long long* d_hist64, unsigned long long* d_vcost, cudaStream_t st,
                           unsigned long long* d_phase, const uint32_t* split) {
    const bool is_old = old != nullptr;
    TriParams P;
    std::memset(&P, 0, sizeof(P));
    P.g = gd;
    P.items = items;
    P.n_items = n_items;
    P.warp_begin = warp_begin;
    P.warp_end = warp_end;
    P.wshift = warp_block_shift(warp_end - warp_begin, (unsigned)census_grid(o));
    P.chunk = o.chunk;
    P.ctr = ctr;
    P.old = old;
    P.perm_state = d_perm_state;
    P.hist = d_hist64;
    P.vcost = d_vcost;
    P.phase = d_phase;
    unsigned grid = (unsigned)census_grid(o);
    P.stamps = grid;
    P.marks = d_phase ? 7u : 0u;
    if (split && !is_old) return walk16_launch(P, split, grid, ctr + 4, st);
    const size_t smem = tri_smem(o.chunk, is_old);
    if (!is_old && n_items >= kItemsApart) {
        TC_TRY(tri_prepare(4, smem));
        P.marks = d_phase ? 3u : 0u;
        k_triangles<false, kTriItems><<<std::min(grid, (unsigned)(sm_count() * kCtasItems)), kThreads, smem, st>>>(P);
        TC_LAUNCH("k_triangles (items)");
        P.marks = d_phase ? 4u : 0u;
        P.n_items = 0;
    }
    TC_TRY(tri_prepare(is_old ? 1 : 0, smem));
    grid = std::min(grid, (unsigned)(sm_count() * (is_old ? kCtasOld : kCtasTri)));
    if (is_old) k_triangles<true, kTriSingle><<<grid, kThreads, smem, st>>>(P);
    else k_triangles<false, kTriSingle><<<grid, kThreads, smem, st>>>(P);
    TC_LAUNCH("k_triangles");
    return TC_OK;
}

// The 16-bit lists are made with a graph's first plan of this form, so that a census that has its plan only
// launches.  One that is captured cannot make them (its plan may be another call's: the 64-state census
// and the server read no such lists), and a device without room for them need not: the general kernel
// counts the same.  The next plan tries again.
tc_status census_plan(GraphStore& g, const Opts& o, cudaStream_t st, Plan** out) {
    if (!has_plan(g, o)) g.no_lists16 = false;
    TC_TRY(get_plan(g, o, st, out));
    if (o.algo != TC_ALGO_TRIANGLE || g.blk16.p || g.no_lists16 || !walk16_takes(g) || captured(st)) return TC_OK;
    const tc_status made = lists16_build(g, st);
    if (made != TC_ERR_OOM) return made;
    g.rec.release();
    g.no_lists16 = true;
    return TC_OK;
}

tc_status triangle_census_enqueue(GraphStore& g, const Opts& o, const Plan& p, uint32_t item0, uint32_t n_items,
                                  uint32_t warp_begin, uint32_t warp_end, cudaStream_t st, unsigned long long* d_out16,
                                  unsigned long long* d_vcost, unsigned long long* d_phase) {
    if (g.e_sym == 0) {
        TC_CUDA(cudaMemsetAsync(d_out16, 0, sizeof(unsigned long long) * 16, st));
        return TC_OK;
    }
    if (!g.vs.p) return fail(TC_ERR_ARG, "the triangle form needs the per upper pair tables");
    // [0, 21) bulk sums, [32, 96) triangle tricodes, then 8 work counters: zeroed at once (g.tri holds them)
    constexpr size_t kScratch = sizeof(unsigned long long) * kBatchStride + sizeof(uint32_t) * 8;
    unsigned long long* raw = g.tri.as<unsigned long long>();
    unsigned long long* hist = raw + 32;
    uint32_t* ctr = reinterpret_cast<uint32_t*>(raw + kBatchStride);
    TC_CUDA(cudaMemsetAsync(raw, 0, kScratch, st));
    const Item* items = p.items.as<Item>() + item0;
    // the range's part of each of the plan's splits
    const uint32_t split[2] = {std::min(std::max(p.split[0], item0) - item0, n_items),
                               std::min(std::max(p.split[1], item0) - item0, n_items)};
    // without the lists (census_plan) the general kernel counts the same
    const bool walk16 = walk16_takes(g) && g.blk16.p;
    const GraphDev gd = g.dev();
    const uint64_t units = (uint64_t)n_items + (warp_end - warp_begin + 31u) / 32u;
    if (units) {
        BulkParams B;
        std::memset(&B, 0, sizeof(B));
        B.g = gd;
        B.items = items;
        B.n_items = n_items;
        B.wb = warp_begin;
        B.we = warp_end;
        B.ctr = ctr;
        B.raw = raw;
        k_pair_bulk<kTriSingle><<<grid_for(units * 32, 256, 4u * (unsigned)sm_count()), 256, 0, st>>>(B);
        TC_LAUNCH("k_pair_bulk");
    }
    TC_TRY(triangles_launch(gd, o, items, n_items, warp_begin, warp_end, ctr, nullptr, nullptr, hist,
                            d_vcost, st, d_phase, walk16 ? split : nullptr));
    Table64 T;
    TC_TRY(fold_table(&T));
    k_tri_fold<<<1, 64, 0, st>>>(raw, hist, T, d_out16);
    TC_LAUNCH("k_tri_fold");
    return TC_OK;
}

tc_status triangle_census_batch(const GraphDev* d_graphs, uint32_t k, const Item* items, uint32_t n_items,
                                const uint4* wblocks, uint32_t n_wblocks, const Opts& o, uint32_t* ctr,
                                unsigned long long* d_scratch, unsigned long long* d_out, cudaStream_t st) {
    if (k == 0) return TC_OK;
    const size_t smem = tri_smem(o.chunk, false);
    TC_TRY(tri_prepare(2, smem));
    TC_CUDA(cudaMemsetAsync(d_scratch, 0, sizeof(unsigned long long) * kBatchStride * k, st));
    const uint64_t units = (uint64_t)n_items + n_wblocks;
    if (units) {
        BulkParams B;
        std::memset(&B, 0, sizeof(B));
        B.items = items;
        B.n_items = n_items;
        B.graphs = d_graphs;
        B.wblocks = wblocks;
        B.n_wblocks = n_wblocks;
        B.ctr = ctr;
        B.raw = d_scratch;
        k_pair_bulk<kTriBatch><<<grid_for(units * 32, 256, 4u * (unsigned)sm_count()), 256, 0, st>>>(B);
        TC_LAUNCH("k_pair_bulk (batched)");
        TriParams P;
        std::memset(&P, 0, sizeof(P));
        P.items = items;
        P.n_items = n_items;
        P.chunk = o.chunk;
        P.ctr = ctr;
        P.hist = d_scratch + 32;
        P.graphs = d_graphs;
        P.wblocks = wblocks;
        P.n_wblocks = n_wblocks;
        k_triangles<false, kTriBatch><<<(unsigned)census_grid(o), kThreads, smem, st>>>(P);
        TC_LAUNCH("k_triangles (batched)");
    }
    Table64 T;
    TC_TRY(fold_table(&T));
    k_tri_fold<<<k, 64, 0, st>>>(d_scratch, d_scratch + 32, T, d_out);
    TC_LAUNCH("k_tri_fold (batched)");
    return TC_OK;
}

tc_status triangle_census_wave(const WaveReq* d_reqs, uint32_t n_reqs, uint32_t total_items, uint32_t total_blocks,
                               const Opts& o, unsigned grid, uint32_t* ctr, cudaStream_t st) {
    if (n_reqs > kMaxWave) return fail(TC_ERR_RANGE, "wave larger than kMaxWave requests");
    const size_t smem = tri_smem(o.chunk, false);
    TC_TRY(tri_prepare(3, smem));
    BulkParams B;
    std::memset(&B, 0, sizeof(B));
    B.n_items = total_items;
    B.n_wblocks = total_blocks;
    B.reqs = d_reqs;
    B.n_reqs = n_reqs;
    B.ctr = ctr;
    const uint64_t units = (uint64_t)total_items + total_blocks;
    k_pair_bulk<kTriWave><<<grid_for(units * 32, 256, 4u * (unsigned)sm_count()), 256, 0, st>>>(B);
    TC_LAUNCH("k_pair_bulk (wave)");
    TriParams P;
    std::memset(&P, 0, sizeof(P));
    P.n_items = total_items;
    P.n_wblocks = total_blocks;
    P.reqs = d_reqs;
    P.n_reqs = n_reqs;
    P.chunk = o.chunk;
    P.ctr = ctr;
    k_triangles<false, kTriWave><<<grid, kThreads, smem, st>>>(P);
    TC_LAUNCH("k_triangles (wave)");
    return TC_OK;
}

tc_status triangle_collect(unsigned long long* const* scratch, uint32_t n, unsigned long long* d_dst, cudaStream_t st) {
    if (n == 0) return TC_OK;
    if (n > kMaxWave) return fail(TC_ERR_RANGE, "more finished requests than a wave holds");
    TriCollect a;
    std::memset(&a, 0, sizeof(a));
    for (uint32_t k = 0; k < n; ++k) a.src[k] = scratch[k];
    a.dst = d_dst;
    a.n = n;
    Table64 T;
    TC_TRY(fold_table(&T));
    k_tri_collect<<<n, 64, 0, st>>>(a, T);
    TC_LAUNCH("k_tri_collect");
    return TC_OK;
}

}  // namespace tc
