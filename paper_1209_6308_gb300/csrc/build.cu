// build.cu - device construction of the compact graph structure of Sec. 6 (Fig. 7):
// one edge array holding every vertex's sorted neighbour list, a start offset per vertex,
// and the two low bits of each stored id giving the arc direction (01 owner->neighbour,
// 10 neighbour->owner, 11 both).
//
// From an arc list: validate ids, drop self-loops, key each arc by its unordered pair with
// one direction bit, radix sort, merge equal pairs by OR-ing their direction bits, count
// degrees, relabel vertices by descending degree (ties by original id), emit both
// directions of every pair in the new ids, radix sort by (owner, neighbour), and read off
// the offsets.  A CSR input is validated (sorted, flagged, loop-free, symmetric) and then
// goes through the same relabel.
#include <algorithm>

#include "graph.cuh"
#include "rows.cuh"
#include "tc_internal.cuh"

namespace tc {
namespace {

constexpr int kB = 256;
constexpr int kStats = 15;   // of the build: what each kernel adds where is said at the kernel

__device__ __forceinline__ uint32_t swap_dir(uint32_t d) { return ((d & 1u) << 1) | ((d >> 1) & 1u); }

// stats[0] self-loops, stats[1] ids out of range
__global__ void k_make_keys(const uint32_t* src, const uint32_t* dst, uint64_t m, uint32_t n, int B,
                            uint64_t* keys, unsigned long long* stats) {
    uint32_t loops = 0, bad = 0;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < m; i += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t a = src[i], b = dst[i];
        uint64_t key = ~0ull;
        if (a >= n || b >= n) ++bad;
        else if (a == b) ++loops;
        else {
            uint64_t lo = a < b ? a : b, hi = a < b ? b : a;
            uint64_t dir = a < b ? 1u : 2u;           // 01: lo->hi, 10: hi->lo
            key = (lo << (B + 2)) | (hi << 2) | dir;
        }
        keys[i] = key;
    }
    for (int o = 16; o; o >>= 1) {
        loops += __shfl_xor_sync(0xffffffffu, loops, o);
        bad += __shfl_xor_sync(0xffffffffu, bad, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (loops) atomicAdd(&stats[0], (unsigned long long)loops);
        if (bad) atomicAdd(&stats[1], (unsigned long long)bad);
    }
}

__global__ void k_head_flags(const uint64_t* keys, uint64_t cnt, uint32_t* flag) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < cnt; i += (uint64_t)gridDim.x * blockDim.x)
        flag[i] = keys[i] != ~0ull && (i == 0 || (keys[i] >> 2) != (keys[i - 1] >> 2)) ? 1u : 0u;
}

// Runs of equal pairs -> one pair key (lo<<B | hi) and the OR of their direction bits.
__global__ void k_unique(const uint64_t* keys, uint64_t cnt, const uint32_t* flag, const uint32_t* pos,
                         uint64_t* ukey, uint32_t* udir) {
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < cnt; i += (uint64_t)gridDim.x * blockDim.x) {
        if (keys[i] == ~0ull) continue;   // a dropped arc's key, past the others
        uint32_t r = pos[i] + flag[i] - 1u;
        if (flag[i]) ukey[r] = keys[i] >> 2;
        atomicOr(&udir[r], (uint32_t)(keys[i] & 3u));
    }
}

// degrees; stats[2] mutual pairs.  The pairs are sorted by their smaller id, so the lanes of a
// warp mostly share it: one atomic per run of equal ids (a hub's run would otherwise serialise
// thousands of atomics on one address).
__global__ void k_degrees(const uint64_t* ukey, const uint32_t* udir, uint64_t E, int B, uint32_t* deg,
                          unsigned long long* stats) {
    const uint64_t mask = (1ull << B) - 1;
    const uint32_t lane = threadIdx.x & 31;
    uint32_t mut = 0;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    for (uint64_t r0 = blockIdx.x * (uint64_t)blockDim.x + (threadIdx.x & ~31u); r0 < E; r0 += stride) {
        const uint64_t r = r0 + lane;   // uniform loop over the warp: every lane takes part in the match
        const bool ok = r < E;
        const uint64_t k = ok ? ukey[r] : ~0ull;
        const uint32_t lo = (uint32_t)(k >> B);
        const uint32_t peers = __match_any_sync(0xffffffffu, ok ? lo : 0xffffffffu);
        if (ok && (peers & ((1u << lane) - 1u)) == 0) atomicAdd(&deg[lo], (uint32_t)__popc(peers));
        if (ok) {
            atomicAdd(&deg[k & mask], 1u);
            mut += (udir[r] == 3u);
        }
    }
    for (int o = 16; o; o >>= 1) mut += __shfl_xor_sync(0xffffffffu, mut, o);
    if ((threadIdx.x & 31) == 0 && mut) atomicAdd(&stats[2], (unsigned long long)mut);
}

__global__ void k_relabel_keys(const uint32_t* deg, uint32_t n, int B, uint64_t* rk) {
    const uint64_t top = (1ull << B) - 1;
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < n; x += (uint64_t)gridDim.x * blockDim.x)
        rk[x] = ((top - deg[x]) << B) | x;
}

__global__ void k_perm(const uint64_t* rk, uint32_t n, int B, uint32_t* new_of_old) {
    const uint64_t mask = (1ull << B) - 1;
    for (uint64_t r = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; r < n; r += (uint64_t)gridDim.x * blockDim.x)
        new_of_old[rk[r] & mask] = (uint32_t)r;
}

// Each pair once in the new ids, from its smaller one: (lo << (B+2)) | (hi << 2) | dir(lo).
__global__ void k_upper_keys(const uint64_t* ukey, const uint32_t* udir, uint64_t E, int B, const uint32_t* new_of_old,
                             uint64_t* key) {
    const uint64_t mask = (1ull << B) - 1;
    for (uint64_t r = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; r < E; r += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t k = ukey[r];
        const uint64_t a = new_of_old[k >> B], b = new_of_old[k & mask];
        const uint32_t d = udir[r];
        key[r] = a < b ? (a << (B + 2)) | (b << 2) | d : (b << (B + 2)) | (a << 2) | swap_dir(d);
    }
}

// With the pairs sorted by (lo, hi), pair p's key in the transpose: (hi << 32) | p.  Sorted by hi,
// stably, vertex v's pairs stand in the order of their lo: its lower list.
__global__ void k_transpose_keys(const uint64_t* __restrict__ key, uint64_t E, int B, uint64_t* __restrict__ tkey) {
    const uint64_t mask = (1ull << B) - 1;
    for (uint64_t p = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; p < E; p += (uint64_t)gridDim.x * blockDim.x)
        tkey[p] = ((key[p] >> 2) & mask) << 32 | p;
}

// start[x] = the first of the E > 0 sorted keys whose row (key >> shift) is >= x, for x in [0, n]: a
// search per vertex, whose neighbours in the warp take the same path but for its end; the rows before
// the first key's and past the last one's (vertices without entries) need none.  Filling the rows
// between two keys from the keys' side leaves a run of rows without keys to one thread: a build of
// 10 M vertices in pairs (i, i + n/2), whose first half has no lower entry, took 24.1 ms so and takes
// 2.9 (pairs anywhere 2.8 and 3.1; R-MAT 20, 15 pairs per vertex, 3.57 and 3.46).
__global__ void k_row_starts(const uint64_t* __restrict__ key, uint64_t E, int shift, uint32_t n, uint64_t* __restrict__ start) {
    const uint64_t first = key[0] >> shift, last = key[E - 1] >> shift;
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x <= n; x += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t lo = x <= first ? 0ull : x > last ? E : 1ull, hi = x > first && x <= last ? E - 1ull : lo;
        while (lo < hi) {   // key lo - 1 is of a row below x, key hi of none
            const uint64_t mid = (lo + hi) >> 1;
            if (key[mid] >> shift < x) lo = mid + 1;
            else hi = mid;
        }
        start[x] = lo;
    }
}

// off and up from the starts of the upper pairs (ub) and of the lower entries (lb) of each vertex.
__global__ void k_offsets(const uint64_t* __restrict__ ub, const uint64_t* __restrict__ lb, uint32_t n, uint64_t* __restrict__ off,
                          uint32_t* __restrict__ up) {
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x <= n; x += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t l = lb[x];
        off[x] = ub[x] + l;
        if (x < n) up[x] = (uint32_t)(lb[x + 1] - l);
    }
}

// The lists: the i-th sorted pair is u's upper entry (behind the lower entries of the vertices up to
// u), the i-th transposed one v's lower entry (behind the upper entries of the vertices below v),
// whose position in v's list is its pair's rp.
__global__ void k_lists(const uint64_t* __restrict__ key, const uint64_t* __restrict__ tkey, uint64_t E, int B,
                        const uint64_t* __restrict__ ub, const uint64_t* __restrict__ lb, uint32_t* __restrict__ adj,
                        uint32_t* __restrict__ rp) {
    const uint64_t mask = (1ull << (B + 2)) - 1;
    for (uint64_t i = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; i < E; i += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t k = key[i], t = tkey[i], v = t >> 32;
        adj[i + lb[(k >> (B + 2)) + 1]] = (uint32_t)(k & mask);
        const uint32_t p = (uint32_t)t;
        const uint64_t kt = key[p];
        adj[i + ub[v]] = (uint32_t)(kt >> (B + 2)) << 2 | swap_dir((uint32_t)kt & 3u);
        rp[p] = (uint32_t)(i - lb[v]);
    }
}

// stats[3] sum deg^2, stats[4] sum over upper pairs of deg(v), stats[5] max degree,
// stats[7] vertices with deg > 0, stats[10] sum of up (up - 1) / 2 (the entries the triangle form
// walks: for every upper pair (b, c), the neighbours of c below b), stats[11] vertices with deg > kHubDeg,
// stats[12] vertices with deg > 32, stats[13] with deg > 64
__global__ void k_graph_sums(const uint64_t* off, const uint32_t* adj, const uint32_t* up, uint32_t n,
                             unsigned long long* stats) {
    unsigned long long d2 = 0, dv = 0, tw = 0;
    uint32_t mx = 0, act = 0, hub = 0, wide = 0, gt64 = 0;
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < n; x += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t d = off[x + 1] - off[x];
        d2 += d * d;
        mx = max(mx, (uint32_t)d);
        act += (d > 0);
        hub += (d > kHubDeg);
        wide += (d > 32);
        gt64 += (d > 64);
        // x is the v of every pair (u, x) with u < x: the first up[x] neighbours
        dv += (unsigned long long)up[x] * d;
        tw += (unsigned long long)up[x] * (up[x] ? up[x] - 1ull : 0ull) / 2ull;
    }
    for (int o = 16; o; o >>= 1) {
        d2 += __shfl_xor_sync(0xffffffffu, d2, o);
        dv += __shfl_xor_sync(0xffffffffu, dv, o);
        tw += __shfl_xor_sync(0xffffffffu, tw, o);
        mx = max(mx, __shfl_xor_sync(0xffffffffu, mx, o));
        act += __shfl_xor_sync(0xffffffffu, act, o);
        hub += __shfl_xor_sync(0xffffffffu, hub, o);
        wide += __shfl_xor_sync(0xffffffffu, wide, o);
        gt64 += __shfl_xor_sync(0xffffffffu, gt64, o);
    }
    if ((threadIdx.x & 31) == 0) {
        if (act) atomicAdd(&stats[7], (unsigned long long)act);
        if (hub) atomicAdd(&stats[11], (unsigned long long)hub);
        if (wide) atomicAdd(&stats[12], (unsigned long long)wide);
        if (gt64) atomicAdd(&stats[13], (unsigned long long)gt64);
        atomicAdd(&stats[3], d2);
        atomicAdd(&stats[4], dv);
        atomicAdd(&stats[10], tw);
        atomicMax(&stats[5], (unsigned long long)mx);
    }
}

constexpr uint32_t kLongList = 4096;   // longer lists: k_pair_tables_long, a CTA per vertex
constexpr int kLongThreads = 1024;

// Per upper pair tables, lists of at most kLongList entries (longer ones are k_pair_tables_long's).
// The lane at position k of N[v] counts the direction classes of the entries after k.  At a lower
// neighbour u = N[v][k] (k < up[v]) those are the third vertices w > u reached from v: vs of the
// upper pair (u, v), whose index is the low half of tkey[lb[v] + k] (k_transpose_keys; lb[v] = the
// lower entries of the vertices before v).  At an upper neighbour (k >= up[v]) they are
// the third vertices w > N[v][k] reached from v, the u side of the pair (v, N[v][k]): us = (class-1,
// class-2 counts).  wk[0] += the suffix lengths at lower neighbours (the N[v] entries a census
// walks), wk[1] += those of them with ids below kMapIdsSuffix: with c the entries of N[v] below it
// (a prefix), the walk past position k meets max(0, c - k - 1) of them.
// The n_wide lists of more than 32 entries go a warp each, in 32-entry blocks from the end with
// running counts; for the others a warp takes 32 vertices (rows.cuh) whose lists share its lanes
// and are counted by one ballot per class.
// Bound by its table writes and, per warp, by the loads' latency: at scale 20 a warp per vertex
// took 0.68 ms.
__global__ void __launch_bounds__(kB) k_pair_tables(const uint64_t* __restrict__ off, const uint32_t* __restrict__ adj,
                              const uint32_t* __restrict__ up, const uint64_t* __restrict__ ub,
                              const uint64_t* __restrict__ lb, uint32_t n,
                              const unsigned long long* __restrict__ n_wide, const uint64_t* __restrict__ tkey, uint2* vs,
                              uint2* us,
                              unsigned long long* wk) {
    __shared__ uint8_t s_at[kB / 32][32];
    const uint32_t lane = threadIdx.x & 31;
    const uint32_t after = lane == 31 ? 0u : ~((2u << lane) - 1u);   // lanes above this one
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    unsigned long long walk = 0, walk_map = 0;
    // the lists of more than 32 entries, a prefix of the ids, a warp each
    const uint64_t wide = *n_wide;
    for (uint64_t v = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5; v < wide; v += stride >> 5) {
        const uint64_t ob = off[v], ubv = ub[v], lbv = lb[v];
        const uint32_t dv = (uint32_t)(off[v + 1] - ob), lv = up[v];
        if (dv > kLongList) continue;                                 // k_pair_tables_long's
        uint32_t c1 = 0, c2 = 0, cmap = 0;
        for (uint32_t cs = dv & ~31u; cs <= dv; cs -= 32) {   // blocks from the last one down
            const uint32_t k = cs + lane;
            const uint32_t e = k < dv ? adj[ob + k] : 0u;
            const uint32_t b1 = __ballot_sync(0xffffffffu, (e & 3u) == 1u);
            const uint32_t b2 = __ballot_sync(0xffffffffu, (e & 3u) == 2u);
            if (k < lv) {
                vs[(uint32_t)tkey[lbv + k]] = make_uint2(c1 + __popc(b1 & after), c2 + __popc(b2 & after));
                walk += dv - k - 1;
            } else if (k < dv) {
                us[ubv + (k - lv)] = make_uint2(c1 + __popc(b1 & after), c2 + __popc(b2 & after));
            }
            c1 += __popc(b1);
            c2 += __popc(b2);
            cmap += __popc(__ballot_sync(0xffffffffu, k < dv && (e >> 2) < kMapIdsSuffix));
            if (cs == 0) break;
        }
        const unsigned long long m = min(lv, cmap);
        if (lane == 0) walk_map += m * cmap - m * (m + 1) / 2;
    }
    for (uint64_t x0 = wide + blockIdx.x * (uint64_t)blockDim.x + (threadIdx.x & ~31u); x0 < n; x0 += stride) {
        const uint64_t x = x0 + lane;
        const bool ok = x < n;
        const uint64_t vob = ok ? off[x] : 0ull, vub = ok ? ub[x] : 0ull, vlb = ok ? lb[x] : 0ull;
        const uint32_t vd = ok ? (uint32_t)(off[x + 1] - vob) : 0u, vl = ok ? up[x] : 0u;
        for_rows(vd, s_at[threadIdx.x >> 5],
            [&](const PackedEntry& p) {
                const uint64_t ob = __shfl_sync(0xffffffffu, vob, p.row), ubv = __shfl_sync(0xffffffffu, vub, p.row);
                const uint64_t lbv = __shfl_sync(0xffffffffu, vlb, p.row);
                const uint32_t dv = __shfl_sync(0xffffffffu, vd, p.row), lv = __shfl_sync(0xffffffffu, vl, p.row);
                const uint32_t k = lane - p.first;
                const uint32_t e = p.valid ? adj[ob + k] : 0u;
                const uint32_t m1 = __ballot_sync(0xffffffffu, (e & 3u) == 1u) & p.lanes;
                const uint32_t m2 = __ballot_sync(0xffffffffu, (e & 3u) == 2u) & p.lanes;
                const uint32_t mm = __ballot_sync(0xffffffffu, p.valid && (e >> 2) < kMapIdsSuffix) & p.lanes;
                const uint2 c = make_uint2(__popc(m1 & after), __popc(m2 & after));
                if (p.valid && k < lv) {
                    vs[(uint32_t)tkey[lbv + k]] = c;
                    walk += dv - k - 1;
                    const uint32_t cmap = __popc(mm);
                    walk_map += cmap > k ? cmap - k - 1u : 0u;
                } else if (p.valid) {
                    us[ubv + (k - lv)] = c;
                }
            },
            [](uint32_t) {});
    }
    for (int o = 16; o; o >>= 1) walk += __shfl_xor_sync(0xffffffffu, walk, o);
    for (int o = 16; o; o >>= 1) walk_map += __shfl_xor_sync(0xffffffffu, walk_map, o);
    if (lane == 0 && walk) atomicAdd(wk, walk);
    if (lane == 0 && walk_map) atomicAdd(wk + 1, walk_map);
}

// The same tables for the vertices with more than kLongList entries, a prefix of the ids
// (degrees descend), one CTA per vertex: a warp per list walks at most kLongList / 32 blocks in
// series.  Each warp takes a contiguous segment of N[v] (a multiple of 32 entries), counts its
// class-1 and class-2 entries, and then walks it backward from the counts of the segments after
// it, as k_pair_tables walks a whole list.
__global__ void __launch_bounds__(kLongThreads) k_pair_tables_long(
        const uint64_t* __restrict__ off, const uint32_t* __restrict__ adj, const uint32_t* __restrict__ up,
        const uint64_t* __restrict__ ub, const uint64_t* __restrict__ lb, uint32_t n, const uint64_t* __restrict__ tkey,
        uint2* vs, uint2* us, unsigned long long* wk) {
    __shared__ uint32_t s_c1[kLongThreads / 32], s_c2[kLongThreads / 32], s_map[kLongThreads / 32];
    const uint64_t v = blockIdx.x;
    if (v >= n) return;
    const uint64_t ob = off[v];
    const uint32_t dv = (uint32_t)(off[v + 1] - ob), lv = up[v];
    if (dv <= kLongList) return;                                      // the same for the whole CTA
    const uint32_t lane = threadIdx.x & 31, wid = threadIdx.x >> 5, nw = blockDim.x >> 5;
    const uint32_t after = lane == 31 ? 0u : ~((2u << lane) - 1u);
    const uint32_t seg = ((dv + nw - 1) / nw + 31u) & ~31u;
    const uint32_t s0 = min(dv, wid * seg), s1 = min(dv, s0 + seg);
    uint32_t a1 = 0, a2 = 0, am = 0;
#pragma unroll 4
    for (uint32_t k = s0 + lane; k < s1; k += 32) {
        const uint32_t e = adj[ob + k];
        a1 += (e & 3u) == 1u;
        a2 += (e & 3u) == 2u;
        am += (e >> 2) < kMapIdsSuffix;
    }
    a1 = __reduce_add_sync(0xffffffffu, a1);
    a2 = __reduce_add_sync(0xffffffffu, a2);
    am = __reduce_add_sync(0xffffffffu, am);
    if (lane == 0) {
        s_c1[wid] = a1;
        s_c2[wid] = a2;
        s_map[wid] = am;
    }
    __syncthreads();
    uint32_t c1 = 0, c2 = 0, cmap = 0;
    for (uint32_t w = 0; w < nw; ++w) {
        if (w > wid) {
            c1 += s_c1[w];
            c2 += s_c2[w];
        }
        cmap += s_map[w];
    }
    unsigned long long walk = 0;
    if (s1 > s0) {
        for (uint32_t cs = (s1 - 1) & ~31u;; cs -= 32) {            // s0 is a multiple of 32
            const uint32_t k = cs + lane;
            const uint32_t e = k < s1 ? adj[ob + k] : 0u;
            const uint32_t b1 = __ballot_sync(0xffffffffu, (e & 3u) == 1u);
            const uint32_t b2 = __ballot_sync(0xffffffffu, (e & 3u) == 2u);
            if (k < lv) {
                vs[(uint32_t)tkey[lb[v] + k]] = make_uint2(c1 + __popc(b1 & after), c2 + __popc(b2 & after));
                walk += dv - k - 1;
            } else if (k < s1) {
                us[ub[v] + (k - lv)] = make_uint2(c1 + __popc(b1 & after), c2 + __popc(b2 & after));
            }
            c1 += __popc(b1);
            c2 += __popc(b2);
            if (cs == s0) break;
        }
    }
    for (int o = 16; o; o >>= 1) walk += __shfl_xor_sync(0xffffffffu, walk, o);
    if (lane == 0 && walk) atomicAdd(wk, walk);
    if (threadIdx.x == 0) {
        const unsigned long long m = min(lv, cmap);
        const unsigned long long wm = m * cmap - m * (m + 1) / 2;
        if (wm) atomicAdd(wk + 1, wm);
    }
}

// ---- CSR input validation: stats[6] = number of violations
__global__ void k_check_csr(const uint64_t* off, const uint32_t* adj, uint32_t n, uint64_t total,
                            unsigned long long* stats) {
    uint32_t badc = 0;
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < n; x += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t b = off[x], e = off[x + 1];
        if (e < b || e > total) { ++badc; continue; }
        for (uint64_t i = b; i < e; ++i) {
            uint32_t w = adj[i], id = w >> 2, d = w & 3u;
            if (id >= n || id == x || d == 0 || (i > b && (adj[i - 1] >> 2) >= id)) { ++badc; break; }
            // symmetry: x must appear in N[id] with mirrored direction bits
            uint64_t lo = off[id], hi = off[id + 1];
            if (hi < lo || hi > total) { ++badc; break; }
            uint32_t key = (uint32_t)x << 2;
            while (lo < hi) {
                uint64_t mid = (lo + hi) >> 1;
                if ((adj[mid] & ~3u) < key) lo = mid + 1; else hi = mid;
            }
            if (lo >= off[id + 1] || adj[lo] != (key | swap_dir(d))) { ++badc; break; }
        }
    }
    for (int o = 16; o; o >>= 1) badc += __shfl_xor_sync(0xffffffffu, badc, o);
    if ((threadIdx.x & 31) == 0 && badc) atomicAdd(&stats[6], (unsigned long long)badc);
}

// Upper entries (x < id) of a valid CSR -> pair keys and direction bits relative to lo = x.
__global__ void k_csr_pairs(const uint64_t* off, const uint32_t* adj, uint32_t n, int B, const uint32_t* upos,
                            uint64_t* ukey, uint32_t* udir, uint32_t* deg, unsigned long long* stats) {
    uint32_t mut = 0;
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < n; x += (uint64_t)gridDim.x * blockDim.x) {
        uint64_t b = off[x], e = off[x + 1];
        deg[x] = (uint32_t)(e - b);
        uint32_t r = upos[x];
        for (uint64_t i = b; i < e; ++i) {
            uint32_t w = adj[i], id = w >> 2;
            if (id > x) {
                ukey[r] = ((uint64_t)x << B) | id;
                udir[r] = w & 3u;
                mut += ((w & 3u) == 3u);
                ++r;
            }
        }
    }
    for (int o = 16; o; o >>= 1) mut += __shfl_xor_sync(0xffffffffu, mut, o);
    if ((threadIdx.x & 31) == 0 && mut) atomicAdd(&stats[2], (unsigned long long)mut);
}

__global__ void k_upper_counts(const uint64_t* off, const uint32_t* adj, uint32_t n, uint32_t* cnt) {
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < n; x += (uint64_t)gridDim.x * blockDim.x) {
        uint32_t c = 0;
        for (uint64_t i = off[x]; i < off[x + 1]; ++i) c += ((adj[i] >> 2) > x);
        cnt[x] = c;
    }
}


// Below this many vertices and pairs a build takes its graph's memory first, while the stream is idle:
// a later allocation that outlives the stream waits for the sorts.
constexpr uint64_t kStoreFirst = 1ull << 22;

// Steps shared by both inputs: E unique pairs (ukey = lo<<B | hi, udir relative to lo) and
// degrees -> relabel, CSR, up[], stats.  Each input is released after its last use, and a large
// graph's own memory is taken after the sorts, in place of the buffer they leave over: 44 B per pair and
// 32 B per vertex at most (up front, with the inputs kept, it was 64 B per pair).
tc_status finish_graph(GraphStore& g, uint64_t E, int B, DevBuf& ukey, DevBuf& udir, DevBuf& deg, DevBuf& stats,
                       cudaStream_t st) {
    const uint32_t n = g.n;
    // the lists hold 2E entries, and the 64-state census sorts them all: 32-bit counts
    if (E >= (1ull << 31)) return fail(TC_ERR_RANGE, "more than 2^31-1 connected pairs");
    const unsigned gridE = grid_for(E, kB, 1u << 16), gridN = grid_for(n, kB, 1u << 16);
    // relabel by descending degree
    DevBuf rk, rtmp;
    TC_TRY(rk.alloc(sizeof(uint64_t) * n, st));
    TC_TRY(rtmp.alloc(sizeof(uint64_t) * n, st));
    // the graph's buffers, carved from one (an allocation that outlives its stream is synchronised)
    const bool store_first = n + E < kStoreFirst;
    auto make_store = [&]() -> tc_status {
        struct { DevBuf* b; size_t bytes; } parts[] = {
            {&g.off, sizeof(uint64_t) * (n + 1ull)}, {&g.ub, sizeof(uint64_t) * (n + 1ull)},
            {&g.adj, sizeof(uint32_t) * (2 * E + 4)},   // read in aligned blocks of four
            {&g.up, sizeof(uint32_t) * n}, {&g.rp, sizeof(uint32_t) * E},
            {&g.vs, sizeof(uint2) * E}, {&g.us, sizeof(uint2) * E},
            {&g.new_of_old, store_first ? sizeof(uint32_t) * n : 0u}};   // last: else it has memory of its own
        size_t total = 0;
        for (const auto& q : parts) total += (q.bytes + 255u) & ~(size_t)255u;
        TC_TRY(g.store.alloc_persistent(total));
        size_t at = 0;
        for (const auto& q : parts) {
            if (q.b != &g.new_of_old || store_first) q.b->carve(g.store, at, q.bytes);
            at += (q.bytes + 255u) & ~(size_t)255u;
        }
        return TC_OK;
    };
    if (store_first) TC_TRY(make_store());
    else TC_TRY(g.new_of_old.alloc_persistent(sizeof(uint32_t) * n));
    k_relabel_keys<<<gridN, kB, 0, st>>>(deg.as<uint32_t>(), n, B, rk.as<uint64_t>());
    TC_LAUNCH("k_relabel_keys");
    deg.release();
    uint64_t* kp = rk.as<uint64_t>();
    uint64_t* tp = rtmp.as<uint64_t>();
    TC_TRY(radix_sort_u64(&kp, &tp, n, B, 2 * B, st));   // stable: ties stay in id order
    k_perm<<<gridN, kB, 0, st>>>(kp, n, B, g.new_of_old.as<uint32_t>());
    TC_LAUNCH("k_perm");
    rk.release();
    rtmp.release();
    unsigned long long* d_stats = stats.as<unsigned long long>();
    // the pairs in the new ids, sorted by (lo, hi): the upper lists in order, a pair's place its table
    // index; and their transpose, sorted by hi: the lower lists in order
    DevBuf key, tmp, tkey, lbuf;
    const uint64_t* ks = nullptr;
    const uint64_t* ts = nullptr;
    if (E) {
        TC_TRY(key.alloc(sizeof(uint64_t) * E, st));
        k_upper_keys<<<gridE, kB, 0, st>>>(ukey.as<uint64_t>(), udir.as<uint32_t>(), E, B, g.new_of_old.as<uint32_t>(),
                                           key.as<uint64_t>());
        TC_LAUNCH("k_upper_keys");
        ukey.release();
        udir.release();
        TC_TRY(tmp.alloc(sizeof(uint64_t) * E, st));
        TC_TRY(tkey.alloc(sizeof(uint64_t) * E, st));
        kp = key.as<uint64_t>();
        tp = tmp.as<uint64_t>();
        TC_TRY(radix_sort_u64(&kp, &tp, E, 2, 2 * B + 2, st));
        ks = kp;
        kp = tkey.as<uint64_t>();   // tp, the buffer the sort left over, is the transpose's second one
        k_transpose_keys<<<gridE, kB, 0, st>>>(ks, E, B, kp);
        TC_LAUNCH("k_transpose_keys");
        TC_TRY(radix_sort_u64(&kp, &tp, E, 32, 32 + B, st));
        ts = kp;
        for (DevBuf* b : {&key, &tmp, &tkey})
            if (b->p != ks && b->p != ts) b->release();
    }
    if (!store_first) TC_TRY(make_store());
    TC_TRY(lbuf.alloc(sizeof(uint64_t) * (n + 1ull), st));
    uint64_t *off = g.off.as<uint64_t>(), *ub = g.ub.as<uint64_t>(), *lb = lbuf.as<uint64_t>();
    if (E) {
        const unsigned gridS = grid_for(n + 1ull, kB, 1u << 16);
        k_row_starts<<<gridS, kB, 0, st>>>(ks, E, B + 2, n, ub);
        TC_LAUNCH("k_row_starts (upper)");
        k_row_starts<<<gridS, kB, 0, st>>>(ts, E, 32, n, lb);
        TC_LAUNCH("k_row_starts (lower)");
    } else {
        TC_CUDA(cudaMemsetAsync(ub, 0, sizeof(uint64_t) * (n + 1ull), st));
        TC_CUDA(cudaMemsetAsync(lb, 0, sizeof(uint64_t) * (n + 1ull), st));
    }
    k_offsets<<<grid_for(n + 1ull, kB, 1u << 16), kB, 0, st>>>(ub, lb, n, off, g.up.as<uint32_t>());
    TC_LAUNCH("k_offsets");
    if (E) {
        k_lists<<<gridE, kB, 0, st>>>(ks, ts, E, B, ub, lb, g.adj.as<uint32_t>(), g.rp.as<uint32_t>());
        TC_LAUNCH("k_lists");
    }
    k_graph_sums<<<gridN, kB, 0, st>>>(off, g.adj.as<uint32_t>(), g.up.as<uint32_t>(), n, d_stats);
    TC_LAUNCH("k_graph_sums");
    if (E) {
        // the suffix counts of the per upper pair tables; the walk lengths go to stats[8..9]
        // (at most 2E / 33 lists have more than 32 entries)
        k_pair_tables<<<grid_lists(n, std::min<uint64_t>(n, 2ull * E / 33)), kB, 0, st>>>(off, g.adj.as<uint32_t>(), g.up.as<uint32_t>(), ub, lb, n,
                                            d_stats + 12, ts, g.vs.as<uint2>(), g.us.as<uint2>(), d_stats + 8);
        TC_LAUNCH("k_pair_tables");
        // lists longer than kLongList: at most 2E / kLongList of them, the first ids
        const uint64_t n_long = std::min<uint64_t>(n, 2ull * E / kLongList + 1);
        k_pair_tables_long<<<(unsigned)n_long, kLongThreads, 0, st>>>(off, g.adj.as<uint32_t>(), g.up.as<uint32_t>(), ub, lb, n,
                                                                      ts, g.vs.as<uint2>(), g.us.as<uint2>(), d_stats + 8);
        TC_LAUNCH("k_pair_tables_long");
    }
    unsigned long long hs[kStats];
    TC_CUDA(cudaMemcpyAsync(hs, stats.p, sizeof(hs), cudaMemcpyDeviceToHost, st));
    TC_CUDA(cudaStreamSynchronize(st));
    g.sum_tri_walk = hs[10];
    g.n_hub = (uint32_t)hs[11];
    g.n_wide = (uint32_t)hs[12];
    g.n_gt64 = (uint32_t)hs[13];
    g.sum_walk = hs[8];
    g.sum_walk_map = hs[9];
    g.e_sym = E;
    g.mutual = hs[2];
    g.arcs = E + hs[2];
    g.sum_d2 = hs[3];
    g.sum_dv_upper = hs[4];
    g.max_deg = (uint32_t)hs[5];
    g.loops = hs[0];
    // degrees descend with the new id, so the vertices with deg > 0 are [0, n_active)
    g.n_active = (uint32_t)hs[7];
    return TC_OK;
}

}  // namespace

int bits_for(uint32_t n) {
    int B = 1;
    while ((1ull << B) < n) ++B;
    return B;
}

namespace {

// Runs of one pair among m keys sorted by pair (direction bits in bits 0..1, runs adjacent, the
// all-ones keys of dropped arcs last) -> E unique pairs (ukey = lo<<B | hi) with the OR of their
// direction bits.  hs receives the stats so far (synchronises st).
tc_status pairs_from_sorted(const uint64_t* kp, uint64_t m, DevBuf& ukey, DevBuf& udir, uint32_t& E, DevBuf& stats,
                            unsigned long long hs[kStats], cudaStream_t st) {
    DevBuf flag, pos;
    TC_TRY(flag.alloc(sizeof(uint32_t) * (m ? m : 1), st));
    TC_TRY(pos.alloc(sizeof(uint32_t) * (m ? m : 1), st));
    if (m) {
        k_head_flags<<<grid_for(m, kB, 1u << 16), kB, 0, st>>>(kp, m, flag.as<uint32_t>());
        TC_LAUNCH("k_head_flags");
        TC_TRY(scan_u32(flag.as<uint32_t>(), pos.as<uint32_t>(), m, reinterpret_cast<uint32_t*>(stats.as<uint64_t>() + 14), st));
    }
    TC_CUDA(cudaMemcpyAsync(hs, stats.p, sizeof(unsigned long long) * kStats, cudaMemcpyDeviceToHost, st));
    TC_CUDA(cudaStreamSynchronize(st));
    E = (uint32_t)hs[14];   // little-endian: the scan's total in the low half
    TC_TRY(ukey.alloc(sizeof(uint64_t) * (E ? E : 1), st));
    TC_TRY(udir.alloc(sizeof(uint32_t) * (E ? E : 1), st));
    TC_CUDA(cudaMemsetAsync(udir.p, 0, sizeof(uint32_t) * (E ? E : 1), st));
    if (E) {
        k_unique<<<grid_for(m, kB, 1u << 16), kB, 0, st>>>(kp, m, flag.as<uint32_t>(), pos.as<uint32_t>(),
                                                          ukey.as<uint64_t>(), udir.as<uint32_t>());
        TC_LAUNCH("k_unique");
    }
    return TC_OK;
}

// Degrees of the E unique pairs, then the relabelled CSR and its tables.
tc_status graph_from_pairs(GraphStore& g, int B, uint32_t E, DevBuf& ukey, DevBuf& udir, DevBuf& stats,
                           cudaStream_t st) {
    DevBuf deg;
    TC_TRY(deg.alloc(sizeof(uint32_t) * (g.n ? g.n : 1), st));
    TC_CUDA(cudaMemsetAsync(deg.p, 0, sizeof(uint32_t) * (g.n ? g.n : 1), st));
    if (E) {
        k_degrees<<<grid_for(E, kB, 1u << 16), kB, 0, st>>>(ukey.as<uint64_t>(), udir.as<uint32_t>(), E, B,
                                                             deg.as<uint32_t>(), stats.as<unsigned long long>());
        TC_LAUNCH("k_degrees");
    }
    return finish_graph(g, E, B, ukey, udir, deg, stats, st);
}

}  // namespace

tc_status build_from_arcs(GraphStore& g, uint64_t m, const uint32_t* d_src, const uint32_t* d_dst, cudaStream_t st) {
    const uint32_t n = g.n;
    const int B = bits_for(n);
    if (m >= (1ull << 32)) return fail(TC_ERR_RANGE, "more than 2^32-1 arcs");
    DevBuf stats, keys, tmp;
    TC_TRY(stats.alloc(sizeof(unsigned long long) * kStats, st));
    TC_CUDA(cudaMemsetAsync(stats.p, 0, sizeof(unsigned long long) * kStats, st));
    TC_TRY(keys.alloc(sizeof(uint64_t) * (m ? m : 1), st));
    TC_TRY(tmp.alloc(sizeof(uint64_t) * (m ? m : 1), st));
    if (m) {
        k_make_keys<<<grid_for(m, kB, 1u << 16), kB, 0, st>>>(d_src, d_dst, m, n, B, keys.as<uint64_t>(),
                                                               stats.as<unsigned long long>());
        TC_LAUNCH("k_make_keys");
    }
    uint64_t* kp = keys.as<uint64_t>();
    uint64_t* tp = tmp.as<uint64_t>();
    TC_TRY(radix_sort_u64(&kp, &tp, m, 2, 2 * B + 2, st));
    // unique pairs (the keys of self-loops and of ids out of range are all ones and sort past the others)
    DevBuf ukey, udir;
    uint32_t E = 0;
    unsigned long long hs[kStats];
    TC_TRY(pairs_from_sorted(kp, m, ukey, udir, E, stats, hs, st));
    if (hs[1]) return fail(TC_ERR_RANGE, "arc list holds a vertex id >= n");
    keys.release();
    tmp.release();
    TC_TRY(graph_from_pairs(g, B, E, ukey, udir, stats, st));
    g.dups = m - g.loops - g.arcs;
    return TC_OK;
}

tc_status build_from_sorted_arcs(GraphStore& g, const uint64_t* d_keys, uint64_t m, cudaStream_t st) {
    const int B = bits_for(g.n);
    if (m >= (1ull << 32)) return fail(TC_ERR_RANGE, "more than 2^32-1 arcs");
    DevBuf stats, ukey, udir;
    TC_TRY(stats.alloc(sizeof(unsigned long long) * kStats, st));
    TC_CUDA(cudaMemsetAsync(stats.p, 0, sizeof(unsigned long long) * kStats, st));
    uint32_t E = 0;
    unsigned long long hs[kStats];
    TC_TRY(pairs_from_sorted(d_keys, m, ukey, udir, E, stats, hs, st));
    TC_TRY(graph_from_pairs(g, B, E, ukey, udir, stats, st));
    g.dups = m - g.arcs;
    return TC_OK;
}

tc_status build_from_csr(GraphStore& g, const uint64_t* d_off, const uint32_t* d_adj, cudaStream_t st) {
    const uint32_t n = g.n;
    const int B = bits_for(n);
    uint64_t total_h = 0, first = 0;
    TC_CUDA(cudaMemcpyAsync(&total_h, d_off + n, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
    TC_CUDA(cudaMemcpyAsync(&first, d_off, sizeof(uint64_t), cudaMemcpyDeviceToHost, st));
    TC_CUDA(cudaStreamSynchronize(st));
    if (first != 0) return fail(TC_ERR_ARG, "CSR offsets must start at 0");
    if (total_h & 1) return fail(TC_ERR_ARG, "CSR is not symmetric (odd number of entries)");
    if (total_h >= (1ull << 32)) return fail(TC_ERR_RANGE, "more than 2^32-1 CSR entries");
    DevBuf stats;
    TC_TRY(stats.alloc(sizeof(unsigned long long) * kStats, st));
    TC_CUDA(cudaMemsetAsync(stats.p, 0, sizeof(unsigned long long) * kStats, st));
    const unsigned gridN = grid_for(n, kB, 1u << 16);
    k_check_csr<<<gridN, kB, 0, st>>>(d_off, d_adj, n, total_h, stats.as<unsigned long long>());
    TC_LAUNCH("k_check_csr");
    unsigned long long hs[8];
    TC_CUDA(cudaMemcpyAsync(hs, stats.p, sizeof(hs), cudaMemcpyDeviceToHost, st));
    TC_CUDA(cudaStreamSynchronize(st));
    if (hs[6]) return fail(TC_ERR_ARG, "CSR is not canonical (unsorted, loop, zero direction, id >= n or asymmetric)");
    uint64_t E = total_h / 2;
    DevBuf cnt, upos, ukey, udir, deg, etot;
    TC_TRY(cnt.alloc(sizeof(uint32_t) * n, st));
    TC_TRY(upos.alloc(sizeof(uint32_t) * n, st));
    TC_TRY(etot.alloc(sizeof(uint32_t), st));
    k_upper_counts<<<gridN, kB, 0, st>>>(d_off, d_adj, n, cnt.as<uint32_t>());
    TC_LAUNCH("k_upper_counts");
    TC_TRY(scan_u32(cnt.as<uint32_t>(), upos.as<uint32_t>(), n, etot.as<uint32_t>(), st));
    TC_TRY(ukey.alloc(sizeof(uint64_t) * (E ? E : 1), st));
    TC_TRY(udir.alloc(sizeof(uint32_t) * (E ? E : 1), st));
    TC_TRY(deg.alloc(sizeof(uint32_t) * n, st));
    k_csr_pairs<<<gridN, kB, 0, st>>>(d_off, d_adj, n, B, upos.as<uint32_t>(), ukey.as<uint64_t>(),
                                      udir.as<uint32_t>(), deg.as<uint32_t>(), stats.as<unsigned long long>());
    TC_LAUNCH("k_csr_pairs");
    cnt.release();
    upos.release();
    TC_TRY(finish_graph(g, E, B, ukey, udir, deg, stats, st));
    g.dups = 0;
    g.loops = 0;
    return TC_OK;
}

}  // namespace tc
