// census64.cu - the 64-state triad census (Sec. 3, Fig. 2): how many triads are in each of the
// 64 labelled states, before isomorphic states are merged into the 16 classes.  A triad's
// actors take the roles (x, y, z) in increasing vertex id of the caller's labels, and the state
// has the tricode's bits: 1 y->x, 2 x->y, 4 y->z, 8 z->y, 16 x->z, 32 z->x.
//
// Every triad is counted by its links, in bulk where its state allows it:
//   - two links (a wedge with centre c): the state depends only on the two links' direction
//     classes seen from c and on where the ends' ids fall against c's.  With c's neighbours
//     sorted by the caller's ids, ordered class-pair counts among the neighbours below c
//     (c is z), among those above c (c is x), and the products of the class counts below and
//     above (c is y) count every pair of neighbours of c once;
//   - three links (a triangle): found once each by the triangle walk of triangles.cu, its
//     state read in the caller's id order.  Each triangle was also counted as a wedge at each
//     of its three vertices: those three are taken back;
//   - one link (a pair (a, b), a < b, and a third vertex linked to neither): the third vertex
//     below a, between or above b puts the link in the roles (y,z), (x,z) or (x,y).  Per pair
//     the three ranges hold a, b - a - 1 and n - 1 - b vertices; summed per direction class,
//     less the triads with more links that hold the same link in the same roles;
//   - no link: C(n,3) less the rest (128-bit).
// The sorted neighbour lists in caller ids come from one radix sort of (caller id of the row,
// caller id of the neighbour) keys of the stored lists.
#include <algorithm>
#include <cstring>
#include <vector>

#include "graph.cuh"
#include "rows.cuh"

namespace tc {
namespace {

// old[new_of_old[x]] = x: the original id of each stored vertex
__global__ void k_old_of(const uint32_t* __restrict__ new_of_old, uint32_t n, uint32_t* old) {
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < n; x += (uint64_t)gridDim.x * blockDim.x)
        old[new_of_old[x]] = (uint32_t)x;
}

// deg_old[x] = the degree of the vertex with caller id x
__global__ void k_deg_old(const uint64_t* __restrict__ off, const uint32_t* __restrict__ new_of_old, uint32_t n,
                          uint32_t* deg_old) {
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < n; x += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t r = new_of_old[x];
        deg_old[x] = (uint32_t)(off[r + 1] - off[r]);
    }
}

// One key per stored entry (row r, neighbour s): (old[r] << (B + 2)) | (old[s] << 2) | dir, with
// dir seen from r (1 r->s, 2 s->r).  The entries of the n_wide rows of more than 32 come first:
// kKeyChunk of them to a warp; then a warp takes 32 rows (rows.cuh).
constexpr uint32_t kKeyChunk = 1024;
__global__ void __launch_bounds__(256) k_keys64(GraphDev g, uint32_t n_wide, const uint32_t* __restrict__ old, int B,
                                                uint64_t* keys) {
    __shared__ uint8_t s_at[8][32];
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t stride = (uint64_t)gridDim.x * blockDim.x;
    auto put = [&](uint64_t row, uint64_t k) {
        const uint32_t x = g.adj[k];
        keys[k] = row << (B + 2) | ((uint64_t)old[x >> 2] << 2) | (x & 3u);
    };
    const uint64_t wide = g.off[n_wide];
    for (uint64_t k0 = ((blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5) * kKeyChunk; k0 < wide;
         k0 += (stride >> 5) * kKeyChunk) {
        const uint64_t end = k0 + kKeyChunk < wide ? k0 + kKeyChunk : wide;
        uint32_t r = 0, hi = n_wide;   // the row of entry k0: the last one with off <= k0
        while (hi - r > 1u) {
            const uint32_t mid = (r + hi) >> 1;
            if (g.off[mid] <= k0) r = mid;
            else hi = mid;
        }
        for (uint64_t k = k0; k < end; ++r) {
            const uint64_t e = g.off[r + 1] < end ? g.off[r + 1] : end, row = old[r];
#pragma unroll 4
            for (uint64_t i = k + lane; i < e; i += 32) put(row, i);
            k = e;
        }
    }
    for (uint64_t x0 = n_wide + blockIdx.x * (uint64_t)blockDim.x + (threadIdx.x & ~31u); x0 < g.n; x0 += stride) {
        const bool ok = x0 + lane < g.n;
        const uint64_t base = ok ? g.off[x0 + lane] : 0ull;
        const uint32_t deg = ok ? (uint32_t)(g.off[x0 + lane + 1] - base) : 0u, mine = ok ? old[x0 + lane] : 0u;
        for_rows(deg, s_at[threadIdx.x >> 5],
            [&](const PackedEntry& p) {
                const uint64_t row = __shfl_sync(0xffffffffu, mine, p.row), b = __shfl_sync(0xffffffffu, base, p.row);
                if (p.valid) put(row, b + (lane - p.first));
            },
            [](uint32_t) {});
    }
}

// The raw sums, per class pair (d1, d2), d = 1..3 (index 3 (d1-1) + d2-1):
//   raw[0..9)   PB: pairs p < q < c of neighbours of c, class(p) = d1, class(q) = d2 (c is z)
//   raw[9..18)  PA: pairs c < p < q                                         (c is x)
//   raw[18..27) X:  (neighbours below c of class d1) x (above c of class d2)  (c is y)
//   raw[27..36) R:  per pair (a, b), a < b, of direction class k = d1 (1 a->b, 2 b->a, 3 both):
//               position d2 = 1 above b (n - 1 - b), 2 between (b - a - 1), 3 below a (a)
// Classes are seen from c (1 c->nbr, 2 nbr->c).
struct Wedges {
    unsigned long long pb[3][3] = {}, pa[3][3] = {}, xx[3][3] = {}, rr[3][3] = {};

    // One block of entries: this lane's key of centre c (n vertices, ids of B bits), its row's lanes, and
    // the counts of the row's earlier blocks by side and class, which it advances.
    __device__ __forceinline__ void block(bool valid, uint64_t key, uint32_t c, uint32_t n, int B, uint32_t lanes,
                                          uint32_t (&rb)[3], uint32_t (&ra)[3]) {
        const uint32_t lt = (1u << (threadIdx.x & 31u)) - 1u;
        const uint32_t nb = (uint32_t)((key >> 2) & ((1ull << B) - 1ull)), d = (uint32_t)(key & 3ull);
        const bool below = valid && nb < c, above = valid && nb > c;
#pragma unroll
        for (int q1 = 0; q1 < 3; ++q1) {
            const uint32_t bb = __ballot_sync(0xffffffffu, below && d == (uint32_t)(q1 + 1)) & lanes;
            const uint32_t ba = __ballot_sync(0xffffffffu, above && d == (uint32_t)(q1 + 1)) & lanes;
            const uint32_t before_b = rb[q1] + __popc(bb & lt), before_a = ra[q1] + __popc(ba & lt);
#pragma unroll
            for (int q2 = 0; q2 < 3; ++q2) {
                if (below && d == (uint32_t)(q2 + 1)) pb[q1][q2] += before_b;
                if (above && d == (uint32_t)(q2 + 1)) pa[q1][q2] += before_a;
            }
            rb[q1] += __popc(bb);
            ra[q1] += __popc(ba);
        }
        if (above) {
            const unsigned long long vals[3] = {(unsigned long long)n - 1ull - nb, (unsigned long long)(nb - c - 1u),
                                                (unsigned long long)c};
#pragma unroll
            for (int q1 = 0; q1 < 3; ++q1)
                if (d == (uint32_t)(q1 + 1))
#pragma unroll
                    for (int q2 = 0; q2 < 3; ++q2) rr[q1][q2] += vals[q2];
        }
    }
    // A row's counts below and above its centre (one lane per row).
    __device__ __forceinline__ void products(const uint32_t (&rb)[3], const uint32_t (&ra)[3]) {
#pragma unroll
        for (int q1 = 0; q1 < 3; ++q1)
#pragma unroll
            for (int q2 = 0; q2 < 3; ++q2) xx[q1][q2] += (unsigned long long)rb[q1] * ra[q2];
    }
    __device__ __forceinline__ void flush(unsigned long long* raw) const {
#pragma unroll
        for (int q1 = 0; q1 < 3; ++q1)
#pragma unroll
            for (int q2 = 0; q2 < 3; ++q2) {
                const unsigned long long v[4] = {pb[q1][q2], pa[q1][q2], xx[q1][q2], rr[q1][q2]};
#pragma unroll
                for (int t = 0; t < 4; ++t) {
                    unsigned long long s = v[t];
                    for (int o = 16; o; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
                    if ((threadIdx.x & 31u) == 0 && s) atomicAdd(&raw[9 * t + 3 * q1 + q2], s);
                }
            }
    }
};

// Rows of at most kHubDeg entries: a warp over `rows` <= 32 vertices (caller ids, rows.cuh); the rows of
// more than 32 entries go one after another, so a small graph's warps take fewer vertices (the caller).
// The warps' 36 sums meet in shared memory first: as global atomics of every warp they took longer than
// the rows did.  64-state census of G(1024, 0.1) with 32 rows to a warp 0.274 ms, so 0.202.
__global__ void __launch_bounds__(256) k_wedges64(const uint64_t* __restrict__ keys, const uint64_t* __restrict__ off_old,
                                                  uint32_t n, uint32_t rows, int B, unsigned long long* raw) {
    __shared__ uint8_t s_at[8][32];
    __shared__ unsigned long long s_raw[36];
    if (threadIdx.x < 36u) s_raw[threadIdx.x] = 0ull;
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    Wedges W;
    for (uint64_t x0 = ((blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5) * rows; x0 < n; x0 += warps * rows) {
        const bool ok = lane < rows && x0 + lane < n;
        const uint64_t vb = ok ? off_old[x0 + lane] : 0ull;
        const uint32_t vd = ok ? (uint32_t)(off_old[x0 + lane + 1] - vb) : 0u;
        for_rows(vd > kHubDeg ? 0u : vd, s_at[threadIdx.x >> 5],
            [&](const PackedEntry& p) {
                const uint64_t b = __shfl_sync(0xffffffffu, vb, p.row);
                uint32_t rb[3] = {0u, 0u, 0u}, ra[3] = {0u, 0u, 0u};
                const uint64_t key = p.valid ? keys[b + (lane - p.first)] : 0ull;
                W.block(p.valid, key, (uint32_t)x0 + p.row, n, B, p.lanes, rb, ra);
                if (p.valid && lane == p.first) W.products(rb, ra);   // the row's totals
            },
            [&](uint32_t row) {
                const uint64_t b = __shfl_sync(0xffffffffu, vb, row);
                const uint32_t d = __shfl_sync(0xffffffffu, vd, row);
                uint32_t rb[3] = {0u, 0u, 0u}, ra[3] = {0u, 0u, 0u};
                uint64_t next = keys[b + lane];   // more than 32 entries
                for (uint32_t k0 = 0; k0 < d; k0 += 32) {
                    const uint64_t key = next;
                    const uint32_t k = k0 + lane;
                    next = k + 32u < d ? keys[b + k + 32u] : 0ull;
                    W.block(k < d, key, (uint32_t)x0 + row, n, B, 0xffffffffu, rb, ra);
                }
                if (lane == 0) W.products(rb, ra);
            });
    }
    W.flush(s_raw);
    __syncthreads();
    if (threadIdx.x < 36u && s_raw[threadIdx.x]) atomicAdd(&raw[threadIdx.x], s_raw[threadIdx.x]);
}

// The longer rows, those of the first n_hub stored vertices: a CTA each, its warps over segments of the
// row from the counts of the segments before.  (One warp per row made the largest hub's 65 k entries
// the kernel's length: scale 20 1.16 ms.)
__global__ void __launch_bounds__(256) k_wedges64_hub(const uint64_t* __restrict__ keys, const uint64_t* __restrict__ off_old,
                                                      const uint32_t* __restrict__ old, uint32_t n_hub, uint32_t n, int B,
                                                      unsigned long long* raw) {
    __shared__ uint32_t s_cnt[8][6];
    const uint32_t lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const uint64_t idmask = (1ull << B) - 1ull;
    Wedges W;
    for (uint32_t r = blockIdx.x; r < n_hub; r += gridDim.x) {
        const uint32_t c = old[r];
        const uint64_t b = off_old[c];
        const uint32_t d = (uint32_t)(off_old[c + 1] - b), seg = ((d + 7u) / 8u + 31u) & ~31u;
        const uint32_t s0 = min(d, warp * seg), s1 = min(d, s0 + seg);
        uint32_t cnt[6] = {0u, 0u, 0u, 0u, 0u, 0u};   // below by class, above by class
#pragma unroll 4
        for (uint32_t k = s0 + lane; k < s1; k += 32) {
            const uint64_t key = keys[b + k];
            const uint32_t q = (uint32_t)(key & 3ull) + ((uint32_t)((key >> 2) & idmask) < c ? 0u : 3u);
#pragma unroll
            for (uint32_t i = 0; i < 6; ++i) cnt[i] += q == i + 1u;
        }
#pragma unroll
        for (uint32_t i = 0; i < 6; ++i) {
            cnt[i] = __reduce_add_sync(0xffffffffu, cnt[i]);
            if (lane == 0) s_cnt[warp][i] = cnt[i];
        }
        __syncthreads();
        uint32_t rb[3] = {0u, 0u, 0u}, ra[3] = {0u, 0u, 0u};
        for (uint32_t w = 0; w < warp; ++w)
#pragma unroll
            for (uint32_t i = 0; i < 3; ++i) {
                rb[i] += s_cnt[w][i];
                ra[i] += s_cnt[w][3 + i];
            }
        uint64_t next = s0 + lane < s1 ? keys[b + s0 + lane] : 0ull;
        for (uint32_t k0 = s0; k0 < s1; k0 += 32) {
            const uint64_t key = next;
            const uint32_t k = k0 + lane;
            next = k + 32u < s1 ? keys[b + k + 32u] : 0ull;
            W.block(k < s1, key, c, n, B, 0xffffffffu, rb, ra);
        }
        if (warp == 7u && lane == 0) W.products(rb, ra);   // the last segment ends with the row's totals
        __syncthreads();   // the counts are read before the next row writes its own
    }
    W.flush(raw);
}

// states of wedges and one-link triads (see the file comment); d = direction class seen
// from the centre (1 centre->end, 2 end->centre)
inline uint32_t st_center_z(uint32_t d1, uint32_t d2) {   // ends p < q < c: p = x, q = y
    return (d1 & 2u ? 16u : 0u) | (d1 & 1u ? 32u : 0u) | (d2 & 2u ? 4u : 0u) | (d2 & 1u ? 8u : 0u);
}
inline uint32_t st_center_x(uint32_t d1, uint32_t d2) {   // c < p < q: p = y, q = z
    return (d1 & 1u ? 2u : 0u) | (d1 & 2u ? 1u : 0u) | (d2 & 1u ? 16u : 0u) | (d2 & 2u ? 32u : 0u);
}
inline uint32_t st_center_y(uint32_t dp, uint32_t dq) {   // p < c < q: p = x, q = z
    return (dp & 2u ? 2u : 0u) | (dp & 1u ? 1u : 0u) | (dq & 1u ? 4u : 0u) | (dq & 2u ? 8u : 0u);
}

// The state of a triangle tricode (roles (a, b, c) of the walk) once its actors are ordered by
// caller id: rank pattern 3 ra + rb (ra, rb = the ranks of a and b, c's is the rest).
std::vector<uint8_t> perm_states() {
    // bit b of a tricode is the arc kArc[b] between the roles a = 0, b = 1, c = 2; in sorted
    // roles x = 0, y = 1, z = 2 the arc (i -> j) has the state bit kBit[i][j]
    const int kArc[6][2] = {{1, 0}, {0, 1}, {1, 2}, {2, 1}, {0, 2}, {2, 0}};
    const int kBit[3][3] = {{0, 2, 16}, {1, 0, 4}, {32, 8, 0}};
    std::vector<uint8_t> t(9 * 64, 0);
    for (int ra = 0; ra < 3; ++ra)
        for (int rb = 0; rb < 3; ++rb) {
            if (ra == rb) continue;
            const int rank[3] = {ra, rb, 3 - ra - rb};
            for (int code = 0; code < 64; ++code) {
                int s = 0;
                for (int b = 0; b < 6; ++b)
                    if (code >> b & 1) s |= kBit[rank[kArc[b][0]]][rank[kArc[b][1]]];
                t[(3 * ra + rb) * 64 + code] = (uint8_t)s;
            }
        }
    return t;
}

}  // namespace
}  // namespace tc

using namespace tc;

extern "C" {

tc_status tc_census64(tc_graph* g, void* stream, tc_u128 out[64]) {
    if (!g || !out) return fail(TC_ERR_ARG, "null argument");
    cudaStream_t st = (cudaStream_t)stream;
    std::unique_lock<std::mutex> lk(g->s.busy, std::try_to_lock);
    if (!lk.owns_lock()) return fail(TC_ERR_BUSY, "graph is in use by another call");
    GraphStore& G = g->s;
    unsigned long long raw[36] = {}, tri[64] = {};
    if (G.e_sym) {
        int B = 1;
        while (B < 32 && (1ull << B) < G.n) ++B;
        const uint64_t E2 = 2ull * G.e_sym;
        DevBuf old, deg, offo, keys, tmp, acc, perm;
        TC_TRY(old.alloc(sizeof(uint32_t) * G.n, st));
        TC_TRY(deg.alloc(sizeof(uint32_t) * G.n, st));
        TC_TRY(offo.alloc(sizeof(uint64_t) * (G.n + 1ull), st));
        TC_TRY(keys.alloc(sizeof(uint64_t) * E2, st));
        TC_TRY(tmp.alloc(sizeof(uint64_t) * E2, st));
        TC_TRY(acc.alloc(sizeof(unsigned long long) * (36 + 64), st));
        TC_TRY(perm.alloc(9 * 64, st));
        const std::vector<uint8_t> ps = perm_states();
        TC_CUDA(cudaMemcpyAsync(perm.p, ps.data(), ps.size(), cudaMemcpyHostToDevice, st));
        TC_CUDA(cudaMemsetAsync(acc.p, 0, sizeof(unsigned long long) * (36 + 64), st));
        const GraphDev gd = G.dev();
        k_old_of<<<grid_for(G.n, 256, 4096), 256, 0, st>>>(G.new_of_old.as<uint32_t>(), G.n, old.as<uint32_t>());
        TC_LAUNCH("k_old_of");
        k_deg_old<<<grid_for(G.n, 256, 4096), 256, 0, st>>>(gd.off, G.new_of_old.as<uint32_t>(), G.n,
                                                            deg.as<uint32_t>());
        TC_LAUNCH("k_deg_old");
        TC_TRY(scan_u32_to_u64(deg.as<uint32_t>(), offo.as<uint64_t>(), G.n, st));
        k_keys64<<<grid_for(std::max<uint64_t>(G.n, E2 / (kKeyChunk / 32)), 256, 1u << 16), 256, 0, st>>>(gd, G.n_wide, old.as<uint32_t>(), B,
                                                                          keys.as<uint64_t>());
        TC_LAUNCH("k_keys64");
        uint64_t* kp = keys.as<uint64_t>();
        uint64_t* tp = tmp.as<uint64_t>();
        TC_TRY(radix_sort_u64(&kp, &tp, E2, 2, 2 * B + 2, st));
        unsigned long long* d_raw = acc.as<unsigned long long>();
        const unsigned wgrid = 4u * (unsigned)sm_count();
        uint32_t rows = 32;
        while (rows > 1u && (uint64_t)G.n < 8ull * wgrid * rows) rows /= 2u;   // as long as warps are left over
        k_wedges64<<<grid_for((G.n + rows - 1ull) / rows * 32u, 256, wgrid), 256, 0, st>>>(kp, offo.as<uint64_t>(), G.n, rows,
                                                                                         B, d_raw);
        TC_LAUNCH("k_wedges64");
        if (G.n_hub) {
            k_wedges64_hub<<<grid_for(256ull * G.n_hub, 256, 2u * (unsigned)sm_count()), 256, 0, st>>>(
                kp, offo.as<uint64_t>(), old.as<uint32_t>(), G.n_hub, G.n, B, d_raw);
            TC_LAUNCH("k_wedges64_hub");
        }
        // triangles, in caller-id states, through the triangle form's plan
        tc_options to;
        std::memset(&to, 0, sizeof(to));
        to.algo = TC_ALGO_TRIANGLE;
        to.chunk_entries = 1024;
        to.ctas_per_sm = 5;   // the caller-id hash doubles the shared memory of a CTA
        Opts o;
        TC_TRY(resolve_opts(&to, nullptr, &o));
        Plan* p = nullptr;
        TC_TRY(get_plan(G, o, st, &p));
        TC_CUDA(cudaMemsetAsync(G.ctr.p, 0, sizeof(uint32_t) * 4, st));
        TC_TRY(triangles_launch(gd, o, p->items.as<Item>(), p->n_items, p->warp_begin, p->warp_end,
                                G.ctr.as<uint32_t>(), old.as<uint32_t>(), perm.as<uint8_t>(), d_raw + 36, nullptr, st));
        unsigned long long h[100];
        TC_CUDA(cudaMemcpyAsync(h, acc.p, sizeof(h), cudaMemcpyDeviceToHost, st));
        TC_CUDA(cudaStreamSynchronize(st));
        std::memcpy(raw, h, sizeof(raw));
        std::memcpy(tri, h + 36, sizeof(tri));
    }
    // assemble the states in 128-bit signed arithmetic
    __int128 C[64] = {};
    for (uint32_t d1 = 1; d1 <= 3; ++d1)
        for (uint32_t d2 = 1; d2 <= 3; ++d2) {
            const uint32_t i = 3 * (d1 - 1) + (d2 - 1);
            C[st_center_z(d1, d2)] += raw[i];
            C[st_center_x(d1, d2)] += raw[9 + i];
            C[st_center_y(d1, d2)] += raw[18 + i];
        }
    for (uint32_t t = 0; t < 64; ++t) {
        if (!tri[t]) continue;
        C[t] += tri[t];
        C[t & ~3u] -= tri[t];    // the wedge at z (x-y unlinked)
        C[t & ~12u] -= tri[t];   // at x (y-z unlinked)
        C[t & ~48u] -= tri[t];   // at y (x-z unlinked)
    }
    // one link: per direction class k of the pair (a, b), the range counts less the connected
    // triads holding that link in those roles
    __int128 S[64] = {};
    for (uint32_t s = 0; s < 64; ++s) S[s] = C[s];
    for (uint32_t k = 1; k <= 3; ++k) {
        const uint32_t ab = k & 1u, ba = k >> 1;
        const uint32_t s_above = (ab ? 2u : 0u) | (ba ? 1u : 0u);      // roles (x, y)
        const uint32_t s_between = (ab ? 16u : 0u) | (ba ? 32u : 0u);  // roles (x, z)
        const uint32_t s_below = (ab ? 4u : 0u) | (ba ? 8u : 0u);      // roles (y, z)
        __int128 a = raw[27 + 3 * (k - 1) + 0], b = raw[27 + 3 * (k - 1) + 1], c = raw[27 + 3 * (k - 1) + 2];
        for (uint32_t s = 0; s < 64; ++s) {
            if (!C[s]) continue;
            if ((s & 3u) == s_above) a -= C[s];
            if ((s & 48u) == s_between) b -= C[s];
            if ((s & 12u) == s_below) c -= C[s];
        }
        S[s_above] += a;
        S[s_between] += b;
        S[s_below] += c;
    }
    __int128 rest = 0;
    for (int s = 1; s < 64; ++s) rest += S[s];
    out[0] = to_u128(choose3(G.n) - (unsigned __int128)rest);
    for (int s = 1; s < 64; ++s) out[s] = to_u128((unsigned __int128)S[s]);
    return TC_OK;
}

}  // extern "C"
