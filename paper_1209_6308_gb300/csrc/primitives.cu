// primitives.cu - device scans and a stable LSD radix sort, used by the graph builder
// (symmetrise, dedupe, relabel and sort steps of the Sec. 6 compact structure).
//
// Both read their input once per pass: a tile learns what comes before it from its predecessors
// ("decoupled look-back", Merrill and Garland 2016).  A tile publishes its own sum at once and, when
// it knows it, the sum of everything up to its end; a tile looks back over its predecessors' sums
// until it meets such an inclusive one.  Tiles are handed out by an atomic ticket, so every
// predecessor is already running and the look-back ends; after kPatience looks at one word a tile
// stops waiting and sums its predecessors' input itself.
// Scan: tiles of 4096 values, one kernel.
// Radix sort: 8-bit digits; one kernel counts every digit of every pass, then one kernel per pass
// ranks a tile's keys stably (per warp: the lanes sharing a digit, by eight ballots, against the
// running counts of its half of the warp's keys), looks back per digit, stages the tile in shared memory in digit order
// and writes contiguous runs per digit ("onesweep", Adinets and Merrill 2022).  16 bytes per key and
// pass where a histogram, a scan and a scatter per pass moved 24 in five kernels.
#include <algorithm>

#include "tc_internal.cuh"

namespace tc {
namespace {

constexpr int kScanThreads = 256;
constexpr int kScanPer = 16;
constexpr int kScanTile = kScanThreads * kScanPer;
// A pass over the 20 M keys of scale 20 takes 133 us (2.4 TB/s): issue 57%, the load/store data pipe 63%,
// DRAM a third; per issue 2.8 warps wait at a barrier, 2.3 for global loads, 2.1 for shared memory.
// (scale-25 build in ms with 512 / 384 / 256 threads of 16 keys: 139.5 / 137.3 / 147.7; 384 of 12 keys or
// __match_any_sync in place of the ballots are slower.)
constexpr int kSortThreads = 384;
constexpr int kSortWarps = kSortThreads / 32;
constexpr int kSortPer = 16;
constexpr int kSortTile = kSortThreads * kSortPer;
constexpr int kPasses = 8;                      // of 8 bits
#ifndef TC_LOOKS   // a test build sets 1, so that tiles do give up
#define TC_LOOKS (1u << 16)
#endif
constexpr uint32_t kPatience = TC_LOOKS;
constexpr int kLook = 4;   // predecessors a sort tile looks at together

// A tile's published sums: the value, and in the top bits which one it is.
constexpr unsigned long long kOwn = 1ull << 62, kUpTo = 2ull << 62, kValue = kOwn - 1ull;

__device__ __forceinline__ unsigned long long peek(const unsigned long long* p) {
    unsigned long long v;
    asm volatile("ld.relaxed.gpu.global.u64 %0, [%1];" : "=l"(v) : "l"(p) : "memory");
    return v;
}
__device__ __forceinline__ void post(unsigned long long* p, unsigned long long v) {
    asm volatile("st.relaxed.gpu.global.u64 [%0], %1;" :: "l"(p), "l"(v) : "memory");
}

template <typename T>
__device__ __forceinline__ T warp_incl_scan(T v) {
    const int lane = threadIdx.x & 31;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
        T y = __shfl_up_sync(0xffffffffu, v, o);
        if (lane >= o) v += y;
    }
    return v;
}

// Exclusive block scan of one value per thread (blockDim.x == 256 or 1024); returns the
// exclusive prefix and writes the block total to *total.
template <typename T>
__device__ __forceinline__ T block_excl_scan(T v, T* total) {
    __shared__ T warp_sums[32];
    __shared__ T s_total;
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = blockDim.x >> 5;
    T inc = warp_incl_scan(v);
    if (lane == 31) warp_sums[warp] = inc;
    __syncthreads();
    if (warp == 0) {
        T w = lane < nw ? warp_sums[lane] : T(0);
        T wi = warp_incl_scan(w);
        warp_sums[lane] = wi - w;
        if (lane == nw - 1) s_total = wi;
    }
    __syncthreads();
    T res = inc - v + warp_sums[warp];
    *total = s_total;
    __syncthreads();
    return res;
}

// state[0]: the ticket; state[1 + t]: tile t's sums (all zero before the launch).  total may be null.
template <typename Tout>
__global__ void __launch_bounds__(kScanThreads) k_scan(const uint32_t* __restrict__ in, uint64_t n, Tout* __restrict__ out,
                                                       Tout* total, unsigned long long* state) {
    __shared__ uint32_t tile_in[kScanTile];
    __shared__ unsigned long long s_before;
    __shared__ uint32_t s_tile;
    const int tid = threadIdx.x, lane = tid & 31;
    if (tid == 0) s_tile = (uint32_t)atomicAdd(state, 1ull);
    __syncthreads();
    const uint32_t tile = s_tile;
    const uint64_t base = (uint64_t)tile * kScanTile;
#pragma unroll
    for (int r = 0; r < kScanPer; ++r) {
        const uint64_t i = base + (uint64_t)r * kScanThreads + tid;
        tile_in[r * kScanThreads + tid] = i < n ? in[i] : 0u;
    }
    __syncthreads();
    // thread t owns the 16 consecutive values [16t, 16t+16) of the tile
    unsigned long long loc[kScanPer], s = 0;
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        loc[k] = s;
        s += tile_in[tid * kScanPer + k];
    }
    unsigned long long own;
    const unsigned long long ex = block_excl_scan<unsigned long long>(s, &own);
    if (tid < 32) {
        if (lane == 0) post(&state[1 + tile], (tile ? kOwn : kUpTo) | own);
        unsigned long long before = 0;
        bool gave_up = false;
        // 32 predecessors at a time, the nearest in lane 0
        for (int64_t t = (int64_t)tile - 1; t >= 0 && !gave_up; t -= 32) {
            unsigned long long v = kUpTo;   // before the first tile: nothing
            if (t - lane >= 0) {
                uint32_t looks = 0;
                while ((v = peek(&state[1 + t - lane])) < kOwn && ++looks < kPatience) {}
            }
            gave_up = __any_sync(0xffffffffu, v < kOwn);
            const uint32_t done = __ballot_sync(0xffffffffu, v >= kUpTo);
            const int last = done ? __ffs(done) - 1 : 31;   // the nearest inclusive sum ends the look-back
            unsigned long long part = lane <= last ? v & kValue : 0ull;
            for (int o = 16; o; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
            before += part;
            if (done) break;
        }
        if (lane == 0) s_before = gave_up ? ~0ull : before;
    }
    __syncthreads();
    if (s_before == ~0ull) {   // uniform: the predecessors' input itself
        unsigned long long sum = 0, all;
        for (uint64_t i = tid; i < base; i += kScanThreads) sum += in[i];
        block_excl_scan<unsigned long long>(sum, &all);
        if (tid == 0) s_before = all;
        __syncthreads();
    }
    const unsigned long long before = s_before;
    if (tid == 0) {
        if (tile) post(&state[1 + tile], kUpTo | (before + own));
        if (total && base + kScanTile >= n) *total = (Tout)(before + own);
    }
#pragma unroll
    for (int k = 0; k < kScanPer; ++k) {
        const uint64_t i = base + (uint64_t)tid * kScanPer + k;
        if (i < n) out[i] = (Tout)(before + ex + loc[k]);
    }
}

template <typename Tout>
tc_status scan_impl(const uint32_t* in, Tout* out, uint64_t n, Tout* total, cudaStream_t st) {
    if (n == 0) {
        if (total) TC_CUDA(cudaMemsetAsync(total, 0, sizeof(Tout), st));
        return TC_OK;
    }
    const uint64_t tiles = (n + kScanTile - 1) / kScanTile;
    if (tiles > 0x7fffffffull) return fail(TC_ERR_RANGE, "scan: too many elements");
    DevBuf state;
    TC_TRY(state.alloc(sizeof(unsigned long long) * (tiles + 1), st));
    TC_CUDA(cudaMemsetAsync(state.p, 0, sizeof(unsigned long long) * (tiles + 1), st));
    k_scan<Tout><<<(unsigned)tiles, kScanThreads, 0, st>>>(in, n, out, total, state.as<unsigned long long>());
    TC_LAUNCH("k_scan");
    return TC_OK;
}

// ------------------------------------------------------------------ radix sort
// hist[256 p + d] += the keys whose digit p (bits lo + 8 p and up) is d, for every pass.
__global__ void __launch_bounds__(kSortThreads) k_digit_counts(const uint64_t* __restrict__ keys, uint64_t n, int lo,
                                                               int passes, uint32_t* hist) {
    __shared__ uint32_t h[kPasses][256];
    for (int k = threadIdx.x; k < passes * 256; k += kSortThreads) (&h[0][0])[k] = 0u;
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t stride = (uint64_t)gridDim.x * kSortThreads;
    constexpr int kAhead = 4;
    for (uint64_t i0 = blockIdx.x * (uint64_t)kSortThreads + (threadIdx.x & ~31u); i0 < n; i0 += kAhead * stride) {
        uint64_t key[kAhead];
#pragma unroll
        for (int r = 0; r < kAhead; ++r) {
            const uint64_t i = i0 + r * stride + lane;
            key[r] = i < n ? keys[i] : 0ull;
        }
#pragma unroll
        for (int r = 0; r < kAhead; ++r) {
            const uint64_t i = i0 + r * stride;
            if (i >= n) break;
            const bool ok = i + lane < n;
            const uint32_t live = __ballot_sync(0xffffffffu, ok);
            for (int p = 0; p < passes; ++p) {
                const uint32_t d = (uint32_t)(key[r] >> (lo + 8 * p)) & 255u;
                const uint32_t d0 = __shfl_sync(0xffffffffu, d, 0);
                // sorted input has one digit in the whole warp: one add instead of 32 on one address
                if (__all_sync(0xffffffffu, !ok || d == d0)) {
                    if (lane == 0) atomicAdd(&h[p][d], (uint32_t)__popc(live));
                } else if (ok) {
                    atomicAdd(&h[p][d], 1u);
                }
            }
        }
    }
    __syncthreads();
    for (int k = threadIdx.x; k < passes * 256; k += kSortThreads)
        if ((&h[0][0])[k]) atomicAdd(&hist[k], (&h[0][0])[k]);
}

struct SortShared {
    uint64_t keys[kSortTile];
    uint16_t wh[2 * kSortWarps][256];   // a half warp-segment's keys per digit; then its first place in the tile
    uint32_t to[256];                   // first place of a digit of this tile in the output, less that in the tile
    uint32_t tile, gave_up;
};

// One pass: out = in stably sorted by its digit at `shift`; hist = the digit's counts, ticket and
// state (256 words per tile) as for k_scan but state words of other passes are left over: they
// carry their pass in bits 32..39 of the value.
__global__ void __launch_bounds__(kSortThreads, 3) k_radix_pass(const uint64_t* __restrict__ in, uint64_t* __restrict__ out,
                                                                uint64_t n, int shift, const uint32_t* __restrict__ hist,
                                                                uint32_t* ticket, unsigned long long* state, uint32_t pass) {
    extern __shared__ __align__(16) unsigned char raw[];
    SortShared& S = *reinterpret_cast<SortShared*>(raw);
    const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
    const uint32_t lt_mask = (1u << lane) - 1u;
    if (tid == 0) {
        S.tile = atomicAdd(ticket, 1u);
        S.gave_up = 0u;
    }
    for (int k = tid; k < kSortWarps * 256; k += kSortThreads) reinterpret_cast<uint32_t*>(&S.wh[0][0])[k] = 0u;
    __syncthreads();
    const uint32_t tile = S.tile;
    const uint64_t base = (uint64_t)tile * kSortTile, wbase = base + (uint64_t)warp * (32 * kSortPer);
    const uint32_t tile_n = n - base < (uint64_t)kSortTile ? (uint32_t)(n - base) : (uint32_t)kSortTile;
    // keys past the end read as all ones: the last of the last digit, never written
    uint64_t key[kSortPer];
#pragma unroll
    for (int r = 0; r < kSortPer; ++r) {
        const uint64_t i = wbase + 32 * r + lane;
        key[r] = i < n ? in[i] : ~0ull;
    }
    // the first and the second half of the warp's keys are ranked side by side, each against its own
    // counts: two independent chains of ballots, a count read and a count written
    uint32_t rank[kSortPer / 2];   // 16 bits each: the key's place among its half's keys of its digit
    uint16_t *w0 = S.wh[2 * warp], *w1 = S.wh[2 * warp + 1];
#pragma unroll
    for (int r = 0; r < kSortPer / 2; ++r) {
        const uint32_t d0 = (uint32_t)(key[r] >> shift) & 255u, d1 = (uint32_t)(key[r + kSortPer / 2] >> shift) & 255u;
        uint32_t p0 = 0xffffffffu, p1 = 0xffffffffu;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
            const uint32_t b0 = __ballot_sync(0xffffffffu, (d0 >> b) & 1u), b1 = __ballot_sync(0xffffffffu, (d1 >> b) & 1u);
            p0 &= ((d0 >> b) & 1u) ? b0 : ~b0;
            p1 &= ((d1 >> b) & 1u) ? b1 : ~b1;
        }
        const uint32_t c0 = w0[d0], c1 = w1[d1];
        __syncwarp();
        if ((p0 & lt_mask) == 0u) w0[d0] = (uint16_t)(c0 + __popc(p0));
        if ((p1 & lt_mask) == 0u) w1[d1] = (uint16_t)(c1 + __popc(p1));
        __syncwarp();
        rank[r] = (c0 + __popc(p0 & lt_mask)) | (c1 + __popc(p1 & lt_mask)) << 16;
    }
    __syncthreads();
    const unsigned long long mark = (unsigned long long)(pass + 1u) << 32;
    uint32_t count = 0, first = 0;
    if (tid < 256) {
#pragma unroll
        for (int w = 0; w < 2 * kSortWarps; ++w) count += S.wh[w][tid];
    }
    const uint32_t all = count;
    if (tid == 255) count -= (uint32_t)kSortTile - tile_n;
    if (tid < 256) post(&state[256ull * tile + tid], (tile ? kOwn : kUpTo) | mark | count);
    uint32_t unused;
    const uint32_t start = block_excl_scan<uint32_t>(all, &unused);
    const uint32_t digit0 = block_excl_scan<uint32_t>(tid < 256 ? hist[tid] : 0u, &unused);
    if (tid < 256) {
        uint32_t at = start;
#pragma unroll
        for (int w = 0; w < 2 * kSortWarps; ++w) {
            const uint32_t c = S.wh[w][tid];
            S.wh[w][tid] = (uint16_t)at;
            at += c;
        }
    }
    __syncthreads();
#pragma unroll
    for (int r = 0; r < kSortPer / 2; ++r) {
        S.keys[w0[(uint32_t)(key[r] >> shift) & 255u] + (rank[r] & 0xffffu)] = key[r];
        S.keys[w1[(uint32_t)(key[r + kSortPer / 2] >> shift) & 255u] + (rank[r] >> 16)] = key[r + kSortPer / 2];
    }
    if (tid < 256) {
        // kLook predecessors' words on their way at a time: many tiles run at once, so the nearest
        // inclusive sum is often tens of tiles back
        bool waits = tile != 0u;
        for (int64_t t = (int64_t)tile - 1; waits; t -= kLook) {
            unsigned long long v[kLook];
#pragma unroll
            for (int j = 0; j < kLook; ++j) v[j] = t >= j ? peek(&state[256ull * (uint64_t)(t - j) + tid]) : kUpTo | mark;
#pragma unroll
            for (int j = 0; j < kLook; ++j) {
                if (!waits) continue;
                uint32_t looks = 0;
                while ((v[j] & (0xffull << 32)) != mark && ++looks < kPatience) v[j] = peek(&state[256ull * (uint64_t)(t - j) + tid]);
                if (looks == kPatience) {
                    S.gave_up = 1u;
                    waits = false;
                }
                first += (uint32_t)v[j];
                waits = waits && v[j] < kUpTo;   // tile 0's sum is inclusive
            }
        }
    }
    __syncthreads();
    if (S.gave_up) {   // uniform: count the predecessors' keys themselves
        __shared__ uint32_t h[256];
        if (tid < 256) h[tid] = 0u;
        __syncthreads();
        for (uint64_t i = tid; i < base; i += kSortThreads) atomicAdd(&h[(uint32_t)(in[i] >> shift) & 255u], 1u);
        __syncthreads();
        if (tid < 256) first = h[tid];
    }
    if (tid < 256) {
        if (tile) post(&state[256ull * tile + tid], kUpTo | mark | (uint32_t)(first + count));
        S.to[tid] = digit0 + first - start;
    }
    __syncthreads();
    for (uint32_t i = tid; i < tile_n; i += kSortThreads) {
        const uint64_t k = S.keys[i];
        out[(uint32_t)(S.to[(uint32_t)(k >> shift) & 255u] + i)] = k;
    }
}

}  // namespace

tc_status scan_u32(const uint32_t* in, uint32_t* out, uint64_t n, uint32_t* total, cudaStream_t st) {
    return scan_impl<uint32_t>(in, out, n, total, st);
}

tc_status scan_u32_to_u64(const uint32_t* in, uint64_t* out, uint64_t n, cudaStream_t st) {
    return scan_impl<uint64_t>(in, out, n, out + n, st);
}

tc_status radix_sort_u64(uint64_t** keys, uint64_t** tmp, uint64_t n, int lo_bit, int hi_bit, cudaStream_t st) {
    if (n <= 1 || hi_bit <= lo_bit) return TC_OK;
    if (n >= (1ull << 32)) return fail(TC_ERR_RANGE, "radix sort: more than 2^32-1 keys");
    const int passes = (hi_bit - lo_bit + 7) / 8;
    if (passes > kPasses) return fail(TC_ERR_ARG, "radix sort: more than 64 bits");
    const uint64_t tiles = (n + kSortTile - 1) / kSortTile;
    // a count per digit and a ticket per pass, then the tiles' sums
    const size_t counts = sizeof(uint32_t) * 257ull * kPasses;
    DevBuf work;
    TC_TRY(work.alloc(counts + sizeof(unsigned long long) * 256ull * tiles, st));
    TC_CUDA(cudaMemsetAsync(work.p, 0, work.bytes, st));
    uint32_t* hist = work.as<uint32_t>();
    uint32_t* ticket = hist + 256 * kPasses;
    unsigned long long* state = reinterpret_cast<unsigned long long*>(work.as<unsigned char>() + counts);
    k_digit_counts<<<grid_for(n, kSortThreads * 4, 4u * (unsigned)sm_count()), kSortThreads, 0, st>>>(*keys, n, lo_bit, passes, hist);
    TC_LAUNCH("k_digit_counts");
    TC_CUDA(cudaFuncSetAttribute((const void*)k_radix_pass, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(SortShared)));
    for (int p = 0; p < passes; ++p) {
        k_radix_pass<<<(unsigned)tiles, kSortThreads, sizeof(SortShared), st>>>(*keys, *tmp, n, lo_bit + 8 * p, hist + 256 * p,
                                                                              ticket + p, state, (uint32_t)p);
        TC_LAUNCH("k_radix_pass");
        std::swap(*keys, *tmp);
    }
    return TC_OK;
}

}  // namespace tc
