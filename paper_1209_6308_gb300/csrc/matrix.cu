// matrix.cu - the matrix form of the census (paper Sec. 4 names Moody's matrix census as the
// dense way to compute it): every class count as sums of elementwise products of 0/1 dyad
// matrices with matrix products of them.  With S the one-way arcs (S[i][j] = 1 for i -> j
// only), M the mutual dyads and N the null dyads (i != j, no arc):
//   003 = sum(N o NN)/6    012 = sum(S o NN)        102 = sum(M o NN)/2
//   021D = sum(N o S'S)/2  021U = sum(N o SS')/2    021C = sum(N o SS)
//   111D = sum(S o NM)     111U = sum(S' o NM)      030T = sum(S o SS)      030C = sum(S' o SS)/3
//   201 = sum(N o MM)/2    120D = sum(M o S'S)/2    120U = sum(M o SS')/2   120C = sum(M o SS)
//   210 = sum(S o MM)      300 = sum(M o MM)/6
// (each a labelled count of the class's arc pattern over its symmetries; S' = S transposed).
// The matrices are 0/1 and held bit-packed, 64 columns per word.  A masked sum is a trace
// sum_ijk Z_ij X_ik Y_kj and can be taken over the ones of any of its three factors: at a one of
// the sparsest factor the other two meet in the popcount of one bit row AND another.  Every sum
// but 003's has S or M as a factor, so for a sparse graph k_sampled_sums takes them all in one pass
// over the connected pairs: O(e n / 64) instead of O(n^3 / 64) each.  003 has none but N: with U
// the strictly upper triangle of N, it is sum(U o (U U')), a dense product on the tensor cores
// (k_masked_product: tcgen05, 0/1 values in FP8 with FP32 accumulation, exact up to 2^24 > n), half
// of its tiles and two thirds of their depth empty by the triangle.  For a dense graph the same
// kernel takes the six products whole.  All 16 counts come from their own sums (the null count
// too), independently of the Fig. 5 method.
#include <cuda.h>

#include <cstring>

#include "graph.cuh"

namespace tc {
namespace {

constexpr uint32_t kMatrixMaxN = 1u << 14;
// the masked product's tile: kTileI x kTileJ entries, kDepth columns per stage
constexpr int kTileI = 128, kTileJ = 256, kDepth = 128, kStages = 4;
constexpr int kThreadsM = 192;   // a warp for the copies, a warp for the products, four for the sums
constexpr uint32_t kStageBytes = (kTileI + kTileJ) * kDepth;

// Bit rows of S, S', M for the relabelled graph (one warp per row), then N from them.  W words
// per row, a multiple of 2 x 64 columns; the columns past n stay 0.
__global__ void k_dyad_bits(const uint64_t* __restrict__ off, const uint32_t* __restrict__ adj, uint32_t n, uint32_t W,
                            unsigned long long* S, unsigned long long* St, unsigned long long* M) {
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t i = (blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5; i < n; i += warps) {
        const uint64_t row = i * W;
        for (uint64_t k = off[i] + lane; k < off[i + 1]; k += 32) {
            const uint32_t e = adj[k], j = e >> 2, dir = e & 3u;   // dir seen from i: 1 i->j, 2 j->i
            unsigned long long* dst = dir == 3u ? M : (dir == 1u ? S : St);
            atomicOr(&dst[row + (j >> 6)], 1ull << (j & 63u));
        }
    }
}

__global__ void k_null_bits(uint32_t n, uint32_t W, const unsigned long long* __restrict__ S,
                            const unsigned long long* __restrict__ St, const unsigned long long* __restrict__ M,
                            unsigned long long* N) {
    const uint64_t total = (uint64_t)n * W;
    for (uint64_t x = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; x < total; x += (uint64_t)gridDim.x * blockDim.x) {
        const uint32_t i = (uint32_t)(x / W), w = (uint32_t)(x % W);
        unsigned long long v = ~(S[x] | St[x] | M[x]);
        const uint32_t lo = w * 64u;
        if (lo + 64u > n) v &= (n > lo) ? ((1ull << (n - lo)) - 1ull) : 0ull;   // columns past n
        if ((i >> 6) == w) v &= ~(1ull << (i & 63u));                           // no self-dyad
        N[x] = v;
    }
}

// The sums with S or M as a factor, in the layout of the host's h[24].
constexpr int kSums = 15;
__device__ constexpr int kSumAt[kSums] = {0, 1, 4, 5, 8, 9, 12, 13, 14, 15, 16, 17, 20, 21, 22};

// A warp takes 32 consecutive list entries at a time, its lanes over the words of the rows: at an
// arc i -> k of S or a dyad of M, popcounts of a row of i AND a row of k.  i's words stay in
// registers over the entries it owns.  Bound by the popcounts (two 32-bit ones per word and sum)
// and by reading the rows of k from the L2.
__global__ void __launch_bounds__(256) k_sampled_sums(const uint64_t* __restrict__ off, const uint32_t* __restrict__ adj,
                                                      uint32_t n, uint32_t W, const unsigned long long* __restrict__ S,
                                                      const unsigned long long* __restrict__ St,
                                                      const unsigned long long* __restrict__ M,
                                                      const unsigned long long* __restrict__ N, unsigned long long* sums) {
    __shared__ unsigned long long tot[kSums];
    if (threadIdx.x < kSums) tot[threadIdx.x] = 0ull;
    __syncthreads();
    const uint32_t lane = threadIdx.x & 31;
    const uint64_t total = off[n], warps = ((uint64_t)gridDim.x * blockDim.x) >> 5;
    for (uint64_t p0 = ((blockIdx.x * (uint64_t)blockDim.x + threadIdx.x) >> 5) * 32u; p0 < total; p0 += warps * 32u) {
        const uint64_t p = p0 + lane;
        const uint32_t e = p < total ? adj[p] : 2u;   // class 2 is taken from its other end
        uint32_t lo = 0, hi = n;                      // the row of entry p: the last one with off <= p
        while (hi - lo > 1u) {
            const uint32_t mid = (lo + hi) >> 1;
            if (off[mid] <= p) lo = mid;
            else hi = mid;
        }
        const uint32_t live = __ballot_sync(0xffffffffu, (e & 3u) != 2u);
        uint32_t acc[kSums];
#pragma unroll
        for (int s = 0; s < kSums; ++s) acc[s] = 0u;
        for (uint32_t w0 = 0; w0 < W; w0 += 32u) {
            const uint32_t w = w0 + lane;
            const bool in = w < W;
            uint32_t row = 0xffffffffu;
            unsigned long long Ni = 0, Si = 0, Ti = 0, Mi = 0;
            for (uint32_t m = live; m; m &= m - 1u) {
                const int t = __ffs(m) - 1;
                const uint32_t i = __shfl_sync(0xffffffffu, lo, t), ek = __shfl_sync(0xffffffffu, e, t);
                if (i != row) {   // uniform over the warp
                    row = i;
                    const uint64_t a = (uint64_t)i * W + w;
                    Ni = in ? N[a] : 0ull;
                    Si = in ? S[a] : 0ull;
                    Ti = in ? St[a] : 0ull;
                    Mi = in ? M[a] : 0ull;
                }
                const uint64_t b = (uint64_t)(ek >> 2) * W + w;
                const unsigned long long Nk = in ? N[b] : 0ull, Mk = in ? M[b] : 0ull;
                if ((ek & 3u) == 1u) {   // uniform: i -> k
                    const unsigned long long Sk = in ? S[b] : 0ull, Tk = in ? St[b] : 0ull;
                    acc[0] += __popcll(Ni & Nk);    // S o NN
                    acc[2] += __popcll(Si & Nk);    // N o S'S
                    acc[3] += __popcll(Si & Mk);    // M o S'S
                    acc[4] += __popcll(Ni & Tk);    // N o SS'
                    acc[5] += __popcll(Mi & Tk);    // M o SS'
                    acc[6] += __popcll(Ni & Sk);    // N o SS
                    acc[7] += __popcll(Si & Sk);    // S o SS
                    acc[8] += __popcll(Ti & Sk);    // S' o SS
                    acc[9] += __popcll(Mi & Sk);    // M o SS
                    acc[10] += __popcll(Ni & Mk);   // S o NM
                    acc[11] += __popcll(Mi & Nk);   // S' o NM
                    acc[13] += __popcll(Mi & Mk);   // S o MM
                } else {                 // i <-> k
                    acc[1] += __popcll(Ni & Nk);    // M o NN
                    acc[12] += __popcll(Ni & Mk);   // N o MM
                    acc[14] += __popcll(Mi & Mk);   // M o MM
                }
            }
        }
#pragma unroll
        for (int s = 0; s < kSums; ++s) {   // at most 32 entries x n per warp: 32 bits
            const uint32_t v = __reduce_add_sync(0xffffffffu, acc[s]);
            if (lane == 0 && v) atomicAdd(&tot[s], (unsigned long long)v);
        }
    }
    __syncthreads();
    if (threadIdx.x < kSums && tot[threadIdx.x]) atomicAdd(&sums[kSumAt[threadIdx.x]], tot[threadIdx.x]);
}

// FP8 (E4M3) 0/1 rows of a bit matrix, 64 W columns; upper: only the columns past the row's own.
__global__ void k_expand_fp8(const unsigned long long* __restrict__ bits, uint64_t words, uint32_t W, bool upper,
                             uint4* out) {
    constexpr uint32_t kOne = 0x38u;   // 1.0
    for (uint64_t q = blockIdx.x * (uint64_t)blockDim.x + threadIdx.x; q < 4ull * words; q += (uint64_t)gridDim.x * blockDim.x) {
        const uint64_t x = q >> 2;
        const uint32_t i = (uint32_t)(x / W), c0 = (uint32_t)(x % W) * 64u + 16u * (uint32_t)(q & 3u);
        uint32_t b = (uint32_t)(bits[x] >> (16u * (q & 3u))) & 0xffffu;
        if (upper && i >= c0) b &= i >= c0 + 15u ? 0u : 0xfffffffeu << (i - c0);
        uint32_t v[4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
            const uint32_t f = b >> (4 * k);   // four bits to four bytes
            v[k] = ((f & 1u) | (f & 2u) << 7 | (f & 4u) << 14 | (f & 8u) << 21) * kOne;
        }
        out[q] = make_uint4(v[0], v[1], v[2], v[3]);
    }
}

// ------------------------------------------------------------------ the masked product
__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// Wait for the phase of a barrier, a bounded number of tries (each suspends for a while by itself).
__device__ __forceinline__ bool bar_wait(uint32_t bar, uint32_t parity) {
    for (uint32_t i = 0; i < (1u << 20); ++i) {
        uint32_t done;
        asm volatile("{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}"
                     : "=r"(done) : "r"(bar), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void tma_rows(uint32_t dst, const CUtensorMap* map, uint32_t col, uint32_t row, uint32_t bar) {
    asm volatile("cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3}], [%4];"
                 :: "r"(dst), "l"(map), "r"(col), "r"(row), "r"(bar) : "memory");
}

// Shared-memory operand of rows of 128 bytes in the 128-byte swizzle, 8-row groups 1024 bytes apart.
__device__ __forceinline__ uint64_t operand_desc(uint32_t addr) {
    return (uint64_t)((addr & 0x3ffffu) >> 4) | (1ull << 16) | (64ull << 32) | (1ull << 46) | (2ull << 61);
}

// sums[m] += sum over i, j < n of Z_m[i][j] (A B')[i][j], m < n_masks, for 0/1 matrices A, B (FP8 rows)
// and Z (bit rows of W words).  tri: A, B and Z are strictly upper triangles (Z's lower part is
// dropped here), so tiles below the diagonal and depths up to the tile's first j hold nothing.
struct MaskedProduct {
    CUtensorMap a, b;
    const unsigned long long* Z[4];
    uint32_t n_masks, n, W, tri;
    unsigned long long* sums;
    uint32_t* error;
};

// One 128 x 256 tile per CTA.  A warp keeps kStages stages of 128 columns of both operands on their
// way by TMA, a warp issues the products (tcgen05.mma, 128 x 256 x 32 each, accumulated in 256
// columns of tensor memory), and four warps read the tile back, a row per lane, and add the
// entries their masks select.  At n = 16384 a whole product takes 3.1 ms, 2.8 PFLOP/s; the triangle
// of 003 at n = 16001 0.47 ms with the tensor pipe 65% busy and the L2 half: the stages' 48 KB for 590
// clocks of products come from the L2.  (16-bit products would double both; 1-bit ones the tensor cores don't have.)  Every
// wait is bounded; one that runs out sets *error and the
// CTA ends without the sums.
__global__ void __launch_bounds__(kThreadsM, 1) k_masked_product(const __grid_constant__ MaskedProduct P) {
    extern __shared__ unsigned char raw[];
    __shared__ __align__(8) unsigned long long s_full[kStages], s_empty[kStages], s_done;
    __shared__ uint32_t s_tmem, s_fail;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    // in a triangle the first j tiles are the deepest, and the CTAs come in that order
    const uint32_t i0 = blockIdx.x * kTileI, jt = blockIdx.y * kTileJ;
    if (P.tri && i0 + 1u >= jt + kTileJ) return;   // no j > i in the tile (uniform over the CTA)
    const uint32_t d0 = P.tri ? jt / kDepth : 0u, d1 = P.W * 64u / kDepth;
    const uint32_t stages = (smem_u32(raw) + 1023u) & ~1023u;
    if (threadIdx.x == 0) {
        for (int s = 0; s < kStages; ++s) {
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&s_full[s])) : "memory");
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&s_empty[s])) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" :: "r"(smem_u32(&s_done)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
        s_fail = 0u;
    }
    if (warp == 1) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;"
                     :: "r"(smem_u32(&s_tmem)), "r"((uint32_t)kTileJ) : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
    const uint32_t tmem = *(volatile uint32_t*)&s_tmem;
    if (warp == 0 && lane == 0) {
        uint32_t it = 0;
        for (uint32_t d = d0; d < d1; ++d, ++it) {
            const uint32_t s = it % kStages;
            if (it >= kStages && !bar_wait(smem_u32(&s_empty[s]), (it / kStages - 1u) & 1u)) {
                *(volatile uint32_t*)&s_fail = 1u;
                break;
            }
            const uint32_t at = stages + s * kStageBytes, bar = smem_u32(&s_full[s]);
            asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" :: "r"(bar), "r"(kStageBytes) : "memory");
            tma_rows(at, &P.a, d * kDepth, i0, bar);
            tma_rows(at + kTileI * kDepth, &P.b, d * kDepth, jt, bar);
        }
        // no copy is in flight past this point, also where the products gave up
        for (uint32_t k = it > kStages ? it - kStages : 0u; k < it; ++k)
            bar_wait(smem_u32(&s_full[k % kStages]), (k / kStages) & 1u);
    } else if (warp == 1 && lane == 0) {
        // D FP32, A and B E4M3, both rows along the depth; 128 x 256
        const uint32_t idesc = (1u << 4) | ((uint32_t)(kTileJ / 8) << 17) | ((uint32_t)(kTileI / 16) << 24);
        uint32_t it = 0;
        bool ok = true;
        for (uint32_t d = d0; d < d1; ++d, ++it) {
            const uint32_t s = it % kStages;
            ok = bar_wait(smem_u32(&s_full[s]), (it / kStages) & 1u);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint64_t da = operand_desc(stages + s * kStageBytes);
            const uint64_t db = operand_desc(stages + s * kStageBytes + kTileI * kDepth);
#pragma unroll
            for (uint32_t k = 0; k < kDepth / 32; ++k) {   // 32 bytes of depth: 2 in the descriptor's address
                const uint32_t add = it != 0u || k != 0u;
                asm volatile("{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
                             "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], %1, %2, %3, p;\n}"
                             :: "r"(tmem), "l"(da + 2ull * k), "l"(db + 2ull * k), "r"(idesc), "r"(add) : "memory");
            }
            asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                         :: "r"(smem_u32(&s_empty[s])) : "memory");
        }
        if (!ok) *(volatile uint32_t*)&s_fail = 1u;
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];"
                     :: "r"(smem_u32(&s_done)) : "memory");
    }
    __syncwarp();
    if (warp >= 2) {
        const uint32_t quarter = (uint32_t)warp & 3u;   // the lanes of tensor memory a warp may read
        const bool ok = bar_wait(smem_u32(&s_done), 0u) && *(volatile uint32_t*)&s_fail == 0u;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        if (!ok) {
            if (lane == 0) atomicOr(P.error, 1u);
        } else {
            const uint32_t i = i0 + 32u * quarter + lane;
            float sum[4] = {0.f, 0.f, 0.f, 0.f};   // at most 256 entries of at most n: below 2^24
            for (uint32_t c = 0; c < kTileJ; c += 32u) {
                uint32_t v[32];
                asm volatile("tcgen05.ld.sync.aligned.32x32b.x32.b32 "
                    "{%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, "
                    "%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];"
                    : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
                      "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]),
                      "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]),
                      "=r"(v[24]), "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
                    : "r"(tmem + ((32u * quarter) << 16) + c));
                asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
                const uint32_t j = jt + c;
#pragma unroll
                for (int m = 0; m < 4; ++m) {
                    if ((uint32_t)m >= P.n_masks) break;
                    uint32_t z = 0;
                    if (i < P.n && j < P.W * 64u) z = reinterpret_cast<const uint32_t*>(P.Z[m])[(uint64_t)i * (2u * P.W) + (j >> 5)];
                    if (P.tri && i >= j) z &= i >= j + 31u ? 0u : 0xfffffffeu << (i - j);
#pragma unroll
                    for (int b = 0; b < 32; ++b) sum[m] += (z >> b) & 1u ? __uint_as_float(v[b]) : 0.f;
                }
            }
#pragma unroll
            for (int m = 0; m < 4; ++m) {
                if ((uint32_t)m >= P.n_masks) break;
                const uint32_t t = __reduce_add_sync(0xffffffffu, (uint32_t)sum[m]);   // 32 x 2^22 at most
                if (lane == 0 && t) atomicAdd(&P.sums[m], (unsigned long long)t);
            }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
    }
    __syncthreads();
    if (warp == 1) {
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" :: "r"(tmem), "r"((uint32_t)kTileJ) : "memory");
    }
}

// A map over n rows of 64 W bytes, boxes of `rows` rows and kDepth columns in the 128-byte swizzle;
// rows past n read as 0.
tc_status fp8_map(const void* p, uint32_t n, uint32_t W, uint32_t rows, CUtensorMap* map) {
    void* fn = nullptr;
    cudaDriverEntryPointQueryResult found;
    TC_CUDA(cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &fn, 12000, cudaEnableDefault, &found));
    if (found != cudaDriverEntryPointSuccess || !fn) return fail(TC_ERR_CUDA, "cuTensorMapEncodeTiled is not available");
    using Encode = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*, const cuuint64_t*,
                                const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                CUtensorMapL2promotion, CUtensorMapFloatOOBfill);
    const cuuint64_t dim[2] = {64ull * W, n}, pitch[1] = {64ull * W};
    const cuuint32_t box[2] = {(cuuint32_t)kDepth, rows}, step[2] = {1, 1};
    const CUresult r = reinterpret_cast<Encode>(fn)(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 2, const_cast<void*>(p), dim, pitch,
                                                    box, step, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                                    CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
    return r == CUDA_SUCCESS ? TC_OK : fail(TC_ERR_CUDA, "cuTensorMapEncodeTiled failed");
}

tc_status masked_product(const void* A, const void* B, MaskedProduct P, cudaStream_t st) {
    TC_TRY(fp8_map(A, P.n, P.W, kTileI, &P.a));
    TC_TRY(fp8_map(B, P.n, P.W, kTileJ, &P.b));
    const size_t smem = kStages * kStageBytes + 1024;
    TC_CUDA(cudaFuncSetAttribute((const void*)k_masked_product, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem));
    const dim3 grid((P.n + kTileI - 1) / kTileI, (P.n + kTileJ - 1) / kTileJ);
    k_masked_product<<<grid, kThreadsM, smem, st>>>(P);
    TC_LAUNCH("k_masked_product");
    return TC_OK;
}

// The sampled sums cost e n / 64 words of up to 12 popcounts, the six products their tensor work
// whatever e: random graphs with 24 e / n^2 = 0.24, 0.70, 1.36, 2.65 take, sampled / whole, 0.76 / 2.50,
// 1.74 / 2.51, 3.16 / 2.53, 5.89 / 2.54 ms at n = 8192 (the popcount products of before: 20.9) and
// 5.7 / 19.4, 14.5 / 19.2, 26.6 / 19.3, 50.6 / 19.5 at n = 16384 (166).
bool dense_pays(uint64_t n, uint64_t e) { return 24ull * e > n * n; }

}  // namespace
}  // namespace tc

using namespace tc;

extern "C" tc_status tc_census_matrix(tc_graph* g, void* stream, tc_u128 out[16]) {
    if (!g || !out) return fail(TC_ERR_ARG, "null argument");
    GraphStore& G = g->s;
    if (G.n > kMatrixMaxN)
        return fail(TC_ERR_RANGE, "tc_census_matrix: n = " + std::to_string(G.n) + " exceeds its limit of " +
                                      std::to_string(kMatrixMaxN) + " vertices");
    cudaStream_t st = (cudaStream_t)stream;
    std::unique_lock<std::mutex> lk(G.busy, std::try_to_lock);
    if (!lk.owns_lock()) return fail(TC_ERR_BUSY, "graph is in use by another call");
    const uint32_t n = G.n;
    unsigned long long h[25] = {};
    if (n >= 3) {
        const uint32_t W = (n + 127) / 128 * 2;
        const uint64_t words = (uint64_t)n * W;
        const bool dense = dense_pays(n, G.e_sym);
        // the bit rows of S, S', M and N, the sums, and an error word
        DevBuf bits, sums, fp8;
        TC_TRY(bits.alloc(sizeof(unsigned long long) * 4ull * words, st));
        TC_TRY(sums.alloc(sizeof(unsigned long long) * 25, st));
        TC_TRY(fp8.alloc(64ull * words * (dense ? 5u : 1u), st));
        unsigned long long *S = bits.as<unsigned long long>(), *St = S + words, *M = St + words, *N = M + words;
        unsigned long long* d_sums = sums.as<unsigned long long>();
        TC_CUDA(cudaMemsetAsync(S, 0, sizeof(unsigned long long) * 3ull * words, st));
        TC_CUDA(cudaMemsetAsync(sums.p, 0, sizeof(unsigned long long) * 25, st));
        if (G.e_sym) {
            k_dyad_bits<<<grid_for((uint64_t)n * 32, 256, 4096), 256, 0, st>>>(G.off.as<uint64_t>(), G.adj.as<uint32_t>(),
                                                                            n, W, S, St, M);
            TC_LAUNCH("k_dyad_bits");
        }
        k_null_bits<<<grid_for(words, 256, 8192), 256, 0, st>>>(n, W, S, St, M, N);
        TC_LAUNCH("k_null_bits");
        auto expand = [&](const unsigned long long* b, bool upper, uint32_t at) -> tc_status {
            k_expand_fp8<<<grid_for(4ull * words, 256, 1u << 16), 256, 0, st>>>(b, words, W, upper,
                                                                              fp8.as<uint4>() + 4ull * words * at);
            TC_LAUNCH("k_expand_fp8");
            return TC_OK;
        };
        MaskedProduct P;
        std::memset(&P, 0, sizeof(P));
        P.n = n;
        P.W = W;
        P.error = reinterpret_cast<uint32_t*>(d_sums + 24);
        // 003 itself: sum over i < j < k of N_ij N_jk N_ik
        TC_TRY(expand(N, true, 0));
        P.tri = 1;
        P.n_masks = 1;
        P.Z[0] = N;
        P.sums = d_sums + 2;
        TC_TRY(masked_product(fp8.p, fp8.p, P, st));
        if (!dense) {
            if (G.e_sym) {
                k_sampled_sums<<<grid_for(2ull * G.e_sym, 256, 8u * (unsigned)sm_count()), 256, 0, st>>>(
                    G.off.as<uint64_t>(), G.adj.as<uint32_t>(), n, W, S, St, M, N, d_sums);
                TC_LAUNCH("k_sampled_sums");
            }
        } else {
            // the products whole, and their masks (S' as the rows of a product's right factor means the
            // factor is S, and so on; M and N are symmetric)
            const unsigned long long* bit[4] = {S, St, M, N};
            for (uint32_t q = 0; q < 4; ++q) TC_TRY(expand(bit[q], false, q + 1u));
            enum { kS, kSt, kM, kN };
            const struct { int x, yt, z[4], masks, at; } prods[6] = {
                {kN, kN, {kS, kM}, 2, 0},             // NN:   012, 2 x 102
                {kSt, kSt, {kN, kM}, 2, 4},           // S'S:  2 x 021D, 2 x 120D
                {kS, kS, {kN, kM}, 2, 8},             // SS':  2 x 021U, 2 x 120U
                {kS, kSt, {kN, kS, kSt, kM}, 4, 12},  // SS:   021C, 030T, 3 x 030C, 120C
                {kN, kM, {kS, kSt}, 2, 16},           // NM:   111D, 111U
                {kM, kM, {kN, kS, kM}, 3, 20},        // MM:   2 x 201, 210, 6 x 300
            };
            P.tri = 0;
            for (const auto& pr : prods) {
                for (int m = 0; m < 4; ++m) P.Z[m] = m < pr.masks ? bit[pr.z[m]] : nullptr;
                P.n_masks = (uint32_t)pr.masks;
                P.sums = d_sums + pr.at;
                const uint4* f = fp8.as<uint4>();
                TC_TRY(masked_product(f + 4ull * words * (pr.x + 1), f + 4ull * words * (pr.yt + 1), P, st));
            }
        }
        TC_CUDA(cudaMemcpyAsync(h, sums.p, sizeof(h), cudaMemcpyDeviceToHost, st));
        TC_CUDA(cudaStreamSynchronize(st));
        if (h[24]) return fail(TC_ERR_TIMEOUT, "a wait of the matrix census's product kernel ran out");
    }
    const unsigned long long c[16] = {
        h[2],      h[0],      h[1] / 2,  h[4] / 2,  h[8] / 2,  h[12],     h[16],     h[17],
        h[13],     h[14] / 3, h[20] / 2, h[5] / 2,  h[9] / 2,  h[15],     h[21],     h[22] / 6};
    for (int t = 0; t < 16; ++t) out[t] = to_u128(c[t]);
    if (n < 3) out[0] = to_u128(0);
    return TC_OK;
}
