// The decoder's projections on tcgen05, with what follows them fused in:
//
//   PLAIN   y  = bf16(x W^T)                      q, k, v in one
//   RESID   h2 = h + x W^T        (fp32)          attention output, MLP output;
//                                                 without h, logits
//   SWIGLU  y  = bf16(silu(x Wg^T) * (x Wu^T))    gate and up in one
//
// x [M][K], W [N][K] bf16, both K-major; sums in fp32, rounded to bf16 only
// where stated.
//
// Few rows read W once and reuse it little: the bound is the rate at which W
// streams from HBM; from some 250 rows on it is the MMAs.  W is the 256-row
// operand of a pair of CTAs (D = W x^T: 256 rows of W by 32 to 256 rows of x),
// so few rows cost few MMAs.  Each CTA of the pair loads its 128 rows of W and
// half of x's, 64 of K at a time: an SM takes half the bytes of x from L2, and
// reads half as many from shared memory per MMA, as one CTA to a tile did
// (512 rows, gate and up of 12288 x 4096: 82 us so, 60 in pairs, 1.7 PFLOP/s;
// 2048 rows 1.97-1.99).  The grid is one pair to two SMs, each going
// through its tiles (those of the same rows of W next to one another in time)
// with two accumulators, a tile's epilogue under the next one's MMAs.  Too few
// tiles for that share K over the 2 to 4 pairs of a cluster, whose sums are
// added through distributed shared memory in share order.  Warp 0 loads by TMA
// into a ring, warp 1 of the even CTA issues the MMAs, warps 2-9 take the
// accumulator out, lanes along the features, two warps to a quarter of them.
//
// Gate and up are one operand: 16 rows of gate, 16 of up, and so on, so that a
// warp's 32 lanes hold both of 16 features and trade half their rows by a
// shuffle.
//
// The other point is the host: a library GEMM takes 20 us of host time here, a
// launch 2.5.  Against the library's GEMMs with decoder.cu's kernels between,
// two layers of a prefill (d_model 4096, F 12288, 32 heads of 128 and 8 for
// keys): 768 rows 855 -> 545 us, 1024 858 -> 682, 1536 970 -> 965, 4096 2870 ->
// 2767; d_model 5120, F 17408: 1024 1054 -> 1066, 4096 4356 -> 4227 (all before
// the smaller tiles of the last wave, see plan).  A decoder layer of 512 cells
// took 317 so, 248 with one CTA to a tile, 216 now.
//
// Every wait is bounded; one that runs out sets the error word, and every role
// leaves its loop (see decoder_error).
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "../csrc/per_device.h"
#include "../csrc/tc_ptx.cuh"
#include "decoder.h"

namespace cg = cooperative_groups;
namespace tc = splice::tc;

namespace {

using decoder::kPlain;
using decoder::kResid;
using decoder::kSwiglu;

constexpr int kFeat = 128, kBK = 64, kOutWarps = 8, kThreads = 64 + 32 * kOutWarps, kMaxStages = 8;
constexpr uint32_t kWBytes = kFeat * kBK * 2;    // 128 rows of W, one K block
constexpr uint32_t kChunkBytes = 16 * kFeat * 4;  // 16 rows' sums of a tile
constexpr int kSmemMax = 226 * 1024;
constexpr unsigned kErrLoad = 1, kErrMma = 2, kErrOut = 4, kErrDrain = 8;

__device__ unsigned g_error;

struct GemmParams {
    int M, N, K;
    int mp;                 // rows of x per tile, the MMA's columns: a multiple of 32, 256 at the most
    int tiles, tiles_m;     // of 256 rows of W (gate and up of 128 features); of mp rows of x
    int tail, tail_mp, tail_m;  // tiles of W from `tail` on are taken tail_mp rows of x at a time, tail_m times
    int kblocks, split;     // K blocks; pairs of CTAs that share them
    int clusters;           // of `split` pairs, in the grid
    int stages, bufs;       // ring; accumulators in TMEM
    uint32_t stage_bytes, tmem_cols;
    const float* h;
    void* y;
};

// g / (1 + e^-g), a quarter of both so that the divisor stays where the short
// division works: within 3 units in the last place of the exact division of
// the same.  That costs 72.2 us against 67.7 for 512 rows of 12288 x 4096, 16.9
// against 11.6 for 400 of 3072 x 1024; __expf, 67.2, is off by 2 + 1.2 |g| units.
__device__ __forceinline__ float silu(float g) { return __fdividef(0.25f * g, fmaf(0.25f, expf(-g), 0.25f)); }

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float (&v)[16]) {
    uint32_t r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, "
        "[%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    tc::tmem_wait_ld();
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

// The residual of 16 rows of x from m on (RESID), before it is needed.
template <int MODE>
__device__ __forceinline__ void load_h(const GemmParams& P, int m, int feature, float (&h)[16]) {
    if constexpr (MODE == kResid) {
#pragma unroll
        for (int e = 0; e < 16; ++e) h[e] = 0.f;
        if (!P.h || feature >= P.N || m >= P.M) return;
        const size_t at = size_t(m) * P.N + feature;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            if (m + e >= P.M) break;
            h[e] = P.h[at + size_t(e) * P.N];
        }
    }
}

// Lane's outputs for 16 rows of x from m on; `feature` per lane (SWIGLU: lanes
// 0-15 gate and 16-31 up of the same 16 features).
template <int MODE>
__device__ __forceinline__ void store16(const GemmParams& P, int m, int feature, const float (&v)[16], const float (&h)[16]) {
    // (the row test as a branch: predicated, the stores of a tile of 192 rows
    // took 2.5 us longer)
    if constexpr (MODE != kSwiglu) {
        if (feature >= P.N || m >= P.M) return;
        const size_t at = size_t(m) * P.N + feature;
#pragma unroll
        for (int e = 0; e < 16; ++e) {
            if (m + e >= P.M) break;
            if constexpr (MODE == kPlain)
                static_cast<__nv_bfloat16*>(P.y)[at + size_t(e) * P.N] = __float2bfloat16_rn(v[e]);
            else
                static_cast<float*>(P.y)[at + size_t(e) * P.N] = h[e] + v[e];
        }
    } else {
        const bool up = threadIdx.x & 16;
        float o[8];
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            const float other = __shfl_xor_sync(0xffffffffu, up ? v[e] : v[8 + e], 16);
            o[e] = silu(up ? other : v[e]) * (up ? v[8 + e] : other);
        }
        if (up) m += 8;
        if (feature >= P.N || m >= P.M) return;
        const size_t at = size_t(m) * P.N + feature;
#pragma unroll
        for (int e = 0; e < 8; ++e) {
            if (m + e >= P.M) break;
            static_cast<__nv_bfloat16*>(P.y)[at + size_t(e) * P.N] = __float2bfloat16_rn(o[e]);
        }
    }
}

// Tile t: its tile of W, first row of x and rows of x.
struct Tile {
    int n, m0, mp;
};
__device__ __forceinline__ Tile tile_of(const GemmParams& P, int t) {
    const int whole = P.tail * P.tiles_m;
    if (t < whole) return {t / P.tiles_m, t % P.tiles_m * P.mp, P.mp};
    t -= whole;
    return {P.tail + t / P.tail_m, t % P.tail_m * P.tail_mp, P.tail_mp};
}

template <int MODE, bool JOINT>
__global__ void __launch_bounds__(kThreads, 1)
    gemm_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_xt,
                const __grid_constant__ CUtensorMap tm_w, const __grid_constant__ CUtensorMap tm_w1, const GemmParams P) {
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * kMaxStages + 5];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t sbase = tc::smem_u32(smem), bar0 = tc::smem_u32(bars);
    auto full = [&](int i) { return bar0 + 8u * i; };                           // the even CTA's counts for both
    auto empty = [&](int i) { return bar0 + 8u * (kMaxStages + i); };
    auto sums = [&](int i) { return bar0 + 8u * (2 * kMaxStages + i); };        // an accumulator is complete
    auto taken = [&](int i) { return bar0 + 8u * (2 * kMaxStages + 2 + i); };   // and read out, by both CTAs (even's)
    const uint32_t drain = bar0 + 8u * (2 * kMaxStages + 4);
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    cg::cluster_group cluster = cg::this_cluster();
    const uint32_t rank = cluster.block_rank(), odd = rank & 1u, even = rank & ~1u, both = 3u << even;
    const int share = int(rank >> 1);          // of K

    if (threadIdx.x == 0) {
        for (int i = 0; i < P.stages; ++i) {
            tc::mbar_init(full(i), 1);
            tc::mbar_init(empty(i), 1);
        }
        for (int i = 0; i < 2; ++i) {
            tc::mbar_init(sums(i), 1);
            tc::mbar_init(taken(i), 2 * kOutWarps);
        }
        tc::mbar_init(drain, 1);
        s_abort = 0;
        tc::fence_mbar_init();
        tc::prefetch_tmap(&tm_x);
        tc::prefetch_tmap(&tm_w);
        if (MODE == kSwiglu) tc::prefetch_tmap(&tm_w1);
    }
    if (warp == 1) {
        tc::tmem_alloc_pair(tc::smem_u32(&s_tmem), P.tmem_cols);
        tc::tmem_relinquish_pair();
    }
    __syncwarp();
    tc::tc_fence_before();
    cluster.sync();
    tc::tc_fence_after();
    // Launched as a programmatic dependent of what precedes it on the stream:
    // everything above needs none of its results.  What follows may be
    // launched now, as it waits for this grid the same way.  (W read before
    // this wait, for the first stages, made no layer faster.)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t tmem = s_tmem;
    const int kb0 = P.kblocks * share / P.split, kb1 = P.kblocks * (share + 1) / P.split;
    const int first = int(blockIdx.x) / (2 * P.split), ntiles = P.tail * P.tiles_m + (P.tiles - P.tail) * P.tail_m;
    const uint32_t quarter = warp & 3;             // TMEM lanes this warp may read
    const uint32_t acc0 = tmem + ((quarter * 32) << 16);
    const int c_first = (warp - 2) / 4, c_step = kOutWarps / 4;   // this warp's 16-row chunks
    const int r = int(quarter) * 32 + lane;
    // this lane's feature in a tile
    const int f0 = MODE == kSwiglu ? int(odd) * 64 + int(quarter) * 16 + (lane & 15) : int(odd) * kFeat + r;
    constexpr int FEAT = MODE == kSwiglu ? kFeat : 2 * kFeat;     // features of a tile
    bool ok = true;
    constexpr int AHEAD = MODE == kResid ? 4 : 1;  // chunks whose residual is loaded ahead
    float h[AHEAD][16];

    // Both roles run as whole warps over warp-uniform values, one elected lane
    // issuing: in a one-lane branch every descriptor goes through non-uniform
    // registers (57 clocks per MMA issued).
    if (warp == 0) {
        const bool leader = tc::elect_one();
        const uint32_t lead = tc::map_cta(bar0, even);   // the even CTA's barriers, for both CTAs' loads
        int s = 0, issued = 0;
        uint32_t phase = 1;     // a fresh stage is empty
        for (int t = first; t < ntiles && ok; t += P.clusters) {
            const Tile tile = tile_of(P, t);
            const int n = tile.n, m0 = tile.m0 + int(odd) * (tile.mp / 2);
            const bool in_tail = n >= P.tail;
            const uint32_t bytes = 2 * (kWBytes + uint32_t(tile.mp) * kBK);
            for (int kb = kb0; kb < kb1; ++kb) {
                ok = __all_sync(0xffffffffu, tc::mbar_wait(empty(s), phase, &s_abort, &g_error, kErrLoad));
                if (!ok) break;
                if (leader) {
                    const uint32_t at = sbase + s * P.stage_bytes, bar = lead + 8u * s;
                    const int k = kb * kBK;
                    if (!odd) tc::mbar_arrive_expect_tx(full(s), bytes);
                    if constexpr (MODE != kSwiglu) {
                        tc::tma_load_2d_pair(at, &tm_w, k, n * FEAT + int(odd) * kFeat, bar);
                    } else if constexpr (JOINT) {
                        tc::tma_load_4d_pair(at, &tm_w, k, 0, 0, n * 8 + int(odd) * 4, bar);
                    } else {
#pragma unroll
                        for (int g = 0; g < 4; ++g) {
                            const int row = n * FEAT + int(odd) * 64 + g * 16;
                            tc::tma_load_2d_pair(at + g * 4096, &tm_w, k, row, bar);
                            tc::tma_load_2d_pair(at + g * 4096 + 2048, &tm_w1, k, row, bar);
                        }
                    }
                    tc::tma_load_2d_pair(at + kWBytes, in_tail ? &tm_xt : &tm_x, k, m0, bar);
                }
                ++issued;
                if (++s == P.stages) {
                    s = 0;
                    phase ^= 1u;
                }
            }
        }
        // Every copy issued must land before the CTAs may exit: the even CTA
        // waits for both.  (The odd one's last copies without a partner, if the
        // even CTA gave up, have had that CTA's second to land.)
        if (!odd) {
            for (int j = max(0, issued - P.stages); j < issued; ++j) {
                volatile int no_abort = 0;
                tc::mbar_wait(full(j % P.stages), uint32_t(j / P.stages) & 1u, &no_abort, &g_error, kErrDrain);
            }
        }
        // So must the even CTA's commits arrive on this CTA's barriers: the
        // sums' commit comes after the stages', but nothing says that two
        // commits arrive in their order.
        for (int j = max(0, issued - P.stages); ok && j < issued; ++j)
            ok = tc::mbar_wait(empty(j % P.stages), uint32_t(j / P.stages) & 1u, &s_abort, &g_error, kErrDrain);
    } else if (warp == 1) {
        if (!odd) {
            const bool leader = tc::elect_one();
            const uint64_t w0 = tc::sw128_desc(sbase, 16, 1024), x0 = tc::sw128_desc(sbase + kWBytes, 16, 1024);
            const uint32_t stage_step = P.stage_bytes >> 4;   // descriptor units of 16 bytes
            int s = 0, buf = 0;
            uint32_t phase = 0, taken_phase = 1;
            bool any = false;
            for (int t = first; t < ntiles && ok; t += P.clusters) {
                ok = __all_sync(0xffffffffu, tc::mbar_wait(taken(buf), taken_phase, &s_abort, &g_error, kErrMma));
                if (!ok) break;
                tc::tc_fence_after();
                const uint32_t acc = tmem + buf * P.mp;
                const uint32_t idesc = tc::idesc_bf16_f32(2 * kFeat, 0, false) | (uint32_t(tile_of(P, t).mp >> 3) << 17);
                for (int kb = kb0; kb < kb1; ++kb) {
                    ok = __all_sync(0xffffffffu, tc::mbar_wait(full(s), phase, &s_abort, &g_error, kErrMma));
                    if (!ok) break;
                    tc::tc_fence_after();
                    if (leader) {
                        const uint64_t w = w0 + s * stage_step, x = x0 + s * stage_step;
#pragma unroll
                        for (int kk = 0; kk < kBK / 16; ++kk)
                            tc::mma_f16_ss_pair(acc, w + kk * 2, x + kk * 2, idesc, kk > 0 || kb > kb0 ? 1u : 0u);
                        tc::mma_commit_pair(empty(s), both);
                    }
                    any = true;
                    if (++s == P.stages) {
                        s = 0;
                        phase ^= 1u;
                    }
                }
                if (ok && leader) tc::mma_commit_pair(sums(buf), both);
                if (++buf == P.bufs) {
                    buf = 0;
                    taken_phase ^= 1u;
                }
            }
            if (!ok && any && leader) {
                // let the MMAs already issued finish before TMEM is freed
                tc::mma_commit_pair(drain, 1u << rank);
                volatile int no_abort = 0;
                tc::mbar_wait(drain, 0, &no_abort, &g_error, kErrDrain);
            }
        }
    } else {
        int buf = 0;
        uint32_t phase = 0;
        // (with shares of K, this CTA's chunks of the cluster's one tile)
        if (P.split > 1) {
#pragma unroll
            for (int i = 0; i < AHEAD; ++i) {
                const int j = share + (c_first + i * c_step) * P.split;
                load_h<MODE>(P, 16 * j < P.mp ? first % P.tiles_m * P.mp + 16 * j : P.M, first / P.tiles_m * FEAT + f0, h[i]);
            }
        }
        for (int t = first; t < ntiles; t += P.clusters) {
            const Tile tile = tile_of(P, t);
            const int feature = tile.n * FEAT + f0, m0 = tile.m0, mp = tile.mp;
            if (P.split == 1) {
#pragma unroll
                for (int i = 0; i < AHEAD; ++i) load_h<MODE>(P, m0 + 16 * (c_first + i * c_step), feature, h[i]);
            }
            ok = __all_sync(0xffffffffu, tc::mbar_wait(sums(buf), phase, &s_abort, &g_error, kErrOut));
            if (!ok) break;
            tc::tc_fence_after();
            if (P.split > 1) break;    // the cluster's one tile: below
            for (int j = c_first; 16 * j < mp; j += AHEAD * c_step) {
#pragma unroll
                for (int i = 0; i < AHEAD; ++i) {
                    const int c = 16 * (j + i * c_step);
                    if (c >= mp) break;
                    float v[16];
                    tmem_ld16(acc0 + buf * P.mp + c, v);
                    store16<MODE>(P, m0 + c, feature, v, h[i]);
                    load_h<MODE>(P, c + 16 * AHEAD * c_step < mp ? m0 + c + 16 * AHEAD * c_step : P.M, feature, h[i]);
                }
            }
            tc::tc_fence_before();
            __syncwarp();
            if (lane == 0) tc::mbar_arrive_cluster(tc::map_cta(taken(buf), even));
            if (++buf == P.bufs) {
                buf = 0;
                phase ^= 1u;
            }
        }
    }
    __syncwarp();
    if (P.split > 1) {
        // The rows of x, 16 at a time, go round the shares: each adds up its
        // part of everyone's sums, in share order, even CTA with even, odd with
        // odd.  No CTA of the cluster has a copy or an MMA in flight any more,
        // so the ring is their inbox: [from share][part][16][128] fp32.
        float* inbox = reinterpret_cast<float*>(smem);
        const int chunks = P.mp / 16, mine = (chunks + P.split - 1) / P.split;
        constexpr int CHUNK = 16 * kFeat;
        const int feature = first / P.tiles_m * FEAT + f0, m0 = first % P.tiles_m * P.mp;
        cluster.sync();
        if (warp >= 2 && ok) {
            for (int j = c_first; j < chunks; j += c_step) {
                if (j % P.split == share) continue;
                float v[16];
                tmem_ld16(acc0 + j * 16, v);
                float* box = cluster.map_shared_rank(inbox, 2 * (j % P.split) + odd) + size_t(share * mine + j / P.split) * CHUNK + r;
#pragma unroll
                for (int e = 0; e < 16; ++e) box[e * kFeat] = v[e];
            }
        }
        cluster.sync();
        if (warp >= 2 && ok) {
            // (4 chunks a warp at the most: 256 rows over two shares and two warps)
#pragma unroll
            for (int i = 0; i < 4; ++i) {
                const int j = share + (c_first + i * c_step) * P.split;
                if (j >= chunks) break;
                float own[16], sum[16];
                tmem_ld16(acc0 + j * 16, own);
#pragma unroll
                for (int e = 0; e < 16; ++e) sum[e] = 0.f;
                for (int from = 0; from < P.split; ++from) {
                    const float* box = inbox + size_t(from * mine + j / P.split) * CHUNK + r;
#pragma unroll
                    for (int e = 0; e < 16; ++e) sum[e] += from == share ? own[e] : box[e * kFeat];
                }
                store16<MODE>(P, m0 + j * 16, feature, sum, h[i % AHEAD]);
            }
        }
    }
    __syncwarp();
    tc::tc_fence_before();
    cluster.sync();
    tc::tc_fence_after();
    if (warp == 1) tc::tmem_dealloc_pair(tmem, P.tmem_cols);
}

// [rows][K] bf16, contiguous; box of 64 x box_rows, 128-byte swizzle, zeros outside.
bool make_map(CUtensorMap* m, const void* base, int rows, int K, int box_rows) {
    decoder::EncodeFn enc = decoder::encode_fn();
    const cuuint64_t dims[2] = {cuuint64_t(K), cuuint64_t(rows)};
    const cuuint64_t strides[1] = {cuuint64_t(K) * 2};
    const cuuint32_t box[2] = {64, cuuint32_t(box_rows)}, es[2] = {1, 1};
    return enc && enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Gate and up [rows][K] bf16 each as one operand: boxes of 4 groups of 16 rows
// of gate and the same 16 of up.  See joint().
bool make_map_joint(CUtensorMap* m, const void* gate, const void* up, int rows, int K) {
    decoder::EncodeFn enc = decoder::encode_fn();
    const cuuint64_t dims[4] = {cuuint64_t(K), 16, 2, cuuint64_t(rows / 16)};
    const cuuint64_t strides[3] = {cuuint64_t(K) * 2, cuuint64_t(static_cast<const char*>(up) - static_cast<const char*>(gate)),
                                   cuuint64_t(K) * 32};
    const cuuint32_t box[4] = {64, 16, 2, 4}, es[4] = {1, 1, 1, 1};
    return enc && enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void*>(gate), dims, strides, box, es,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Clusters of 1 to 4 pairs that are resident together.
struct Resident {
    int n[4];
};

// A K block of 64 for mp rows of x, in clocks.
double block_clocks(int mp) { return std::max(2.0 * mp, (16384.0 + 64.0 * mp) / 75.0) + 20.0; }

// The launch's shape (host arithmetic only): tiles of 32 to 256 rows of x and
// shares of K, of the least time in clocks by what a K block of 64 takes (2 per
// row of x in MMAs, or its bytes at the 75 a clock that an SM gets from L2),
// whole waves of tiles and 6000 for adding up shares.  At 512 rows that is two
// tiles of 256 for 12288 gates (2.5 waves of 76 pairs) and three of 192 for 6144
// features (72 tiles).
void plan(int mode, GemmParams& p, const int (&resident)[4]) {
    const int feat = mode == kSwiglu ? kFeat : 2 * kFeat;
    p.tiles = (p.N + feat - 1) / feat;
    p.kblocks = (p.K + kBK - 1) / kBK;
    p.tail = p.tiles;
    p.tail_mp = 32;
    p.tail_m = 1;
    double least = 0;
    GemmParams best = p;
    for (int mp = 256; mp >= 32; mp -= 32) {
        if (mp - 32 >= p.M) continue;
        GemmParams c = p;
        c.mp = mp;
        c.tiles_m = (p.M + mp - 1) / mp;
        c.stage_bytes = kWBytes + uint32_t(c.mp) * kBK;
        c.stages = std::min(kMaxStages, int((kSmemMax - 1024) / c.stage_bytes));
        const long tiles = long(c.tiles) * c.tiles_m;
        for (c.split = 1; c.split <= 4; ++c.split) {
            if (c.split > 1 && (tiles > resident[c.split - 1] || c.kblocks < 2 * c.split)) break;
            c.clusters = int(std::min(tiles, long(resident[0])));
            c.bufs = tiles > c.clusters ? 2 : 1;
            c.tmem_cols = 32;
            while (c.tmem_cols < uint32_t(c.mp * c.bufs)) c.tmem_cols *= 2;
            const double clocks = double((tiles + c.clusters - 1) / c.clusters) * block_clocks(c.mp) * c.kblocks / c.split +
                                  8.0 * c.mp / c.split + (c.split > 1 ? 6000.0 : 0.0);
            if (least == 0 || clocks < least) {
                least = clocks;
                best = c;
            }
        }
        // The tiles past the last whole wave, in smaller ones that make up
        // one wave (4096 deep, gate and up of 12288: 512 rows, 2.53 waves, 63.7
        // -> 61.8 us; 1024, 5.05 waves, 117.9 -> 111.9; 6144 features, 2048
        // rows 60.9 -> 56.1; 4096 by 12288 deep, 2048 rows 136 -> 122).
        c.split = 1;
        c.clusters = resident[0];
        const long waves = tiles / c.clusters;
        if (waves < 1 || tiles % c.clusters == 0) continue;
        c.tail = int(waves * c.clusters / c.tiles_m);
        c.bufs = 2;
        c.tmem_cols = 32;
        while (c.tmem_cols < uint32_t(c.mp * c.bufs)) c.tmem_cols *= 2;
        for (c.tail_mp = 32; c.tail_mp < mp; c.tail_mp += 32) {
            c.tail_m = (p.M + c.tail_mp - 1) / c.tail_mp;
            if (long(c.tail) * c.tiles_m + long(c.tiles - c.tail) * c.tail_m > (waves + 1) * c.clusters) continue;
            const double clocks = (waves * block_clocks(mp) + block_clocks(c.tail_mp)) * c.kblocks + 8.0 * mp;
            if (clocks < least) {
                least = clocks;
                best = c;
            }
            break;
        }
    }
    p = best;
}

// Whether two weight matrices can be one operand of make_map_joint: whole
// groups of 16 rows and up behind gate, as the halves of one matrix are (else
// a stage takes eight loads of 16 rows).
bool joint(const void* gate, const void* up, int rows) {
    const intptr_t d = static_cast<const char*>(up) - static_cast<const char*>(gate);
    return rows % 16 == 0 && d > 0 && d % 16 == 0 && d < intptr_t(1) << 40;
}

template <int MODE, bool JOINT>
int launch(const void* x, const void* w0, const void* w1, GemmParams p, cudaStream_t st) {
    static splice::PerDevice<Resident> kept;
    Resident resident;
    const cudaError_t e = kept.get(&resident, [](int, Resident* r) {
        cudaError_t err = cudaFuncSetAttribute(gemm_kernel<MODE, JOINT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
        for (int i = 0; i < 4 && err == cudaSuccess; ++i) {
            cudaLaunchConfig_t cfg = {};
            cfg.gridDim = dim3(2u * (i + 1));
            cfg.blockDim = dim3(kThreads);
            cfg.dynamicSmemBytes = kSmemMax;
            cudaLaunchAttribute attr;
            attr.id = cudaLaunchAttributeClusterDimension;
            attr.val.clusterDim.x = 2u * (i + 1);
            attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
            cfg.attrs = &attr;
            cfg.numAttrs = 1;
            err = cudaOccupancyMaxActiveClusters(&r->n[i], gemm_kernel<MODE, JOINT>, &cfg);
        }
        r->n[0] = std::max(r->n[0], 1);
        return err;
    });
    if (e != cudaSuccess) return int(e);
    plan(MODE, p, resident.n);
    CUtensorMap mx, mt, m0, m1;
    if (!make_map(&mx, x, p.M, p.K, p.mp / 2)) return int(cudaErrorInvalidValue);
    mt = mx;
    if (p.tail < p.tiles && !make_map(&mt, x, p.M, p.K, p.tail_mp / 2)) return int(cudaErrorInvalidValue);
    if (!(JOINT ? make_map_joint(&m0, w0, w1, p.N, p.K) : make_map(&m0, w0, p.N, p.K, MODE == kSwiglu ? 16 : kFeat)))
        return int(cudaErrorInvalidValue);
    m1 = m0;
    if (MODE == kSwiglu && !JOINT && !make_map(&m1, w1, p.N, p.K, 16)) return int(cudaErrorInvalidValue);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(p.clusters) * 2u * unsigned(p.split));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = size_t(p.stages) * p.stage_bytes + 1024;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = 2u * unsigned(p.split);
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return int(cudaLaunchKernelEx(&cfg, gemm_kernel<MODE, JOINT>, mx, mt, m0, m1, p));
}

}  // namespace

namespace decoder {

EncodeFn encode_fn() {
    static EncodeFn fn = [] {
        void* p = nullptr;
        cudaDriverEntryPointQueryResult q;
        if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault, &q) != cudaSuccess ||
            q != cudaDriverEntryPointSuccess)
            p = nullptr;
        return reinterpret_cast<EncodeFn>(p);
    }();
    return fn;
}

unsigned* error_word() {
    void* p = nullptr;
    return cudaGetSymbolAddress(&p, g_error) == cudaSuccess ? static_cast<unsigned*>(p) : nullptr;
}

bool gemm_takes(int M, int N, int K) {
    // TMA rows are multiples of 16 bytes.
    return M >= 1 && M <= 65536 && N >= 1 && K >= 8 && K % 8 == 0;
}

int gemm(int mode, const void* x, const void* w0, const void* w1, const void* h, void* y, int M, int N, int K,
         cudaStream_t st) {
    if (!gemm_takes(M, N, K)) return int(cudaErrorInvalidValue);
    GemmParams p{};
    p.M = M;
    p.N = N;
    p.K = K;
    p.h = static_cast<const float*>(h);
    p.y = y;
    if (mode == kPlain) return launch<kPlain, false>(x, w0, nullptr, p, st);
    if (mode == kResid) return launch<kResid, false>(x, w0, nullptr, p, st);
    return joint(w0, w1, N) ? launch<kSwiglu, true>(x, w0, w1, p, st) : launch<kSwiglu, false>(x, w0, w1, p, st);
}

}  // namespace decoder

extern "C" {

// mode 0: y bf16 [M][N] = x w0^T; 1: y fp32 [M][N] = h + x w0^T (h NULL: 0); 2: y bf16
// [M][N] = silu(x w0^T) * (x w1^T).  All contiguous, 16-byte aligned; shapes
// that gemm_takes.  Returns a cudaError_t.
int decoder_gemm(int mode, const void* x, const void* w0, const void* w1, const void* h, void* y, int M, int N, int K,
                 void* stream) {
    if (mode < 0 || mode > 2) return int(cudaErrorInvalidValue);
    return decoder::gemm(mode, x, w0, w1, h, y, M, N, K, static_cast<cudaStream_t>(stream));
}

// The shape a launch would take where `resident` clusters of 1 to 4 pairs of
// CTAs are resident together, for tests (no CUDA call): out = {rows of x per
// tile, K blocks, shares of K, tiles of W, tiles of rows of x, clusters, ring
// stages, bytes per stage, TMEM columns, accumulators, bytes of the sums traded,
// shared memory, tiles of W before the tail, the tail's rows of x per tile, and
// tiles of rows of x}.
int decoder_gemm_plan(int mode, int M, int N, int K, const int* resident, long* out) {
    if (mode < 0 || mode > 2 || resident[0] < 1 || !decoder::gemm_takes(M, N, K)) return int(cudaErrorInvalidValue);
    GemmParams p{};
    p.M = M;
    p.N = N;
    p.K = K;
    const int r[4] = {resident[0], resident[1], resident[2], resident[3]};
    plan(mode, p, r);
    const long traded = p.split > 1 ? long(p.split) * ((p.mp / 16 + p.split - 1) / p.split) * kChunkBytes : 0;
    const long v[15] = {p.mp, p.kblocks, p.split, p.tiles, p.tiles_m, p.clusters, p.stages, long(p.stage_bytes),
                        long(p.tmem_cols), p.bufs, traded, long(p.stages) * long(p.stage_bytes) + 1024, p.tail, p.tail_mp, p.tail_m};
    for (int i = 0; i < 15; ++i) out[i] = v[i];
    return 0;
}

// The error word of the current device's launches (a wait ran out), and
// clears it; synchronises the device.
int decoder_error(unsigned* word) {
    const unsigned zero = 0;
    cudaError_t e = cudaDeviceSynchronize();    // (the copy waits for blocking streams only)
    if (e == cudaSuccess) e = cudaMemcpyFromSymbol(word, g_error, sizeof zero);
    if (e == cudaSuccess && *word) e = cudaMemcpyToSymbol(g_error, &zero, sizeof zero);
    return int(e);
}

}  // extern "C"
