// The decoder's projections of few rows on tcgen05, with what follows them
// fused in:
//
//   PLAIN   y  = bf16(x W^T)                      q, k, v in one
//   RESID   h2 = h + x W^T        (fp32)          attention output, MLP output
//   SWIGLU  y  = bf16(silu(x Wg^T) * (x Wu^T))    gate and up in one
//
// x [M][K], W [N][K] bf16, both K-major; sums in fp32, rounded to bf16 only
// where stated.
//
// So few rows read W once and reuse it little: the bound is the rate at which
// W streams from HBM.  W is the 128-row operand (a CTA makes 128 output
// features for all rows of x: D = W x^T), so one MMA takes 4 KB of W whatever
// M is, and the K dimension is shared out over a cluster of CTAs until every
// SM streams; the CTAs add their accumulators through distributed shared
// memory in rank order.  (With x as the 128-row operand the same kernel was
// held up by its MMA issue: 32 to 64 rows of W per MMA.)  Warp 0 loads 64-wide K
// blocks by TMA into a ring, warp 1 issues the MMAs, warps 2-9 take the
// accumulator out, lanes along the features, two warps to a quarter of them.
//
// The point beside the fusion is the host: a library GEMM takes 20 us of host
// time here, a launch 2.5, and with few rows the GPU is done sooner.  So 128
// rows, or as many as the GPU takes no longer for (see gemm_takes), come here;
// larger batches stay with the library, whose kernels reuse both operands.  A
// layer of 78 cells (d_model 1888) takes 115 us where the library's GEMMs and
// the kernels of decoder.cu between them took about 300 and torch's
// expressions 1034.  Alone, on cold weights, 16 rows: 6144 x 4096 12.4 us, 4.1
// TB/s (the library 10.1), gate and up of 12288 x 4096 with SwiGLU 37.2, 5.4
// TB/s (31.9 and the SwiGLU kernel).
//
// Every wait is bounded; one that runs out sets the error word, and every role
// leaves its loop (see decoder_error).
#include <cooperative_groups.h>
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "../csrc/tc_ptx.cuh"
#include "decoder.h"

namespace cg = cooperative_groups;
namespace tc = splice::tc;

namespace {

using decoder::kPlain;
using decoder::kResid;
using decoder::kSwiglu;

constexpr int kFeat = 128, kBK = 64, kOutWarps = 8, kThreads = 64 + 32 * kOutWarps, kMaxStages = 8, kMaxSplit = 8;
constexpr uint32_t kWBytes = kFeat * kBK * 2;    // 128 rows of W, one K block
constexpr uint32_t kChunkBytes = 16 * kFeat * 4;  // 16 rows' sums of a tile
constexpr int kSmemMax = 226 * 1024;
constexpr unsigned kErrLoad = 1, kErrMma = 2, kErrOut = 4, kErrDrain = 8;

__device__ unsigned g_error;

struct GemmParams {
    int M, N, K;
    int mp;                 // rows of x per CTA, the MMA's columns: a multiple of 16, 256 at the most
    int ctas_per_sm;        // 2 up to 128 rows, else 1
    int tiles_m;            // of mp rows
    int kblocks, split;     // K blocks; CTAs that share them
    int stages;
    int tiles;              // of 128 features
    uint32_t stage_bytes, tmem_cols;
    const float* h;
    void* y;
};

// (a few units of 2^-24 off, far inside the output's bf16 rounding; the exact
// division and expf cost a tile of 144 rows 3.4 us of its epilogue warps)
__device__ __forceinline__ float silu(float g) { return __fdividef(g, 1.f + __expf(-g)); }

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

// One feature's outputs for 16 rows of x from row m on (lanes: consecutive features).
template <int MODE>
__device__ __forceinline__ void store16(const GemmParams& P, int m, int feature, const float (&v)[16], const float (&u)[16]) {
    if (feature >= P.N || m >= P.M) return;
    const size_t at = size_t(m) * P.N + feature;
    float h[16];
    if constexpr (MODE == kResid) {
#pragma unroll
        for (int e = 0; e < 16; ++e) h[e] = m + e < P.M ? P.h[at + size_t(e) * P.N] : 0.f;   // (all loads before any store)
    }
#pragma unroll
    for (int e = 0; e < 16; ++e) {
        if (m + e >= P.M) break;
        if constexpr (MODE == kResid)
            static_cast<float*>(P.y)[at + size_t(e) * P.N] = h[e] + v[e];
        else
            static_cast<__nv_bfloat16*>(P.y)[at + size_t(e) * P.N] =
                __float2bfloat16_rn(MODE == kSwiglu ? silu(v[e]) * u[e] : v[e]);
    }
}

template <int MODE>
__global__ void __launch_bounds__(kThreads, 2)
    gemm_kernel(const __grid_constant__ CUtensorMap tm_x, const __grid_constant__ CUtensorMap tm_w0,
                const __grid_constant__ CUtensorMap tm_w1, const GemmParams P) {
    constexpr int PARTS = MODE == kSwiglu ? 2 : 1;     // W matrices, accumulators
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[2 * kMaxStages + 2];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
    const uint32_t sbase = tc::smem_u32(smem), bar0 = tc::smem_u32(bars);
    auto full = [&](int i) { return bar0 + 8u * i; };
    auto empty = [&](int i) { return bar0 + 8u * (kMaxStages + i); };
    const uint32_t done = bar0 + 8u * (2 * kMaxStages), drain = done + 8u;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = P.split > 1 ? int(cluster.block_rank()) : 0;

    if (threadIdx.x == 0) {
        for (int i = 0; i < P.stages; ++i) {
            tc::mbar_init(full(i), 1);
            tc::mbar_init(empty(i), 1);
        }
        tc::mbar_init(done, 1);
        tc::mbar_init(drain, 1);
        s_abort = 0;
        tc::fence_mbar_init();
        tc::prefetch_tmap(&tm_x);
        tc::prefetch_tmap(&tm_w0);
        if (MODE == kSwiglu) tc::prefetch_tmap(&tm_w1);
    }
    if (warp == 1) {
        tc::tmem_alloc(tc::smem_u32(&s_tmem), P.tmem_cols);
        tc::tmem_relinquish();
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    // Launched as a programmatic dependent of what precedes it on the stream:
    // everything above needs none of its results.  What follows may be
    // launched now, as it waits for this grid the same way.
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t tmem = s_tmem;
    const int kb0 = P.kblocks * rank / P.split, kb1 = P.kblocks * (rank + 1) / P.split;
    const int n0 = int(blockIdx.x) / P.split * kFeat, m0 = int(blockIdx.y) * P.mp;
    constexpr uint32_t x_at = PARTS * kWBytes;     // a stage: W (, the other W), x

    // Both roles run as whole warps over warp-uniform values, one elected lane
    // issuing: in a one-lane branch every descriptor goes through non-uniform
    // registers (57 clocks per MMA issued).
    if (warp == 0) {
        const bool leader = tc::elect_one();
        int s = 0, issued = 0;
        uint32_t phase = 1;     // a fresh stage is empty
        const uint32_t bytes = PARTS * kWBytes + uint32_t(P.mp) * kBK * 2;
        for (int kb = kb0; kb < kb1; ++kb) {
            if (!__all_sync(0xffffffffu, tc::mbar_wait(empty(s), phase, &s_abort, &g_error, kErrLoad))) break;
            if (leader) {
                const uint32_t at = sbase + s * P.stage_bytes, bar = full(s);
                const int k = kb * kBK;
                tc::mbar_arrive_expect_tx(bar, bytes);
                tc::tma_load_2d(at, &tm_w0, k, n0, bar);
                if (MODE == kSwiglu) tc::tma_load_2d(at + kWBytes, &tm_w1, k, n0, bar);
                tc::tma_load_2d(at + x_at, &tm_x, k, m0, bar);
            }
            ++issued;
            if (++s == P.stages) {
                s = 0;
                phase ^= 1u;
            }
        }
        // every copy issued must land before the CTA may exit
        for (int j = max(0, issued - P.stages); j < issued; ++j) {
            volatile int no_abort = 0;
            tc::mbar_wait(full(j % P.stages), uint32_t(j / P.stages) & 1u, &no_abort, &g_error, kErrDrain);
        }
    } else if (warp == 1) {
        const bool leader = tc::elect_one();
        const uint32_t idesc = tc::idesc_bf16_f32(kFeat, 0, false) | (uint32_t(P.mp >> 3) << 17);
        const uint64_t w0 = tc::sw128_desc(sbase, 16, 1024), x0 = tc::sw128_desc(sbase + x_at, 16, 1024);
        const uint32_t stage_step = P.stage_bytes >> 4;   // descriptor units of 16 bytes
        int s = 0;
        uint32_t phase = 0;
        bool ok = true, any = false;
        for (int kb = kb0; kb < kb1; ++kb) {
            if (!__all_sync(0xffffffffu, tc::mbar_wait(full(s), phase, &s_abort, &g_error, kErrMma))) {
                ok = false;
                break;
            }
            tc::tc_fence_after();
            if (leader) {
                const uint64_t w = w0 + s * stage_step, x = x0 + s * stage_step;
                const uint32_t acc = kb > kb0 ? 1u : 0u;
#pragma unroll
                for (int kk = 0; kk < kBK / 16; ++kk)
#pragma unroll
                    for (int part = 0; part < PARTS; ++part)
                        tc::mma_f16_ss(tmem + part * P.mp, w + part * (kWBytes / 16) + kk * 2, x + kk * 2, idesc,
                                       kk == 0 ? acc : 1u);
                tc::mma_commit(empty(s));
            }
            any = true;
            if (++s == P.stages) {
                s = 0;
                phase ^= 1u;
            }
        }
        if (ok && leader) tc::mma_commit(done);
        if (!ok && any && leader) {
            // let the MMAs already issued finish before TMEM is freed
            tc::mma_commit(drain);
            volatile int no_abort = 0;
            tc::mbar_wait(drain, 0, &no_abort, &g_error, kErrDrain);
        }
    }
    __syncwarp();
    const int quarter = warp & 3;                  // TMEM lanes this warp may read
    const int r = quarter * 32 + lane, feature = n0 + r;
    const uint32_t acc = tmem + (uint32_t(quarter * 32) << 16);
    const bool out = warp >= 2;
    const int c_first = (warp - 2) / 4, c_step = kOutWarps / 4;   // this warp's 16-row chunks
    bool ok = true;
    if (out) ok = __all_sync(0xffffffffu, tc::mbar_wait(done, 0, &s_abort, &g_error, kErrOut));
    tc::tc_fence_after();
    if (P.split == 1) {
        if (out && ok) {
            for (int c = 16 * c_first; c < P.mp; c += 16 * c_step) {
                float v[16], u[16];
                tmem_ld16(acc + c, v);
                if (MODE == kSwiglu) tmem_ld16(acc + P.mp + c, u);
                store16<MODE>(P, m0 + c, feature, v, u);
            }
        }
    } else {
        // The rows of x, 16 at a time, go round the ranks: each adds up its
        // share of everyone's sums, in rank order.  No CTA of the cluster has
        // a copy or an MMA in flight any more, so the ring is their inbox:
        // [from rank][share][part][16][128 features] fp32.
        float* inbox = reinterpret_cast<float*>(smem);
        const int chunks = P.mp / 16, mine = (chunks + P.split - 1) / P.split;
        constexpr int CHUNK = 16 * kFeat;
        cluster.sync();
        if (out && ok) {
            for (int j = c_first; j < chunks; j += c_step) {
                if (j % P.split == rank) continue;
                float* box = cluster.map_shared_rank(inbox, j % P.split) + size_t(rank * mine + j / P.split) * PARTS * CHUNK + r;
#pragma unroll
                for (int part = 0; part < PARTS; ++part) {
                    float v[16];
                    tmem_ld16(acc + part * P.mp + j * 16, v);
#pragma unroll
                    for (int e = 0; e < 16; ++e) box[part * CHUNK + e * kFeat] = v[e];
                }
            }
        }
        cluster.sync();
        if (out && ok) {
            for (int j = rank + c_first * P.split; j < chunks; j += c_step * P.split) {
                float sum[PARTS][16];
#pragma unroll
                for (int part = 0; part < PARTS; ++part) {
                    float own[16];
                    tmem_ld16(acc + part * P.mp + j * 16, own);
#pragma unroll
                    for (int e = 0; e < 16; ++e) sum[part][e] = 0.f;
#pragma unroll 2
                    for (int from = 0; from < P.split; ++from) {
                        const float* box = inbox + (size_t(from * mine + j / P.split) * PARTS + part) * CHUNK + r;
#pragma unroll
                        for (int e = 0; e < 16; ++e) sum[part][e] += from == rank ? own[e] : box[e * kFeat];
                    }
                }
                store16<MODE>(P, m0 + j * 16, feature, sum[0], sum[PARTS - 1]);
            }
        }
    }
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == 1) tc::tmem_dealloc(tmem, P.tmem_cols);
}

using EncodeFn = CUresult (*)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                              const cuuint64_t*, const cuuint32_t*, const cuuint32_t*, CUtensorMapInterleave,
                              CUtensorMapSwizzle, CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

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

// [rows][K] bf16, contiguous; box of 64 x box_rows, 128-byte swizzle, zeros outside.
bool make_map(CUtensorMap* m, const void* base, int rows, int K, int box_rows) {
    EncodeFn enc = encode_fn();
    const cuuint64_t dims[2] = {cuuint64_t(K), cuuint64_t(rows)};
    const cuuint64_t strides[1] = {cuuint64_t(K) * 2};
    const cuuint32_t box[2] = {64, cuuint32_t(box_rows)}, es[2] = {1, 1};
    return enc && enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(base), dims, strides, box, es,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Ring and split of tiles of p.mp rows (host arithmetic only).
void plan_tiles(int mode, GemmParams& p, int sms) {
    const int parts = mode == kSwiglu ? 2 : 1;
    p.tiles_m = (p.M + p.mp - 1) / p.mp;
    p.ctas_per_sm = p.mp <= 128 ? 2 : 1;
    p.stage_bytes = parts * kWBytes + uint32_t(p.mp) * kBK * 2;
    p.stages = std::min(kMaxStages, int((kSmemMax / p.ctas_per_sm - 1024) / p.stage_bytes));
    p.tmem_cols = 32;
    while (p.tmem_cols < uint32_t(p.mp * parts)) p.tmem_cols *= 2;
    // CTAs per tile: as many as are resident together (clusters do not pack
    // the SMs whole, hence the eighth left over), each with two K blocks
    // at least, and few enough that the ring holds the sums they trade.
    const int room = p.ctas_per_sm * sms * 7 / 8;
    p.split = std::max(1, std::min(std::min(kMaxSplit, int(room / (long(p.tiles) * p.tiles_m))), p.K / (2 * kBK)));
    const int chunks = p.mp / 16;
    while (p.split > 1 && uint32_t(p.split * ((chunks + p.split - 1) / p.split) * parts) * kChunkBytes >
                              uint32_t(p.stages) * p.stage_bytes)
        --p.split;
}

// The launch's shape (host arithmetic only).  Up to 128 rows one tile of rows
// (W streams from HBM once).  More rows are bound by the MMAs, a tile of 256
// rows and a K block of 64 taking 640 clocks: even tiles of 128 to 256 rows,
// of the least time in whole waves (512 rows, gate and up of 12288: 96 tiles
// of features by two of rows are 1.26 waves of 256 rows, by three 1.9 of 176).
void plan(int mode, GemmParams& p, int sms) {
    p.tiles = (p.N + kFeat - 1) / kFeat;
    p.kblocks = (p.K + kBK - 1) / kBK;
    GemmParams best = p;
    double least = 0;
    for (int tm = (p.M + 255) / 256; tm <= (p.M + 127) / 128; ++tm) {
        GemmParams c = p;
        c.mp = ((p.M + tm - 1) / tm + 15) / 16 * 16;
        plan_tiles(mode, c, sms);
        const long ctas = long(c.tiles) * c.tiles_m * c.split, at_once = long(c.ctas_per_sm) * sms;
        const double block = (mode == kSwiglu ? 2 : 1) * 2.5 * c.mp + 130.0;
        const double clocks = double((ctas + at_once - 1) / at_once) *
                                  (c.ctas_per_sm * block * c.kblocks / c.split + 6000.0) + (c.split > 1 ? 5000.0 : 0.0);
        if (least == 0 || clocks < least) {
            least = clocks;
            best = c;
        }
    }
    p = best;
}

template <int MODE>
int launch(const void* x, const void* w0, const void* w1, GemmParams p, cudaStream_t st) {
    static const int sms = [] {
        int dev = 0, n = 0;
        cudaFuncSetAttribute(gemm_kernel<MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
        cudaGetDevice(&dev);
        cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
        return n > 0 ? n : 1;
    }();
    plan(MODE, p, sms);
    CUtensorMap mx, m0, m1;
    if (!make_map(&mx, x, p.M, p.K, p.mp) || !make_map(&m0, w0, p.N, p.K, kFeat)) return int(cudaErrorInvalidValue);
    if (MODE == kSwiglu) {
        if (!make_map(&m1, w1, p.N, p.K, kFeat)) return int(cudaErrorInvalidValue);
    } else {
        m1 = m0;
    }
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(p.tiles) * unsigned(p.split), unsigned(p.tiles_m));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = size_t(p.stages) * p.stage_bytes + 1024;
    cfg.stream = st;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = unsigned(p.split);
    attr[1].val.clusterDim.y = attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return int(cudaLaunchKernelEx(&cfg, gemm_kernel<MODE>, mx, m0, m1, p));
}

}  // namespace

namespace decoder {

bool gemm_takes(int M, int N, int K) {
    // TMA rows are multiples of 16 bytes.
    if (M < 1 || M > 65536 || N < 1 || K < 8 || K % 8 != 0) return false;
    return M <= kGemmRows || (M + 255L) / 256 * N * K * 2 <= 64L << 20;
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
    if (mode == kPlain) return launch<kPlain>(x, w0, nullptr, p, st);
    if (mode == kResid) return launch<kResid>(x, w0, nullptr, p, st);
    return launch<kSwiglu>(x, w0, w1, p, st);
}

}  // namespace decoder

extern "C" {

// mode 0: y bf16 [M][N] = x w0^T; 1: y fp32 [M][N] = h + x w0^T; 2: y bf16
// [M][N] = silu(x w0^T) * (x w1^T).  All contiguous, 16-byte aligned; shapes
// that gemm_takes.  Returns a cudaError_t.
int decoder_gemm(int mode, const void* x, const void* w0, const void* w1, const void* h, void* y, int M, int N, int K,
                 void* stream) {
    if (mode < 0 || mode > 2) return int(cudaErrorInvalidValue);
    return decoder::gemm(mode, x, w0, w1, h, y, M, N, K, static_cast<cudaStream_t>(stream));
}

// The shape a launch on `sms` multiprocessors would take, for tests (no CUDA
// call): out = {x rows per MMA, K blocks, CTAs per tile, tiles, ring stages,
// bytes per stage, TMEM columns, bytes of the sums traded, shared memory, tiles
// of rows of x}.
int decoder_gemm_plan(int mode, int M, int N, int K, int sms, long* out) {
    if (mode < 0 || mode > 2 || sms < 1 || !decoder::gemm_takes(M, N, K)) return int(cudaErrorInvalidValue);
    GemmParams p{};
    p.M = M;
    p.N = N;
    p.K = K;
    plan(mode, p, sms);
    const int chunks = p.mp / 16;
    const long traded = p.split > 1 ? long(p.split) * ((chunks + p.split - 1) / p.split) * (mode == kSwiglu ? 2 : 1) * kChunkBytes : 0;
    const long v[10] = {p.mp, p.kblocks, p.split, p.tiles, p.stages, long(p.stage_bytes), long(p.tmem_cols), traded,
                       long(p.stages) * long(p.stage_bytes) + 1024, p.tiles_m};
    for (int i = 0; i < 10; ++i) out[i] = v[i];
    return 0;
}

// The error word of the current device's launches (a wait ran out), and
// clears it; synchronises.
int decoder_error(unsigned* word) {
    const unsigned zero = 0;
    cudaError_t e = cudaMemcpyFromSymbol(word, g_error, sizeof zero);
    if (e == cudaSuccess && *word) e = cudaMemcpyToSymbol(g_error, &zero, sizeof zero);
    return int(e);
}

}  // extern "C"
