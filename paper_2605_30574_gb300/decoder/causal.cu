// Causal attention of one sequence over itself, for the prefill: q [T][Hq][d],
// k, v [Hkv][T][d], out [T][Hq][d], all bf16; scores, sums and outputs in fp32,
// probabilities rounded to bf16 for their product with V (a tensor-core
// operand).
//
// A CTA takes 128 rows of one query head, on tcgen05, over key blocks of 64:
// S = Q K^T into one of two TMEM slots, softmax by four warps (a thread per
// row), P over S in its slot as the A operand of P V, O in TMEM.  The next
// block's Q K^T is issued before a block's softmax is waited for, and two CTAs
// share an SM (d <= 128), so that MMAs of one run under the softmax of the
// other; that softmax, 64 exponentials per thread and block at a quarter of a
// warp per clock, is the bound.  Tiles of many blocks come first, the heads of a
// kv head next to one another.  O is rescaled where a row's maximum grows, so
// that the largest weight is 1 exactly (left up to 2^8 behind, 7% faster but 3%
// further from 64 bits).  32 heads of 128, 8 for keys, against the flash kernel
// that torch picks: 256 tokens 7.2 us, 16.2; 1024 22.9, 53.4; 4096 143, 427; no
// further from 64 bits at any size.
//
// Every wait is bounded, as in gemm.cu.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "../csrc/per_device.h"
#include "../csrc/tc_ptx.cuh"
#include "decoder.h"

namespace tc = splice::tc;

namespace {

constexpr int kRows = 128, kBN = 64, kThreads = 192;     // softmax: warps 0-3
constexpr int kLoadWarp = 4, kMmaWarp = 5;
constexpr unsigned kErrLoad = 16, kErrMma = 32, kErrOut = 64, kErrDrain = 128;

template <int D>
struct Cfg {
    static constexpr int PANELS = D / 64;
    static constexpr uint32_t Q_BYTES = kRows * D * 2, KV_BYTES = kBN * D * 2;
    static constexpr uint32_t OFF_K = Q_BYTES, OFF_V = OFF_K + 2 * KV_BYTES, BYTES = OFF_V + 2 * KV_BYTES;
    static constexpr int CTAS = D == 256 ? 1 : 2;        // per SM, by TMEM (and no third by shared memory)
    static constexpr uint32_t SMEM = (BYTES + 1024 > 80 * 1024 ? BYTES + 1024 : 80 * 1024);
    static constexpr uint32_t COL_O = 2 * kBN;
    static constexpr uint32_t TMEM = D == 256 ? 512 : 256;
    static_assert(COL_O + D <= TMEM && CTAS * TMEM <= 512 && (CTAS + 1) * (SMEM + 1024) > 228 * 1024);
};

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// A = P (bf16 pairs, in TMEM), B = V (smem descriptor).
__device__ __forceinline__ void mma_f16_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc, uint32_t accumulate) {
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], [%1], %2, %3, p;\n\t}" ::"r"(d_tmem),
        "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
        : "memory");
}

__device__ __forceinline__ void tma_load_3d(uint32_t dst, const void* tmap, int32_t x, int32_t y, int32_t z, uint32_t bar) {
    asm volatile(
        "cp.async.bulk.tensor.3d.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
        "l"(tmap), "r"(x), "r"(y), "r"(z), "r"(bar)
        : "memory");
}

// 32 columns of this thread's lane, complete when it returns (one statement, so
// that nothing that uses the values can be moved between load and wait).
__device__ __forceinline__ void tmem_ld32_done(uint32_t taddr, float (&v)[32]) {
    uint32_t r[32];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%32];\n\t"
        "tcgen05.wait::ld.sync.aligned;"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
        : "r"(taddr)
        : "memory");
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

template <int D>
__global__ void __launch_bounds__(kThreads, Cfg<D>::CTAS)
    causal_kernel(const __grid_constant__ CUtensorMap tm_q, const __grid_constant__ CUtensorMap tm_k,
                  const __grid_constant__ CUtensorMap tm_v, __nv_bfloat16* out, int T, int Hq, int G, float scale_log2,
                  unsigned* err) {
    using C = Cfg<D>;
    extern __shared__ uint8_t smem_raw[];
    __shared__ __align__(8) uint64_t bars[15];
    __shared__ uint32_t s_tmem;
    __shared__ volatile int s_abort;
    const uint32_t sbase = (tc::smem_u32(smem_raw) + 1023) & ~1023u, bar0 = tc::smem_u32(bars);
    const uint32_t qfull = bar0, pvdone = bar0 + 8, drain = bar0 + 16;
    auto kfull = [&](int i) { return bar0 + 24 + 8u * i; };
    auto vfull = [&](int i) { return bar0 + 40 + 8u * i; };
    auto kempty = [&](int i) { return bar0 + 56 + 8u * i; };
    auto vempty = [&](int i) { return bar0 + 72 + 8u * i; };
    auto sfull = [&](int i) { return bar0 + 88 + 8u * i; };
    auto pfull = [&](int i) { return bar0 + 104 + 8u * i; };
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int head = int(blockIdx.x) % Hq, row0 = ((T + kRows - 1) / kRows - 1 - int(blockIdx.x) / Hq) * kRows;
    const int nblk = (min(T, row0 + kRows) + kBN - 1) / kBN;

    if (threadIdx.x == 0) {
        for (int i = 0; i < 13; ++i) tc::mbar_init(bar0 + 8u * i, 1);
        for (int i = 0; i < 2; ++i) tc::mbar_init(pfull(i), kRows);
        s_abort = 0;
        tc::fence_mbar_init();
        tc::prefetch_tmap(&tm_q);
        tc::prefetch_tmap(&tm_k);
        tc::prefetch_tmap(&tm_v);
    }
    if (warp == kMmaWarp) {
        tc::tmem_alloc(tc::smem_u32(&s_tmem), C::TMEM);
        tc::tmem_relinquish();
    }
    __syncwarp();
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    // (a programmatic dependent of what precedes it, as the other kernels are)
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    const uint32_t tmem = s_tmem;

    if (warp == kLoadWarp) {
        const bool leader = tc::elect_one();
        const int hk = head / G;
        if (leader) {
            tc::mbar_arrive_expect_tx(qfull, C::Q_BYTES);
#pragma unroll
            for (int p = 0; p < C::PANELS; ++p) tma_load_3d(sbase + p * (kRows * 128), &tm_q, p * 64, head, row0, qfull);
        }
        int j = 0;
        for (; j < nblk; ++j) {
            const int s = j & 1;
            const uint32_t phase = (uint32_t(j >> 1) & 1u) ^ 1u;
            if (!__all_sync(0xffffffffu, tc::mbar_wait(kempty(s), phase, &s_abort, err, kErrLoad))) break;
            if (leader) {
                tc::mbar_arrive_expect_tx(kfull(s), C::KV_BYTES);
#pragma unroll
                for (int p = 0; p < C::PANELS; ++p)
                    tma_load_3d(sbase + C::OFF_K + s * C::KV_BYTES + p * (kBN * 128), &tm_k, p * 64, j * kBN, hk, kfull(s));
            }
            if (!__all_sync(0xffffffffu, tc::mbar_wait(vempty(s), phase, &s_abort, err, kErrLoad))) break;
            if (leader) {
                tc::mbar_arrive_expect_tx(vfull(s), C::KV_BYTES);
#pragma unroll
                for (int p = 0; p < C::PANELS; ++p)
                    tma_load_3d(sbase + C::OFF_V + s * C::KV_BYTES + p * (kBN * 128), &tm_v, p * 64, j * kBN, hk, vfull(s));
            }
        }
        // Every copy issued must land before the CTA may exit.  (A broken-off
        // round's own K block has had the second of the wait that ran out.)
        volatile int no_abort = 0;
        tc::mbar_wait(qfull, 0, &no_abort, err, kErrDrain);
        for (int i = max(0, j - 2); i < j; ++i) {
            tc::mbar_wait(kfull(i & 1), uint32_t(i >> 1) & 1u, &no_abort, err, kErrDrain);
            tc::mbar_wait(vfull(i & 1), uint32_t(i >> 1) & 1u, &no_abort, err, kErrDrain);
        }
        // So must the commits arrive: the last P V's comes after the stages',
        // but nothing says that two commits arrive in their order.
        bool ok = j == nblk;
        for (int i = max(0, j - 2); ok && i < j; ++i)
            ok = tc::mbar_wait(kempty(i & 1), uint32_t(i >> 1) & 1u, &s_abort, err, kErrDrain) &&
                 tc::mbar_wait(vempty(i & 1), uint32_t(i >> 1) & 1u, &s_abort, err, kErrDrain);
    } else if (warp == kMmaWarp) {
        const bool leader = tc::elect_one();
        constexpr uint32_t idesc_qk = tc::idesc_bf16_f32(kRows, kBN, false), idesc_pv = tc::idesc_bf16_f32(kRows, D, true);
        bool ok = __all_sync(0xffffffffu, tc::mbar_wait(qfull, 0, &s_abort, err, kErrMma)), any = false;
        for (int j = -1; ok && j < nblk; ++j) {
            if (j + 1 < nblk) {
                // S of block j + 1, once P V of block j - 1 has read P from
                // its slot (under the softmax of block j)
                const int s = (j + 1) & 1;
                ok = __all_sync(0xffffffffu, tc::mbar_wait(kfull(s), uint32_t((j + 1) >> 1) & 1u, &s_abort, err, kErrMma)) &&
                     (j < 1 || __all_sync(0xffffffffu, tc::mbar_wait(pvdone, uint32_t(j - 1) & 1u, &s_abort, err, kErrMma)));
                if (!ok) break;
                tc::tc_fence_after();
                if (leader) {
#pragma unroll
                    for (int kk = 0; kk < D / 16; ++kk) {
                        const uint64_t a = tc::sw128_desc(sbase + (kk / 4) * (kRows * 128) + (kk % 4) * 32, 16, 1024);
                        const uint64_t b = tc::sw128_desc(sbase + C::OFF_K + s * C::KV_BYTES + (kk / 4) * (kBN * 128) + (kk % 4) * 32, 16, 1024);
                        tc::mma_f16_ss(tmem + s * kBN, a, b, idesc_qk, kk > 0 ? 1u : 0u);
                    }
                    tc::mma_commit(sfull(s));
                    tc::mma_commit(kempty(s));
                }
                any = true;
            }
            if (j < 0) continue;
            const int s = j & 1;
            const uint32_t phase = uint32_t(j >> 1) & 1u;
            ok = __all_sync(0xffffffffu, tc::mbar_wait(vfull(s), phase, &s_abort, err, kErrMma)) &&
                 __all_sync(0xffffffffu, tc::mbar_wait(pfull(s), phase, &s_abort, err, kErrMma));
            if (!ok) break;
            tc::tc_fence_after();
            if (leader) {
#pragma unroll
                for (int kk = 0; kk < kBN / 16; ++kk) {
                    const uint64_t b = tc::sw128_desc(sbase + C::OFF_V + s * C::KV_BYTES + kk * 16 * 128, kBN * 128, 1024);
                    mma_f16_ts(tmem + C::COL_O, tmem + s * kBN + kk * 8, b, idesc_pv, j > 0 || kk > 0 ? 1u : 0u);
                }
                tc::mma_commit(vempty(s));
                tc::mma_commit(pvdone);
            }
        }
        if (!ok && any && leader) {
            // let the MMAs already issued finish before TMEM is freed
            tc::mma_commit(drain);
            volatile int no_abort = 0;
            tc::mbar_wait(drain, 0, &no_abort, err, kErrDrain);
        }
    } else {
        const int row = row0 + warp * 32 + lane;
        const uint32_t mine = tmem + (uint32_t(warp * 32) << 16);
        float m = 0.f, l = 0.f;
        bool ok = true;
        // A positive scale goes in with the exponent's fma, past the masking and
        // the maximum; one of zero or below would make NaN or +inf of a masked
        // score and turn the order round, so it goes in first.
        const bool scale_first = !(scale_log2 > 0.f);
        const float scale_later = scale_first ? 1.f : scale_log2;
        for (int j = 0; j < nblk; ++j) {
            const int s = j & 1;
            ok = __all_sync(0xffffffffu, tc::mbar_wait(sfull(s), uint32_t(j >> 1) & 1u, &s_abort, err, kErrOut));
            if (!ok) break;
            tc::tc_fence_after();
            float v[2][32];
            tmem_ld32_done(mine + s * kBN, v[0]);
            tmem_ld32_done(mine + s * kBN + 32, v[1]);
            if (scale_first) {
#pragma unroll
                for (int i = 0; i < kBN; ++i) v[i >> 5][i & 31] *= scale_log2;
            }
            if ((j + 1) * kBN > row0 + 1) {          // the diagonal's blocks
                const int last = row - j * kBN;      // this row's last key in the block
#pragma unroll
                for (int i = 0; i < kBN; ++i)
                    if (i > last) v[i >> 5][i & 31] = -INFINITY;
            }
            float top = v[0][0];
#pragma unroll
            for (int i = 1; i < kBN; ++i) top = fmaxf(top, v[i >> 5][i & 31]);
            top *= scale_later;
            if (j == 0) {
                m = top;
            } else if (__any_sync(0xffffffffu, top > m)) {
                const float to = fmaxf(m, top), alpha = ex2(m - (to == -INFINITY ? 0.f : to));
                m = to;
                l *= alpha;
                // O is at rest: the last P V issued is the previous block's
                ok = __all_sync(0xffffffffu, tc::mbar_wait(pvdone, uint32_t(j - 1) & 1u, &s_abort, err, kErrOut));
                if (!ok) break;
                tc::tc_fence_after();
#pragma unroll
                for (int c = 0; c < D; c += 32) {
                    float o[32];
                    tmem_ld32_done(mine + C::COL_O + c, o);
#pragma unroll
                    for (int i = 0; i < 32; ++i) o[i] *= alpha;
                    tc::tmem_st32(mine + C::COL_O + c, o);
                }
                tc::tmem_wait_st();
            }
            // a row whose every score so far is -inf has no weights yet
            const float ref = m == -INFINITY ? 0.f : m;
            // (the weights as they are used, rounded: their sum then makes up
            // for part of the rounding)
            float part[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
            for (int half = 0; half < 2; ++half) {
                uint32_t pk[16];
#pragma unroll
                for (int i = 0; i < 16; ++i) {
                    const float a = ex2(fmaf(v[half][2 * i], scale_later, -ref)), b = ex2(fmaf(v[half][2 * i + 1], scale_later, -ref));
                    const __nv_bfloat162 p2 = __floats2bfloat162_rn(a, b);
                    pk[i] = *reinterpret_cast<const uint32_t*>(&p2);
                    part[i & 3] += __low2float(p2) + __high2float(p2);
                }
                asm volatile(
                    "tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, "
                    "%14, %15, %16};" ::"r"(mine + s * kBN + half * 16),
                    "r"(pk[0]), "r"(pk[1]), "r"(pk[2]), "r"(pk[3]), "r"(pk[4]), "r"(pk[5]), "r"(pk[6]), "r"(pk[7]), "r"(pk[8]),
                    "r"(pk[9]), "r"(pk[10]), "r"(pk[11]), "r"(pk[12]), "r"(pk[13]), "r"(pk[14]), "r"(pk[15])
                    : "memory");
            }
            l += (part[0] + part[1]) + (part[2] + part[3]);
            tc::tmem_wait_st();
            // Each warp sees each of pvdone's phases (long complete by now):
            // one that went on without could take the last but one for the
            // last, as a wait tells a phase by its parity.
            if (j > 0) {
                ok = __all_sync(0xffffffffu, tc::mbar_wait(pvdone, uint32_t(j - 1) & 1u, &s_abort, err, kErrOut));
                if (!ok) break;
            }
            tc::tc_fence_before();
            tc::mbar_arrive(pfull(s));
        }
        if (ok) ok = __all_sync(0xffffffffu, tc::mbar_wait(pvdone, uint32_t(nblk - 1) & 1u, &s_abort, err, kErrOut));
        if (ok) {
            tc::tc_fence_after();
            const float inv = l == 0.f ? 0.f : 1.f / l;   // (no weights at all: zeros)
            uint4* dst = reinterpret_cast<uint4*>(out + (size_t(row) * Hq + head) * D);
#pragma unroll
            for (int c = 0; c < D; c += 32) {
                float o[32];
                tmem_ld32_done(mine + C::COL_O + c, o);
                if (row < T) {
#pragma unroll
                    for (int i = 0; i < 4; ++i) {
                        uint32_t w[4];
#pragma unroll
                        for (int e = 0; e < 4; ++e) {
                            const __nv_bfloat162 p2 = __floats2bfloat162_rn(o[8 * i + 2 * e] * inv, o[8 * i + 2 * e + 1] * inv);
                            w[e] = *reinterpret_cast<const uint32_t*>(&p2);
                        }
                        dst[c / 8 + i] = make_uint4(w[0], w[1], w[2], w[3]);
                    }
                }
            }
        }
    }
    __syncwarp();
    tc::tc_fence_before();
    __syncthreads();
    tc::tc_fence_after();
    if (warp == kMmaWarp) tc::tmem_dealloc(tmem, C::TMEM);
}

// [z][y][x] bf16, strides in elements (x: 1); box of bz x by x 64, 128-byte
// swizzle, zeros outside.
bool make_map(CUtensorMap* m, const void* base, int x, int y, int z, size_t sy, size_t sz, int by, int bz) {
    decoder::EncodeFn enc = decoder::encode_fn();
    const cuuint64_t dims[3] = {cuuint64_t(x), cuuint64_t(y), cuuint64_t(z)}, strides[2] = {sy * 2, sz * 2};
    const cuuint32_t box[3] = {64, cuuint32_t(by), cuuint32_t(bz)}, es[3] = {1, 1, 1};
    return enc && enc(m, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3, const_cast<void*>(base), dims, strides, box, es,
                      CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
                      CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <int D>
int launch(const void* q, const void* k, const void* v, void* out, int T, int Hq, int Hkv, float scale, cudaStream_t st) {
    using C = Cfg<D>;
    static splice::PerDevice<bool> kept;
    bool set = false;
    const cudaError_t e = kept.get(&set, [](int, bool* done) {
        *done = true;
        return cudaFuncSetAttribute(causal_kernel<D>, cudaFuncAttributeMaxDynamicSharedMemorySize, int(C::SMEM));
    });
    if (e != cudaSuccess) return int(e);
    unsigned* err = decoder::error_word();
    CUtensorMap mq, mk, mv;
    if (!err || !make_map(&mq, q, D, Hq, T, D, size_t(Hq) * D, 1, kRows) ||
        !make_map(&mk, k, D, T, Hkv, D, size_t(T) * D, kBN, 1) || !make_map(&mv, v, D, T, Hkv, D, size_t(T) * D, kBN, 1))
        return int(cudaErrorInvalidValue);
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned((T + kRows - 1) / kRows) * unsigned(Hq));
    cfg.blockDim = dim3(kThreads);
    cfg.dynamicSmemBytes = C::SMEM;
    cfg.stream = st;
    cudaLaunchAttribute a;
    a.id = cudaLaunchAttributeProgrammaticStreamSerialization;
    a.val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = &a;
    cfg.numAttrs = 1;
    return int(cudaLaunchKernelEx(&cfg, causal_kernel<D>, mq, mk, mv, static_cast<__nv_bfloat16*>(out), T, Hq, Hq / Hkv,
                                  scale * 1.4426950408889634f, err));
}

}  // namespace

extern "C" {

// See the head of this file; 16-byte aligned.  Returns a cudaError_t.
int decoder_causal(const void* q, const void* k, const void* v, void* out, long T, int Hq, int Hkv, int d, float scale,
                   void* stream) {
    if (T < 1 || T > (1 << 20) || Hq < 1 || Hkv < 1 || Hq % Hkv != 0) return int(cudaErrorInvalidValue);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (d == 64) return launch<64>(q, k, v, out, int(T), Hq, Hkv, scale, st);
    if (d == 128) return launch<128>(q, k, v, out, int(T), Hq, Hkv, scale, st);
    if (d == 256) return launch<256>(q, k, v, out, int(T), Hq, Hkv, scale, st);
    return int(cudaErrorInvalidValue);
}

}  // extern "C"
