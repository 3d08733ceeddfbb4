// Shared by the two generated-span kernels: work items and the merge of a
// row's two partial states.
#pragma once

#include <cuda_runtime.h>

#include <cmath>

#include "splice_internal.h"

namespace splice {
namespace gs {

constexpr unsigned kFull = 0xffffffffu;
constexpr float kTau = 8.0f;

__device__ __forceinline__ float ex2(float x) {
    float y;
    asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// Generated-span K/V is read once: the copy marks its L2 lines first to be
// evicted, so the streamed bytes do not push out the partial states the
// merge reads right after.
__device__ __forceinline__ uint64_t l2_evict_first_policy() {
    uint64_t pol;
    asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(pol));
    return pol;
}

__device__ __forceinline__ unsigned ld_relaxed_gpu(const unsigned* p) {
    unsigned v;
    asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p));
    return v;
}

// The merge of a row's two partial states -- the prompt-span pass's (when
// has_span) and this pass's -- with a ZERO span's closed form, in exactly
// the operations and order of the merge kernel for a row of at most two
// states (merge_row.cuh): the same bits.  Returns the factor of the
// weighted sum (0 for a row with nothing live) and the two weights.
__device__ __forceinline__ float merge_two_weights(bool has_span, float2 ml_span, float m_gen, float l_gen,
                                                   bool zero_span, int n_zero, float* w_span, float* w_gen) {
    const bool live_s = has_span && ml_span.y > 0.f, live_g = l_gen > 0.f;
    float M = fmaxf(live_s ? ml_span.x : -INFINITY, live_g ? m_gen : -INFINITY);
    if (zero_span) M = fmaxf(M, 0.f);
    *w_span = live_s ? exp2f(ml_span.x - M) : 0.f;
    *w_gen = live_g ? exp2f(m_gen - M) : 0.f;
    float den = __fadd_rn(has_span ? __fmul_rn(*w_span, ml_span.y) : 0.f, __fmul_rn(*w_gen, l_gen));
    if (zero_span) den = fmaf(float(n_zero), exp2f(0.f - M), den);
    return den > 0.f ? 1.f / den : 0.f;
}

__device__ __forceinline__ float merge_two(bool has_span, float w_span, float o_span, float w_gen, float o_gen,
                                           float inv) {
    float acc = 0.f;
    if (has_span && w_span != 0.f) acc = fmaf(w_span, o_span, acc);
    if (w_gen != 0.f) acc = fmaf(w_gen, o_gen, acc);
    return __fmul_rn(acc, inv);
}

// Items a warp may leave unmerged until its end (with P.gs_merge): those
// that end before the prompt-span pass has completed.
constexpr int kPend = kMaxPending;

// n / d for 0 <= n < 2^31 by a multiply and a shift, for a divisor fixed
// per launch (Granlund and Montgomery, "Division by invariant integers using
// multiplication", 1994, the round-up method): with s = ceil(log2 d) and
// m = floor(2^32 (2^s - d) / d) + 1, n / d = (umulhi(n, m) + n) >> s; the
// sum stays below 2^32 because umulhi(n, m) < n < 2^31.
struct FastDiv {
    uint32_t d, m, s;
    __device__ explicit FastDiv(int divisor) : d(uint32_t(divisor)), m(1), s(0) {
        while ((1u << s) < d) ++s;
        m = uint32_t((((uint64_t(1) << s) - d) << 32) / d + 1);
    }
    __device__ __forceinline__ int div(int n) const { return int((__umulhi(uint32_t(n), m) + uint32_t(n)) >> s); }
};

struct ItemDivs {
    FastDiv nss, chunks, hkv;
};

// One work item: where its rows and keys are.  The issue cursor decodes
// each item once and hands it to the consumer through the warp's ring
// (eight ints, idx -1 for the end of the walk).
struct Item {
    int idx, s, h, split, k0, k1, nblk, rc;
};

// Work item idx = ((sequence * Hkv + kv head) * row chunks + row chunk) *
// splits + key split.
__device__ __forceinline__ void item_of(const AttnParams& P, const ItemDivs& dv, int idx, Item& it) {
    it.idx = idx;
    const int rem = dv.nss.div(idx);
    it.split = idx - rem * P.nss;
    const int sh = dv.chunks.div(rem);
    it.rc = rem - sh * P.gs_chunks;
    it.s = dv.hkv.div(sh);
    it.h = sh - it.s * P.Hkv;
    it.k0 = P.s_lo + it.split * P.s_chunk;
    it.k1 = min(P.s_hi, it.k0 + P.s_chunk);
    it.nblk = it.k1 > it.k0 ? (it.k1 - it.k0 + 15) / 16 : 0;
}

// Offset (in elements) of the generated-span K/V rows of (sequence, kv head)
// at this layer.
template <int D>
__device__ __forceinline__ size_t span_base(const AttnParams& P, int s, int h) {
    return ((size_t(s) * P.N + P.layer) * P.Hkv + h) * size_t(P.T) * D;
}

// Both kernels' arguments: the call's parameters, the number of items and
// the number of multiprocessors.
int launch_mma(const AttnParams& p, cudaStream_t stream, bool overlap_previous);
// Warps of the tensor-core kernel that an SM holds, and whether it is built
// with its merge path, at `rows` query rows per item.
int mma_warps_per_sm(int d, int rows);
bool mma_can_merge(int d, int rows);

}  // namespace gs
}  // namespace splice
