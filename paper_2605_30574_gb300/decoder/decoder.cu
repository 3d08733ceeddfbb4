// Elementwise and normalisation kernels of the decoder that drives Algorithm 1
// (model.py): RMSNorm, the per-head norm and RoPE of q and k, the residual
// additions, SwiGLU's product and the attention output's conversion.  The
// projections between them are gemm.cu's (library GEMMs for shapes that those
// do not take), the prefill's attention is causal.cu's, the decode attention
// libsplice.so's.
//
// Every kernel reads its inputs once and writes its outputs once, computes in
// fp32 and rounds to bf16 only where the decoder's definition does (model.py's
// torch expressions: the norm's output, q and k after RoPE, the SwiGLU product,
// the attention output), with the same order of the element operations; only
// the order of the row sums differs.
//
// At a decode batch each of them moves 10-50 MB: one wave or a few of blocks
// that are bound by their loads' latency, not by bandwidth.  Their point is
// their number: in a Qwen3-8B-shaped layer of 512 cells they take the place
// of 62 launches by 7 (980 -> 317 us with library GEMMs; a step of two layers and
// the head 2149 -> 797, a prefill of 1024 tokens 2376 -> 890; 216, 705 and 773
// with gemm.cu and causal.cu).  Times below are a launch's
// on cold caches at 512 rows of 4096 (32 + 2 x 8 heads of 128, F = 12288).
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <initializer_list>

#include "decoder.h"

namespace {

constexpr int kThreads = 256;
constexpr int kKeep = 4;        // float4 of a row that a thread keeps in registers between the passes

// Every kernel here is launched as a programmatic dependent of what precedes
// it on the stream: its blocks may be set up while that still runs, wait for
// all of it before they read or write anything, and let what follows do the
// same.
__device__ __forceinline__ void wait_for_previous() {
    asm volatile("griddepcontrol.wait;" ::: "memory");
    asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
}

template <class... Params, class... Args>
int launch(void (*kernel)(Params...), dim3 grid, cudaStream_t stream, Args... args) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = grid;
    cfg.blockDim = dim3(kThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return int(cudaLaunchKernelEx(&cfg, kernel, args...));
}

__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
    for (int off = 16; off > 0; off >>= 1) x += __shfl_xor_sync(0xffffffffu, x, off);
    return x;
}

__device__ __forceinline__ uint2 pack4(float a, float b, float c, float d) {
    const __nv_bfloat162 lo = __floats2bfloat162_rn(a, b), hi = __floats2bfloat162_rn(c, d);
    return make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}

__device__ __forceinline__ float4 unpack4(uint2 w) {
    return make_float4(__uint_as_float(w.x << 16), __uint_as_float(w.x & 0xffff0000u), __uint_as_float(w.y << 16),
                       __uint_as_float(w.y & 0xffff0000u));
}

__device__ __forceinline__ float4 add4(float4 a, float4 b) {
    return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w);
}

// x = bf16(h / rms(h) * w), one block per row; ADD: h + o first (o bf16, the
// output of a projection), the sum written to h2.  6 bytes per element (ADD:
// 12): 6.9 us, ADD 5.8 (the five torch passes it replaces: 33).  A thread keeps its first kKeep float4 of the row in
// registers, so rows of up to 4096 elements are read once; what is beyond is
// read again for the second pass (from L1 or L2).
template <bool ADD, bool VEC>
__global__ void __launch_bounds__(kThreads)
    rms_norm_kernel(const float* __restrict__ h, const __nv_bfloat16* __restrict__ o,
                    const __nv_bfloat16* __restrict__ w, float* __restrict__ h2, __nv_bfloat16* __restrict__ x, int D,
                    float eps) {
    __shared__ float part[kThreads / 32];
    wait_for_previous();
    const size_t base = size_t(blockIdx.x) * D;
    const int t = threadIdx.x;
    float sum = 0.f;
    float4 keep[kKeep];
    const int n4 = VEC ? D / 4 : 0;
    auto load4 = [&](int i) -> float4 {
        float4 v = reinterpret_cast<const float4*>(h + base)[i];
        if (ADD) v = add4(v, unpack4(reinterpret_cast<const uint2*>(o + base)[i]));
        return v;
    };
    auto load1 = [&](int i) -> float { return ADD ? h[base + i] + __bfloat162float(o[base + i]) : h[base + i]; };
    if constexpr (VEC) {
#pragma unroll
        for (int k = 0; k < kKeep; ++k) {
            const int i = t + k * kThreads;
            keep[k] = i < n4 ? load4(i) : make_float4(0.f, 0.f, 0.f, 0.f);
        }
#pragma unroll
        for (int k = 0; k < kKeep; ++k) {
            const int i = t + k * kThreads;
            if (ADD && i < n4) reinterpret_cast<float4*>(h2 + base)[i] = keep[k];
            sum += (keep[k].x * keep[k].x + keep[k].y * keep[k].y) + (keep[k].z * keep[k].z + keep[k].w * keep[k].w);
        }
        for (int i = t + kKeep * kThreads; i < n4; i += kThreads) {
            const float4 v = load4(i);
            if (ADD) reinterpret_cast<float4*>(h2 + base)[i] = v;
            sum += (v.x * v.x + v.y * v.y) + (v.z * v.z + v.w * v.w);
        }
    } else {
        for (int i = t; i < D; i += kThreads) {
            const float v = load1(i);
            if (ADD) h2[base + i] = v;
            sum += v * v;
        }
    }
    sum = warp_sum(sum);
    if ((t & 31) == 0) part[t >> 5] = sum;
    __syncthreads();
    sum = 0.f;
#pragma unroll
    for (int k = 0; k < kThreads / 32; ++k) sum += part[k];
    const float r = rsqrtf(sum / float(D) + eps);
    if constexpr (VEC) {
        auto out4 = [&](int i, float4 v) {
            const float4 g = unpack4(reinterpret_cast<const uint2*>(w)[i]);
            reinterpret_cast<uint2*>(x + base)[i] =
                pack4(__fmul_rn(v.x * r, g.x), __fmul_rn(v.y * r, g.y), __fmul_rn(v.z * r, g.z), __fmul_rn(v.w * r, g.w));
        };
#pragma unroll
        for (int k = 0; k < kKeep; ++k) {
            const int i = t + k * kThreads;
            if (i < n4) out4(i, keep[k]);
        }
        for (int i = t + kKeep * kThreads; i < n4; i += kThreads) out4(i, load4(i));
    } else {
        for (int i = t; i < D; i += kThreads)
            x[base + i] = __float2bfloat16_rn(__fmul_rn(load1(i) * r, __bfloat162float(w[i])));
    }
}

// h2 = h + o (o bf16); h2 may be h.  10 bytes per element: 5.0 us.
template <bool VEC>
__global__ void __launch_bounds__(kThreads)
    add_kernel(const float* h, const __nv_bfloat16* __restrict__ o, float* h2, long n) {
    wait_for_previous();
    const long i = long(blockIdx.x) * kThreads + threadIdx.x;
    if constexpr (VEC) {
        if (i < n / 4)
            reinterpret_cast<float4*>(h2)[i] =
                add4(reinterpret_cast<const float4*>(h)[i], unpack4(reinterpret_cast<const uint2*>(o)[i]));
    } else {
        if (i < n) h2[i] = h[i] + __bfloat162float(o[i]);
    }
}

// y = bf16(x): 6 bytes per element, 4.2 us.
template <bool VEC>
__global__ void __launch_bounds__(kThreads)
    to_bf16_kernel(const float* __restrict__ x, __nv_bfloat16* __restrict__ y, long n) {
    wait_for_previous();
    const long i = long(blockIdx.x) * kThreads + threadIdx.x;
    if constexpr (VEC) {
        if (i < n / 4) {
            const float4 v = reinterpret_cast<const float4*>(x)[i];
            reinterpret_cast<uint2*>(y)[i] = pack4(v.x, v.y, v.z, v.w);
        }
    } else {
        if (i < n) y[i] = __float2bfloat16_rn(x[i]);
    }
}

__device__ __forceinline__ float silu(float g) { return g / (1.f + expf(-g)); }

// y[r][i] = bf16(silu(gate[r][i]) * up[r][i]); gate and up rows are `ld`
// elements apart (2 F when one GEMM made both).  6 bytes per output: 9.9 us
// (38 MB, 3.8 TB/s).
template <bool VEC>
__global__ void __launch_bounds__(kThreads)
    silu_mul_kernel(const __nv_bfloat16* __restrict__ gate, const __nv_bfloat16* __restrict__ up, long ld,
                    __nv_bfloat16* __restrict__ y, int F) {
    wait_for_previous();
    const long r = blockIdx.y;
    const int i = blockIdx.x * kThreads + threadIdx.x;
    if constexpr (VEC) {
        if (i >= F / 4) return;
        const float4 g = unpack4(reinterpret_cast<const uint2*>(gate + r * ld)[i]);
        const float4 u = unpack4(reinterpret_cast<const uint2*>(up + r * ld)[i]);
        reinterpret_cast<uint2*>(y + r * F)[i] = pack4(silu(g.x) * u.x, silu(g.y) * u.y, silu(g.z) * u.z, silu(g.w) * u.w);
    } else {
        if (i >= F) return;
        y[r * F + i] = __float2bfloat16_rn(silu(__bfloat162float(gate[r * ld + i])) * __bfloat162float(up[r * ld + i]));
    }
}

struct HeadRows {
    const __nv_bfloat16* src;   // rows [row][head][d], rows `ld` elements apart
    long ld;
    __nv_bfloat16* dst;         // element (row, head, c) at row * row_stride + head * head_stride + c
    long row_stride, head_stride;
};

// V bf16 values, loaded and stored as one word.
template <int V>
struct alignas(2 * V) Vec {
    __nv_bfloat16 x[V];
};

// q and k: bf16(rope(rms_norm over the head dim)); v: copied.  A warp per
// (row, head), eight heads of a row per block; the row's D / 2 rotation
// angles are computed once per block into shared memory.  Lane i holds
// elements V i .. V i + V - 1 of both halves of the head (V = D / 64), so the
// rotation needs no exchange.  4 bytes per element and one head per warp, so
// that a row's 48 heads are in flight at once: 8.0 us, where torch made 36
// launches.  Rows of heads and the norms' weights are
// read and written V elements at a time: see qkv_post_takes.
template <int D>
__global__ void __launch_bounds__(kThreads)
    qkv_post_kernel(HeadRows q, HeadRows k, HeadRows v, const __nv_bfloat16* __restrict__ q_norm,
                    const __nv_bfloat16* __restrict__ k_norm, const float* __restrict__ inv_freq,
                    const void* __restrict__ pos, int pos_kind, int Hq, int Hkv, float eps) {
    constexpr int HALF = D / 2, V = D / 64;
    __shared__ float2 cs[HALF];
    wait_for_previous();
    const long row = blockIdx.x;
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int j = blockIdx.y * (kThreads / 32) + warp;
    const bool live = j < Hq + 2 * Hkv, turn = j < Hq + Hkv;
    const __nv_bfloat16* src = nullptr;
    __nv_bfloat16* dst = nullptr;
    if (j < Hq) {
        src = q.src + row * q.ld + long(j) * D;
        dst = q.dst + row * q.row_stride + j * q.head_stride;
    } else if (turn) {
        src = k.src + row * k.ld + long(j - Hq) * D;
        dst = k.dst + row * k.row_stride + (j - Hq) * k.head_stride;
    } else if (live) {
        src = v.src + row * v.ld + long(j - Hq - Hkv) * D;
        dst = v.dst + row * v.row_stride + (j - Hq - Hkv) * v.head_stride;
    }
    Vec<V> lo, hi, g_lo, g_hi;
    if (live) {
        lo = reinterpret_cast<const Vec<V>*>(src)[lane];
        hi = reinterpret_cast<const Vec<V>*>(src + HALF)[lane];
    }
    if (turn) {
        const __nv_bfloat16* g = j < Hq ? q_norm : k_norm;
        g_lo = reinterpret_cast<const Vec<V>*>(g)[lane];
        g_hi = reinterpret_cast<const Vec<V>*>(g + HALF)[lane];
    }
    float p;
    if (pos_kind == 0)
        p = float(reinterpret_cast<const int64_t*>(pos)[row]);
    else if (pos_kind == 1)
        p = float(reinterpret_cast<const int32_t*>(pos)[row]);
    else
        p = reinterpret_cast<const float*>(pos)[row];
    for (int i = threadIdx.x; i < HALF; i += kThreads) {
        float s, c;
        sincosf(p * inv_freq[i], &s, &c);
        cs[i] = make_float2(c, s);
    }
    __syncthreads();
    if (!live) return;
    if (turn) {
        float a[V], b[V], sum = 0.f;
#pragma unroll
        for (int i = 0; i < V; ++i) {
            a[i] = __bfloat162float(lo.x[i]);
            b[i] = __bfloat162float(hi.x[i]);
            sum += a[i] * a[i] + b[i] * b[i];
        }
        const float r = rsqrtf(warp_sum(sum) / float(D) + eps);
#pragma unroll
        for (int i = 0; i < V; ++i) {
            const float x1 = __fmul_rn(a[i] * r, __bfloat162float(g_lo.x[i]));
            const float x2 = __fmul_rn(b[i] * r, __bfloat162float(g_hi.x[i]));
            const float2 f = cs[lane * V + i];
            lo.x[i] = __float2bfloat16_rn(__fsub_rn(__fmul_rn(x1, f.x), __fmul_rn(x2, f.y)));
            hi.x[i] = __float2bfloat16_rn(__fadd_rn(__fmul_rn(x2, f.x), __fmul_rn(x1, f.y)));
        }
    }
    reinterpret_cast<Vec<V>*>(dst)[lane] = lo;
    reinterpret_cast<Vec<V>*>(dst + HALF)[lane] = hi;
}

bool vec_ok(const void* a, const void* b, const void* c, const void* d, long n) {
    const uintptr_t bits = reinterpret_cast<uintptr_t>(a) | reinterpret_cast<uintptr_t>(b) |
                           reinterpret_cast<uintptr_t>(c) | reinterpret_cast<uintptr_t>(d);
    return (bits & 15u) == 0 && n % 4 == 0;
}

unsigned blocks_for(long n) { return unsigned((n + kThreads - 1) / kThreads); }

using bf = __nv_bfloat16;

int rms_norm(const float* h, const bf* w, bf* x, long rows, int D, float eps, cudaStream_t st) {
    const dim3 grid{unsigned(rows)};
    const bf* none = nullptr;
    float* no_sum = nullptr;
    if (vec_ok(h, w, x, nullptr, D)) return launch(rms_norm_kernel<false, true>, grid, st, h, none, w, no_sum, x, D, eps);
    return launch(rms_norm_kernel<false, false>, grid, st, h, none, w, no_sum, x, D, eps);
}

int to_bf16(const float* x, bf* y, long n, cudaStream_t st) {
    if (vec_ok(x, y, nullptr, nullptr, n)) return launch(to_bf16_kernel<true>, dim3(blocks_for(n / 4)), st, x, y, n);
    return launch(to_bf16_kernel<false>, dim3(blocks_for(n)), st, x, y, n);
}

size_t align256(size_t n) { return (n + 255) / 256 * 256; }

bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

// Whether every word of d / 64 elements that qkv_post_kernel<d> takes is aligned.
bool qkv_post_takes(std::initializer_list<const void*> ptrs, const long* strides, int n_strides, int d) {
    if (d != 64 && d != 128 && d != 256) return false;
    for (const void* p : ptrs)
        if (reinterpret_cast<uintptr_t>(p) % unsigned(d / 32)) return false;
    for (int i = 0; i < n_strides; ++i)
        if (strides[i] % (d / 64)) return false;
    return true;
}

}  // namespace

// Every call returns the cudaError_t of its launches and takes contiguous rows
// unless strides are given; rows and sizes >= 1.  rows < 2^31, n < 2^39.
extern "C" {

int decoder_rms_norm(const void* h, const void* w, void* x, long rows, int D, float eps, void* stream) {
    return rms_norm(static_cast<const float*>(h), static_cast<const bf*>(w), static_cast<bf*>(x), rows, D, eps,
                    static_cast<cudaStream_t>(stream));
}

int decoder_add_rms_norm(const void* h, const void* o, const void* w, void* h2, void* x, long rows, int D, float eps,
                         void* stream) {
    const bool vec = vec_ok(h, w, x, h2, D) && vec_ok(o, nullptr, nullptr, nullptr, D);
    return launch(vec ? rms_norm_kernel<true, true> : rms_norm_kernel<true, false>, dim3(unsigned(rows)),
                  static_cast<cudaStream_t>(stream), static_cast<const float*>(h), static_cast<const bf*>(o),
                  static_cast<const bf*>(w), static_cast<float*>(h2), static_cast<bf*>(x), D, eps);
}

int decoder_add(const void* h, const void* o, void* h2, long n, void* stream) {
    const bool vec = vec_ok(h, o, h2, nullptr, n);
    return launch(vec ? add_kernel<true> : add_kernel<false>, dim3(blocks_for(vec ? n / 4 : n)),
                  static_cast<cudaStream_t>(stream), static_cast<const float*>(h), static_cast<const bf*>(o),
                  static_cast<float*>(h2), n);
}

int decoder_to_bf16(const void* x, void* y, long n, void* stream) {
    return to_bf16(static_cast<const float*>(x), static_cast<bf*>(y), n, static_cast<cudaStream_t>(stream));
}

int decoder_silu_mul(const void* gate, const void* up, long ld, void* y, long rows, int F, void* stream) {
    // (blockIdx.y holds a row: at most 65535 rows per launch)
    for (long r0 = 0; r0 < rows; r0 += 65535) {
        const unsigned n = unsigned(rows - r0 < 65535 ? rows - r0 : 65535);
        const bf* g = static_cast<const bf*>(gate) + r0 * ld;
        const bf* u = static_cast<const bf*>(up) + r0 * ld;
        bf* out = static_cast<bf*>(y) + r0 * F;
        const bool vec = vec_ok(g, u, out, nullptr, F) && ld % 8 == 0;
        const int e = launch(vec ? silu_mul_kernel<true> : silu_mul_kernel<false>, dim3(blocks_for(vec ? F / 4 : F), n),
                             static_cast<cudaStream_t>(stream), g, u, ld, out, F);
        if (e != 0) return e;
    }
    return 0;
}

// strides: {q, k, v source row strides, q row, q head, k row, k head, v row, v
// head destination strides}, in elements.  pos_kind: 0 int64, 1 int32, 2 fp32.
int decoder_qkv_post(const void* q, const void* k, const void* v, void* q_out, void* k_out, void* v_out,
                     const long* strides, const void* q_norm, const void* k_norm, const void* inv_freq,
                     const void* pos, int pos_kind, long rows, int Hq, int Hkv, int d, float eps, void* stream) {
    const HeadRows a{static_cast<const bf*>(q), strides[0], static_cast<bf*>(q_out), strides[3], strides[4]};
    const HeadRows b{static_cast<const bf*>(k), strides[1], static_cast<bf*>(k_out), strides[5], strides[6]};
    const HeadRows c{static_cast<const bf*>(v), strides[2], static_cast<bf*>(v_out), strides[7], strides[8]};
    if (!qkv_post_takes({q, k, v, q_out, k_out, v_out, q_norm, k_norm}, strides, 9, d)) return int(cudaErrorInvalidValue);
    auto kernel = d == 64 ? qkv_post_kernel<64> : (d == 128 ? qkv_post_kernel<128> : qkv_post_kernel<256>);
    const dim3 grid(unsigned(rows), unsigned((Hq + 2 * Hkv + kThreads / 32 - 1) / (kThreads / 32)));
    return launch(kernel, grid, static_cast<cudaStream_t>(stream), a, b, c, static_cast<const bf*>(q_norm),
                  static_cast<const bf*>(k_norm), static_cast<const float*>(inv_freq), pos, pos_kind, Hq, Hkv, eps);
}

// ---- a layer's two halves in one call each, for the shapes gemm.cu takes ----

// Bytes of scratch that decoder_qkv (half = 0) and decoder_block (1) need, 0
// where the shape is not one for them.  nqkv: outputs of the joined
// projection; nq: of q's.
long decoder_scratch_bytes(int half, long rows, int D, int nq, int nqkv, int F) {
    const int M = int(rows < 1 << 20 ? rows : 1 << 20);
    if (half == 0)
        return decoder::gemm_takes(M, nqkv, D) ? long(align256(size_t(rows) * D * 2) + size_t(rows) * nqkv * 2) : 0;
    if (!decoder::gemm_takes(M, D, nq) || !decoder::gemm_takes(M, F, D) || !decoder::gemm_takes(M, D, F)) return 0;
    return long(align256(size_t(rows) * nq * 2) + align256(size_t(rows) * D * 4) + align256(size_t(rows) * D * 2) +
                size_t(rows) * F * 2);
}

// Input norm, joined projection, per-head norm and RoPE.  strides: {q row, q
// head, k row, k head, v row, v head} of the outputs.
int decoder_qkv(const void* h, const void* in_norm, const void* wqkv, void* scratch, void* q_out, void* k_out, void* v_out,
                const long* strides, const void* q_norm, const void* k_norm, const void* inv_freq, const void* pos,
                int pos_kind, long rows, int D, int Hq, int Hkv, int d, float eps, void* stream) {
    const int nq = Hq * d, nk = Hkv * d, n = nq + 2 * nk;
    if (!aligned16(wqkv) || !aligned16(scratch) || !qkv_post_takes({q_out, k_out, v_out, q_norm, k_norm}, strides, 6, d))
        return int(cudaErrorInvalidValue);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    bf* x = static_cast<bf*>(scratch);
    bf* y = reinterpret_cast<bf*>(static_cast<char*>(scratch) + align256(size_t(rows) * D * 2));
    int e = rms_norm(static_cast<const float*>(h), static_cast<const bf*>(in_norm), x, rows, D, eps, st);
    if (e == 0) e = decoder::gemm(decoder::kPlain, x, wqkv, nullptr, nullptr, y, int(rows), n, D, st);
    if (e != 0) return e;
    const long all[9] = {n, n, n, strides[0], strides[1], strides[2], strides[3], strides[4], strides[5]};
    return decoder_qkv_post(y, y + nq, y + nq + nk, q_out, k_out, v_out, all, q_norm, k_norm, inv_freq, pos, pos_kind, rows,
                            Hq, Hkv, d, eps, stream);
}

// Output projection and residual, norm, SwiGLU, down projection and residual.
// attn: [rows][nq] fp32 or bf16; out: fp32 [rows][D].
int decoder_block(const void* h, const void* attn, int attn_bf16, const void* wo, const void* post_norm, const void* w_gate,
                  const void* w_up, const void* w_down, void* scratch, void* out, long rows, int D, int nq, int F, float eps,
                  void* stream) {
    for (const void* p : {attn, wo, w_gate, w_up, w_down, static_cast<const void*>(scratch)})
        if (!aligned16(p)) return int(cudaErrorInvalidValue);
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    char* at = static_cast<char*>(scratch);
    bf* a = reinterpret_cast<bf*>(at);
    at += align256(size_t(rows) * nq * 2);
    float* h2 = reinterpret_cast<float*>(at);
    at += align256(size_t(rows) * D * 4);
    bf* x = reinterpret_cast<bf*>(at);
    at += align256(size_t(rows) * D * 2);
    bf* y = reinterpret_cast<bf*>(at);
    const int M = int(rows);
    int e = attn_bf16 ? 0 : to_bf16(static_cast<const float*>(attn), a, rows * nq, st);
    if (e == 0) e = decoder::gemm(decoder::kResid, attn_bf16 ? attn : a, wo, nullptr, h, h2, M, D, nq, st);
    if (e == 0) e = rms_norm(h2, static_cast<const bf*>(post_norm), x, rows, D, eps, st);
    if (e == 0) e = decoder::gemm(decoder::kSwiglu, x, w_gate, w_up, nullptr, y, M, F, D, st);
    if (e == 0) e = decoder::gemm(decoder::kResid, y, w_down, nullptr, h2, out, M, D, F, st);
    return e;
}

}  // extern "C"
