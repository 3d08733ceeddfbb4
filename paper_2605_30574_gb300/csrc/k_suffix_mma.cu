// Generated-span pass: attention of the G query rows of one (sequence, kv
// head) over that sequence's own generated-span K/V (§3: the decode step
// attends over the prompt span and the t generated entries).
//
// HBM-bound streaming kernel:
//   * persistent warps walking work items (sequence, kv head, row chunk, key
//     split; one chunk but for more than eight rows in a small launch) and,
//     inside an item, blocks of 16 keys: a fixed stream per warp when this
//     pass goes first, items claimed at run time (one ahead) when it runs
//     behind the prompt-span pass, so warps that start late (on SMs that pass
//     still holds) simply take fewer; the issue cursor decodes each item once
//     and hands it to the consumer through a per-warp ring;
//   * every block's K and V rows (contiguous in the generated-span store) are
//     fetched by 16-byte asynchronous copies into a two-stage per-warp ring,
//     chunks swizzled by row so the matrix loads are free of bank conflicts,
//     rows past the split's end zero-filled; the next block -- of this item
//     or the next one -- is in flight while the current one is computed; an
//     item's first block brings the item's query rows with it, so no item
//     starts on a load from global memory;
//   * both contractions run on mma.sync with the keys or dims on the 16-row
//     side and the (padded) query rows on the 8-column side: S^T = K Q^T,
//     then O^T += V^T P^T.  All G <= 8 rows (two column tiles for G <= 16)
//     share one read of K and V;
//   * fp32 throughout: the bf16 products are exact; a probability is split
//     into three bf16 terms that hold all of its bits; the tensor core's sums
//     are at most three products long and are added to the running sums by
//     fp32 additions (the tensor core truncates where an addition rounds, and
//     a truncated running sum would drift);
//   * online softmax with a lazily moved reference max: the common path
//     needs no rescale and no cross-lane max; row sums are reduced once per
//     item.
// Alone, 512 sequences x 8 heads x 512 keys of 128 dims at four rows per kv
// head: 168 us, 6.4 TB/s (the FMA kernel of k_suffix_gs.cu: 173); eight rows,
// 300 x 8 heads x 277 keys: 58 us, 5.9 TB/s (110, where four rows at a time
// each read K and V); sixteen rows, 64 x 8 x 500 keys: 46-50 us (87).  A block
// takes about 290 instructions (128 dims), a fifth of the issue slots; warps
// mostly wait for their copies.  The error against fp64 is that of the FMA
// kernel or less: 1.6e-7 against 2.0e-7 in the 2-norm at 500 keys.
// Emits the partial state (m, l, o) of every row, like the prompt-span pass
// -- or, behind the prompt-span pass with one split of each span, merges
// the rows itself and writes the output (no merge kernel then).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>

#include "gs_common.cuh"
#include "per_device.h"
#include "tc_ptx.cuh"

namespace splice {
namespace gs {
namespace {

// 16 bytes to shared memory; FULL = false: `bytes` of them (0 or 16), the
// rest zeros.
template <bool FULL>
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, int bytes, uint64_t pol) {
    if constexpr (FULL)
        asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "l"(pol)
                     : "memory");
    else
        asm volatile("cp.async.cg.shared.global.L2::cache_hint [%0], [%1], 16, %2, %3;" ::"r"(dst), "l"(src), "r"(bytes),
                     "l"(pol)
                     : "memory");
}
// The same without a hint: the query rows are read again by the prompt-span
// pass of the call.
__device__ __forceinline__ void cp16_plain(uint32_t dst, const void* src) {
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(dst), "l"(src) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
    asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
__device__ __forceinline__ void ldsm4_t(uint32_t (&r)[4], uint32_t addr) {
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0, %1, %2, %3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}
// 8x8 transpose of 16-bit values across the warp.
__device__ __forceinline__ uint32_t movm_t(uint32_t x) {
    uint32_t y;
    asm("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;" : "=r"(y) : "r"(x));
    return y;
}
// d = a b + c, bf16 in, fp32 out (m16n8k16).
__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], uint32_t b0, uint32_t b1, const float (&c)[4]) {
    asm("mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
        "{%10, %11, %12, %13};"
        : "=f"(d[0]), "=f"(d[1]), "=f"(d[2]), "=f"(d[3])
        : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b0), "r"(b1), "f"(c[0]), "f"(c[1]), "f"(c[2]), "f"(c[3]));
}

// (x, y) -> three words of bf16 pairs whose sum is (x, y) to all 24 bits.
__device__ __forceinline__ void split3(float x, float y, uint32_t (&w)[3]) {
#pragma unroll
    for (int i = 0; i < 3; ++i) {
        const __nv_bfloat162 h = __floats2bfloat162_rn(x, y);
        w[i] = *reinterpret_cast<const uint32_t*>(&h);
        x -= __uint_as_float(w[i] << 16);
        y -= __uint_as_float(w[i] & 0xffff0000u);
    }
}

__device__ __forceinline__ float4 merge_two4(bool has_span, float w_span, float4 s, float w_gen, float4 g, float inv) {
    return make_float4(merge_two(has_span, w_span, s.x, w_gen, g.x, inv), merge_two(has_span, w_span, s.y, w_gen, g.y, inv),
                       merge_two(has_span, w_span, s.z, w_gen, g.z, inv), merge_two(has_span, w_span, s.w, w_gen, g.w, inv));
}

// NT: column tiles of eight query rows (1 for G <= 8, 2 for G <= 16).
template <int D, int NT>
struct GM {
    static constexpr int BK = 16;                             // keys per block
    static constexpr int CH = D / 8;                          // 16-byte chunks per K (or V) row
    static constexpr int RPI = 32 / CH;                       // rows per copy instruction
    static constexpr uint32_t ROW = D * 2;                    // bytes of one row
    static constexpr uint32_t KBYTES = BK * ROW;              // K (or V) of one block
    static constexpr uint32_t STAGE = 2 * KBYTES;
    static constexpr int NQ = 8 * NT;                         // padded query rows
    static constexpr int HALF = D / 2;                        // dims staged at a time by the epilogue
    static constexpr int LDO = HALF + 4;                      // floats per staged row: rows 2 t apart start 8 banks apart
    // Q fragments in registers where they fit beside the accumulators, else
    // loaded from shared memory for every block
    static constexpr bool QREG = D / 16 * NT <= 16;
    // the merge path is built where a warp's prompt-span states fit in registers
    static constexpr bool MERGE = NT * D <= 256;
    // warps per SM that the registers allow (128, 168 or 255 a thread)
    static constexpr int REG_WARPS = D == 64 ? (NT == 1 ? 16 : 12) : 8;
    static constexpr int MAX_WARPS = D == 256 ? REG_WARPS : 4;      // per CTA
    // per-warp shared memory: two stages, [4] items (decoded) in the order
    // they were taken, [kPend] items whose merge waits for the warp's end,
    // [2] query rows of the items in flight (G rows each), [G][LDO] fp32 staged
    static constexpr uint32_t OFF_TAKEN = 2 * STAGE;
    static constexpr uint32_t OFF_PEND = OFF_TAKEN + 4 * 32;
    static constexpr uint32_t OFF_Q = OFF_PEND + kPend * 4 + 96;
    static_assert(OFF_Q % 128 == 0, "query rows start on a swizzle period");
    __host__ __device__ static constexpr uint32_t off_stg(int G) { return OFF_Q + 2 * G * ROW; }
    __host__ __device__ static constexpr uint32_t per_warp(int G) {
        return (off_stg(G) + G * LDO * 4 + 1023) / 1024 * 1024;
    }
    static constexpr int LPR = HALF / 4;                      // lanes per staged row (16-byte units)
    static constexpr int RPP = 32 / LPR;                      // rows per epilogue pass
    static constexpr int NP = NQ / RPP;                       // epilogue passes
    // prompt-span states fetched ahead for both halves of the dims, where
    // registers allow, else for the half at hand
    static constexpr int AHEAD = NT * D <= 128 ? 2 : 1;
};

template <int D, int NT>
__global__ void __launch_bounds__(GM<D, NT>::MAX_WARPS * 32, GM<D, NT>::REG_WARPS / GM<D, NT>::MAX_WARPS)
    gs_mma_kernel(const AttnParams P, int n_items, int sm_count) {
    using C = GM<D, NT>;
    extern __shared__ __align__(1024) uint8_t smem[];
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, WARPS = blockDim.x >> 5;
    // The call's first pass: launched as a programmatic dependent of
    // whatever precedes it on the stream, this grid may start before that
    // work has finished, so it waits for it (its writes visible) before
    // reading or writing anything.  Only then may the pass queued behind it
    // launch: the prompt-span pass reads the queries and the prompt stores
    // without a wait of its own, and it reads nothing this grid writes, so it
    // may take the SMs this grid's last CTAs leave.  (Behind the prompt-span
    // pass instead, that pass has waited before it let this grid launch, and
    // this grid reads what it writes only after that pass's completion flag,
    // with P.gs_merge; see the end of the kernel.)  No-ops for a plain
    // launch.
    if (!P.gs_after_prefix) {
        asm volatile("griddepcontrol.wait;" ::: "memory");
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    uint8_t* ws = smem + warp * C::per_warp(P.gs_rows);
    const uint32_t wbase = tc::smem_u32(ws);
    float* stg = reinterpret_cast<float*>(ws + C::off_stg(P.gs_rows));
    int4* ring = reinterpret_cast<int4*>(ws + C::OFF_TAKEN);
    int* pend = reinterpret_cast<int*>(ws + C::OFF_PEND);
    int npend = 0;
    const int g8 = lane >> 2, t4 = lane & 3;     // fragment row and column pair

    // ---- work items: the warp of rank r starts on item r.  As the call's
    // first pass (all warps start together) it then walks items r + k *
    // (warps of the grid): the extra items of an uneven share land on the
    // lowest ranks, so the other SMs come free whole and early for the
    // prompt-span pass queued behind.  Behind the prompt-span pass (CTAs
    // start as that pass's CTAs leave) every later item is claimed from the
    // launch-wide counter (numbered from the grid's warp count on), one
    // ahead: lane 0 holds the claim in flight, whose value is needed only
    // when the next item starts (the prompt-span pass clears the counter
    // before this grid can launch) ----
    const unsigned nwarps = gridDim.x * WARPS;
    // The warps' ranks.  With the prompt-span pass queued behind, SM-major
    // when the grid is whole waves of sm_count CTAs: the first wave's CTAs
    // land on distinct SMs and each later wave stacks one more CTA on each
    // in the same order, so CTAs b, b + sm_count, ... share an SM and get
    // consecutive ranks -- the extra items of an uneven share then fill
    // whole SMs, and the others come free together for that pass.  With
    // nothing queued behind, CTA-major, which spreads the extra items over
    // the SMs.
    int rank = int(blockIdx.x) * WARPS + warp;
    if (P.prefix_after_gs && sm_count > 0 && gridDim.x % unsigned(sm_count) == 0) {
        const int cps = int(gridDim.x) / sm_count;
        rank = ((int(blockIdx.x) % sm_count) * cps + int(blockIdx.x) / sm_count) * WARPS + warp;
    }
    const int first_item = rank;
    const bool claims = P.gs_after_prefix != 0;
    unsigned claim = unsigned(first_item) + nwarps;
    // d = 256 (fewer, longer items per warp): the claim goes out two blocks
    // before the item's end instead, so no warp holds an item it will not
    // start soon.
    constexpr bool kLateClaim = D == 256;
    bool have_claim = !claims || !kLateClaim;
    if (!kLateClaim && claims && lane == 0) claim = nwarps + atomicAdd(P.sched + 2, 1u);
    auto request = [&]() {
        if (!have_claim) {
            if (lane == 0) claim = nwarps + atomicAdd(P.sched + 2, 1u);
            have_claim = true;
        }
    };
    auto next_item = [&]() -> int {
        if constexpr (kLateClaim) {
            request();   // an item too short for the early request
            const int i = int(__shfl_sync(kFull, claim, 0));
            if (claims) {
                have_claim = false;
            } else {
                claim += nwarps;
            }
            return i < n_items ? i : -1;
        } else {
            const int i = int(__shfl_sync(kFull, claim, 0));
            if (i >= n_items) return -1;
            if (claims) {
                if (lane == 0) claim = nwarps + atomicAdd(P.sched + 2, 1u);
            } else {
                claim += nwarps;
            }
            return i;
        }
    };

    // ---- issue cursor: walks (item, block) in claim order and records every
    // item it takes, decoded (then the end, idx -1), for the consumer.  It
    // runs two blocks ahead and every item has a block (the host makes no
    // empty split), so it is at most two items ahead ----
    const ItemDivs dv{FastDiv(P.nss), FastDiv(P.gs_chunks), FastDiv(P.Hkv)};
    Item iss;
    int iss_idx = first_item < n_items ? first_item : -1, iss_b = 0, recorded = 0;
    bool iss_ok = false;
    auto record = [&](const Item& e) {
        if (lane == 0) {
            ring[2 * (recorded & 3)] = make_int4(e.idx, e.s, e.h, e.split);
            ring[2 * (recorded & 3) + 1] = make_int4(e.k0, e.k1, e.nblk, e.rc);
        }
        ++recorded;
    };
    auto seek = [&]() {   // the first block at or after item iss_idx
        iss_ok = false;
        while (iss_idx >= 0) {
            item_of(P, dv, iss_idx, iss);
            record(iss);
            if (iss.nblk > 0) {
                iss_ok = true;
                return;
            }
            iss_idx = next_item();
        }
        iss.idx = -1;
        record(iss);
    };
    seek();
    int issued = 0, iss_items = 0;
    // a copy instruction covers RPI rows: this lane's place in the first
    const uint32_t c_at = (lane / C::CH) * C::ROW + (((lane % C::CH) ^ (lane / C::CH)) * 16);
    const uint64_t pol = l2_evict_first_policy();
    size_t iss_base = iss_ok ? span_base<D>(P, iss.s, iss.h) : 0;
    // One commit group per call, empty once the walk has ended, so that a
    // block is always the second-newest group when it is waited for.
    auto issue_next = [&]() {
        if (iss_ok) {
            // an item's first block also brings the item's query rows
            // (contiguous in q) into its query buffer
            if (iss_b == 0) {
                const uint32_t qd = wbase + C::OFF_Q + (iss_items & 1) * (P.gs_rows * C::ROW);
                const uint16_t* qs = P.q + (size_t(iss.s) * P.Hq + iss.h * P.G + iss.rc * P.gs_rows) * D;
                const int rows = min(P.gs_rows, P.G - iss.rc * P.gs_rows);
                for (int e = lane; e < rows * C::CH; e += 32) {
                    const int r = e / C::CH, c = e % C::CH;
                    cp16_plain(qd + r * C::ROW + ((c ^ (r & 7)) * 16), qs + e * 8);
                }
                ++iss_items;
            }
            const int j = iss.k0 + iss_b * 16;
            int nk = min(16, iss.k1 - j);
            // fused append: entry step - 1 (the block's last row) is not in the
            // store yet; the consumer writes that row of the stage from registers
            if (P.fuse_append && j + nk == P.s_hi) --nk;
            const size_t src = iss_base + size_t(j) * D + lane * 8;
            const uint32_t at = wbase + (issued & 1) * C::STAGE + c_at;
            if (nk == 16) {
#pragma unroll
                for (int i = 0; i < C::BK / C::RPI; ++i) {
                    const uint32_t to = (at ^ ((i * C::RPI & 7) * 16)) + i * C::RPI * C::ROW;
                    cp16<true>(to, P.ks + src + i * 256, 16, pol);
                    cp16<true>(to + C::KBYTES, P.vs + src + i * 256, 16, pol);
                }
            } else {
#pragma unroll
                for (int i = 0; i < C::BK / C::RPI; ++i) {
                    const uint32_t to = (at ^ ((i * C::RPI & 7) * 16)) + i * C::RPI * C::ROW;
                    const bool live = i * C::RPI + lane / C::CH < nk;
                    const size_t from = live ? src + i * 256 : iss_base;
                    cp16<false>(to, P.ks + from, live ? 16 : 0, pol);
                    cp16<false>(to + C::KBYTES, P.vs + from, live ? 16 : 0, pol);
                }
            }
            ++issued;
            if constexpr (kLateClaim) {
                if (claims && iss_b + 2 >= iss.nblk) request();
            }
            if (++iss_b >= iss.nblk) {
                iss_b = 0;
                iss_idx = next_item();
                seek();
                if (iss_ok) iss_base = span_base<D>(P, iss.s, iss.h);
            }
        }
        cp_commit();
    };
    issue_next();
    issue_next();

    int consumed = 0, cons_items = 0;
    bool ps_ready = false;   // the prompt-span pass's states are complete and visible
    // matrix-load lanes: lane i gives the row address of matrix i / 8
    const int k_row = (lane & 7) + ((lane >> 3) & 1) * 8, k_ch = lane >> 4;     // K: keys 0-7, 8-15; chunk lo, hi
    const int v_row = (lane & 7) + (lane >> 4) * 8, v_ch = (lane >> 3) & 1;     // V (transposed)
    const int q_ch = lane >> 3;                                                 // Q: four chunks of eight rows
    const uint32_t k_at = k_row * C::ROW + ((k_ch ^ (k_row & 7)) * 16), v_at = v_row * C::ROW + ((v_ch ^ (v_row & 7)) * 16);
    // chunk 2 c + (0, 1) of a swizzled row, given the row's chunk 0 (or 1)
    auto chunk2 = [](uint32_t at, int c) { return (at ^ ((c & 3) * 32)) + (c >> 2) * 128; };
    // the epilogue's lanes: row e_row of a pass, 16 bytes e_c
    const int e_row = lane / C::LPR, e_c = lane % C::LPR;
    for (int taken = 0;; ++taken) {
        __syncwarp();
        const int4 e0 = ring[2 * (taken & 3)];
        if (e0.x < 0) break;
        const int4 e1 = ring[2 * (taken & 3) + 1];
        const Item it{e0.x, e0.y, e0.z, e0.w, e1.x, e1.y, e1.z, e1.w};
        // merges in this pass: the rows' source (a ZERO row needs no
        // prompt-span state) and, until it has been seen set, the prompt-span
        // pass's completion flag, read now and used at the item's end
        unsigned code = 0, poll = 0;
        if (C::MERGE && P.gs_merge) {
            code = P.src[it.s];
            if (!ps_ready) poll = ld_relaxed_gpu(P.sched + 4);
        }
        // fused append: this item's split ends at the step's own entry (step
        // - 1), which comes from the new K/V rows, loaded now (lanes take
        // 16-byte chunks: the K row's D / 8, then the V row's)
        constexpr int NCH = D / 4;                       // 16-byte chunks of the K and V rows
        constexpr int CPL = NCH >= 32 ? NCH / 32 : 1;    // chunks per lane
        const bool tail = P.fuse_append && it.k1 == P.s_hi && it.nblk > 0;
        uint4 nkv[CPL];
        if (tail) {
            const size_t rowc = (size_t(it.s) * P.Hkv + it.h) * (D / 8);
#pragma unroll
            for (int i = 0; i < CPL; ++i) {
                const int c = lane + 32 * i;
                if (c < NCH)
                    nkv[i] = c < D / 8 ? reinterpret_cast<const uint4*>(P.kn)[rowc + c]
                                       : reinterpret_cast<const uint4*>(P.vn)[rowc + c - D / 8];
            }
        }
        const uint32_t qaddr = wbase + C::OFF_Q + (cons_items & 1) * (P.gs_rows * C::ROW);
        // (columns past the item's rows read its last row again and are not used)
        const int rows = min(P.gs_rows, P.G - it.rc * P.gs_rows);
        uint32_t q_at[NT];
#pragma unroll
        for (int n = 0; n < NT; ++n) {
            const int r = min(8 * n + (lane & 7), rows - 1);
            q_at[n] = r * C::ROW + ((q_ch ^ (r & 7)) * 16);
        }
        if (it.nblk > 0) ++cons_items;
        // Q as the column operand: fragment kk covers dims 16 kk .. 16 kk + 15
        uint32_t qf[C::QREG ? NT : 1][C::QREG ? D / 16 : 1][2];
        // m, l of query rows 2 t4, 2 t4 + 1 of every column tile: m the same
        // in the eight lanes of a column pair, l each lane's own share
        float m[NT][2], l[NT][2];
        float o[NT][D / 16][4];                          // O^T: dims 16 i + g8 (+ 8), rows 2 t4, 2 t4 + 1
#pragma unroll
        for (int n = 0; n < NT; ++n) {
#pragma unroll
            for (int e = 0; e < 2; ++e) {
                m[n][e] = -INFINITY;
                l[n][e] = 0.f;
            }
#pragma unroll
            for (int i = 0; i < D / 16; ++i)
#pragma unroll
                for (int e = 0; e < 4; ++e) o[n][i][e] = 0.f;
        }

        for (int b = 0; b < it.nblk; ++b) {
            cp_wait<1>();
            __syncwarp();
            const int stg_i = consumed & 1;
            const uint32_t kst = wbase + stg_i * C::STAGE, vst = kst + C::KBYTES;
            const int jb = it.k0 + b * 16;
            if (C::QREG && b == 0) {
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int kk = 0; kk < D / 16; kk += 2) {
                        uint32_t r[4];
                        ldsm4(r, chunk2(qaddr + q_at[n], kk));
                        qf[n][kk][0] = r[0];
                        qf[n][kk][1] = r[1];
                        qf[n][kk + 1][0] = r[2];
                        qf[n][kk + 1][1] = r[3];
                    }
            }
            if (tail && b == it.nblk - 1) {
                // the step's own entry: its row of the stage from registers,
                // and (once per (sequence, kv head)) into the store
                const int rj = P.s_hi - 1 - jb;
                const size_t ent = ((size_t(it.s) * P.N + P.layer) * P.Hkv + it.h) * size_t(P.T) + (P.s_hi - 1);
#pragma unroll
                for (int i = 0; i < CPL; ++i) {
                    const int c = lane + 32 * i;
                    if (c < NCH) {
                        const bool isk = c < D / 8;
                        const int cc = isk ? c : c - D / 8;
                        *reinterpret_cast<uint4*>(ws + stg_i * C::STAGE + (isk ? 0u : C::KBYTES) + rj * C::ROW +
                                                  ((cc ^ (rj & 7)) * 16)) = nkv[i];
                        if (it.rc == 0)
                            reinterpret_cast<uint4*>(isk ? P.ks_w : P.vs_w)[ent * (D / 8) + cc] = nkv[i];
                    }
                }
                __syncwarp();
            }

            // ---- S^T = K Q^T: 16 keys x 8 rows per column tile; every two
            // products of the tensor core are added by an fp32 addition ----
            // (several pairs at a time, so that the products overlap)
            constexpr int QI = NT == 1 ? (D == 64 ? 2 : 4) : 2;
            float s[NT][4];
#pragma unroll
            for (int k0 = 0; k0 < D / 16; k0 += 2 * QI) {
                uint32_t a[2 * QI][4], q4[NT][QI][4];
                float x[NT][QI][4] = {};
#pragma unroll
                for (int i = 0; i < 2 * QI; ++i) ldsm4(a[i], chunk2(kst + k_at, k0 + i));
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int i = 0; i < QI; ++i) {
                        if constexpr (C::QREG) {
                            q4[n][i][0] = qf[n][k0 + 2 * i][0];
                            q4[n][i][1] = qf[n][k0 + 2 * i][1];
                            q4[n][i][2] = qf[n][k0 + 2 * i + 1][0];
                            q4[n][i][3] = qf[n][k0 + 2 * i + 1][1];
                        } else {
                            ldsm4(q4[n][i], chunk2(qaddr + q_at[n], k0 + 2 * i));
                        }
                    }
#pragma unroll
                for (int h = 0; h < 2; ++h)
#pragma unroll
                    for (int n = 0; n < NT; ++n)
#pragma unroll
                        for (int i = 0; i < QI; ++i)
                            mma(x[n][i], a[2 * i + h], q4[n][i][2 * h], q4[n][i][2 * h + 1], x[n][i]);
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int e = 0; e < 4; ++e) {
#pragma unroll
                        for (int w = QI / 2; w > 0; w >>= 1)
#pragma unroll
                            for (int i = 0; i < w; ++i) x[n][i][e] += x[n][i + w][e];
                        s[n][e] = k0 == 0 ? x[n][0][e] : s[n][e] + x[n][0][e];
                    }
            }
            // ---- logits in log2 units; keys past the split's end weigh nothing ----
            const bool live0 = jb + g8 < it.k1, live1 = jb + 8 + g8 < it.k1;
            bool need = false;
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    s[n][e] = (e < 2 ? live0 : live1) ? s[n][e] * P.scale_log2 : -INFINITY;
                    need |= s[n][e] > m[n][e & 1] + kTau;
                }
            if (__any_sync(kFull, need)) {
                // rare: some row's reference max moves
#pragma unroll
                for (int n = 0; n < NT; ++n)
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        float mb = fmaxf(s[n][e], s[n][e + 2]);
#pragma unroll
                        for (int off = 4; off < 32; off <<= 1) mb = fmaxf(mb, __shfl_xor_sync(kFull, mb, off));
                        if (mb > m[n][e] + kTau) {
                            const float alpha = ex2(m[n][e] - mb);
                            l[n][e] *= alpha;
#pragma unroll
                            for (int i = 0; i < D / 16; ++i) {
                                o[n][i][e] *= alpha;
                                o[n][i][e + 2] *= alpha;
                            }
                            m[n][e] = mb;
                        }
                    }
            }
            // ---- probabilities, as the column operand P^T in three terms ----
            uint32_t pf[NT][3][2];
#pragma unroll
            for (int n = 0; n < NT; ++n) {
                float p[4];
#pragma unroll
                for (int e = 0; e < 4; ++e) {
                    const float mr = m[n][e & 1] == -INFINITY ? 0.f : m[n][e & 1];
                    p[e] = ex2(s[n][e] - mr);
                    l[n][e & 1] += p[e];
                }
                uint32_t w0[3], w1[3];
                split3(p[0], p[1], w0);
                split3(p[2], p[3], w1);
#pragma unroll
                for (int i = 0; i < 3; ++i) {
                    pf[n][i][0] = movm_t(w0[i]);
                    pf[n][i][1] = movm_t(w1[i]);
                }
            }
            // ---- O^T += V^T P^T, the smallest terms first; four tiles of
            // dims at a time, so that their chains of three overlap ----
            constexpr int IL = NT == 1 ? 4 : 2;
#pragma unroll
            for (int i0 = 0; i0 < D / 16; i0 += IL) {
                uint32_t a[IL][4];
#pragma unroll
                for (int i = 0; i < IL; ++i)
                    ldsm4_t(a[i], chunk2(vst + v_at, i0 + i));
                float x[IL][NT][4] = {};
#pragma unroll
                for (int w = 2; w >= 0; --w)
#pragma unroll
                    for (int i = 0; i < IL; ++i)
#pragma unroll
                        for (int n = 0; n < NT; ++n) mma(x[i][n], a[i], pf[n][w][0], pf[n][w][1], x[i][n]);
#pragma unroll
                for (int i = 0; i < IL; ++i)
#pragma unroll
                    for (int n = 0; n < NT; ++n)
#pragma unroll
                        for (int e = 0; e < 4; e += 2) {
                            const float2 y = __fadd2_rn(make_float2(o[n][i0 + i][e], o[n][i0 + i][e + 1]),
                                                        make_float2(x[i][n][e], x[i][n][e + 1]));
                            o[n][i0 + i][e] = y.x;
                            o[n][i0 + i][e + 1] = y.y;
                        }
            }
            // stage free: every lane is done reading it
            __syncwarp();
            ++consumed;
            issue_next();
        }

        // ---- merge here?  Always for a ZERO row; for the others once the
        // prompt-span pass has completed, whose states are fetched now, under
        // the row sums below.  An item that ends before then writes its
        // partial state and is merged at the warp's end (up to kPend of
        // them; past that the warp waits for the prompt-span grid here) ----
        bool merge_here = false;
        const bool has_span = code != SPLICE_SRC_ZERO;
        const size_t row0 = size_t(it.s) * P.Hq + it.h * P.G + it.rc * P.gs_rows;
        constexpr int NPM = C::MERGE ? C::NP : 1;
        float2 ml_span[NPM];
        float4 o_span[C::AHEAD][NPM];
        if (C::MERGE && P.gs_merge) {
            if (!ps_ready && __all_sync(kFull, poll != 0u)) {
                asm volatile("fence.acq_rel.gpu;" ::: "memory");
                ps_ready = true;
            }
            merge_here = !has_span || ps_ready;
            if (!merge_here) {
                if (npend < kPend) {
                    if (lane == 0) pend[npend] = it.idx;
                    ++npend;
                } else {
                    asm volatile("griddepcontrol.wait;" ::: "memory");
                    ps_ready = true;
                    merge_here = true;
                }
            }
            if (merge_here && has_span) {
#pragma unroll
                for (int k = 0; k < NPM; ++k) {
                    const int r = k * C::RPP + e_row;
                    if (r < rows) {
                        ml_span[k] = __ldcg(P.ws_ml + row0 + r);     // split 0's slot
                        const float4* sp = reinterpret_cast<const float4*>(P.ws_o + (row0 + r) * D) + e_c;
#pragma unroll
                        for (int hh = 0; hh < C::AHEAD; ++hh) o_span[hh][k] = __ldcg(sp + hh * C::LPR);
                    }
                }
            }
        }

        // ---- row sums over the lanes of a column pair ----
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int e = 0; e < 2; ++e)
#pragma unroll
                for (int off = 4; off < 32; off <<= 1) l[n][e] += __shfl_xor_sync(kFull, l[n][e], off);

        // ---- an infinite or NaN sum: the three terms of a probability
        // times an infinite value need not add up to what their sum times it
        // is (0 x inf among them), so such sums are made again term by term ----
        float2 nan0 = make_float2(0.f, 0.f), nan1 = nan0;    // 0 x o: NaN where o is not finite
#pragma unroll
        for (int n = 0; n < NT; ++n)
#pragma unroll
            for (int i = 0; i < D / 16; ++i) {
                nan0 = __ffma2_rn(make_float2(o[n][i][0], o[n][i][1]), make_float2(0.f, 0.f), nan0);
                nan1 = __ffma2_rn(make_float2(o[n][i][2], o[n][i][3]), make_float2(0.f, 0.f), nan1);
            }
        if (__any_sync(kFull, !((nan0.x + nan0.y) + (nan1.x + nan1.y) == 0.f))) {
            const size_t base = span_base<D>(P, it.s, it.h);
            const size_t nrow = (size_t(it.s) * P.Hkv + it.h) * D;
#pragma unroll
            for (int n = 0; n < NT; ++n) {
#pragma unroll
                for (int i = 0; i < D / 16; ++i)
#pragma unroll
                    for (int e = 0; e < 4; ++e) o[n][i][e] = 0.f;
#pragma unroll 1
                for (int j = it.k0; j < it.k1; ++j) {
                    const bool own = P.fuse_append && j == P.s_hi - 1;
                    const uint16_t* kr = own ? P.kn + nrow : P.ks + base + size_t(j) * D;
                    const uint16_t* vr = own ? P.vn + nrow : P.vs + base + size_t(j) * D;
                    float p[2];
#pragma unroll
                    for (int e = 0; e < 2; ++e) {
                        const int r = 8 * n + 2 * t4 + e;
                        float z = 0.f;
                        if (r < rows) {
                            const uint16_t* qr = P.q + (row0 + r) * D;
#pragma unroll 1
                            for (int c = 0; c < D; ++c)
                                z = fmaf(__uint_as_float(uint32_t(qr[c]) << 16), __uint_as_float(uint32_t(kr[c]) << 16), z);
                        }
                        p[e] = ex2(z * P.scale_log2 - (m[n][e] == -INFINITY ? 0.f : m[n][e]));
                    }
#pragma unroll
                    for (int i = 0; i < D / 16; ++i)
#pragma unroll
                        for (int e = 0; e < 4; ++e)
                            o[n][i][e] = fmaf(p[e & 1], __uint_as_float(uint32_t(vr[16 * i + g8 + (e >> 1) * 8]) << 16),
                                              o[n][i][e]);
                }
            }
        }

        // ---- the rows' (m, l) on the epilogue's lanes, and the weights of a
        // merge; then O, staged half the dims at a time so that it leaves
        // (and, merged, meets the prompt-span states) row by row ----
        float mr[C::NP], lr[C::NP], w_span[NPM], w_gen[NPM], inv[NPM];
#pragma unroll
        for (int k = 0; k < C::NP; ++k) {
            if (k * C::RPP >= rows) break;
            const int r = k * C::RPP + e_row, src = (r & 7) >> 1;
            float mm = 0.f, ll = 0.f;
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int e = 0; e < 2; ++e) {
                    const float a = __shfl_sync(kFull, m[n][e], src), c = __shfl_sync(kFull, l[n][e], src);
                    if ((r >> 3) == n && (r & 1) == e) {
                        mm = a;
                        ll = c;
                    }
                }
            mr[k] = mm;
            lr[k] = ll;
            if (C::MERGE && merge_here)
                inv[k % NPM] = merge_two_weights(has_span, has_span ? ml_span[k % NPM] : make_float2(-INFINITY, 0.f), mm, ll,
                                                 !has_span && P.p_hi > P.p_lo, P.p_hi - P.p_lo, &w_span[k % NPM],
                                                 &w_gen[k % NPM]);
        }
        const size_t gen0 = size_t(kMaxPrefixSplits + it.split) * P.B * P.Hq + row0;
#pragma unroll
        for (int hh = 0; hh < 2; ++hh) {
            if (C::MERGE && hh >= C::AHEAD && merge_here && has_span) {
#pragma unroll
                for (int k = 0; k < NPM; ++k) {
                    const int r = k * C::RPP + e_row;
                    if (r < rows) o_span[0][k] = __ldcg(reinterpret_cast<const float4*>(P.ws_o + (row0 + r) * D) + C::LPR + e_c);
                }
            }
            __syncwarp();
#pragma unroll
            for (int n = 0; n < NT; ++n)
#pragma unroll
                for (int i = 0; i < D / 32; ++i)
#pragma unroll
                    for (int e = 0; e < 4; ++e)
                        if (8 * n + 2 * t4 + (e & 1) < rows)
                            stg[(8 * n + 2 * t4 + (e & 1)) * C::LDO + 16 * i + g8 + (e >> 1) * 8] = o[n][hh * (D / 32) + i][e];
            __syncwarp();
#pragma unroll
            for (int k = 0; k < C::NP; ++k) {
                const int r = k * C::RPP + e_row;
                if (r < rows) {
                    const float4 x = *reinterpret_cast<const float4*>(stg + r * C::LDO + 4 * e_c);
                    if (C::MERGE && merge_here) {
                        const float4 sp = has_span ? o_span[hh % C::AHEAD][k % NPM] : make_float4(0.f, 0.f, 0.f, 0.f);
                        reinterpret_cast<float4*>(P.out + (row0 + r) * D)[hh * C::LPR + e_c] =
                            merge_two4(has_span, w_span[k % NPM], sp, w_gen[k % NPM], x, inv[k % NPM]);
                    } else {
                        reinterpret_cast<float4*>(P.ws_o + (gen0 + r) * D)[hh * C::LPR + e_c] = x;
                        if (hh == 0 && e_c == 0) P.ws_ml[gen0 + r] = make_float2(mr[k], lr[k]);
                    }
                }
            }
        }
    }
    cp_wait<0>();
    if (P.gs_after_prefix && (blockIdx.x == 0 || npend > 0)) {
        // Behind the prompt-span pass: this grid's completion must imply that
        // pass's, so the merge queued behind this grid sees both (with
        // P.gs_merge no merge is queued: this grid writes every output).  One
        // CTA that waits for that pass is enough; the others go, and leave
        // their SMs to this grid's CTAs that found none beside that pass (36 x
        // 8 heads, sixteen rows of 256 dims, three keys each, beside 48
        // prompt-span CTAs: 30.6 us when all waited, 25.3 so).
        // Then the work behind may launch (the merge waits for this whole
        // grid before it reads anything); every CTA of this grid is running
        // by the time all of them have signalled or gone, so those CTAs never
        // hold an SM it still needs.
        asm volatile("griddepcontrol.wait;" ::: "memory");
        // The items left unmerged: the prompt-span states are complete and
        // visible now; this warp's own partial states are re-read (the same
        // bits it stored) and merged as at an item's end.
        if constexpr (C::MERGE) {
            if (P.gs_merge && npend > 0) {
                __syncwarp();
                for (int k = 0; k < npend; ++k) {
                    Item it;
                    item_of(P, dv, pend[k], it);
                    const size_t row0 = size_t(it.s) * P.Hq + it.h * P.G + it.rc * P.gs_rows;
                    const int rows = min(P.gs_rows, P.G - it.rc * P.gs_rows);
                    const size_t gen0 = size_t(kMaxPrefixSplits) * P.B * P.Hq + row0;
                    // (the loads of all passes go out before any is used)
                    constexpr int K = C::NP;
                    for (int r0 = e_row; r0 - e_row < rows; r0 += K * C::RPP) {
                        float2 ml_gen[K], ml_span[K];
                        float4 og[K][2], os[K][2];
#pragma unroll
                        for (int i = 0; i < K; ++i) {
                            const int r = r0 + i * C::RPP;
                            if (r < rows) {
                                ml_gen[i] = __ldcg(P.ws_ml + gen0 + r);
                                ml_span[i] = __ldcg(P.ws_ml + row0 + r);
#pragma unroll
                                for (int hh = 0; hh < 2; ++hh) {
                                    og[i][hh] = __ldcg(reinterpret_cast<const float4*>(P.ws_o + (gen0 + r) * D) + hh * C::LPR + e_c);
                                    os[i][hh] = __ldcg(reinterpret_cast<const float4*>(P.ws_o + (row0 + r) * D) + hh * C::LPR + e_c);
                                }
                            }
                        }
#pragma unroll
                        for (int i = 0; i < K; ++i) {
                            const int r = r0 + i * C::RPP;
                            if (r < rows) {
                                float w_span, w_gen;
                                const float inv = merge_two_weights(true, ml_span[i], ml_gen[i].x, ml_gen[i].y, false, 0,
                                                                    &w_span, &w_gen);
                                float4* op = reinterpret_cast<float4*>(P.out + (row0 + r) * D) + e_c;
#pragma unroll
                                for (int hh = 0; hh < 2; ++hh)
                                    op[hh * C::LPR] = merge_two4(true, w_span, os[i][hh], w_gen, og[i][hh], inv);
                            }
                        }
                    }
                }
            }
        }
        asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
    }
    // (Run-time claims: the prompt-span pass ahead of this grid cleared the
    // item counter before this grid could launch.)
}

// Launch shape for G query rows: warps per CTA and CTAs per SM, as many warps
// as the registers and the shared memory of an SM allow.
template <int D, int NT>
struct Shape {
    int warps = 1, ctas = 1;
    explicit Shape(int G) {
        using C = GM<D, NT>;
        for (int w = C::MAX_WARPS; w > 0; --w) {
            const int fit = int((228u * 1024u) / (w * C::per_warp(G) + 1024u));
            const int c = fit < C::REG_WARPS / w ? fit : C::REG_WARPS / w;
            if (c * w > ctas * warps) {
                warps = w;
                ctas = c;
            }
        }
    }
};

template <int D, int NT>
int launch_mma_t(const AttnParams& p, int n_items, cudaStream_t st, bool overlap_previous) {
    using C = GM<D, NT>;
    static PerDevice<int> kept;
    int sms = 0;
    const cudaError_t e = kept.get(&sms, [](int dev, int* n) {
        const cudaError_t err = cudaFuncSetAttribute(gs_mma_kernel<D, NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
        return err != cudaSuccess ? err : cudaDeviceGetAttribute(n, cudaDevAttrMultiProcessorCount, dev);
    });
    if (e != cudaSuccess) return int(e);
    Shape<D, NT> sh(p.gs_rows);
    // few items: spread over the SMs rather than a CTA's warps
    sh.warps = int(std::min<long>(sh.warps, (long(n_items) + sms - 1) / sms));
    const long want = (long(n_items) + sh.warps - 1) / sh.warps;
    const long cap = long(sh.ctas) * sms;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(want < cap ? want : cap));
    cfg.blockDim = dim3(unsigned(sh.warps) * 32);
    cfg.dynamicSmemBytes = sh.warps * C::per_warp(p.gs_rows);
    cfg.stream = st;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = attr;
    cfg.numAttrs = overlap_previous ? 1 : 0;
    return int(cudaLaunchKernelEx(&cfg, gs_mma_kernel<D, NT>, p, n_items, sms));
}

}  // namespace

int launch_mma(const AttnParams& p, cudaStream_t stream, bool overlap_previous) {
    const int n_items = int(long(p.B) * p.Hkv * p.gs_chunks * p.nss);
    const bool two = p.gs_rows > 8;
    switch (p.D) {
        case 64:
            return two ? launch_mma_t<64, 2>(p, n_items, stream, overlap_previous)
                       : launch_mma_t<64, 1>(p, n_items, stream, overlap_previous);
        case 128:
            return two ? launch_mma_t<128, 2>(p, n_items, stream, overlap_previous)
                       : launch_mma_t<128, 1>(p, n_items, stream, overlap_previous);
        case 256:
            return two ? launch_mma_t<256, 2>(p, n_items, stream, overlap_previous)
                       : launch_mma_t<256, 1>(p, n_items, stream, overlap_previous);
        default: return int(cudaErrorInvalidValue);
    }
}

namespace {
template <int D, int NT>
int warps_per_sm(int rows) {
    const Shape<D, NT> s(rows);
    return s.warps * s.ctas;
}
}  // namespace

int mma_warps_per_sm(int d, int rows) {
    if (rows > 8) return d == 64 ? warps_per_sm<64, 2>(rows) : (d == 128 ? warps_per_sm<128, 2>(rows) : warps_per_sm<256, 2>(rows));
    return d == 64 ? warps_per_sm<64, 1>(rows) : (d == 128 ? warps_per_sm<128, 1>(rows) : warps_per_sm<256, 1>(rows));
}

bool mma_can_merge(int d, int rows) { return d * (rows > 8 ? 2 : 1) <= 256; }   // GM::MERGE

}  // namespace gs
}  // namespace splice
