// Delta encoding of the stored donor spans against the clean spans.
//
// A stored donor span (prompt p, stored slot st, layer l, kv head h) is
// aligned position by position with the clean span of (p, l, h): §3 trims
// donor and target prompts to the same length.  Position j is encoded iff
// the donor's K row or V row at j differs bit for bit from the clean span's.
// Attention over the donor span is then the log-sum-exp merge of attention
// over the clean span without the encoded positions and attention over the
// encoded rows, so readers of a donor that shares most positions with the
// clean prompt read the clean span (which its clean readers read anyway)
// plus a short run of encoded rows.
//
// A cluster of CTAs per span, one pass over it in rounds of consecutive
// chunks of positions, one chunk per CTA:
//   1. each warp loads its rows of the chunk -- the donor's and the clean
//      span's K and V, eight pairs of 16-byte loads per lane in flight --
//      and compares them; the row's bit goes into the chunk's mask words;
//   2. the CTAs of the cluster trade their chunks' counts through
//      distributed shared memory (one cluster barrier per round, the counts
//      double-buffered by round parity), so every warp knows the output row
//      of its first encoded row;
//   3. the encoded rows are stored from the registers they were compared in.
// After the last round the rows count .. T_p-1 are zeroed, so a 128-row tile
// that runs past the count reads zeros, never stale memory.
//
// HBM-bound: every donor row is read once and every output row written once;
// the clusters of one clean span's donors are neighbours in launch order, so
// that span comes from HBM about once and from L2 for the others.  (One CTA
// per span that compared a row per warp at a time and read the encoded rows
// again for the copy took 1.33 ms for six prompts of 4096 positions, four
// donors, four layers, 8 heads of 128: 3.6 GB.  This takes 0.62 ms, 5.8 TB/s;
// splice_delta_build as a whole 1.44 -> 0.74 ms, the rest host work on the tables.)
#include <cooperative_groups.h>
#include <cuda_runtime.h>

#include "splice_internal.h"

namespace cg = cooperative_groups;

namespace splice {
namespace {

constexpr int kDeltaThreads = 256, kDeltaWarps = kDeltaThreads / 32;
constexpr int kMaxCluster = 8;

template <int D>
struct DeltaCfg {
    static constexpr int C = D / 8;                            // 16-byte chunks of a K (or V) row
    static constexpr int LPR = 2 * C < 32 ? 2 * C : 32;        // lanes of one row's K and V
    static constexpr int RPI = 32 / LPR;                       // rows per load instruction
    static constexpr int IPR = 2 * C / LPR;                    // load instructions per row
    static constexpr int LOADS = 8;                            // load pairs in flight per lane
    static constexpr int ROWS = LOADS * RPI / IPR;             // rows per warp and round: 16, 8, 4
    static constexpr int CHUNK = ROWS * kDeltaWarps;           // positions per CTA and round: 128, 64, 32
};

// The donor's row pair, clean row pair and output row pair of one position
// are C chunks of K and C of V; lane i of a row's LPR lanes holds chunks i,
// i + LPR, ... of the 2 C.
template <int D>
__global__ void __launch_bounds__(kDeltaThreads, 3) delta_build_kernel(
    const uint4* __restrict__ kc, const uint4* __restrict__ vc, const uint4* __restrict__ kd,
    const uint4* __restrict__ vd, uint32_t* __restrict__ mask, int32_t* __restrict__ count, uint4* __restrict__ xk,
    uint4* __restrict__ xv, int Dst, int N, int Hkv, int Tp, int w32) {
    using F = DeltaCfg<D>;
    __shared__ uint32_t words[F::CHUNK / 32];
    __shared__ int peers[2][kMaxCluster];              // [round parity][rank] encoded rows of the peers' chunks
    cg::cluster_group cluster = cg::this_cluster();
    const int rank = int(cluster.block_rank()), nrank = int(cluster.num_blocks());
    // span number in launch order: ((p * N + l) * Hkv + h) * Dst + st
    const long id = long(blockIdx.x) / nrank;
    const long st = id % Dst, clean = id / Dst;
    const long h = clean % Hkv, l = (clean / Hkv) % N, p = clean / (long(Hkv) * N);
    const long sp = ((p * Dst + st) * N + l) * Hkv + h;         // span number in the stores
    const size_t crow = size_t(clean) * size_t(Tp);             // first row of the clean span
    const size_t drow = size_t(sp) * size_t(Tp);                // of the donor span and of its delta rows
    const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
    const int sub = lane / F::LPR, rl = lane % F::LPR;
    const int chunks = w32 * 32 / F::CHUNK;                     // whole: w32 is a multiple of 4
    if (nrank > 1) cluster.sync();                              // the peers' shared memory is there
    int done = 0;                                               // encoded rows of the chunks before this round's
    for (int c0 = 0, round = 0; c0 < chunks; c0 += nrank, ++round) {
        const int chunk = c0 + rank;
        const int j0 = chunk * F::CHUNK + warp * F::ROWS;       // the warp's first position
        uint4 a[F::LOADS], b[F::LOADS];
#pragma unroll
        for (int i = 0; i < F::LOADS; ++i) {
            const int j = j0 + (i / F::IPR) * F::RPI + sub;
            const int c = rl + (i % F::IPR) * F::LPR;
            const bool is_k = c < F::C;
            const int cc = is_k ? c : c - F::C;
            a[i] = b[i] = make_uint4(0u, 0u, 0u, 0u);
            if (j < Tp && chunk < chunks) {
                a[i] = __ldcs((is_k ? kd : vd) + (drow + j) * F::C + cc);
                b[i] = __ldg((is_k ? kc : vc) + (crow + j) * F::C + cc);
            }
        }
        uint32_t bits = 0;                                      // bit r: row j0 + r is encoded
#pragma unroll
        for (int i = 0; i < F::LOADS; i += F::IPR) {
            bool diff = false;
#pragma unroll
            for (int k = 0; k < F::IPR; ++k)
                diff |= (a[i + k].x != b[i + k].x) | (a[i + k].y != b[i + k].y) | (a[i + k].z != b[i + k].z) |
                        (a[i + k].w != b[i + k].w);
            const uint32_t vote = __ballot_sync(0xffffffffu, diff);
#pragma unroll
            for (int r = 0; r < F::RPI; ++r) {
                const uint32_t lanes = F::LPR == 32 ? 0xffffffffu : ((1u << F::LPR) - 1u) << (r * F::LPR);
                bits |= (vote & lanes) ? 1u << ((i / F::IPR) * F::RPI + r) : 0u;
            }
        }
        __syncthreads();                                        // the previous round's words have been read
        if (lane == 0) {
            if constexpr (F::ROWS == 16)
                reinterpret_cast<uint16_t*>(words)[warp] = uint16_t(bits);
            else if constexpr (F::ROWS == 8)
                reinterpret_cast<uint8_t*>(words)[warp] = uint8_t(bits);
            else if (warp == 0)
                words[0] = 0u;
        }
        __syncthreads();
        if constexpr (F::ROWS == 4) {
            if (lane == 0) atomicOr(words, bits << (4 * warp));
            __syncthreads();
        }
        // encoded rows of the chunk, and those before this warp's rows
        int total = 0, before = 0;
#pragma unroll
        for (int w = 0; w < F::CHUNK / 32; ++w) {
            const uint32_t v = words[w];
            const int lo = warp * F::ROWS - 32 * w;             // rows of the word before the warp's
            total += __popc(v);
            before += lo >= 32 ? __popc(v) : (lo > 0 ? __popc(v & ((1u << lo) - 1u)) : 0);
        }
        if (threadIdx.x < F::CHUNK / 32 && chunk < chunks)
            mask[size_t(sp) * w32 + chunk * (F::CHUNK / 32) + threadIdx.x] = words[threadIdx.x];
        if (nrank > 1) {
            if (threadIdx.x < nrank) cluster.map_shared_rank(&peers[round & 1][0], threadIdx.x)[rank] = total;
            cluster.sync();
            int all = 0;
            for (int r = 0; r < nrank; ++r) {
                const int n = peers[round & 1][r];
                if (r < rank) before += n;
                all += n;
            }
            total = all;
        }
        const size_t first = drow + size_t(done + before);
#pragma unroll
        for (int i = 0; i < F::LOADS; ++i) {
            const int r = (i / F::IPR) * F::RPI + sub;
            const int c = rl + (i % F::IPR) * F::LPR;
            const bool is_k = c < F::C;
            const int cc = is_k ? c : c - F::C;
            if ((bits >> r) & 1u)
                __stcs((is_k ? xk : xv) + (first + __popc(bits & ((1u << r) - 1u))) * F::C + cc, a[i]);
        }
        done += total;
    }
    const uint4 z = make_uint4(0u, 0u, 0u, 0u);
    const size_t end = (drow + Tp) * F::C;
    for (size_t i = (drow + done) * F::C + size_t(rank) * kDeltaThreads + threadIdx.x; i < end;
         i += size_t(nrank) * kDeltaThreads) {
        __stcs(xk + i, z);
        __stcs(xv + i, z);
    }
    if (rank == 0 && threadIdx.x == 0) count[sp] = done;
}

template <int D>
int launch_delta_t(const uint4* kc, const uint4* vc, const uint4* kd, const uint4* vd, uint32_t* mask, int32_t* count,
                   uint4* xk, uint4* xv, long spans, int Dst, int N, int Hkv, int Tp, int w32, cudaStream_t stream) {
    int dev = 0, sms = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return int(e);
    // CTAs per span: enough for eight waves of three CTAs per SM (a last wave
    // that is nearly empty then costs little, and few spans still fill the
    // GPU), no more than the span has chunks.
    const int chunks = w32 * 32 / DeltaCfg<D>::CHUNK;
    int nrank = 1;
    while (nrank < kMaxCluster && 2 * nrank <= chunks && spans * nrank < 8L * 3 * sms) nrank *= 2;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(unsigned(spans * nrank));
    cfg.blockDim = dim3(kDeltaThreads);
    cfg.stream = stream;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeClusterDimension;
    attr[0].val.clusterDim.x = unsigned(nrank);
    attr[0].val.clusterDim.y = attr[0].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    return int(cudaLaunchKernelEx(&cfg, delta_build_kernel<D>, kc, vc, kd, vd, mask, count, xk, xv, Dst, N, Hkv, Tp, w32));
}

}  // namespace

int launch_delta_build(const uint16_t* kc, const uint16_t* vc, const uint16_t* kd, const uint16_t* vd,
                       uint32_t* mask, int32_t* count, uint16_t* xk, uint16_t* xv, int P, int Dst, int N,
                       int Hkv, int Tp, int D, int w32, void* stream) {
    const long spans = long(P) * Dst * N * Hkv;
    if (spans <= 0) return 0;
    auto u4 = [](const uint16_t* x) { return reinterpret_cast<const uint4*>(x); };
    auto launch = D == 64 ? launch_delta_t<64> : (D == 128 ? launch_delta_t<128> : launch_delta_t<256>);
    return launch(u4(kc), u4(vc), u4(kd), u4(vd), mask, count, reinterpret_cast<uint4*>(xk),
                  reinterpret_cast<uint4*>(xv), spans, Dst, N, Hkv, Tp, w32, static_cast<cudaStream_t>(stream));
}

}  // namespace splice
