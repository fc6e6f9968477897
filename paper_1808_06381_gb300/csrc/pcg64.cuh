// Conjugate gradients on chip: the building blocks shared by the solves of
// small FP64 and mixed systems (cg_persistent.cu) and the allocation-free solve
// of a caller's CSR system (noalloc.cu), each one cooperative launch.  The
// FP64 ones first:
//
// GB300 issues FP64 at 2 FMA per clock and SM, half an operation per clock on
// each of its four schedulers, so one FP64 instruction of a warp holds its
// scheduler for ~64 clocks: a solve of a few thousand rows is bound by the
// number of FP64 instructions on the longest path of an iteration and by the
// latency of its memory round trips, not by bytes.  Hence:
//   - rows come in chunks of 32; a warp owns one Cartesian component of a
//     chunk (lane = row), so a row's sum needs no shuffles and the update no
//     idle lanes: 32 of 32 lanes do FP64 work (four lanes per row with one
//     component each left a quarter idle and added six shuffled additions);
//   - a thread keeps its components' solver vectors in registers for the
//     whole solve, and the block keeps its chunks' entries (alpha w_ij and the
//     column) in shared memory: an iteration reads only its neighbours'
//     gathered values from global memory (one round trip; before, the slot
//     map, the chunk bounds, the columns and the gathers were a chain of four);
//   - gathered values are published as one 32-byte record per row (x, y, z, 0),
//     so the three warps of a chunk read the same sectors;
//   - the reductions add as little as possible: three values are summed over a
//     warp by 6 additions (15 one by one), the warps' sums by 5, and the blocks'
//     by three warps of their own that do nothing else, while the others gather
//     for the next product; A_ii D^-1_ii = 1 replaces the diagonal product.
#pragma once

#include "internal.cuh"

namespace ss {
namespace p64 {

constexpr int kMaxChunks = 64;      // chunks of 32 rows a block holds at most
constexpr int kMaxGroups = 5;       // chunks in flight (three warps each)
constexpr int kMaxWarps = 3 * kMaxGroups;
constexpr int kScalarWarps = 3;     // warps that sum the grid's partials, one value each
// threads of a block whose threads hold u chunks (from u = 4 on four groups, so that 128 registers are left a thread)
constexpr int max_threads(int u) { return 32 * ((u >= 4 ? 12 : kMaxWarps) + kScalarWarps); }
// an entry in shared memory: alpha w (FP64, or FP32 in the mixed solve) and the column
template <class V>
constexpr int kEntryBytes = (int)sizeof(V) + 4;
constexpr int kChunkSmem = 16 * 1024;        // shared memory planned per chunk (42 FP64 entries a row), one chunk spare
constexpr int kMaxSmem = 200 * 1024;

struct Grid {
    unsigned int* count;            // arrivals of this launch (grows; reset by the last block to leave)
    unsigned int* exits;
    int* error;                     // set to SP_ERR_TIMEOUT by a wait that ran past the limit
    unsigned long long limit_ns;
    double* partials;               // two sets of kScalarWarps * stride sums
    int stride;
    int bid, nb;
};

struct Shared {
    double wsum[kScalarWarps][kMaxWarps + 1];
    double tot[kScalarWarps];
    double alpha, beta;
    int off[kMaxChunks], len[kMaxChunks];   // first entry in shared memory (-1: read from global), entries a row
    int action, flag, bad;
};

__device__ __forceinline__ unsigned long long now_ns()
{
    unsigned long long t;
    asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
    return t;
}

// One arrival (thread 0's release covers the block's writes ordered before it
// by a block barrier), then a bounded wait for `target` arrivals.
__device__ __forceinline__ int arrive_and_wait(const Grid& G, unsigned int target)
{
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(G.count) : "memory");
    const unsigned long long t0 = now_ns();
    for (;;) {
        unsigned int v;
        asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(G.count) : "memory");
        if (v >= target) return 0;
        if (now_ns() - t0 > G.limit_ns) {
            atomicCAS(G.error, 0, (int)SP_ERR_TIMEOUT);
            return (int)SP_ERR_TIMEOUT;
        }
    }
}

__device__ __forceinline__ void leave(const Grid& G)
{
    __syncthreads();
    if (threadIdx.x == 0 && atomicAdd(G.exits, 1u) == (unsigned)G.nb - 1) {
        *G.count = 0u;
        *G.exits = 0u;
    }
}

// The sums of three values over a warp in 6 additions: the first exchange
// leaves value 0 in the lower half and value 1 in the upper, the second adds
// value 2 in the lanes with bit 3 set, three more finish all of them.  Lane 0
// returns the sum of v0, lane 16 of v1, lane 8 of v2.
__device__ __forceinline__ double warp_sum3(double v0, double v1, double v2)
{
    const int lane = threadIdx.x & 31;
    const bool up = lane & 16, third = lane & 8;
    double a = (up ? v1 : v0) + __shfl_xor_sync(0xffffffffu, up ? v0 : v1, 16);
    const double c = v2 + __shfl_xor_sync(0xffffffffu, v2, 16);
    a = (third ? c : a) + __shfl_xor_sync(0xffffffffu, third ? a : c, 8);
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
    return a;
}

// Reads the entries of the block's nc chunks into shared memory.  Sys gives, of
// the block's chunk i, the row of a lane (-1: none), the entries per row and
// the entries; its chunks are bid, bid + nb, ... of the system (strided, so
// that a dense region's long rows are shared out: with contiguous runs the
// densest block had 1.5x the mean entries, and overflowed).  A chunk that
// finds no room keeps off = -1 and is read through Sys in every product.  An
// entry beyond a row's own (weight 0) names the row of lane 0, so the padding
// lanes of a gather share one sector.  Ends with a block barrier.
template <class Sys>
__device__ __forceinline__ void stage(const Sys& S, Shared& sh, unsigned char* dyn, int smem_bytes, int nc)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nwarps = blockDim.x >> 5;
    if (threadIdx.x == 0) sh.bad = 0;
    for (int i = warp; i < nc; i += nwarps) {
        const int len = S.chunk_len(i, lane);
        if (lane == 0) sh.len[i] = len;
    }
    __syncthreads();
    using V = typename Sys::Value;
    const int cap = smem_bytes / kEntryBytes<V>;
    if (threadIdx.x == 0) {
        int at = 0;
        for (int i = 0; i < nc; ++i) {
            const long long want = 32ll * sh.len[i];
            sh.off[i] = at + want <= cap ? at : -1;
            if (sh.off[i] >= 0) at += (int)want;
        }
    }
    __syncthreads();
    V* val = reinterpret_cast<V*>(dyn);
    int* col = reinterpret_cast<int*>(dyn + sizeof(V) * (size_t)cap);
    constexpr int KS = 8;
    for (int i = warp; i < nc; i += nwarps) {
        const int row = S.row(i, lane), len = sh.len[i], off = sh.off[i];
        const auto at = S.entries(i, lane, row);
        const int pad = max(__shfl_sync(0xffffffffu, row, 0), 0);
        bool bad = !at.valid();
        for (int kb = 0; kb < len; kb += KS) {
            if (__any_sync(0xffffffffu, bad)) break;   // refused: no read beyond a malformed row's first bad column
            int j[KS];
            V w[KS];
#pragma unroll
            for (int u = 0; u < KS; ++u) {
                j[u] = 0;
                w[u] = V(0);
                if (kb + u < len) at.get(kb + u, j[u], w[u]);
            }
#pragma unroll
            for (int u = 0; u < KS; ++u) {
                if (!S.in_range(j[u])) {
                    bad = true;
                    j[u] = 0;
                    w[u] = V(0);
                }
                if (off >= 0 && kb + u < len) {
                    const int e = off + 32 * (kb + u) + lane;
                    col[e] = w[u] != V(0) ? j[u] : pad;
                    val[e] = S.alpha() * w[u];
                }
            }
        }
        if (bad) atomicOr(&sh.bad, 1);
    }
    __syncthreads();
}

// sum_j alpha w_ij rec_j of one component of one row (32-byte records)
template <int KB, class Sys>
__device__ __forceinline__ double row_product(const Sys& S, const Shared& sh, const unsigned char* dyn, int cap,
                                              int i, int row, const double* rec, int comp)
{
    const int lane = threadIdx.x & 31, len = sh.len[i], off = sh.off[i];
    const double* rc = rec + comp;
    double s = 0.0;
    if (off >= 0) {
        const double* val = reinterpret_cast<const double*>(dyn) + off + lane;
        const int* col = reinterpret_cast<const int*>(dyn + 8 * (size_t)cap) + off + lane;
        for (int kb = 0; kb < len; kb += KB) {
            double g[KB];
#pragma unroll
            for (int u = 0; u < KB; ++u) g[u] = kb + u < len ? rc[4 * (size_t)col[32 * (kb + u)]] : 0.0;
#pragma unroll
            for (int u = 0; u < KB; ++u)
                if (kb + u < len) s = fma(val[32 * (kb + u)], g[u], s);
        }
        return s;
    }
    if (row < 0) return 0.0;
    const auto at = S.entries(i, lane, row);
    for (int kb = 0; kb < len; kb += KB) {
        int j[KB];
        double w[KB], g[KB];
#pragma unroll
        for (int u = 0; u < KB; ++u) {
            j[u] = 0;
            w[u] = 0.0;
            if (kb + u < len) at.get(kb + u, j[u], w[u]);
        }
#pragma unroll
        for (int u = 0; u < KB; ++u) g[u] = w[u] != 0.0 ? rc[4 * (size_t)j[u]] : 0.0;
#pragma unroll
        for (int u = 0; u < KB; ++u) s = fma(w[u], g[u], s);
    }
    return S.alpha() * s;
}

// Blocks, threads and chunks per thread of a system of nch chunks on num_sms
// SMs: as few chunks per block as one block per SM allows.  Up to 5 chunks a
// block every chunk has its own three warps (one component a thread); above,
// a thread takes 2 (to 10 chunks) or 4 (to 16: the registers' limit), or, where
// the caller has no other form, 16 (to 64, spilling: a device of few SMs).
// u is 0 where the system does not fit.
struct Shape {
    int blocks, threads, u, smem;
};
inline Shape shape_of(int nch, int num_sms, int max_u)
{
    const int c = (nch + num_sms - 1) / num_sms;
    Shape s{};
    s.u = c <= kMaxGroups ? 1 : (c <= 2 * kMaxGroups ? 2 : (c <= 16 ? 4 : 16));
    if (s.u > max_u || c > kMaxChunks) return Shape{};
    const int g = (c + s.u - 1) / s.u;
    s.blocks = (nch + c - 1) / c;
    s.threads = 32 * (3 * g + kScalarWarps);
    s.smem = (c + 1) * kChunkSmem < kMaxSmem ? (c + 1) * kChunkSmem : kMaxSmem;
    return s;
}

// One grid reduction of up to three values, the publication barrier of the
// records written before it, and, while the scalar warps sum the blocks'
// partials and derive the scalars (post, run by one thread with the totals in
// sh.tot), the other warps' work (each thread's).  K = 0 is a barrier only.
// Returns false when the wait ran past the limit.
template <class Work, class Post>
__device__ __forceinline__ bool reduce_overlapped(const Grid& G, Shared& sh, unsigned int& gen, int K, double v0,
                                                  double v1, double v2, Work work, Post post)
{
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ncw = (blockDim.x >> 5) - kScalarWarps;   // compute warps
    double* part = G.partials + (size_t)(gen & 1u) * kScalarWarps * G.stride;
    if (warp < ncw && K > 0) {
        const double a = warp_sum3(v0, v1, v2);
        if ((lane & 7) == 0 && lane < 24) sh.wsum[lane == 0 ? 0 : (lane == 16 ? 1 : 2)][warp] = a;
    }
    __syncthreads();
    if (warp == ncw) {
        if (K > 0) {
            const int k = lane >> 3;
            double a = 0.0;
            if (k < kScalarWarps) {
                a = (lane & 7) < ncw ? sh.wsum[k][lane & 7] : 0.0;
                if (ncw > 8) a += (lane & 7) + 8 < ncw ? sh.wsum[k][(lane & 7) + 8] : 0.0;
            }
#pragma unroll
            for (int o = 4; o > 0; o >>= 1) a += __shfl_xor_sync(0xffffffffu, a, o);
            if ((lane & 7) == 0 && k < K) part[k * G.stride + G.bid] = a;
            __syncwarp();   // lane 0's release covers the other lanes' sums
        }
        if (lane == 0) sh.flag = arrive_and_wait(G, (gen + 1u) * (unsigned int)G.nb);
    }
    __syncthreads();
    gen += 1u;
    if (sh.flag != 0) return false;
    if (warp < ncw) {
        work();
    } else if (K > 0) {
        const int k = warp - ncw;
        if (k < K) {   // all loads are issued before the first sum
            constexpr int U = 5;
            double pv[U];
#pragma unroll
            for (int u = 0; u < U; ++u) pv[u] = lane + 32 * u < G.nb ? __ldcg(part + k * G.stride + lane + 32 * u) : 0.0;
            double a = pv[0];
#pragma unroll
            for (int u = 1; u < U; ++u)
                if (32 * u < G.nb) a += pv[u];
            for (int b = lane + 32 * U; b < G.nb; b += 32) a += __ldcg(part + k * G.stride + b);
            a = warp_sum(a);
            if (lane == 0) sh.tot[k] = a;
        }
        asm volatile("bar.sync 1, %0;" ::"n"(32 * kScalarWarps) : "memory");
        if (k == 0 && lane == 0) post();
    }
    __syncthreads();
    return true;
}

}  // namespace p64
}  // namespace ss
