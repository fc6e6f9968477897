// Learned warm start for the velocity solve: a small message-passing network
// that guesses v = A^-1 b before CG (the paper has no learned part; the
// solve it accelerates is Eq. algebra of arXiv 1808.06381, §Method).
//
// Per node i and Cartesian component c (row r = 3 i + c), shared weights:
//   s = RMS of b;  x0 = (b / A_ii, vprev, b) / s
//   a0 = M x0 with (M u)_i = sum_j alpha w_ij / A_ii u_j       (message pass 1)
//   h1 = tanh([x0, a0] W1);  h2 = tanh(h1 W2);  y = h2 W3       (6 -> 64 -> 64 -> 4)
//   a1 = M y                                                     (message pass 2)
//   guess = s [y, a1, x0] . o
// The message passes run on the narrow features (like an SpMV of the solver);
// the MLP of inference is one kernel on the tcgen05 tensor cores (BF16
// operands in shared memory, FP32 accumulators in tensor memory, 128-row
// tiles; k_mp_mlp_fwd_tc).  Training (MSE to the converged velocities)
// recomputes the forward and runs the backward on the same tensor cores
// (k_mp_mlp_bwd_tc: activation gradients and the weight gradients as
// products over each tile's rows, accumulated in tensor memory across a
// block's tiles), then a deterministic reduction over blocks and Adam on FP32
// master weights.
#include <cuda_bf16.h>
#include <math.h>

#include <cstring>
#include <random>
#include <vector>

#include "sim_impl.cuh"

namespace ss {

namespace {

constexpr int kTileRows = 128;
constexpr int kMaxGradBlocks = 1024;

__device__ __forceinline__ unsigned smem_addr(const void* p)
{
    return static_cast<unsigned>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ unsigned pack_bf16(float lo, float hi)
{
    __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
    return *reinterpret_cast<unsigned*>(&v);
}

// Weight layouts in the packed BF16 array (element offsets).
constexpr int kW1T = 0;                 // [64][16]: W1 transposed, k padded 6 -> 16
constexpr int kW2T = kW1T + 64 * 16;    // [64][64]: W2 transposed
constexpr int kW3T = kW2T + 64 * 64;    // [8][64]:  W3 transposed, n padded 4 -> 8
constexpr int kW2N = kW3T + 8 * 64;     // [64][64]: W2 as is (backward)
constexpr int kW3P = kW2N + 64 * 64;    // [64][16]: W3 as is, k padded 4 -> 16 (backward)
constexpr int kWB = kW3P + 64 * 16;

// tanh by the hardware approximation (one MUFU operation, relative error
// below 2^-10): finer than the BF16 rounding the activations get next.
__device__ __forceinline__ float tanh_fast(float x)
{
    float y;
    asm("tanh.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
    return y;
}

// ------------------------------------------- forward MLP on tcgen05 tensor cores
//
// The three layers of a tile of 128 rows as 5th-generation tensor-core MMAs
// (tcgen05.mma, kind::f16, BF16 operands from shared memory, FP32
// accumulators in tensor memory), M = 128 rows: layer 1 [x0, a0] (K 6 -> 16)
// x W1 (N = 64), layer 2 h1 x W2 (K = N = 64, four K = 16 steps), layer 3 h2 x
// W3 (N 4 -> 16).  One thread issues the MMAs and commits them to an
// mbarrier; the four warps read the accumulators back with tcgen05.ld (warp w
// owns rows 32w..32w+31, its lane quarter of tensor memory), apply tanh, and
// store BF16 into the next layer's operand tile.  Operands use the
// no-swizzle K-major layout of 8 x 16-byte core matrices: element (r, k) of an
// R x K tile sits at ((r / 8) (K / 8) + k / 8) 128 + (r % 8) 16 + (k % 8) 2
// bytes, so the leading (K) core-matrix stride is 128 bytes and the stride
// between 8-row groups K / 8 x 128 bytes.  64 columns of tensor memory are
// reused by the three layers.  Every wait is bounded.
namespace tc {

constexpr int kRows = 128;
constexpr int kTmemCols = 64;
constexpr long long kWaitLimit = 1ll << 24;

__device__ __forceinline__ int core_off(int r, int k, int K)   // byte offset in a core-matrix tile
{
    return ((r >> 3) * (K >> 3) + (k >> 3)) * 128 + (r & 7) * 16 + (k & 7) * 2;
}

__device__ __forceinline__ unsigned long long smem_desc(const void* base, int K)
{
    const unsigned long long addr = smem_addr(base);
    const unsigned long long lbo = 128, sbo = (unsigned long long)(K >> 3) * 128;
    return ((addr >> 4) & 0x3FFFull) | (((lbo >> 4) & 0x3FFFull) << 16) | (((sbo >> 4) & 0x3FFFull) << 32) |
           (1ull << 46);   // descriptor version 1; base offset 0, no swizzle
}

// The same with both strides given: K-major, lbo steps from one core matrix to
// the next along K and sbo along the rows; MN-major (a transposed operand), lbo
// steps along K (8 rows of the stored tile) and sbo along M or N.
__device__ __forceinline__ unsigned long long smem_desc(const void* base, unsigned lbo, unsigned sbo)
{
    const unsigned long long addr = smem_addr(base);
    return ((addr >> 4) & 0x3FFFull) | ((unsigned long long)(lbo >> 4) << 16) |
           ((unsigned long long)(sbo >> 4) << 32) | (1ull << 46);
}

// mn_major: A and B are both stored transposed (MN-major) instead of K-major
__host__ __device__ constexpr unsigned idesc_bf16(int M, int N, bool mn_major = false)
{
    return (1u << 4)                  // D: FP32
           | (1u << 7) | (1u << 10)   // A, B: BF16
           | (mn_major ? (1u << 15) | (1u << 16) : 0u)
           | ((unsigned)(N >> 3) << 17) | ((unsigned)(M >> 4) << 24);
}

__device__ __forceinline__ void mma(unsigned tmem_d, unsigned long long a, unsigned long long b, unsigned idesc,
                                    int accumulate)
{
    asm volatile(
        "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
        "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(tmem_d),
        "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void commit(void* mbar)
{
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(mbar))
                 : "memory");
}

// bounded wait for the mbarrier phase with the given parity; false on timeout
__device__ __forceinline__ bool wait_phase(void* mbar, unsigned parity)
{
    const unsigned a = smem_addr(mbar);
    for (long long it = 0; it < kWaitLimit; ++it) {
        unsigned done;
        asm volatile(
            "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
            "selp.u32 %0, 1, 0, p;\n\t}\n"
            : "=r"(done) : "r"(a), "r"(parity) : "memory");
        if (done) return true;
    }
    return false;
}

__device__ __forceinline__ void ld16(unsigned taddr, float (&v)[16])
{
    unsigned r[16];
    asm volatile(
        "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
        : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
          "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
        : "r"(taddr));
    asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
    for (int k = 0; k < 16; ++k) v[k] = __uint_as_float(r[k]);
}

__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

}  // namespace tc

}  // namespace

// y = h2 W3 with h2 = tanh(tanh([x0, a0] W1) W2), 128 rows per tile (see tc above).
__global__ void __launch_bounds__(128) k_mp_mlp_fwd_tc(int rows, MpBuffers M, DevState* st)
{
    using namespace tc;
    __shared__ __align__(128) unsigned char sA1[kRows * 16 * 2];   // [128][16] inputs
    __shared__ __align__(128) unsigned char sB1[64 * 16 * 2];      // [64][16]  W1^T
    __shared__ __align__(128) unsigned char sA2[kRows * 64 * 2];   // [128][64] h1, then h2
    __shared__ __align__(128) unsigned char sB2[64 * 64 * 2];      // [64][64]  W2^T
    __shared__ __align__(128) unsigned char sB3[16 * 64 * 2];      // [16][64]  W3^T (n padded 4 -> 16)
    __shared__ __align__(8) unsigned long long mbar;
    __shared__ unsigned tmem_base;
    __shared__ int failed;
    const int tid = threadIdx.x, warp = tid >> 5;

    // weights (BF16, already transposed and padded) into core-matrix tiles
    for (int e = tid; e < 64 * 16; e += blockDim.x)
        *reinterpret_cast<__nv_bfloat16*>(sB1 + core_off(e / 16, e % 16, 16)) = M.wb[kW1T + e];
    for (int e = tid; e < 64 * 64; e += blockDim.x)
        *reinterpret_cast<__nv_bfloat16*>(sB2 + core_off(e / 64, e % 64, 64)) = M.wb[kW2T + e];
    for (int e = tid; e < 16 * 64; e += blockDim.x) {
        const int n = e / 64, k = e % 64;
        *reinterpret_cast<__nv_bfloat16*>(sB3 + core_off(n, k, 64)) =
            n < 8 ? M.wb[kW3T + n * 64 + k] : __float2bfloat16_rn(0.f);
    }
    if (tid == 0) {
        failed = 0;
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&mbar)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_base)),
                     "r"(kTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    const unsigned tmem = tmem_base;
    const unsigned tlane = tmem + ((unsigned)(warp * 32) << 16);   // this warp's lane quarter
    const unsigned id1 = idesc_bf16(kRows, 64), id3 = idesc_bf16(kRows, 16);
    unsigned phase = 0;

    for (int base = blockIdx.x * kRows; base < rows && !failed; base += gridDim.x * kRows) {
        const int r = base + tid;   // this thread's row (tile row tid)
        {   // layer-1 operand: [x0, a0] in BF16, k 6..15 zero
            const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
            const float4 x = r < rows ? M.x0[r] : z, a = r < rows ? M.a0[r] : z;
            uint4 lo, hi;
            lo.x = pack_bf16(x.x, x.y);
            lo.y = pack_bf16(x.z, a.x);
            lo.z = pack_bf16(a.y, a.z);
            lo.w = 0u;
            hi = make_uint4(0u, 0u, 0u, 0u);
            *reinterpret_cast<uint4*>(sA1 + core_off(tid, 0, 16)) = lo;
            *reinterpret_cast<uint4*>(sA1 + core_off(tid, 8, 16)) = hi;
        }
        fence_async_smem();
        fence_before();
        __syncthreads();
        fence_after();
        if (tid == 0) {
            mma(tmem, smem_desc(sA1, 16), smem_desc(sB1, 16), id1, 0);
            commit(&mbar);
        }
        if (!wait_phase(&mbar, phase)) atomicExch(&failed, 1);
        phase ^= 1u;
        fence_after();
        // h1 = tanh(D), BF16 into the layer-2 operand
#pragma unroll
        for (int c = 0; c < 64; c += 16) {
            float v[16];
            ld16(tlane + c, v);
#pragma unroll
            for (int q = 0; q < 16; q += 8) {
                uint4 w;
                w.x = pack_bf16(tanh_fast(v[q]), tanh_fast(v[q + 1]));
                w.y = pack_bf16(tanh_fast(v[q + 2]), tanh_fast(v[q + 3]));
                w.z = pack_bf16(tanh_fast(v[q + 4]), tanh_fast(v[q + 5]));
                w.w = pack_bf16(tanh_fast(v[q + 6]), tanh_fast(v[q + 7]));
                *reinterpret_cast<uint4*>(sA2 + core_off(tid, c + q, 64)) = w;
            }
        }
        fence_async_smem();
        fence_before();
        __syncthreads();
        fence_after();
        if (tid == 0) {
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)   // K = 16 per step: two core matrices, 256 bytes
                mma(tmem, smem_desc(sA2 + ks * 256, 64), smem_desc(sB2 + ks * 256, 64), id1, ks > 0);
            commit(&mbar);
        }
        if (!wait_phase(&mbar, phase)) atomicExch(&failed, 1);
        phase ^= 1u;
        fence_after();
        // h2 = tanh(D) overwrites h1 (layer 2 has read it)
#pragma unroll
        for (int c = 0; c < 64; c += 16) {
            float v[16];
            ld16(tlane + c, v);
#pragma unroll
            for (int q = 0; q < 16; q += 8) {
                uint4 w;
                w.x = pack_bf16(tanh_fast(v[q]), tanh_fast(v[q + 1]));
                w.y = pack_bf16(tanh_fast(v[q + 2]), tanh_fast(v[q + 3]));
                w.z = pack_bf16(tanh_fast(v[q + 4]), tanh_fast(v[q + 5]));
                w.w = pack_bf16(tanh_fast(v[q + 6]), tanh_fast(v[q + 7]));
                *reinterpret_cast<uint4*>(sA2 + core_off(tid, c + q, 64)) = w;
            }
        }
        fence_async_smem();
        fence_before();
        __syncthreads();
        fence_after();
        if (tid == 0) {
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                mma(tmem, smem_desc(sA2 + ks * 256, 64), smem_desc(sB3 + ks * 256, 64), id3, ks > 0);
            commit(&mbar);
        }
        if (!wait_phase(&mbar, phase)) atomicExch(&failed, 1);
        phase ^= 1u;
        fence_after();
        {
            float v[16];
            ld16(tlane, v);
            if (r < rows) M.y[r] = make_float4(v[0], v[1], v[2], v[3]);
        }
        fence_before();
        __syncthreads();   // the next tile's MMAs overwrite tensor memory and the operands
        fence_after();
    }
    if (failed && tid == 0) atomicCAS(&st->error, 0, (int)SP_ERR_TIMEOUT);
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTmemCols) : "memory");
}

// ------------------------------------------ training backward on tcgen05
//
// Tiles of 128 rows, one thread per row; every product is a tcgen05.mma with M =
// 128 (BF16 operands in no-swizzle core-matrix tiles as above, FP32 accumulators
// in tensor memory):
//   h1 = tanh(X W1), h2 = tanh(h1 W2)             (forward recomputed; K 16, 64)
//   dp2 = (dY W3^T) (1 - h2^2)                     (A = dY [128][16], B = W3 [64][16])
//   dp1 = (dp2 W2^T) (1 - h1^2)                    (A = dp2 [128][64], B = W2 [64][64])
// and the weight gradients as products over the tile's rows (K = 128), with
// both operands read transposed (MN-major) from the tiles that the products
// above use: H = [h1, h2] and Q = [dp2, dp1], 128 x 128 each,
//   H^T dp2 -> rows 0-63: dW2 = h1^T dp2
//   H^T dY  -> rows 64-127: dW3 = h2^T dY
//   Q^T X   -> rows 64-127: dW1^T = dp1^T X
// so nothing is written twice: a thread stores its row's activations 16 bytes
// at a time (conflict-free) and keeps them packed for the derivatives.
//
// The gradient accumulators stay in tensor memory across all the block's tiles
// and are read back once: one partial gradient per block, summed over blocks in
// order (k_mp_update).  The tensor cores' FP32 accumulation truncates, so the
// order in which an accumulator takes its tiles is part of the result (two
// accumulators per SM instead of one moved a gradient at n = 262,144 by 1e-5 to
// 8e-5 of its norm): one block per SM takes tiles blockIdx + k gridDim in the
// order of k.  Two groups of 128 threads share the block's accumulators and
// weights, each with its own operand tiles and activation columns: group g
// works on tiles k = g, g + 2, ..., one group's epilogues run under the other's
// products, and a group's issuer adds tile k's gradients once those of tile k -
// 1 are complete (the mbarrier in_order, whose phase k ends with tile k's).
// Tensor memory columns: 128 g .. + 63 group g's activations (reused), + 64 ..
// 127 its dY W3^T, 256-319 dW2, 320-335 dW3, 336-351 dW1^T.  The derivative of
// tanh uses the BF16 activations the products use.  Every wait is bounded.
// 786,432 rows: 233 us with transposed copies of every operand written two bytes
// at a time by one group, 89 now (82 with two accumulators per SM, which rounded
// differently).
namespace tcb {
constexpr int kBRows = 128;
constexpr int kBGroups = 2;
constexpr int kBTmemCols = 512;
constexpr int kColH2 = 64, kColGroup = 128, kColW2 = 256, kColW3 = 320, kColW1 = 336;
// dynamic shared memory layout (byte offsets, 128-byte aligned): the weights,
constexpr int oW1T = 0;                      // [64][16]  W1^T          (B, layer 1)
constexpr int oW2T = oW1T + 64 * 16 * 2;     // [64][64]  W2^T          (B, layer 2)
constexpr int oW3P = oW2T + 64 * 64 * 2;     // [64][16]  W3 (k 4 -> 16) (B, dh2)
constexpr int oW2N = oW3P + 64 * 16 * 2;     // [64][64]  W2            (B, dh1)
constexpr int oGroups = oW2N + 64 * 64 * 2;  // and the groups' tiles, each
constexpr int oX = 0;                        // [128][16] [x0, a0]      (A, layer 1; B, dW1^T)
constexpr int oDY = oX + kBRows * 16 * 2;    // [128][16] dY            (A, dh2; B, dW3)
constexpr int oH = oDY + kBRows * 16 * 2;    // [128][128] [h1, h2]     (A, layer 2, dW2 and dW3)
constexpr int oQ = oH + kBRows * 128 * 2;    // [128][128] [dp2, dp1]   (A, dh1 and dW1^T; B, dW2)
constexpr int kGroupSmem = oQ + kBRows * 128 * 2;
constexpr int kSmem = oGroups + kBGroups * kGroupSmem;
constexpr int kHalf = 8 * 128;               // bytes from column 0 to column 64 of a 128-column tile
constexpr int kGroup8 = 16 * 128;            // bytes from one group of 8 rows of it to the next
}  // namespace tcb

int mp_bwd_tc_smem_bytes() { return tcb::kSmem + 128; }

__device__ __forceinline__ float bf16_lo(unsigned v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf16_hi(unsigned v) { return __uint_as_float(v & 0xffff0000u); }

__global__ void __launch_bounds__(128 * tcb::kBGroups, 1) k_mp_mlp_bwd_tc(int rows, MpBuffers M, DevState* st)
{
    using namespace tc;
    using namespace tcb;
    extern __shared__ __align__(128) unsigned char sm_raw[];
    // the operand tiles start on a 128-byte boundary (the launch adds 128 bytes)
    unsigned char* sm = sm_raw + ((128u - (smem_addr(sm_raw) & 127u)) & 127u);
    __shared__ __align__(8) unsigned long long mbars[kBGroups], in_order;
    __shared__ unsigned tmem_base;
    __shared__ int failed_of[kBGroups];   // a group leaves its loop by its own flag alone (its barriers need all of it)
    const int g = threadIdx.x >> 7, tid = threadIdx.x & 127, warp = threadIdx.x >> 5;
    unsigned char* sg = sm + oGroups + g * kGroupSmem;
    unsigned long long* mbar = &mbars[g];
    int& failed = failed_of[g];
    // weights (BF16 layouts of k_mp_update) into core-matrix tiles
    for (int e = threadIdx.x; e < 64 * 16; e += blockDim.x) {
        *reinterpret_cast<__nv_bfloat16*>(sm + oW1T + core_off(e / 16, e % 16, 16)) = M.wb[kW1T + e];
        *reinterpret_cast<__nv_bfloat16*>(sm + oW3P + core_off(e / 16, e % 16, 16)) = M.wb[kW3P + e];
    }
    for (int e = threadIdx.x; e < 64 * 64; e += blockDim.x) {
        *reinterpret_cast<__nv_bfloat16*>(sm + oW2T + core_off(e / 64, e % 64, 64)) = M.wb[kW2T + e];
        *reinterpret_cast<__nv_bfloat16*>(sm + oW2N + core_off(e / 64, e % 64, 64)) = M.wb[kW2N + e];
    }
    if (threadIdx.x == 0) {
        for (int k = 0; k < kBGroups; ++k) {
            failed_of[k] = 0;
            asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&mbars[k])) : "memory");
        }
        asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(smem_addr(&in_order)) : "memory");
        asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    }
    if (warp == 0) {
        asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(&tmem_base)),
                     "r"(kBTmemCols)
                     : "memory");
        asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
    }
    fence_async_smem();
    fence_before();
    __syncthreads();
    fence_after();
    const unsigned tmem = tmem_base, tact = tmem + (unsigned)(g * kColGroup);   // this group's activations
    const unsigned quarter = (unsigned)((warp & 3) * 32) << 16;                  // this warp's lane quarter
    const unsigned tlane = tact + quarter;
    const unsigned id64 = idesc_bf16(kBRows, 64);
    const unsigned idt64 = idesc_bf16(kBRows, 64, true), idt16 = idesc_bf16(kBRows, 16, true);
    unsigned phase = 0;
    auto sync_group = [&]() { asm volatile("bar.sync %0, 128;" ::"r"(1 + g) : "memory"); };
    auto sync_mma = [&]() {   // operands written by all the group's threads -> visible to its MMA issuer
        fence_async_smem();
        fence_before();
        sync_group();
        fence_after();
    };
    auto wait_mma = [&]() {
        if (!wait_phase(mbar, phase)) atomicExch(&failed, 1);
        phase ^= 1u;
        fence_after();
    };
    auto put8 = [&](int off, const unsigned* w) {   // 8 columns of this thread's row of a 128-column tile
        *reinterpret_cast<uint4*>(sg + off + (tid >> 3) * kGroup8 + (tid & 7) * 16) = make_uint4(w[0], w[1], w[2], w[3]);
    };
    // the row's inputs, requested a tile ahead
    float4 x, a, dy;
    auto load = [&](long long tile) {
        const float4 z = make_float4(0.f, 0.f, 0.f, 0.f);
        const long long r = tile * kBRows + tid;
        x = r < rows ? M.x0[r] : z;
        a = r < rows ? M.a0[r] : z;
        dy = r < rows ? M.dy[r] : z;
    };
    const long long ntile = (rows + kBRows - 1) / kBRows;
    auto tile_of = [&](int k) { return (long long)blockIdx.x + (long long)k * gridDim.x; };
    load(tile_of(g));

    for (int k = g; tile_of(k) < ntile && !failed; k += kBGroups) {
        {   // X = [x0, a0] (k 6..15 zero) and dY (k 4..15 zero)
            const uint4 zero = make_uint4(0u, 0u, 0u, 0u);
            *reinterpret_cast<uint4*>(sg + oX + core_off(tid, 0, 16)) =
                make_uint4(pack_bf16(x.x, x.y), pack_bf16(x.z, a.x), pack_bf16(a.y, a.z), 0u);
            *reinterpret_cast<uint4*>(sg + oX + core_off(tid, 8, 16)) = zero;
            *reinterpret_cast<uint4*>(sg + oDY + core_off(tid, 0, 16)) =
                make_uint4(pack_bf16(dy.x, dy.y), pack_bf16(dy.z, dy.w), 0u, 0u);
            *reinterpret_cast<uint4*>(sg + oDY + core_off(tid, 8, 16)) = zero;
        }
        sync_mma();
        if (tid == 0) {   // layer 1, and dh2 = dY W3^T
            mma(tact, smem_desc(sg + oX, 16), smem_desc(sm + oW1T, 16), id64, 0);
            mma(tact + kColH2, smem_desc(sg + oDY, 16), smem_desc(sm + oW3P, 16), id64, 0);
            commit(mbar);
        }
        wait_mma();
        unsigned h1[32];   // the row's activations, packed
#pragma unroll
        for (int c = 0; c < 64; c += 16) {
            float v[16];
            ld16(tlane + c, v);
#pragma unroll
            for (int q = 0; q < 16; q += 2) h1[(c + q) / 2] = pack_bf16(tanh_fast(v[q]), tanh_fast(v[q + 1]));
            put8(oH + c / 8 * 128, h1 + c / 2);
            put8(oH + (c / 8 + 1) * 128, h1 + c / 2 + 4);
        }
        sync_mma();
        if (tid == 0) {
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                mma(tact, smem_desc(sg + oH + ks * 256, 128u, (unsigned)kGroup8), smem_desc(sm + oW2T + ks * 256, 64),
                    id64, ks > 0);
            commit(mbar);
        }
        wait_mma();
        // h2 = tanh(D) and dp2 = dh2 (1 - h2^2)
#pragma unroll
        for (int c = 0; c < 64; c += 16) {
            float v[16], u[16];
            ld16(tlane + c, v);
            ld16(tlane + kColH2 + c, u);
            unsigned h2[8], w[8];
#pragma unroll
            for (int q = 0; q < 16; q += 2) {
                const unsigned h = pack_bf16(tanh_fast(v[q]), tanh_fast(v[q + 1]));
                const float lo = bf16_lo(h), hi = bf16_hi(h);
                h2[q / 2] = h;
                w[q / 2] = pack_bf16(u[q] * (1.f - lo * lo), u[q + 1] * (1.f - hi * hi));
            }
            put8(oH + kHalf + c / 8 * 128, h2);
            put8(oH + kHalf + (c / 8 + 1) * 128, h2 + 4);
            put8(oQ + c / 8 * 128, w);
            put8(oQ + (c / 8 + 1) * 128, w + 4);
        }
        sync_mma();
        if (tid == 0) {   // dh1 = dp2 W2^T
#pragma unroll
            for (int ks = 0; ks < 4; ++ks)
                mma(tact, smem_desc(sg + oQ + ks * 256, 128u, (unsigned)kGroup8), smem_desc(sm + oW2N + ks * 256, 64),
                    id64, ks > 0);
            commit(mbar);
        }
        wait_mma();
        // dp1 = dh1 (1 - h1^2)
#pragma unroll
        for (int c = 0; c < 64; c += 16) {
            float v[16];
            ld16(tlane + c, v);
            unsigned w[8];
#pragma unroll
            for (int q = 0; q < 16; q += 2) {
                const float lo = bf16_lo(h1[(c + q) / 2]), hi = bf16_hi(h1[(c + q) / 2]);
                w[q / 2] = pack_bf16(v[q] * (1.f - lo * lo), v[q + 1] * (1.f - hi * hi));
            }
            put8(oQ + kHalf + c / 8 * 128, w);
            put8(oQ + kHalf + (c / 8 + 1) * 128, w + 4);
        }
        sync_mma();
        if (tid == 0) {   // the weight gradients over the tile's rows (K = 128, 16 a step), behind the tile before
            if (k > 0 && !wait_phase(&in_order, (unsigned)(k - 1) & 1u)) {
                atomicExch(&failed, 1);
            } else {
                fence_after();
#pragma unroll
                for (int ks = 0; ks < 8; ++ks) {
                    const int on = k > 0 || ks > 0;
                    const unsigned long long h = smem_desc(sg + oH + ks * 2 * kGroup8, (unsigned)kGroup8, 128u);
                    const unsigned long long q = smem_desc(sg + oQ + ks * 2 * kGroup8, (unsigned)kGroup8, 128u);
                    mma(tmem + kColW2, h, q, idt64, on);
                    mma(tmem + kColW3, h, smem_desc(sg + oDY + ks * 512, 256u, 128u), idt16, on);
                    mma(tmem + kColW1, q, smem_desc(sg + oX + ks * 512, 256u, 128u), idt16, on);
                }
            }
            commit(&in_order);
            commit(mbar);
        }
        load(tile_of(k + kBGroups));
        wait_mma();   // the next tile overwrites the operands
        fence_before();
        sync_group();
        fence_after();
    }
    fence_before();
    __syncthreads();   // both groups' gradients are in tensor memory
    fence_after();
    const bool bad = failed_of[0] || failed_of[1];
    // this block's partial gradient (zero if it had no tile)
    float* gp = M.gpart + (size_t)blockIdx.x * kMpParams;
    if ((long long)blockIdx.x < ntile && !bad) {
        const unsigned lane0 = tmem + quarter;
        if (g == 0 && warp < 2) {   // rows 0-63: dW2[i][h] (i = row)
            const int i = tid;
#pragma unroll
            for (int c = 0; c < 64; c += 16) {
                float v[16];
                ld16(lane0 + kColW2 + c, v);
#pragma unroll
                for (int q = 0; q < 16; ++q) gp[kMpOffW2 + i * 64 + c + q] = v[q];
            }
        } else if (g == 0) {        // rows 64-127: dW3[h][m] (h = row - 64) and dW1^T[i][f] (i = row - 64)
            const int h = tid - 64;
            float v[16];
            ld16(lane0 + kColW3, v);
#pragma unroll
            for (int m = 0; m < 4; ++m) gp[kMpOffW3 + h * 4 + m] = v[m];
            ld16(lane0 + kColW1, v);
#pragma unroll
            for (int f = 0; f < 6; ++f) gp[kMpOffW1 + f * 64 + h] = v[f];
        }
    } else {
        for (int e = threadIdx.x; e < kMpOffO; e += blockDim.x) gp[e] = 0.f;
    }
    if (bad && threadIdx.x == 0) atomicCAS(&st->error, 0, (int)SP_ERR_TIMEOUT);
    fence_before();
    __syncthreads();
    if (warp == 0)
        asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kBTmemCols) : "memory");
}

// -------------------------------------------------------------- kernels

// Component c of b at row i: the mixed path keeps b as double-floats only.
__device__ __forceinline__ double b_at(const DevBuffers& B, int np, int c, int i)
{
    if (B.bdf) {
        const float4 h = B.bdf[2 * i], l = B.bdf[2 * i + 1];
        return c == 0 ? (double)h.x + (double)l.x : (c == 1 ? (double)h.y + (double)l.y : (double)h.z + (double)l.z);
    }
    return B.b[c * np + i];
}

// s = sqrt(sum b^2 / 3n) (1 if b = 0)
__global__ void k_mp_scale(KParams P, DevBuffers B, MpBuffers M)
{
    const int np = P.npad;
    double acc = 0.0;
    for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < P.n; i += gridDim.x * blockDim.x)
        for (int c = 0; c < 3; ++c) {
            const double b = M.in ? M.in[c * np + i] : b_at(B, np, c, i);
            acc += b * b;
        }
    const double v[1] = {acc};
    if (publish_partials<1>(v, M.part, &M.ticket[0])) {
        double out[1];
        reduce_partials<1>(M.part, out);
        if (threadIdx.x == 0) {
            const double s = sqrt(out[0] / (3.0 * P.n));
            M.scal[0] = s > 0.0 ? s : 1.0;
        }
    }
}

// x0 rows (b / A_ii, vprev, b) / s, with vprev = the current x (the previous velocities).
__global__ void k_mp_input(KParams P, DevBuffers B, MpBuffers M)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.n) return;
    const int np = P.npad;
    const float inv = (float)(1.0 / M.scal[0]);
    const double di = B.bdf ? (double)B.dinv32[i] : B.dinv[i];
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const double b = M.in ? M.in[c * np + i] : b_at(B, np, c, i);
        const float vp = M.zero_vprev ? 0.f : (float)B.x[c * np + i] * inv;
        M.x0[3 * i + c] = make_float4((float)(b * di) * inv, vp, (float)b * inv, 0.f);
    }
}

// This thread's node and its entries' range.  The message passes take the rows
// in row order: neighbouring lanes gather largely the same rows (in slot order
// the entry loads are coalesced, but a pass took 66 us instead of 61).
struct MpNode {
    int i, base, cnt;
};
__device__ __forceinline__ MpNode mp_node(const KParams& P, const DevBuffers& B)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.n) return MpNode{-1, 0, 0};
    const int slot = B.row_slot[i];
    return MpNode{i, B.chunk_off[slot >> 5] + (slot & 31), B.row_cnt[i]};
}

// a0 = M x0; three rows per node.
__global__ void k_mp_aggregate(KParams P, DevBuffers B, const float4* __restrict__ in, float4* __restrict__ out)
{
    const MpNode nd = mp_node(P, B);
    const int i = nd.i;
    if (i < 0) return;
    const float ae = (float)P.alpha;
    float4 s[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) s[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k = 0; k < nd.cnt; ++k) {
        const int e = nd.base + 32 * k;
        const int j = B.col[e];
        const float w = ae * B.val32[e];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float4 u = in[3 * j + c];
            s[c].x = fmaf(w, u.x, s[c].x);
            s[c].y = fmaf(w, u.y, s[c].y);
            s[c].z = fmaf(w, u.z, s[c].z);
            s[c].w = fmaf(w, u.w, s[c].w);
        }
    }
    const float di = B.dinv32[i];
#pragma unroll
    for (int c = 0; c < 3; ++c) out[3 * i + c] = make_float4(s[c].x * di, s[c].y * di, s[c].z * di, s[c].w * di);
}

// dY = dout o[0:4] + M^T (dout o[4:8]), o the readout: the gradient at the second
// message pass is a row's dout times four constants, so an entry gathers the
// partner's three dout and D^-1 (16 bytes) and forms the twelve products again,
// rounded as when they were stored (with them stored, 48 bytes and D^-1 an
// entry: 62 us at 786,432 rows, 48 now).
__global__ void k_mp_pull(KParams P, DevBuffers B, MpBuffers M)
{
    const MpNode nd = mp_node(P, B);
    if (nd.i < 0) return;
    const float ae = (float)P.alpha;
    float o[8];
#pragma unroll
    for (int k = 0; k < 8; ++k) o[k] = M.master[kMpOffO + k];
    float s[3][4];
#pragma unroll
    for (int c = 0; c < 3; ++c)
#pragma unroll
        for (int k = 0; k < 4; ++k) s[c][k] = 0.f;
    for (int k = 0; k < nd.cnt; ++k) {
        const int e = nd.base + 32 * k;
        const float4 v = M.dout[B.col[e]];
        const float w = ae * B.val32[e] * v.w, d[3] = {v.x, v.y, v.z};
#pragma unroll
        for (int c = 0; c < 3; ++c)
#pragma unroll
            for (int q = 0; q < 4; ++q) s[c][q] = fmaf(w, __fmul_rn(d[c], o[4 + q]), s[c][q]);
    }
    const float4 v = M.dout[nd.i];
    const float d[3] = {v.x, v.y, v.z};
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        float r[4];
#pragma unroll
        for (int q = 0; q < 4; ++q) r[q] = __fadd_rn(s[c][q], __fmul_rn(d[c], o[q]));
        M.dy[3 * nd.i + c] = make_float4(r[0], r[1], r[2], r[3]);
    }
}

// Second message pass fused with the output: a1 = M y for node i, then
// guess = s [y, a1, x0] . o written as the start vector of CG (a1 is kept
// for training).
__global__ void k_mp_aggregate_output(KParams P, DevBuffers B, MpBuffers M)
{
    const MpNode nd = mp_node(P, B);
    const int i = nd.i;
    if (i < 0) return;
    const float ae = (float)P.alpha;
    float4 acc[3];
#pragma unroll
    for (int c = 0; c < 3; ++c) acc[c] = make_float4(0.f, 0.f, 0.f, 0.f);
    for (int k = 0; k < nd.cnt; ++k) {
        const int e = nd.base + 32 * k;
        const int j = B.col[e];
        const float w = ae * B.val32[e];
#pragma unroll
        for (int c = 0; c < 3; ++c) {
            const float4 u = M.y[3 * j + c];
            acc[c].x = fmaf(w, u.x, acc[c].x);
            acc[c].y = fmaf(w, u.y, acc[c].y);
            acc[c].z = fmaf(w, u.z, acc[c].z);
            acc[c].w = fmaf(w, u.w, acc[c].w);
        }
    }
    const float di = B.dinv32[i];
    const double s = M.scal[0];
    const float* o = M.master + kMpOffO;
#pragma unroll
    for (int c = 0; c < 3; ++c) {
        const int r = 3 * i + c;
        const float4 a = make_float4(acc[c].x * di, acc[c].y * di, acc[c].z * di, acc[c].w * di);
        M.a1[r] = a;
        const float4 y = M.y[r], x = M.x0[r];
        const float out = y.x * o[0] + y.y * o[1] + y.z * o[2] + y.w * o[3] + a.x * o[4] + a.y * o[5] + a.z * o[6] +
                          a.w * o[7] + x.x * o[8] + x.y * o[9] + x.z * o[10];
        (M.out ? M.out : B.x)[c * P.npad + i] = s * (double)out;
    }
}

// a / b from inv = 1 / b by one correction of the product a inv with its exact
// remainder (Markstein, IBM J. Res. Dev. 34, 1990), three FP64 operations.
__device__ __forceinline__ double quotient(double a, double b, double inv)
{
    const double q = a * inv, r = fma(-q, b, a);
    return isfinite(r) ? fma(r, inv, q) : q;
}

// A sum of FP32 terms in three words: the exact error of every addition goes to
// the second word, the exact error of that addition to the third (72 bits; an
// FP64 sum has 53 and needs two operations a term on the 1/64-rate pipe).
struct Sum3 {
    float a, b, c;
    __device__ void add(float v)
    {
        const dfloat t = two_sum(a, v), u = two_sum(b, t.lo);
        a = t.hi;
        b = u.hi;
        c = __fadd_rn(c, u.lo);
    }
};

// Loss rows: e = out - vstar / s, dout = 2 e / 3n (of each node kept, with D^-1);
// per block: sum e^2 and the readout gradient sum dout [y, a1, x0].  Bound by FP64
// (GB300 issues it at 1/64 of the FP32 rate), which only e, its square's sum and
// dout need: 107 us at 786,432 rows with two FP64 divisions and eleven FP64 sums a
// row, 36 now.
__global__ void __launch_bounds__(kVecBlock) k_mp_loss(KParams P, DevBuffers B, MpBuffers M)
{
    __shared__ double s_inv[2];
    const int rows = 3 * P.n;
    const double scale = M.scal[0], rows_d = (double)rows;
    if (threadIdx.x == 0) {
        s_inv[0] = 1.0 / scale;
        s_inv[1] = 1.0 / rows_d;
    }
    __syncthreads();
    const double inv = s_inv[0], inv_rows = s_inv[1];
    float o[11];
#pragma unroll
    for (int k = 0; k < 11; ++k) o[k] = M.master[kMpOffO + k];
    double ee = 0.0;
    Sum3 acc[11];
#pragma unroll
    for (int k = 0; k < 11; ++k) acc[k] = Sum3{0.f, 0.f, 0.f};
    for (int r = blockIdx.x * blockDim.x + threadIdx.x; r < rows; r += gridDim.x * blockDim.x) {
        const int i = r / 3, c = r - 3 * i;
        const float4 y = M.y[r], a = M.a1[r], x = M.x0[r];
        const float out = y.x * o[0] + y.y * o[1] + y.z * o[2] + y.w * o[3] + a.x * o[4] + a.y * o[5] + a.z * o[6] +
                          a.w * o[7] + x.x * o[8] + x.y * o[9] + x.z * o[10];
        const double e = (double)out - quotient(B.x[c * P.npad + i], scale, inv);
        const float d = (float)quotient(2.0 * e, rows_d, inv_rows);
        ee = fma(e, e, ee);
        float* node = reinterpret_cast<float*>(M.dout + i);
        node[c] = d;
        if (c == 2) node[3] = B.dinv32[i];
        const float f[11] = {y.x, y.y, y.z, y.w, a.x, a.y, a.z, a.w, x.x, x.y, x.z};
#pragma unroll
        for (int k = 0; k < 11; ++k) acc[k].add(__fmul_rn(d, f[k]));
    }
    __shared__ double sh[12][kVecBlock / 32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
    for (int k = 0; k < 11; ++k) {
#pragma unroll
        for (int w = 16; w > 0; w >>= 1) {
            const float a = __shfl_xor_sync(0xffffffffu, acc[k].a, w), b = __shfl_xor_sync(0xffffffffu, acc[k].b, w);
            const float c = __shfl_xor_sync(0xffffffffu, acc[k].c, w);
            acc[k].add(a);
            const dfloat u = two_sum(acc[k].b, b);
            acc[k].b = u.hi;
            acc[k].c = __fadd_rn(acc[k].c, __fadd_rn(u.lo, c));
        }
        if (lane == 0) sh[1 + k][warp] = ((double)acc[k].c + (double)acc[k].b) + (double)acc[k].a;
    }
    ee = warp_sum(ee);
    if (lane == 0) sh[0][warp] = ee;
    __syncthreads();
    if (threadIdx.x < 12) {
        double t = 0.0;
        for (int w = 0; w < kVecBlock / 32; ++w) t += sh[threadIdx.x][w];
        M.dpart[blockIdx.x * 12 + threadIdx.x] = t;
    }
}

// One weight by Adam (Kingma & Ba 2015) on the FP32 masters, then its BF16
// entries of the layouts for the kernels.
__device__ __forceinline__ void mp_adam(const MpBuffers& M, int p, float lr, int t)
{
    if (lr != 0.f) {
        const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
        const float gp = M.grad[p];
        const float m = b1 * M.m[p] + (1.f - b1) * gp;
        const float v = b2 * M.v[p] + (1.f - b2) * gp * gp;
        M.m[p] = m;
        M.v[p] = v;
        const float mh = m / (1.f - powf(b1, (float)t));
        const float vh = v / (1.f - powf(b2, (float)t));
        M.master[p] -= lr * mh / (sqrtf(vh) + eps);
    }
    const __nv_bfloat16 w = __float2bfloat16_rn(M.master[p]);
    if (p < kMpOffW2) {
        const int f = p / 64, i = p % 64;     // W1[f][i]
        M.wb[kW1T + i * 16 + f] = w;
    } else if (p < kMpOffW3) {
        const int q = p - kMpOffW2, i = q / 64, h = q % 64;   // W2[i][h]
        M.wb[kW2T + h * 64 + i] = w;
        M.wb[kW2N + i * 64 + h] = w;
    } else if (p < kMpOffO) {
        const int q = p - kMpOffW3, h = q / 4, m = q % 4;     // W3[h][m]
        M.wb[kW3T + m * 64 + h] = w;
        M.wb[kW3P + h * 16 + m] = w;
    }
}

__global__ void k_mp_convert(MpBuffers M)
{
    const int p = blockIdx.x * blockDim.x + threadIdx.x;
    if (p < kMpParams) mp_adam(M, p, 0.f, 1);
}

// grad = sum over blocks, the readout's gradient and the loss from the loss
// blocks, and the weight's Adam step.  The weights' FP32 partials are added one
// by one in the order of the blocks (the rounding of that order is the
// gradient's): all warps bring a run of them into shared memory and the first
// adds them up (one thread per weight loading all of them in turn took 75 us);
// the FP64 partials are shared out among the warps.
constexpr int kGradRun = 160;
__global__ void __launch_bounds__(256) k_mp_update(MpBuffers M, int nblocks_mlp, int nblocks_loss, int rows, float lr,
                                                   int t)
{
    __shared__ float run[kGradRun][32];
    __shared__ double sh[8][32];
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, p = blockIdx.x * 32 + lane;
    static_assert(kMpOffO % 32 == 0, "a block's weights are all the network's or all the readout's");
    if (p < kMpOffO) {
        float f = 0.f;
        for (int b0 = 0; b0 < nblocks_mlp; b0 += kGradRun) {
            const int m = min(kGradRun, nblocks_mlp - b0);
#pragma unroll 4
            for (int b = warp; b < m; b += 8) run[b][lane] = M.gpart[(size_t)(b0 + b) * kMpParams + p];
            __syncthreads();
            if (warp == 0)
#pragma unroll 8
                for (int b = 0; b < m; ++b) f += run[b][lane];
            __syncthreads();
        }
        if (warp != 0) return;
        M.grad[p] = f;
    } else {   // entry 0 of a loss block: sum e^2; 1 + k: the readout's gradient
        double s = 0.0;
        if (p <= kMpParams) {
            const int k = p < kMpParams ? 1 + (p - kMpOffO) : 0;
#pragma unroll 4
            for (int b = warp; b < nblocks_loss; b += 8) s += M.dpart[b * 12 + k];
        }
        sh[warp][lane] = s;
        __syncthreads();
        if (warp != 0 || p > kMpParams) return;
        double a = 0.0;
        for (int w = 0; w < 8; ++w) a += sh[w][lane];
        if (p == kMpParams) {
            M.scal[1] = a / rows;
            return;
        }
        M.grad[p] = (float)a;
    }
    mp_adam(M, p, lr, t);
}

// ------------------------------------------------------------------ launchers

void launch_mp_infer(const KParams& P, DevBuffers& B, MpBuffers& M, Launch L)
{
    const int rows = 3 * P.n;
    k_mp_scale<<<grid_for(P.n, kVecBlock, L.num_sms * 4), kVecBlock, 0, L.stream>>>(P, B, M);
    k_mp_input<<<grid_for(P.n, kVecBlock, 1 << 30), kVecBlock, 0, L.stream>>>(P, B, M);
    k_mp_aggregate<<<grid_for(P.n, 128, 1 << 30), 128, 0, L.stream>>>(P, B, M.x0, M.a0);
    k_mp_mlp_fwd_tc<<<grid_for(rows, tc::kRows, L.num_sms * 6), tc::kRows, 0, L.stream>>>(rows, M, B.st);
    k_mp_aggregate_output<<<grid_for(P.n, 128, 1 << 30), 128, 0, L.stream>>>(P, B, M);
}

int mp_infer_launches() { return 5; }

void launch_mp_apply(const KParams& P, DevBuffers& B, const MpBuffers& M, const double* in, double* out, Launch L)
{
    MpBuffers A = M;
    A.in = in;
    A.out = out;
    A.zero_vprev = 1;
    launch_mp_infer(P, B, A, L);
}

void launch_mp_train(const KParams& P, DevBuffers& B, MpBuffers& M, float lr, int t, Launch L)
{
    const int rows = 3 * P.n;
    const int nloss = grid_for(rows, kVecBlock, std::min(kMaxGradBlocks, L.num_sms * 2));
    k_mp_loss<<<nloss, kVecBlock, 0, L.stream>>>(P, B, M);
    k_mp_pull<<<grid_for(P.n, 128, 1 << 30), 128, 0, L.stream>>>(P, B, M);
    const int nmlp = grid_for(rows, kTileRows, std::min(kMaxGradBlocks, L.num_sms));
    k_mp_mlp_bwd_tc<<<nmlp, 128 * tcb::kBGroups, mp_bwd_tc_smem_bytes(), L.stream>>>(rows, M, B.st);
    k_mp_update<<<kMpParams / 32 + 1, 256, 0, L.stream>>>(M, nmlp, nloss, rows, lr, t);
}

int mp_prepare()
{
    return (int)cudaFuncSetAttribute(k_mp_mlp_bwd_tc, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     mp_bwd_tc_smem_bytes());
}

int mp_weights_bf16_count() { return kWB; }

void launch_mp_convert(MpBuffers& M, cudaStream_t s)
{
    k_mp_convert<<<grid_for(kMpParams, kVecBlock, 1 << 30), kVecBlock, 0, s>>>(M);
}

}  // namespace ss
