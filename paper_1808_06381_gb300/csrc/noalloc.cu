// sp_solve_csr_noalloc: the velocity solve of Eq. algebra for callers that
// cannot allocate device memory.
//
// Some callers run where cudaMalloc is not available to them: inside a host
// framework that owns every device allocation (a fixed memory pool, a
// real-time or embedded loop that forbids allocation after start-up, or a
// library that must not touch the caller's allocator).  This entry point takes
// the system and the output from the caller and keeps what its blocks exchange
// (the two buffers of published records, the partial sums and the solver's
// state) in one file-scope device array of fixed size, so it never allocates.
//
// The solve is one cooperative launch of the on-chip CG of pcg64.cuh: the
// entries in shared memory, the vectors in registers.  Jacobi-PCG with the
// direction update fused into the product (q = A z + beta q, p = z + beta p),
// two grid reductions per iteration: a caller's matrix may be worse
// conditioned than Eq. algebra's, and pipelined CG (one reduction) drifts
// further from the true residual.  Measured (n = 12,289 clustered rows in
// random order, 62 iterations): one thread per row, four kernels an iteration
// and the host polling every eighth, 3.48 ms; this form 0.96 ms.
//
// Limits and sharing:
//   - at most kNoallocMaxRows rows; larger systems are rejected;
//   - the array (about 2.1 MB) lives in every device context that loads the
//     library, until the process exits;
//   - every call on a device uses the same array: calls that may overlap on
//     the GPU (other streams, other host threads) race and must be serialised
//     by the caller;
//   - the first call on a device looks up the array's device address with that
//     device current; every call reads the solver state back and synchronises
//     its stream, so no call may be made on a stream that is being captured
//     (such a call is rejected);
//   - device ordinals 0 .. 63 (one looked-up address per device).
#include <cuda_runtime.h>

#include <cmath>
#include <cstdlib>
#include <cstring>
#include <mutex>
#include <string>

#include "internal.cuh"
#include "pcg64.cuh"

namespace ss {
namespace {

constexpr long long kNoallocMaxRows = 32768;
constexpr int kNaMaxBlocks = 512;

struct NaState {
    double bnorm2, last_res;
    int iter, status, done, error;
    alignas(128) unsigned int count;   // the launch's grid barriers (pcg64.cuh)
    alignas(128) unsigned int exits;
};

constexpr size_t kRecordDoubles = 2 * 4 * (size_t)kNoallocMaxRows;       // two buffers of (x, y, z, 0) per row
constexpr size_t kPartialDoubles = 2 * p64::kScalarWarps * kNaMaxBlocks;
constexpr size_t kScratchBytes = (kRecordDoubles + kPartialDoubles) * sizeof(double) + sizeof(NaState);

static __device__ __align__(256) unsigned char g_noalloc_scratch[kScratchBytes];

struct NaSystem {   // the caller's arrays, and pcg64's system
    long long n;
    const int* row_ptr;
    const int* col;
    const double* w;
    const double* diag;
    double alpha_e;
    const double* b;
    double* x;
    double tol2;
    int max_iter;
    using Value = double;
    const int* rows;   // the block's rows by length, in its shared memory (-1: none)
    struct Entries {
        const int* col;
        const double* w;
        int cnt;
        bool ok;
        __device__ bool valid() const { return ok; }
        __device__ void get(int k, int& j, double& v) const
        {
            if (k < cnt) {
                j = __ldg(col + k);
                v = __ldg(w + k);
            }
        }
    };
    __device__ double alpha() const { return alpha_e; }
    __device__ bool in_range(int j) const { return j >= 0 && j < n; }
    __device__ int row(int i, int lane) const { return rows[32 * i + lane]; }
    // row_ptr must start at 0 and never decrease; a row that breaks this is
    // not read (and fails the call)
    __device__ Entries entries(int, int, int row) const
    {
        if (row < 0) return Entries{col, w, 0, true};
        const int e0 = row_ptr[row], e1 = row_ptr[row + 1];
        const bool ok = e0 >= 0 && e1 >= e0 && (row != 0 || e0 == 0);
        return Entries{col + (ok ? e0 : 0), w + (ok ? e0 : 0), ok ? e1 - e0 : 0, ok};
    }
    __device__ int chunk_len(int i, int lane) const
    {
        return __reduce_max_sync(0xffffffffu, entries(i, lane, row(i, lane)).cnt);
    }
};

struct NaScalars {
    double rho, bnorm2, last_res;
    int iter, restarts, status;
};

// Every block validates the rows it reads (row_ptr, and every column inside [0,
// n)) while it places them, before anything gathers through a column; the
// first grid reduction carries the verdict, so a malformed system is refused
// by all blocks together and x stays as it was.
template <int U, int KB>
__global__ void __launch_bounds__(p64::max_threads(U), 1) k_na_solve(NaSystem S, double* scratch, int smem_bytes,
                                                                       unsigned long long limit_ns)
{
    extern __shared__ double na_dyn[];
    __shared__ p64::Shared sh;
    __shared__ NaScalars cg;
    __shared__ int rows[32 * p64::kMaxChunks];
    unsigned char* dyn = reinterpret_cast<unsigned char*>(na_dyn);
    NaState* st = reinterpret_cast<NaState*>(scratch + kRecordDoubles + kPartialDoubles);
    const p64::Grid G{&st->count, &st->exits, &st->error, limit_ns, scratch + kRecordDoubles, kNaMaxBlocks,
                      (int)blockIdx.x, (int)gridDim.x};
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    const int ncw = (blockDim.x >> 5) - p64::kScalarWarps, groups = ncw / 3;
    const int grp = warp / 3, comp = warp - 3 * grp;
    const int nch = (int)((S.n + 31) / 32), nc = (nch - G.bid + G.nb - 1) / G.nb;   // chunks bid, bid + nb, ...
    const int cap = smem_bytes / p64::kEntryBytes<double>;
    if (threadIdx.x == 0) {
        sh.flag = 0;
        sh.action = 0;
        cg.status = SP_OK;
        cg.iter = cg.restarts = 0;
        cg.bnorm2 = cg.last_res = 0.0;
    }
    // the block's rows sorted by length, so that a chunk's rows are about
    // equally long (the caller's order is arbitrary: chunks of 32 rows as they
    // come carry ~1.9x the entries of their rows as padding); the keys are
    // ordered in the dynamic space that the entries take afterwards
    {
        unsigned long long* key = reinterpret_cast<unsigned long long*>(na_dyn);
        const int R = 32 * nc;
        for (int k = threadIdx.x; k < R; k += blockDim.x) {
            const long long i = 32ll * (G.bid + (long long)G.nb * (k >> 5)) + (k & 31);
            const unsigned long long len = i < S.n ? 1ull + (unsigned)S.entries(0, 0, (int)i).cnt : 0ull;
            key[k] = (len << 32) | (unsigned)k;
        }
        __syncthreads();
        for (int k = threadIdx.x; k < R; k += blockDim.x) {
            const unsigned long long mine = key[k];
            int before = 0;
            for (int m = 0; m < R; ++m) before += key[m] > mine;
            rows[before] = mine >> 32 ? 32 * (G.bid + G.nb * (k >> 5)) + (k & 31) : -1;
        }
        __syncthreads();
    }
    S.rows = rows;
    p64::stage(S, sh, dyn, smem_bytes, nc);
    unsigned int gen = 0u;
    double* rec[2] = {scratch, scratch + 4 * (size_t)kNoallocMaxRows};
    int cur = 0;   // the buffer of the next product
    int row[U];
    double x[U], r[U], p[U], q[U], di[U], sm[U];
    double v0 = 0.0, v1 = 0.0, v2 = threadIdx.x == 0 && sh.bad ? 1.0 : 0.0;
#pragma unroll
    for (int u = 0; u < U; ++u) {   // x = 0, r = b; z = D^-1 r published; b.b, r.z
        const int i = grp + groups * u;
        row[u] = warp < ncw && i < nc ? S.row(i, lane) : -1;
        x[u] = r[u] = p[u] = q[u] = di[u] = sm[u] = 0.0;
        if (row[u] < 0) continue;
        r[u] = S.b[comp * S.n + row[u]];
        di[u] = 1.0 / S.diag[row[u]];
        const double z = di[u] * r[u];
        v0 = fma(r[u], r[u], v0);
        v1 = fma(r[u], z, v1);
        rec[0][4 * (size_t)row[u] + comp] = z;
    }
    auto publish = [&](int u, double v) { rec[cur ^ 1][4 * (size_t)row[u] + comp] = v; };
    enum { kStart, kDirection, kUpdate, kX, kTrue };   // the values the next reduction carries (kX: none)
    int phase = kStart;
    auto product = [&] {   // sum_j alpha w_ij of the published vector
        if (phase == kDirection || sh.bad) return;
#pragma unroll
        for (int u = 0; u < U; ++u) {
            const int i = grp + groups * u;
            if (i < nc) sm[u] = p64::row_product<KB>(S, sh, dyn, cap, i, row[u], rec[cur], comp);
        }
    };
    auto scalars = [&] {   // one thread per block, the same totals in every block
        const double t0 = sh.tot[0], t1 = sh.tot[1];
        sh.action = 0;
        sh.beta = 0.0;
        if (phase == kStart) {
            cg.bnorm2 = t0;
            cg.rho = t1;
            if (sh.tot[2] != 0.0) {
                cg.status = SP_ERR_INVALID_ARG;
                sh.action = 2;
            } else if (!isfinite(t0)) {
                cg.status = SP_ERR_NONFINITE;
                sh.action = 2;
            } else if (t0 == 0.0) {
                sh.action = 2;   // b = 0: x = 0
            }
        } else if (phase == kDirection) {   // p.q
            if (!(t0 > 0.0) || !isfinite(t0)) {
                cg.status = SP_ERR_NONFINITE;
                sh.action = 2;
            } else {
                sh.alpha = cg.rho / t0;
            }
        } else if (phase == kUpdate) {      // r.r, r.z
            ++cg.iter;
            if (!isfinite(t0)) {
                cg.status = SP_ERR_NONFINITE;
                sh.action = 2;
            } else if (t0 <= S.tol2 * cg.bnorm2 || cg.iter >= S.max_iter) {
                sh.action = 1;   // the true residual decides
            } else {
                sh.beta = t1 / cg.rho;
                cg.rho = t1;
            }
        } else {                            // the true residual's r.r, r.z
            cg.last_res = sqrt(t0 / cg.bnorm2);
            if (t0 <= S.tol2 * cg.bnorm2) {
                sh.action = 2;
            } else if (cg.iter >= S.max_iter || cg.restarts >= kMaxCgRestarts) {
                cg.status = SP_ERR_NOT_CONVERGED;
                sh.action = 2;
            } else {
                ++cg.restarts;
                cg.rho = t1;
            }
        }
    };
    for (;;) {
        const int K = phase == kX ? 0 : (phase == kStart ? 3 : (phase == kDirection ? 1 : 2));
        if (!p64::reduce_overlapped(G, sh, gen, K, v0, v1, v2, product, scalars)) break;
        if (K > 0 && sh.action == 2) break;
        v0 = v1 = v2 = 0.0;
        if (phase == kX) {   // r = b - A x
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (row[u] < 0) continue;
                r[u] = S.b[comp * S.n + row[u]] - (S.diag[row[u]] * x[u] - sm[u]);
                const double z = di[u] * r[u];
                v0 = fma(r[u], r[u], v0);
                v1 = fma(r[u], z, v1);
                publish(u, z);
            }
            cur ^= 1;
            phase = kTrue;
        } else if (phase == kDirection) {   // x += alpha p; r -= alpha q; z published
            const double a = sh.alpha;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (row[u] < 0) continue;
                r[u] = fma(-a, q[u], r[u]);
                const double z = di[u] * r[u];
                publish(u, z);
                x[u] = fma(a, p[u], x[u]);
                v0 = fma(r[u], r[u], v0);
                v1 = fma(r[u], z, v1);
            }
            cur ^= 1;
            phase = kUpdate;
        } else if (sh.action == 1) {        // the true residual: x published
#pragma unroll
            for (int u = 0; u < U; ++u)
                if (row[u] >= 0) publish(u, x[u]);
            cur ^= 1;
            phase = kX;
        } else {                            // q = A z + beta q (A_ii z = r); p = z + beta p
            const double beta = sh.beta;
#pragma unroll
            for (int u = 0; u < U; ++u) {
                if (row[u] < 0) continue;
                q[u] = fma(beta, q[u], r[u] - sm[u]);
                p[u] = fma(beta, p[u], di[u] * r[u]);
                v0 = fma(p[u], q[u], v0);
            }
            phase = kDirection;
        }
    }
    if (cg.status != SP_ERR_INVALID_ARG) {
#pragma unroll
        for (int u = 0; u < U; ++u)
            if (row[u] >= 0) S.x[comp * S.n + row[u]] = x[u];
    }
    if (G.bid == 0 && threadIdx.x == 0) {
        st->bnorm2 = cg.bnorm2;
        st->last_res = cg.last_res;
        st->iter = cg.iter;
        st->status = cg.status;
        st->done = 1;
    }
    p64::leave(G);
}

std::mutex g_na_mutex;
void* g_na_base[64] = {nullptr};

}  // namespace
}  // namespace ss

extern std::string& sp_global_error();

extern "C" int sp_solve_csr_noalloc(int32_t device, void* stream, int64_t n, const int32_t* row_ptr_dev,
                                    const int32_t* col_dev, const double* w_dev, const double* diag_dev,
                                    double alpha, const double* b_dev, double* x_dev, double tol,
                                    int32_t max_iter, sp_solve_info* info)
{
    using namespace ss;
    std::string& err = sp_global_error();
    if (n < 1 || n > kNoallocMaxRows) {
        err = "sp_solve_csr_noalloc: n must be in [1, " + std::to_string(kNoallocMaxRows) + "]";
        return SP_ERR_INVALID_ARG;
    }
    if (!row_ptr_dev || !col_dev || !w_dev || !diag_dev || !b_dev || !x_dev || !(tol > 0) || max_iter < 1 ||
        !(alpha >= 0) || device < 0 || device >= 64) {
        err = "sp_solve_csr_noalloc: null pointer or invalid tol, max_iter, alpha or device";
        return SP_ERR_INVALID_ARG;
    }
    int prev = -1;
    if (cudaGetDevice(&prev) != cudaSuccess || cudaSetDevice(device) != cudaSuccess) {
        cudaGetLastError();
        err = "sp_solve_csr_noalloc: no CUDA device with that ordinal";
        return SP_ERR_NO_DEVICE;
    }
    auto finish = [&](int rc, const char* what) {
        if (what) err = std::string("sp_solve_csr_noalloc: ") + what + ": " + cudaGetErrorString(cudaGetLastError());
        cudaSetDevice(prev);
        return rc;
    };
    // every call reads the solver state back and synchronises, which a stream
    // under capture does not allow (checked before anything else touches the device)
    cudaStreamCaptureStatus cap = cudaStreamCaptureStatusNone;
    if (cudaStreamIsCapturing(static_cast<cudaStream_t>(stream), &cap) != cudaSuccess)
        return finish(SP_ERR_CUDA, "cudaStreamIsCapturing");
    if (cap != cudaStreamCaptureStatusNone) {
        err = "sp_solve_csr_noalloc: the stream is being captured; this call synchronises and cannot be captured";
        cudaSetDevice(prev);
        return SP_ERR_INVALID_ARG;
    }
    void* base = nullptr;
    {
        std::lock_guard<std::mutex> lock(g_na_mutex);
        if (!g_na_base[device]) {
            void* p = nullptr;
            if (cudaGetSymbolAddress(&p, g_noalloc_scratch) != cudaSuccess || !p)
                return finish(SP_ERR_CUDA, "cudaGetSymbolAddress");
            g_na_base[device] = p;
        }
        base = g_na_base[device];
    }
    double* scratch = static_cast<double*>(base);
    NaSystem S{n, row_ptr_dev, col_dev, w_dev, diag_dev, alpha, b_dev, x_dev, tol * tol, max_iter, nullptr};
    cudaStream_t s = static_cast<cudaStream_t>(stream);
    NaState* st = reinterpret_cast<NaState*>(scratch + kRecordDoubles + kPartialDoubles);
    int num_sms = 1;
    if (cudaDeviceGetAttribute(&num_sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess)
        return finish(SP_ERR_CUDA, "cudaDeviceGetAttribute");
    // fewer SMs than the device has: only to exercise the forms that a device of few SMs (a part of a
    // GB300 given out as an instance of its own) takes, four and sixteen chunks a thread
    if (const char* few = std::getenv("SHEARSIM_NOALLOC_SMS")) num_sms = std::max(1, std::min(num_sms, std::atoi(few)));
    p64::Shape sp = p64::shape_of((int)((n + 31) / 32), std::min(num_sms, kNaMaxBlocks), 16);
    // sixteen chunks a thread keep part of their vectors in local memory
    const void* fn = sp.u == 1 ? (const void*)k_na_solve<1, 12>
                               : (sp.u == 2 ? (const void*)k_na_solve<2, 8>
                                            : (sp.u == 4 ? (const void*)k_na_solve<4, 6> : (const void*)k_na_solve<16, 4>));
    if (sp.u == 0) {
        err = "sp_solve_csr_noalloc: too few SMs for this system";
        return finish(SP_ERR_CUDA, nullptr);
    }
    // the state (and the grid barriers' counters) must start at zero on every call
    if (cudaMemsetAsync(st, 0, sizeof(NaState), s) != cudaSuccess) return finish(SP_ERR_CUDA, "cudaMemsetAsync");
    if (sp.smem > 32 * 1024 &&   // with the static arrays, near the 48 KB a kernel has by default
        allow_shared_memory(fn, p64::kMaxSmem) != cudaSuccess)
        return finish(SP_ERR_CUDA, "cudaFuncSetAttribute");
    unsigned long long limit_ns = kDefaultWaitLimitNs;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3((unsigned)sp.blocks);
    cfg.blockDim = dim3((unsigned)sp.threads);
    cfg.dynamicSmemBytes = (size_t)sp.smem;
    cfg.stream = s;
    cudaLaunchAttribute attr[1];
    attr[0].id = cudaLaunchAttributeCooperative;
    attr[0].val.cooperative = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 1;
    void* args[] = {&S, &scratch, &sp.smem, &limit_ns};
    if (cudaLaunchKernelExC(&cfg, fn, args) != cudaSuccess) return finish(SP_ERR_CUDA, "launching the solve");
    NaState h;
    std::memset(&h, 0, sizeof(h));
    if (cudaMemcpyAsync(&h, st, sizeof(NaState), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
        cudaStreamSynchronize(s) != cudaSuccess)
        return finish(SP_ERR_CUDA, "reading the solver state");
    if (h.error != 0) h.status = h.error;
    int status = h.done ? h.status : SP_ERR_NOT_CONVERGED;
    if (info) {
        info->status = status;
        info->iterations = h.iter;
        info->residual = h.last_res;
        info->bnorm = std::sqrt(h.bnorm2);
        info->offchip_blocks = 0;
    }
    if (status == SP_ERR_INVALID_ARG)
        err = "sp_solve_csr_noalloc: row_ptr must start at 0 and not decrease, and every col must lie in [0, n)";
    else if (status == SP_ERR_NOT_CONVERGED)
        err = "sp_solve_csr_noalloc: not converged (max_iter reached, or the true residual stayed above tol "
              "after the restart limit)";
    else if (status == SP_ERR_TIMEOUT)
        err = "sp_solve_csr_noalloc: a grid-barrier wait ran past its limit";
    else if (status != SP_OK)
        err = "sp_solve_csr_noalloc: solve failed";
    return finish(status, nullptr);
}
