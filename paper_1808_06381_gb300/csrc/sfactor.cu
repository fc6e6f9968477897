// Inter-chain structure factor S(q) = (1/n) |sum_c exp(-i q . R_c)|^2 at q_z = 0
// (arXiv 1808.06381, Eq. Sfactor; the paper shows it in the flow-gradient
// plane as S(q_x, q_y)).
//
// Under Lees-Edwards shear the allowed wave vectors form the sheared reciprocal
// lattice q_x = 2 pi kx / L_x, q_y = 2 pi ky / L_y - gamma q_x with gamma =
// delta / L_y: in the sheared frame x' = x - gamma y (mod L_x) the density is
// periodic in (x', y) and q . R = 2 pi (kx x' / L_x + ky y / L_y).
//
// Grid mode: cloud-in-cell deposit of the particles on a G x G grid of the
// sheared frame (z summed, since q_z = 0), in 2^-32 fixed point with integer
// atomics so that the grid does not depend on the order of the deposits; a
// separable DFT of the grid for the requested modes with a precomputed twiddle
// table; division by the CIC window sinc^2(pi kx / G) sinc^2(pi ky / G).  All
// bound by GB300's FP64 pipe (2 FMA per clock and SM), so the FP64 operations
// are counted: the deposit's products are 64-bit integer, the density is real
// (kx >= 0 only, the rest by conjugation), and both transforms sum a point
// together with its mirror G - g (half the multiplications; in y both signs of
// ky from the same products).
// Direct mode: the sum over particles for every requested mode, in FP64.
#include <math.h>

#include "internal.cuh"
#include "sfactor_cell.cuh"

namespace ss {

namespace {

constexpr double kFix = 4294967296.0;   // 2^32

// Fractions of a cell in 2^-50, weights in 2^-32: integer products rounded to
// nearest like the FP64 products they replace, three FP64 operations and two
// conversions a particle instead of ~150 (four divisions, eight products and four
// roundings): 33.6 us at n = 262,144 before, 10.0 now.  Every value of a
// coordinate lands on the grid (grid_cell).
__global__ void k_sq_deposit(KParams P, const double* __restrict__ pos, double gamma, double sx, double sy, int G,
                             unsigned long long* __restrict__ grid)
{
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= P.n) return;
    const double x = pos[i], y = pos[P.npad + i];
    const GridCell u = grid_cell(fma(-gamma, y, x) * sx, G), v = grid_cell(y * sy, G);
    atomicAdd(grid + (size_t)v.i0 * G + u.i0, cell_weight(u.g, v.g));
    atomicAdd(grid + (size_t)v.i0 * G + u.i1, cell_weight(u.f, v.g));
    atomicAdd(grid + (size_t)v.i1 * G + u.i0, cell_weight(u.g, v.f));
    atomicAdd(grid + (size_t)v.i1 * G + u.i1, cell_weight(u.f, v.f));
}

// Block gy: A[kx][gy] = sum_gx rho[gy][gx] exp(-2 pi i kx gx / G) for kx =
// 0..nkx.  The row is folded about gx = 0 as it is read (exact integer sums
// and differences): re = rho_0 + sum_(m >= 1) (rho_m + rho_(G-m)) cos, im = -sum
// (rho_m - rho_(G-m)) sin (for even G the middle point m = G / 2 has cos only).
// A group of kSqSplit neighbouring lanes shares a kx, each taking every
// kSqSplit-th m.  The blocks from G on write the squared inverse windows
// 1 / sinc^4(pi k / G) of k = 0..kmax.  (One thread per (kx, gy) reading a
// column of the grid: 76.7 us at G = 256, nkx = 48; this form 13.4.)
constexpr int kSqSplit = 8;
__global__ void __launch_bounds__(256) k_sq_dft_x(const unsigned long long* __restrict__ grid, int G, int nkx, int kmax,
                                                  const double2* __restrict__ tw, double2* __restrict__ A,
                                                  double* __restrict__ win)
{
    extern __shared__ double2 sq_sm[];
    if ((int)blockIdx.x >= G) {
        const int k = ((int)blockIdx.x - G) * blockDim.x + threadIdx.x;
        if (k > kmax) return;
        double w = 1.0;
        if (k != 0) {
            const double pi = 3.14159265358979323846, s = sin(pi * k / G) / (pi * k / G);
            w = s * s;
        }
        win[k] = 1.0 / (w * w);
        return;
    }
    double2* t = sq_sm;                  // [G] twiddles
    double2* f = sq_sm + G;              // [G / 2 + 1] (rho_m + rho_(G-m), rho_m - rho_(G-m))
    const unsigned long long* row = grid + (size_t)blockIdx.x * G;
    const int half = G / 2, last = (G - 1) / 2;   // the mirrored points are m = 1..last
    for (int m = threadIdx.x; m < G; m += blockDim.x) t[m] = tw[m];
    for (int m = threadIdx.x; m <= half; m += blockDim.x) {
        const long long a = (long long)row[m], b = m >= 1 && m <= last ? (long long)row[G - m] : 0ll;
        f[m] = make_double2((double)(a + b), m >= 1 && m <= last ? (double)(a - b) : 0.0);
    }
    __syncthreads();
    const int sub = threadIdx.x % kSqSplit;
    for (int k0 = 0; k0 <= nkx; k0 += blockDim.x / kSqSplit) {
        const int kx = k0 + threadIdx.x / kSqSplit;
        double re = 0.0, im = 0.0;
        if (kx <= nkx) {
            const int step = (int)((long long)kx * kSqSplit % G);
            int at = (int)((long long)kx * sub % G);
            for (int m = sub; m <= half; m += kSqSplit) {
                const double2 w = t[at], r = f[m];
                re = fma(r.x, w.x, re);
                im = fma(-r.y, w.y, im);
                at += step;
                if (at >= G) at -= G;
            }
        }
#pragma unroll
        for (int o = kSqSplit / 2; o > 0; o >>= 1) {
            re += __shfl_xor_sync(0xffffffffu, re, o);
            im += __shfl_xor_sync(0xffffffffu, im, o);
        }
        if (kx <= nkx && sub == 0) A[(size_t)kx * G + blockIdx.x] = make_double2(re / kFix, im / kFix);
    }
}

// F[kx][ky] = sum_gy A[kx][gy] exp(-2 pi i ky gy / G) for one kx >= 0 (blockIdx.x)
// and kSqKy values of ky >= 0 (blockIdx.y), and with the same products F[kx][-ky]:
// with P = A_m + A_(G-m), Q = A_m - A_(G-m), C = A_0 + sum P cos and D = sum Q
// sin, F[kx][+-ky] = C -+ i D.  S = |F|^2 / n over the window; S[-kx][-ky] = S[kx][ky].
// (One thread per mode, 256 complex products in turn: 126 us at G = 256, 97 x 97
// modes; this form 10.8.)
constexpr int kSqKy = 16;
__global__ void __launch_bounds__(kSqKy * kSqSplit) k_sq_dft_y(const double2* __restrict__ A, int G, int nkx, int nky,
                                                                const double2* __restrict__ tw,
                                                                const double* __restrict__ win, KParams P, double delta,
                                                                double* __restrict__ S, double* __restrict__ qx,
                                                                double* __restrict__ qy, int tw_shared)
{
    extern __shared__ double2 sq_sm[];
    double2* fp = sq_sm;                     // [G / 2 + 1] P (A_0 and the middle point as they are)
    double2* fq = fp + G / 2 + 1;            // [G / 2 + 1] Q
    double2* ts = fq + G / 2 + 1;            // [G] twiddles, where they fit
    const double2* t = tw_shared ? ts : tw;
    const int kx = blockIdx.x, half = G / 2, last = (G - 1) / 2;
    const double2* row = A + (size_t)kx * G;
    if (tw_shared)
        for (int m = threadIdx.x; m < G; m += blockDim.x) ts[m] = tw[m];
    for (int m = threadIdx.x; m <= half; m += blockDim.x) {
        const double2 a = row[m];
        if (m >= 1 && m <= last) {
            const double2 b = row[G - m];
            fp[m] = make_double2(a.x + b.x, a.y + b.y);
            fq[m] = make_double2(a.x - b.x, a.y - b.y);
        } else {
            fp[m] = a;
            fq[m] = make_double2(0.0, 0.0);
        }
    }
    __syncthreads();
    const int ky = blockIdx.y * kSqKy + threadIdx.x / kSqSplit, sub = threadIdx.x % kSqSplit;
    double cr = 0.0, ci = 0.0, dr = 0.0, di = 0.0;
    if (ky <= nky) {
        const int step = (int)((long long)ky * kSqSplit % G);
        int at = (int)((long long)ky * sub % G);
        for (int m = sub; m <= half; m += kSqSplit) {
            const double2 w = t[at], p = fp[m], q = fq[m];
            cr = fma(p.x, w.x, cr);
            ci = fma(p.y, w.x, ci);
            dr = fma(q.x, w.y, dr);
            di = fma(q.y, w.y, di);
            at += step;
            if (at >= G) at -= G;
        }
    }
#pragma unroll
    for (int o = kSqSplit / 2; o > 0; o >>= 1) {
        cr += __shfl_xor_sync(0xffffffffu, cr, o);
        ci += __shfl_xor_sync(0xffffffffu, ci, o);
        dr += __shfl_xor_sync(0xffffffffu, dr, o);
        di += __shfl_xor_sync(0xffffffffu, di, o);
    }
    if (ky > nky || sub >= 4) return;
    // lanes 0..3 of the group: the modes (kx, ky), (kx, -ky), (-kx, ky), (-kx, -ky)
    const int my = 2 * nky + 1;
    const int mx = sub & 2 ? -kx : kx, m_y = sub & 1 ? -ky : ky;
    const double sg = ((sub >> 1) ^ sub) & 1 ? -1.0 : 1.0;   // F[kx][ky sg]: S[-kx][ky] = S[kx][-ky]
    const double re = fma(sg, di, cr), im = fma(-sg, dr, ci);
    const double pi = 3.14159265358979323846;
    const size_t at = (size_t)(mx + nkx) * my + (m_y + nky);
    S[at] = (re * re + im * im) * (win[kx] * win[ky]) / P.n;
    const double q_x = 2.0 * pi * mx / P.L[0];
    qx[at] = q_x;
    qy[at] = 2.0 * pi * m_y / P.L[1] - delta / P.L[1] * q_x;
}

// Direct sum over particles for each mode (one block per mode).
__global__ void k_sq_direct(KParams P, const double* __restrict__ pos, double delta, int nkx, int nky,
                            double* __restrict__ S, double* __restrict__ qx, double* __restrict__ qy)
{
    __shared__ double sh[32];
    const int t = blockIdx.x;
    const int my = 2 * nky + 1;
    const int kx = t / my - nkx, ky = t % my - nky;
    const double pi = 3.14159265358979323846;
    const double q_x = 2.0 * pi * kx / P.L[0];
    const double q_y = 2.0 * pi * ky / P.L[1] - delta / P.L[1] * q_x;
    const int np = P.npad;
    double re = 0.0, im = 0.0;
    for (int i = threadIdx.x; i < P.n; i += blockDim.x) {
        double s, c;
        sincos(q_x * pos[i] + q_y * pos[np + i], &s, &c);
        re += c;
        im -= s;
    }
    re = block_sum(re, sh);
    __syncthreads();
    im = block_sum(im, sh);
    if (threadIdx.x == 0) {
        S[t] = (re * re + im * im) / P.n;
        qx[t] = q_x;
        qy[t] = q_y;
    }
}

}  // namespace

cudaError_t run_structure_factor(const KParams& P, const DevBuffers& B, double delta, int G, int nkx, int nky,
                                 const double* twiddle_dev, unsigned long long* grid_dev, double2* A_dev,
                                 double* S_dev, double* qx_dev, double* qy_dev, cudaStream_t s)
{
    const int m = (2 * nkx + 1) * (2 * nky + 1);
    if (G == 0) {
        k_sq_direct<<<m, 256, 0, s>>>(P, B.pos_s, delta, nkx, nky, S_dev, qx_dev, qy_dev);
        return cudaGetLastError();
    }
    cudaMemsetAsync(grid_dev, 0, sizeof(unsigned long long) * (size_t)G * G, s);
    const double unit = kCellUnit * G;
    k_sq_deposit<<<grid_for(P.n, kVecBlock, 1 << 30), kVecBlock, 0, s>>>(P, B.pos_s, delta / P.L[1], unit / P.L[0],
                                                                            unit / P.L[1], G, grid_dev);
    const double2* tw = reinterpret_cast<const double2*>(twiddle_dev);
    double* win = reinterpret_cast<double*>(A_dev + (size_t)(nkx + 1) * G);
    const int kmax = nkx > nky ? nkx : nky, extra = kmax / 256 + 1;
    const size_t tab = sizeof(double2) * (size_t)G, hf = sizeof(double2) * (size_t)(G / 2 + 1);
    const size_t sx = tab + hf;                                    // at most 192 KB (G = 8,192)
    const int tw_shared = tab + 2 * hf <= 200 * 1024 ? 1 : 0;      // G above ~6,400: the table through L1
    const size_t sy = 2 * hf + (tw_shared ? tab : 0);
    constexpr int kMaxSmem = 200 * 1024;   // sx and sy at every G
    if (tab + 2 * hf > 32 * 1024 && (allow_shared_memory(k_sq_dft_x, kMaxSmem) != cudaSuccess ||
                                     allow_shared_memory(k_sq_dft_y, kMaxSmem) != cudaSuccess))
        return cudaGetLastError();
    k_sq_dft_x<<<G + extra, 256, sx, s>>>(grid_dev, G, nkx, kmax, tw, A_dev, win);
    k_sq_dft_y<<<dim3(nkx + 1, nky / kSqKy + 1), kSqKy * kSqSplit, sy, s>>>(A_dev, G, nkx, nky, tw, win, P, delta, S_dev,
                                                                            qx_dev, qy_dev, tw_shared);
    return cudaGetLastError();
}

}  // namespace ss
