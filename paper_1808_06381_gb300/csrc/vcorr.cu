// Velocity cross-correlation versus distance (arXiv 1808.06381, §Results,
// Fig. vv): the average inter-chain velocity product <v_c . v_c'> / <v_c^2>
// as a function of the inter-chain distance |R_cc'|.
//
// u_c = v_c - kappa (y_c - L_y/2) x is the velocity relative to the imposed
// flow (the Lees-Edwards image of c' moves with v_c' + kappa L_y n x and so
// carries the same u).  Every pair c < c' whose minimum-image distance r is
// below rmax adds u_c . u_c' to bin floor(r nbins / rmax) and counts there.
//
// All pairs are visited (n^2 / 2): one block per 512 particles c (two per
// thread) and a run of 256-particle tiles of c' staged in shared memory, every
// pair in FP32.  The
// decisions that make the result exact are taken in FP64 where FP32 could get
// them wrong: a pair whose FP32 image index, bin or cut-off test lies within
// the FP32 error bound of a boundary is appended to a list, and a second
// kernel decides those pairs with the FP64 operations of the definition, so
// the counts are exact.  The products go into per-warp shared-memory
// histograms as 2^-20-scaled fixed-point integers (scale from the largest
// |u|^2), so the sums do not depend on the order of the additions.
//
// Bound by instruction issue and the histograms' shared-memory atomics.  A
// thread's two particles c go through packed FP32 pairs (two operations an
// instruction); a pair costs two native 32-bit shared atomics, emptied every 64
// tile particles before they can overflow (one 64-bit atomic per pair is a
// compare-and-swap loop); listed pairs are gathered in shared memory and
// appended by one global atomic per 64 tile particles; the order test j > i is
// compiled in for the two diagonal tiles only; the tile keeps every value twice,
// as the packed operations take it, and both pairs' bin decisions are packed and
// predicated.  n = 17,191, 120 bins: 433 us with one 64-bit atomic a pair, 339
// with the packed pairs and 32-bit atomics, 262 with the rest.
#include <math.h>

#include <algorithm>
#include <cstdlib>
#include <cstring>
#include <type_traits>
#include <vector>

#include "internal.cuh"

namespace ss {

namespace {

constexpr int kVcTile = 256;               // particles per tile; threads per block
constexpr int kVcWarps = kVcTile / 32;
constexpr int kVcPrepBlocks = 1024;        // vsq partial sums

struct VcConst {
    int n, nbins, ntile, chunk;
    float Lf[3], iLf[3], df;   // box edges, their inverses, delta (FP32)
    float r2_hi;               // FP32 |R|^2 >= r2_hi: certainly |R| >= rmax
    float r_band;              // FP32 |R| > r_band: decided in FP64
    float inv_f;               // nbins / rmax
    float eb;                  // FP32 bin position within eb of an edge: decided in FP64
    float half[3];             // |component| > half[a] (L_a/2 less the FP32 error): image decided in FP64
    double delta, kappa, rmax2, inv;
    double invL[3];            // 1 / L_a (FP64)
};

// FP32 copies of the positions and of u; FP64 sums of |u|^2 per block and the
// largest FP32 |u|^2 (its bits, non-negative floats order like integers).
__global__ void __launch_bounds__(kVcTile) k_vc_prep(VcConst C, KParams P, const double* __restrict__ pos,
                                                       const double* __restrict__ v, float4* __restrict__ p4,
                                                       float4* __restrict__ u4, double* __restrict__ part,
                                                       unsigned int* __restrict__ umax, int* __restrict__ flag)
{
    __shared__ double ssum[kVcWarps];
    __shared__ float smax[kVcWarps];
    double s = 0.0;
    float m = 0.f;
    for (int i = blockIdx.x * kVcTile + threadIdx.x; i < C.n; i += gridDim.x * kVcTile) {
        const double x = pos[3 * i], y = pos[3 * i + 1], z = pos[3 * i + 2];
        if (!(x >= 0.0 && x < P.L[0] && y >= 0.0 && y < P.L[1] && z >= 0.0 && z < P.L[2])) atomicOr(flag, 1);
        const double ux = v[3 * i] - C.kappa * (y - 0.5 * P.L[1]), uy = v[3 * i + 1], uz = v[3 * i + 2];
        s += ux * ux + uy * uy + uz * uz;
        const float4 uf = make_float4((float)ux, (float)uy, (float)uz, 0.f);
        p4[i] = make_float4((float)x, (float)y, (float)z, 0.f);
        u4[i] = uf;
        m = fmaxf(m, uf.x * uf.x + uf.y * uf.y + uf.z * uf.z);
    }
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    s = warp_sum(s);
    for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    if (lane == 0) {
        ssum[warp] = s;
        smax[warp] = m;
    }
    __syncthreads();
    if (warp == 0) {
        s = lane < kVcWarps ? ssum[lane] : 0.0;
        m = lane < kVcWarps ? smax[lane] : 0.f;
        s = warp_sum(s);
        for (int o = 16; o > 0; o >>= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
        if (lane == 0) {
            part[blockIdx.x] = s;
            atomicMax(umax, __float_as_uint(m));
        }
    }
}

// vsq = (1/n) sum |u|^2 (partials summed in a fixed order) and the
// fixed-point scale S = 2^(20 - e) with max |u_f|^2 < 2^e, so that every FP32
// product times S stays below 2^21 in magnitude.
__global__ void k_vc_scale(int n, int nparts, const double* __restrict__ part, const unsigned int* __restrict__ umax,
                           double* __restrict__ scal)
{
    double s = 0.0;
    for (int k = threadIdx.x; k < nparts; k += 32) s += part[k];
    s = warp_sum(s);
    if (threadIdx.x == 0) {
        scal[0] = s / (double)n;
        const float m = __uint_as_float(*umax);
        int e = 0;
        if (m > 0.f) frexp((double)m, &e);
        scal[1] = ldexp(1.0, 20 - e);
    }
}

// ---- two FP32 values in one register pair (add, multiply and fused
// multiply-add of both in one instruction, each rounded as the scalar one)
typedef unsigned long long f2;
__device__ __forceinline__ f2 f2_make(float lo, float hi)
{
    f2 r;
    asm("mov.b64 %0, {%1, %2};" : "=l"(r) : "f"(lo), "f"(hi));
    return r;
}
__device__ __forceinline__ void f2_get(f2 v, float& lo, float& hi)
{
    asm("mov.b64 {%0, %1}, %2;" : "=f"(lo), "=f"(hi) : "l"(v));
}
__device__ __forceinline__ f2 f2_add(f2 a, f2 b)
{
    f2 r;
    asm("add.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_mul(f2 a, f2 b)
{
    f2 r;
    asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}
__device__ __forceinline__ f2 f2_fma(f2 a, f2 b, f2 c)
{
    f2 r;
    asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(r) : "l"(a), "l"(b), "l"(c));
    return r;
}
__device__ __forceinline__ f2 f2_both(float v) { return f2_make(v, v); }
// rint(x) of both for |x| < 2^22 by the 1.5 2^23 shift (two FP32 additions
// instead of a rounding instruction); ties go to even like rintf
__device__ __forceinline__ f2 f2_rint(f2 x)
{
    return f2_add(f2_add(x, f2_both(12582912.f)), f2_both(-12582912.f));
}

__device__ __forceinline__ f2 f2_add_rd(f2 a, f2 b)   // both rounded down
{
    f2 r;
    asm("add.rm.f32x2 %0, %1, %2;" : "=l"(r) : "l"(a), "l"(b));
    return r;
}

constexpr int kVcSegment = 64;    // tile particles between two emptyings of the histograms
constexpr int kVcListed = 1024;   // listed pairs held in shared memory per segment
constexpr int kVcCountBit = 19;   // histogram word A: 7 low bits of the product (sum below 2^19), count from here

// Block (I, J0): particles i = 512 I + tid and 512 I + 256 + tid against the
// c' tiles J0 .. J0 + chunk - 1 (256 particles each).
__global__ void __launch_bounds__(kVcTile) k_vc_pairs(VcConst C, const float4* __restrict__ p4,
                                                        const float4* __restrict__ u4, const int2* __restrict__ tiles,
                                                        const double* __restrict__ scal,
                                                        unsigned long long* __restrict__ gsum,
                                                        unsigned long long* __restrict__ gcnt,
                                                        int2* __restrict__ band, unsigned int* __restrict__ band_n,
                                                        unsigned int band_cap)
{
    extern __shared__ float4 vc_smem[];
    // the c' tile with every value twice, as the packed operations take it:
    // (-x, -x, -y, -y), (-z, -z, u_x, u_x), (u_y, u_y, u_z, u_z)
    float4* sp = vc_smem;
    const ulonglong2* spd = reinterpret_cast<const ulonglong2*>(sp);
    unsigned int* listed = reinterpret_cast<unsigned int*>(sp + 3 * kVcTile);   // [kVcListed] local codes of listed pairs
    // per-warp histograms of a segment, two 32-bit words per bin: a warp adds at
    // most 64 x 64 = 2^12 pairs to a bin, so word A holds the count above its 7
    // low bits' sum and word B (16 bits a pair) stays below 2^28
    unsigned int* hist = listed + kVcListed;   // [2][warps][nbins]
    __shared__ unsigned int nlisted, list_at;
    const int tid = threadIdx.x, warp = tid >> 5;
    const int hb = kVcWarps * C.nbins;     // words A, then words B
    for (int k = tid; k < 2 * hb; k += kVcTile) hist[k] = 0u;
    if (tid == 0) nlisted = 0u;
    const int2 tb = tiles[blockIdx.x];
    const int I = tb.x, J0 = tb.y, J1 = min(C.ntile - 1, J0 + C.chunk - 1);
    const int i0 = I * 2 * kVcTile + tid, i1 = i0 + kVcTile;
    // a particle past n has NaN coordinates: every comparison of its pairs is
    // false, so they are neither counted nor listed
    const float nan = __int_as_float(0x7fffffff);
    const float4 n4 = make_float4(nan, nan, nan, 0.f), z4 = make_float4(0.f, 0.f, 0.f, 0.f);
    const float4 pi0 = i0 < C.n ? p4[i0] : n4, ui0 = i0 < C.n ? u4[i0] : z4;
    const float4 pi1 = i1 < C.n ? p4[i1] : n4, ui1 = i1 < C.n ? u4[i1] : z4;
    const f2 X = f2_make(pi0.x, pi1.x), Y = f2_make(pi0.y, pi1.y), Z = f2_make(pi0.z, pi1.z);
    const f2 UX = f2_make(ui0.x, ui1.x), UY = f2_make(ui0.y, ui1.y), UZ = f2_make(ui0.z, ui1.z);
    const float S = (float)scal[1];
    unsigned int* hw = hist + warp * C.nbins;
    constexpr int kOwn = kVcMaxBins / kVcTile;   // bins this thread keeps across segments
    long long sum[kOwn];
    unsigned long long cnt[kOwn];
#pragma unroll
    for (int u = 0; u < kOwn; ++u) sum[u] = 0, cnt[u] = 0ull;
    const f2 nLx = f2_both(-C.Lf[0]), nLy = f2_both(-C.Lf[1]), nLz = f2_both(-C.Lf[2]), nDf = f2_both(-C.df);
    const f2 iLx = f2_both(C.iLf[0]), iLy = f2_both(C.iLf[1]), iLz = f2_both(C.iLf[2]);
    const f2 S2 = f2_both(S), magic = f2_both(12582912.f), inv2 = f2_both(C.inv_f), p23 = f2_both(8388608.f);
    const f2 m23 = f2_both(-8388608.f), neg1 = f2_both(-1.f);
    const float hx = C.half[0], hy = C.half[1], hz = C.half[2], one_eb = 1.f - C.eb;
    // a rare pair (a few per thousand) to the segment's list, or straight to the global one
    auto list = [&](unsigned int code, int i, int j) {
        const unsigned int at = atomicAdd(&nlisted, 1u);
        if (at < kVcListed) {
            listed[at] = code;
        } else {
            const unsigned int idx = atomicAdd(band_n, 1u);
            if (idx < band_cap) band[idx] = make_int2(i, j);
        }
    };
    auto segment = [&](auto diag, int J, int b, int e) {
        for (int jj = b; jj < e; ++jj) {
            const int j = J * kVcTile + jj;
            const ulonglong2 ja = spd[jj], jb = spd[kVcTile + jj], jc = spd[2 * kVcTile + jj];
            f2 dx = f2_add(X, ja.x), dy = f2_add(Y, ja.y), dz = f2_add(Z, jb.x);
            const f2 ny = f2_rint(f2_mul(dy, iLy));
            dy = f2_fma(ny, nLy, dy);
            dx = f2_fma(ny, nDf, dx);
            dx = f2_fma(f2_rint(f2_mul(dx, iLx)), nLx, dx);
            dz = f2_fma(f2_rint(f2_mul(dz, iLz)), nLz, dz);
            const f2 r2 = f2_fma(dx, dx, f2_fma(dy, dy, f2_mul(dz, dz)));
            const f2 q = f2_fma(f2_fma(UX, jb.y, f2_fma(UY, jc.x, f2_mul(UZ, jc.y))), S2, magic);
            float ax, ay, az, ar, aq, bx, by, bz, br, bq, as, bs;
            f2_get(dx, ax, bx);
            f2_get(dy, ay, by);
            f2_get(dz, az, bz);
            f2_get(r2, ar, br);
            f2_get(q, aq, bq);
            // |R| from the reciprocal square root (within 3 ulp; the bands allow for it),
            // its bin position t, 2^23 + floor(t) (0 <= t < 2^23) and t's fraction (exact)
            asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(as) : "f"(fmaxf(ar, 1e-30f)));
            asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(bs) : "f"(fmaxf(br, 1e-30f)));
            const f2 r = f2_mul(r2, f2_make(as, bs)), t = f2_mul(r, inv2);
            const f2 tk = f2_add_rd(t, p23), fr = f2_fma(f2_add(tk, m23), neg1, t);
            float ra, rb, ta, tb2, fa, fb;
            f2_get(r, ra, rb);
            f2_get(tk, ta, tb2);
            f2_get(fr, fa, fb);
            // an image index taken within the FP32 error of a tie leaves that component
            // within the same error of half the box edge
            const bool in_a = !decltype(diag)::value || j > i0, in_b = !decltype(diag)::value || j > i1;
            const bool tie_a = fabsf(ax) > hx || fabsf(ay) > hy || fabsf(az) > hz;
            const bool tie_b = fabsf(bx) > hx || fabsf(by) > hy || fabsf(bz) > hz;
            const bool near_a = ra > C.r_band || fa < C.eb || fa > one_eb;
            const bool near_b = rb > C.r_band || fb < C.eb || fb > one_eb;
            const bool cut_a = ar < C.r2_hi, cut_b = br < C.r2_hi;
            // m = round(dot S) + 2^22 (|dot S| < 2^21): its low 7 bits and a count of 1
            // in word A, its high 16 bits in word B
            if (in_a && !tie_a && cut_a && !near_a) {
                unsigned int* h = hw + (__float_as_int(ta) - 0x4B000000);
                atomicAdd(h, (__float_as_uint(aq) & 127u) | (1u << kVcCountBit));
                atomicAdd(h + hb, (__float_as_uint(aq) >> 7) & 0xffffu);
            }
            if (in_b && !tie_b && cut_b && !near_b) {
                unsigned int* h = hw + (__float_as_int(tb2) - 0x4B000000);
                atomicAdd(h, (__float_as_uint(bq) & 127u) | (1u << kVcCountBit));
                atomicAdd(h + hb, (__float_as_uint(bq) >> 7) & 0xffffu);
            }
            const bool push_a = in_a && (tie_a || (cut_a && near_a)), push_b = in_b && (tie_b || (cut_b && near_b));
            if (push_a || push_b) {
                const unsigned int code = (unsigned int)tid | ((unsigned int)jj << 9);
                if (push_a) list(code, i0, j);
                if (push_b) list(code | kVcTile, i1, j);
            }
        }
    };
    for (int J = J0; J <= J1; ++J) {
        const int jt = J * kVcTile + tid;
        __syncthreads();   // the histograms are zeroed; the previous tile is no longer read
        if (jt < C.n) {
            const float4 p = p4[jt], u = u4[jt];
            sp[tid] = make_float4(-p.x, -p.x, -p.y, -p.y);
            sp[kVcTile + tid] = make_float4(-p.z, -p.z, u.x, u.x);
            sp[2 * kVcTile + tid] = make_float4(u.y, u.y, u.z, u.z);
        }
        __syncthreads();
        const int jn = min(kVcTile, C.n - J * kVcTile);
        for (int b = 0; b < jn; b += kVcSegment) {
            const int e = min(b + kVcSegment, jn);
            if (J <= 2 * I + 1)
                segment(std::true_type{}, J, b, e);
            else
                segment(std::false_type{}, J, b, e);
            __syncthreads();
            const unsigned int nl = min(nlisted, (unsigned int)kVcListed);
            if (tid == 0 && nl > 0u) list_at = atomicAdd(band_n, nl);
#pragma unroll
            for (int u = 0; u < kOwn; ++u) {   // empty the histograms into the owning threads' registers
                const int k = tid + u * kVcTile;
                if (k < C.nbins) {
                    unsigned int lo = 0u, c = 0u, hi = 0u;   // 8 warps: below 2^22, 2^16 and 2^31
#pragma unroll
                    for (int w = 0; w < kVcWarps; ++w) {
                        const unsigned int a = hist[w * C.nbins + k];
                        hi += hist[hb + w * C.nbins + k];
                        lo += a & ((1u << kVcCountBit) - 1u);
                        c += a >> kVcCountBit;
                        hist[w * C.nbins + k] = 0u;
                        hist[hb + w * C.nbins + k] = 0u;
                    }
                    sum[u] += (long long)lo + ((long long)hi << 7) - ((long long)c << 22);
                    cnt[u] += c;
                }
            }
            __syncthreads();
            for (unsigned int k = tid; k < nl; k += kVcTile) {
                const unsigned int v = listed[k];
                if (list_at + k < band_cap)
                    band[list_at + k] = make_int2(I * 2 * kVcTile + (int)(v & 511u), J * kVcTile + (int)(v >> 9));
            }
            __syncthreads();
            if (tid == 0) nlisted = 0u;
            __syncthreads();
        }
    }
#pragma unroll
    for (int u = 0; u < kOwn; ++u) {
        const int k = tid + u * kVcTile;
        if (k < C.nbins && cnt[u]) {
            atomicAdd(gsum + k, (unsigned long long)sum[u]);
            atomicAdd(gcnt + k, cnt[u]);
        }
    }
}

// round(a / L) as the definition computes it (quotient rounded to FP64, then
// rounded half away from zero), with the division taken only where the
// product by 1/L (within 2^-50 of the quotient for |a / L| < 2) lies near a
// half-integer.
__device__ __forceinline__ double round_quotient(double a, double L, double invL)
{
    const double q = __dmul_rn(a, invL);
    const double f = fabs(q - trunc(q));
    return fabs(f - 0.5) < 0x1p-46 ? round(__ddiv_rn(a, L)) : round(q);
}

// round(a / L) for |a| < L (the quotient rounds to 1/2 or more exactly when a
// >= L / 2: the next double below L / 2 has a quotient of at most 1/2 - 2^-54):
// two comparisons instead of a product, a truncation and a rounding
__device__ __forceinline__ double round_near(double a, double halfL)
{
    return a >= halfL ? 1.0 : (a <= -halfL ? -1.0 : 0.0);
}

// The Lees-Edwards minimum image with every operation of the definition
// (the same results as min_image(); a product by 0 or +-1 is exact and its
// subtraction of 0 changes nothing).
__device__ __forceinline__ void vc_min_image(const KParams& P, const VcConst& C, double xi, double yi, double zi,
                                             double xj, double yj, double zj, double& dx, double& dy, double& dz)
{
    dx = __dsub_rn(xi, xj);
    dy = __dsub_rn(yi, yj);
    dz = __dsub_rn(zi, zj);
    const double n = round_near(dy, 0.5 * P.L[1]), c = round_near(dz, 0.5 * P.L[2]);
    if (n != 0.0) {
        dy = __dsub_rn(dy, n > 0.0 ? P.L[1] : -P.L[1]);
        dx = __dsub_rn(dx, n > 0.0 ? C.delta : -C.delta);
    }
    const double a = fabs(dx) < P.L[0] ? round_near(dx, 0.5 * P.L[0]) : round_quotient(dx, P.L[0], C.invL[0]);
    if (a != 0.0) dx = __dsub_rn(dx, __dmul_rn(P.L[0], a));
    if (c != 0.0) dz = __dsub_rn(dz, c > 0.0 ? P.L[2] : -P.L[2]);
}

// The listed pairs with the FP64 operations of the definition (the minimum
// image rounded exactly as written, |R|^2 < rmax^2, floor(sqrt(|R|^2) nbins /
// rmax)); products in FP64, rounded to the same fixed point.
__global__ void k_vc_band(VcConst C, KParams P, const double* __restrict__ pos, const double* __restrict__ v,
                          const int2* __restrict__ band, const unsigned int* __restrict__ band_n,
                          unsigned int band_cap, const double* __restrict__ scal,
                          unsigned long long* __restrict__ gsum, unsigned long long* __restrict__ gcnt)
{
    const unsigned int m = min(*band_n, band_cap);
    const double S = scal[1];
    for (unsigned int t = blockIdx.x * blockDim.x + threadIdx.x; t < m; t += gridDim.x * blockDim.x) {
        const int2 pr = band[t];
        const int i = pr.x, j = pr.y;
        double dx, dy, dz;
        vc_min_image(P, C, pos[3 * i], pos[3 * i + 1], pos[3 * i + 2], pos[3 * j], pos[3 * j + 1], pos[3 * j + 2],
                     dx, dy, dz);
        const double r2 = sq_norm_exact(dx, dy, dz);
        if (!(r2 < C.rmax2)) continue;
        long long k = (long long)floor(__dmul_rn(__dsqrt_rn(r2), C.inv));
        if (k > C.nbins - 1) k = C.nbins - 1;
        const double yi = pos[3 * i + 1], yj = pos[3 * j + 1];
        const double uxi = v[3 * i] - C.kappa * (yi - 0.5 * P.L[1]);
        const double uxj = v[3 * j] - C.kappa * (yj - 0.5 * P.L[1]);
        const double dot = uxi * uxj + v[3 * i + 1] * v[3 * j + 1] + v[3 * i + 2] * v[3 * j + 2];
        atomicAdd(gsum + k, (unsigned long long)llrint(dot * S));
        atomicAdd(gcnt + k, 1ull);
    }
}

size_t pairs_smem(int nbins)
{
    return sizeof(float4) * 3 * kVcTile + sizeof(unsigned int) * (kVcListed + 2 * kVcWarps * nbins);
}

template <class T>
cudaError_t vc_alloc(T** p, long long count)
{
    cudaFree(*p);
    *p = nullptr;
    return cudaMalloc(p, sizeof(T) * (size_t)count);
}

}  // namespace

void vc_free(VcBuffers& V)
{
    void* ptrs[] = {V.fixed, V.rows, V.band_own, V.tiles};
    for (void* q : ptrs) cudaFree(q);
    if (V.ev[0]) cudaEventDestroy(V.ev[0]);
    if (V.ev[1]) cudaEventDestroy(V.ev[1]);
    V = VcBuffers{};
}

// Buffers for n particles (kept and reused while n does not grow): one
// allocation for the fixed-size part and one for the rows (an allocation and
// its release cost ~10 us each, and the call from host arrays makes all anew).
cudaError_t vc_reserve(VcBuffers& V, long long n)
{
    cudaError_t e = cudaSuccess;
    auto T = [&](cudaError_t r) { if (e == cudaSuccess) e = r; };
    if (!V.fixed) {
        // initial capacity of the boundary-pair list (grown on demand; a small
        // value set through the environment exercises the growth)
        long long bc = 1 << 20;
        if (const char* env = getenv("SHEARSIM_VCORR_BAND_CAP")) bc = std::max(1ll, atoll(env));
        constexpr size_t words = 2 * kVcMaxBins + kVcPrepBlocks + 2 + 2;   // sum, cnt, part, scal, misc (8 bytes each)
        T(vc_alloc(&V.fixed, (long long)words + bc));
        if (e == cudaSuccess) {
            V.sum = V.fixed;
            V.cnt = V.sum + kVcMaxBins;
            V.part = reinterpret_cast<double*>(V.cnt + kVcMaxBins);
            V.scal = V.part + kVcPrepBlocks;
            V.misc = reinterpret_cast<unsigned int*>(V.scal + 2);
            V.band = reinterpret_cast<int2*>(V.fixed + words);
            V.band_cap = bc;
        }
        T(cudaEventCreate(&V.ev[0]));
        T(cudaEventCreate(&V.ev[1]));
        if (e != cudaSuccess) {
            vc_free(V);
            return e;
        }
    }
    if (n > V.n_cap) {
        V.n_cap = 0;
        T(vc_alloc(&V.rows, 5 * n));   // p4, u4 (16 bytes a row), pos_n3, v_n3 (24)
        if (e == cudaSuccess) {
            V.p4 = V.rows;
            V.u4 = V.p4 + n;
            V.pos_n3 = reinterpret_cast<double*>(V.u4 + n);
            V.v_n3 = V.pos_n3 + 3 * n;
            V.n_cap = n;
        }
    }
    return e;
}

int run_velocity_correlation(VcBuffers& V, long long n, const double L[3], double delta, double kappa, int nbins,
                             double rmax, cudaStream_t s, double* sum_host, long long* cnt_host, double* vsq_host,
                             VcStats* stats, const char** err)
{
    if (n < 1 || n > (1ll << 30) || nbins < 1 || nbins > kVcMaxBins || !(rmax > 0.0) || !std::isfinite(rmax) ||
        !(delta >= 0.0) || !(delta < L[0]) || !std::isfinite(kappa)) {
        if (err) *err = "velocity correlation: needs n >= 1, 1 <= nbins <= 1024, rmax > 0, 0 <= delta < L_x";
        return SP_ERR_INVALID_ARG;
    }
    for (int a = 0; a < 3; ++a)
        if (!(L[a] > 0.0) || !std::isfinite(L[a])) {
            if (err) *err = "velocity correlation: box edges must be positive";
            return SP_ERR_INVALID_ARG;
        }
    if (vc_reserve(V, n) != cudaSuccess) {
        cudaGetLastError();
        return SP_ERR_OOM;
    }
    static bool attr_set = false;
    if (!attr_set) {
        if (cudaFuncSetAttribute(k_vc_pairs, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)pairs_smem(kVcMaxBins)) !=
            cudaSuccess)
            return SP_ERR_CUDA;
        attr_set = true;
    }

    VcConst C{};
    C.n = (int)n;
    C.nbins = nbins;
    C.ntile = (int)((n + kVcTile - 1) / kVcTile);
    C.chunk = C.ntile <= 128 ? 1 : (C.ntile <= 256 ? 4 : 16);
    for (int a = 0; a < 3; ++a) {
        C.Lf[a] = (float)L[a];
        C.iLf[a] = (float)(1.0 / L[a]);
    }
    C.df = (float)delta;
    // E bounds |r_FP32 - r| for positions in [0, L): each FP32 operation rounds
    // by at most 2^-24 of a result no larger than 2 L_x (x), L_y, L_z, plus the
    // relative roundings of the squares, the approximate square root (3 ulp)
    // and the scaling.
    const double u = 5.9604644775390625e-8;
    const double E = u * (20.0 * (L[0] + L[1] + L[2]) + 16.0 * rmax);
    C.r2_hi = nextafterf((float)((rmax + 2.0 * E) * (rmax + 2.0 * E)), INFINITY);
    C.r_band = nextafterf((float)(rmax - 2.0 * E), -INFINITY);
    C.inv = (double)nbins / rmax;
    C.inv_f = (float)C.inv;
    C.eb = (float)std::min(0.5, 2.0 * E * C.inv + 8.0 * u * nbins + 4.0 * u);
    for (int a = 0; a < 3; ++a) {
        C.half[a] = (float)(L[a] * (0.5 - 64.0 * u));
        C.invL[a] = 1.0 / L[a];
    }
    C.delta = delta;
    C.kappa = kappa;
    C.rmax2 = rmax * rmax;

    KParams P{};
    P.L[0] = L[0];
    P.L[1] = L[1];
    P.L[2] = L[2];

    // blocks (I, first J of a run of `chunk` c' tiles): I covers particles
    // [512 I, 512 I + 512), so the tiles below 2 I hold no partner j > i
    std::vector<int2> tl;
    const int ni = (int)((n + 2 * kVcTile - 1) / (2 * kVcTile));
    for (int I = 0; I < ni; ++I)
        for (int J = 2 * I; J < C.ntile; J += C.chunk) tl.push_back(make_int2(I, J));
    if ((long long)tl.size() > V.tiles_cap) {
        V.tiles_cap = 0;
        V.tiles_n = 0;
        if (vc_alloc(&V.tiles, (long long)tl.size()) != cudaSuccess) {
            cudaGetLastError();
            return SP_ERR_OOM;
        }
        V.tiles_cap = (long long)tl.size();
    }
    if (V.tiles_n != (long long)tl.size() || V.tiles_for != n) {
        if (cudaMemcpyAsync(V.tiles, tl.data(), sizeof(int2) * tl.size(), cudaMemcpyHostToDevice, s) != cudaSuccess)
            return SP_ERR_CUDA;
        if (cudaStreamSynchronize(s) != cudaSuccess) return SP_ERR_CUDA;
        V.tiles_n = (long long)tl.size();
        V.tiles_for = n;
    }

    const int prep_blocks = (int)std::min<long long>(kVcPrepBlocks, (n + kVcTile - 1) / kVcTile);
    unsigned int* band_n = reinterpret_cast<unsigned int*>(V.misc);
    unsigned int* umax = band_n + 1;
    int* flag = reinterpret_cast<int*>(band_n + 2);
    std::vector<unsigned long long> hs(nbins), hc(nbins);
    unsigned int misc_h[4];
    double scal_h[2];
    for (int attempt = 0; attempt < 2; ++attempt) {
        const unsigned int cap = (unsigned int)std::min<long long>(V.band_cap, 0xffffffffll);
        if (cudaMemsetAsync(V.sum, 0, sizeof(unsigned long long) * nbins, s) != cudaSuccess ||
            cudaMemsetAsync(V.cnt, 0, sizeof(unsigned long long) * nbins, s) != cudaSuccess ||
            cudaMemsetAsync(V.misc, 0, sizeof(unsigned int) * 4, s) != cudaSuccess)
            return SP_ERR_CUDA;
        k_vc_prep<<<prep_blocks, kVcTile, 0, s>>>(C, P, V.pos_n3, V.v_n3, V.p4, V.u4, V.part, umax, flag);
        k_vc_scale<<<1, 32, 0, s>>>(C.n, prep_blocks, V.part, umax, V.scal);
        cudaEventRecord(V.ev[0], s);
        k_vc_pairs<<<(unsigned)tl.size(), kVcTile, pairs_smem(nbins), s>>>(C, V.p4, V.u4, V.tiles, V.scal, V.sum,
                                                                          V.cnt, V.band, band_n, cap);
        cudaEventRecord(V.ev[1], s);
        k_vc_band<<<4 * 152, 256, 0, s>>>(C, P, V.pos_n3, V.v_n3, V.band, band_n, cap, V.scal, V.sum, V.cnt);
        if (cudaGetLastError() != cudaSuccess) return SP_ERR_CUDA;
        if (cudaMemcpyAsync(hs.data(), V.sum, sizeof(unsigned long long) * nbins, cudaMemcpyDeviceToHost, s) !=
                cudaSuccess ||
            cudaMemcpyAsync(hc.data(), V.cnt, sizeof(unsigned long long) * nbins, cudaMemcpyDeviceToHost, s) !=
                cudaSuccess ||
            cudaMemcpyAsync(misc_h, V.misc, sizeof(misc_h), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaMemcpyAsync(scal_h, V.scal, sizeof(scal_h), cudaMemcpyDeviceToHost, s) != cudaSuccess ||
            cudaStreamSynchronize(s) != cudaSuccess)
            return SP_ERR_CUDA;
        const int bad = (int)misc_h[2];
        if (bad) {
            if (err) *err = "velocity correlation: positions must lie in [0, L) on every axis";
            return SP_ERR_INVALID_ARG;
        }
        if (misc_h[0] <= cap) break;
        // more pairs near a boundary than the list holds: grow it and run again
        const long long want = (long long)misc_h[0] + (misc_h[0] >> 2) + 1024;
        V.band_cap = 0;
        if (attempt == 1 || vc_alloc(&V.band_own, want) != cudaSuccess) {
            cudaGetLastError();
            if (err) *err = "velocity correlation: boundary pair list overflow";
            return SP_ERR_OOM;
        }
        V.band = V.band_own;
        V.band_cap = want;
    }
    const double S = scal_h[1];
    for (int k = 0; k < nbins; ++k) {
        if (sum_host) sum_host[k] = (double)(long long)hs[k] / S;
        if (cnt_host) cnt_host[k] = (long long)hc[k];
    }
    if (vsq_host) *vsq_host = scal_h[0];
    if (stats) {
        float ms = 0.f;
        cudaEventElapsedTime(&ms, V.ev[0], V.ev[1]);
        stats->pairs_ms = ms;
        stats->band_pairs = misc_h[0];
        stats->blocks = (long long)tl.size();
    }
    return SP_OK;
}

}  // namespace ss
