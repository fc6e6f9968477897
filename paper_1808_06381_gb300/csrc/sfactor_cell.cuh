// The grid cell of a coordinate and the cloud-in-cell weights of the structure
// factor's deposit, in integers (also compiled for the host by the CPU tests).
#pragma once

#include <math.h>

#ifdef __CUDACC__
#define SS_CELL_FN __host__ __device__ __forceinline__
#else
#define SS_CELL_FN static inline
#endif

namespace ss {

constexpr double kCellUnit = 1125899906842624.0;   // 2^50 per grid cell

struct GridCell {
    int i0, i1;                  // the cell and the next one, both in [0, G)
    unsigned long long f, g;     // the distances to their points times 2^63: the weights of i1 and i0
};

// v: the coordinate in grid cells times kCellUnit.  For the coordinates of a
// particle in the box |v| < 2^13 2^50 (G <= 8192): one conversion and a shift,
// and at most one addition brings the cell into [0, G) (its fraction keeps 50
// bits; an FP64 coordinate above 8 cells has no more).  Any other value, which
// refused positions or a step longer than the box can leave behind, takes the
// remainder by G; an infinity (beyond ~1e293 cells) or a NaN goes to
// cell 0.
SS_CELL_FN GridCell grid_cell(double v, int G)
{
    constexpr long long kMask = (1ll << 50) - 1;
    GridCell c;
    long long q;
    if (v >= -9223372036854775808.0 && v < 9223372036854775808.0) {   // 2^63
#ifdef __CUDA_ARCH__
        const long long u = __double2ll_rd(v);
#else
        const long long u = (long long)floor(v);
#endif
        q = u >> 50;
        c.f = (unsigned long long)(u & kMask) << 13;
    } else {
        const double whole = floor(v * (1.0 / kCellUnit)), r = fmod(whole, (double)G);   // from 2^63 on v is whole cells
        q = r > -(double)G && r < (double)G ? (long long)r : 0;                           // false for a NaN
        c.f = 0ull;
    }
    c.g = (1ull << 63) - c.f;
    if (q < 0) q += G;
    if (q >= G) q -= G;
    if (q < 0 || q >= G) q = (q % G + G) % G;
    c.i0 = (int)q;
    c.i1 = c.i0 + 1 < G ? c.i0 + 1 : 0;
    return c;
}

// a b in units of 2^-32 (a, b in units of 2^-63), rounded to nearest
SS_CELL_FN unsigned long long cell_weight(unsigned long long a, unsigned long long b)
{
#ifdef __CUDA_ARCH__
    const unsigned long long hi = __umul64hi(a, b);
#else
    const unsigned long long hi = (unsigned long long)(((unsigned __int128)a * b) >> 64);
#endif
    return (hi + (1ull << 29)) >> 30;
}

}  // namespace ss
