// Site coordinates and neighbour offsets of a periodic lattice for kernels
// that walk the sites in memory order.
#pragma once

#include "kernels.h"
#include "su3.cuh"

namespace lqcd {
namespace {

// Site coordinates and neighbour indices in type I: int whenever the site
// loops fit (2 V + a block below 2^31), so that the divisions of the site
// index and the neighbour offsets take 32-bit arithmetic (a 64-bit division
// is a long software sequence); the 16-byte lane addresses stay 64-bit.
// Measured at 32^3x64 FP32: hopping operator 0.176 -> 0.168 ms, force 0.281
// -> 0.246 ms (32-bit lane addresses as well were slower: 0.171, 0.289).
template <typename I> struct Sites {
    int L0, L1, L2, L3;
    I s1, s2, s3, V;
};

template <typename I> __device__ __forceinline__ Sites<I> make_sites(const int dims[4])
{
    Sites<I> g;
    g.L0 = dims[0];
    g.L1 = dims[1];
    g.L2 = dims[2];
    g.L3 = dims[3];
    g.s1 = dims[0];
    g.s2 = g.s1 * dims[1];
    g.s3 = g.s2 * dims[2];
    g.V = g.s3 * dims[3];
    return g;
}

// Coordinates of site n < 2^31 with the strides' division magic (three
// multiply-highs instead of three divisions by run-time values: hopping
// force 0.242 -> 0.234 ms at 32^3x64 FP32).
__device__ __forceinline__ Coord coord_fast(const Sites<int> &g, const DivMagic div[3], int n)
{
    Coord x;
    x.c3 = (int)div_by((unsigned)n, div[2]);
    int r = n - x.c3 * g.s3;
    x.c2 = (int)div_by((unsigned)r, div[1]);
    r -= x.c2 * g.s2;
    x.c1 = (int)div_by((unsigned)r, div[0]);
    x.c0 = r - x.c1 * g.s1;
    return x;
}

template <typename I> __device__ __forceinline__ Coord coord_in(const Sites<I> &g, I n)
{
    Coord x;
    x.c3 = (int)(n / g.s3);
    I r = n - x.c3 * g.s3;
    x.c2 = (int)(r / g.s2);
    r -= x.c2 * g.s2;
    x.c1 = (int)(r / g.s1);
    x.c0 = (int)(r - x.c1 * g.s1);
    return x;
}

// Index offset of the step s * hat(mu) (s = +-1), periodic.
template <typename I>
__device__ __forceinline__ I hop_offset(const Sites<I> &g, const Coord &x, int mu, int s)
{
    const int L = pick(mu, g.L0, g.L1, g.L2, g.L3);
    const int c = pick(mu, x.c0, x.c1, x.c2, x.c3);
    const I st = mu == 0 ? I(1) : (mu == 1 ? g.s1 : (mu == 2 ? g.s2 : g.s3));
    if (s > 0) return c + 1 == L ? (I)(1 - L) * st : st;
    return c == 0 ? (I)(L - 1) * st : -st;
}

// One step up along mu on coordinates.
template <typename I> __device__ __forceinline__ void step_up(const Sites<I> &g, Coord &x, int mu)
{
    if (mu == 0) x.c0 = x.c0 + 1 == g.L0 ? 0 : x.c0 + 1;
    else if (mu == 1) x.c1 = x.c1 + 1 == g.L1 ? 0 : x.c1 + 1;
    else if (mu == 2) x.c2 = x.c2 + 1 == g.L2 ? 0 : x.c2 + 1;
    else x.c3 = x.c3 + 1 == g.L3 ? 0 : x.c3 + 1;
}

// Site loops in int: n + grid stride stays below 2 V + a block.
inline bool sites_fit_int(int64_t V) { return 2 * V + 1024 < ((int64_t)1 << 31); }

// The magic of the strides L0, L0 L1, L0 L1 L2 (1 where they do not fit).
inline void stride_magic(const int dims[4], DivMagic div[3])
{
    int64_t s = 1;
    for (int i = 0; i < 3; ++i) {
        s *= dims[i];
        div[i] = div_magic(s < ((int64_t)1 << 31) ? (unsigned)s : 1u);
    }
}

} // namespace
} // namespace lqcd
