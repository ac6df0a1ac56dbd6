// Fixed-point arithmetic for FP64 fields of SU(3) matrices.
//
// GB300 issues 2 FP64 FMAs per clock and SM but 64 integer multiply-adds of
// 32 x 32 + 64 bits (measured: 1.7 and 63.4).  The entries of an SU(3) matrix
// are at most 1 in modulus, so instead of a floating point they can have a
// fixed one: a real x is the 59-bit integer x 2^58 in two signed limbs,
// x 2^58 = h 2^29 + l with -2^28 <= l < 2^28, and a product is
//     x y 2^58 = h h' + (h l' + l h') 2^-29 + l l' 2^-58,
// three multiply-adds into two 64-bit accumulators (the last term, below
// 2^-60, is left out): 21 real FMAs per clock and SM against 2.  Rounding is
// by half a unit of 2^-58, 1.7e-18, where an FP64 result of that size rounds
// by up to 5.5e-17, so sums of products come out more exact than in FP64.
// Sums that pass 1 are kept in coarser units (2^-56 up to 8, 2^-53 up to 64),
// the unit being fixed by the place in the formula.
//
// Overflow: entries of a product of matrices that are unitary to about 1e-3
// are bounded by 1 + 1e-2 through every partial sum (Cauchy-Schwarz), the
// mixed terms of one product by sqrt(6) 2^58; up to six products share one
// pair of accumulators (below 2^62).  Links that are not within 1e-3 of SU(3)
// or not finite are marked (kPoison) and take the floating-point path.
#pragma once

#include "su3.cuh"

namespace lqcd {

constexpr int kLimb = 29;        // bits of the low limb
constexpr int kUnit = 2 * kLimb; // entries in units of 2^-58

// h of entry (0, 0) of a matrix that has no fixed-point form.
constexpr int kPoison = (int)0x80000000;

struct FMat {
    int rh[3][3], rl[3][3], ih[3][3], il[3][3];
};

// High and mixed sums of a matrix of products.
struct FAcc {
    long long rh[3][3], rl[3][3], ih[3][3], il[3][3];
};

// A matrix of whole numbers (in the units of its place).
struct FInt {
    long long re[3][3], im[3][3];
};

__device__ __forceinline__ void fx_zero(FAcc &y)
{
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) y.rh[i][j] = y.rl[i][j] = y.ih[i][j] = y.il[i][j] = 0;
}

// One real product into a pair of sums.
__device__ __forceinline__ void fx_mad(long long &h, long long &l, int ah, int al, int bh, int bl)
{
    h += (long long)ah * bh;
    l += (long long)ah * bl;
    l += (long long)al * bh;
}

// y += op_a(a) op_b(b), rows 0..ROWS-1.
template <int FA, int FB, int ROWS = 3>
__device__ __forceinline__ void fx_mul_acc(FAcc &y, const FMat &a, const FMat &b)
{
    constexpr int SA = FA == N ? 1 : -1, SB = FB == N ? 1 : -1; // signs of the imaginary parts
#pragma unroll
    for (int i = 0; i < ROWS; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            const int ai = FA == N ? i : k, ak = FA == N ? k : i;
            const int arh = a.rh[ai][ak], arl = a.rl[ai][ak], aih = a.ih[ai][ak], ail = a.il[ai][ak];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int bi = FB == N ? k : j, bk = FB == N ? j : k;
                const int brh = b.rh[bi][bk], brl = b.rl[bi][bk];
                const int bih = b.ih[bi][bk], bil = b.il[bi][bk];
                fx_mad(y.rh[i][j], y.rl[i][j], arh, arl, brh, brl);
                fx_mad(y.rh[i][j], y.rl[i][j], SA * SB > 0 ? -aih : aih, SA * SB > 0 ? -ail : ail, bih, bil);
                fx_mad(y.ih[i][j], y.il[i][j], SB > 0 ? arh : -arh, SB > 0 ? arl : -arl, bih, bil);
                fx_mad(y.ih[i][j], y.il[i][j], SA > 0 ? aih : -aih, SA > 0 ? ail : -ail, brh, brl);
            }
        }
}

// The value of a pair of sums, in the unit of the high one.
__device__ __forceinline__ long long fx_value(long long h, long long l)
{
    return h + ((l + (1ll << (kLimb - 1))) >> kLimb);
}

// v 2^-SH as two limbs.
template <int SH> __device__ __forceinline__ void fx_split(long long v, int &h, int &l)
{
    if constexpr (SH > 0) v = (v + (1ll << (SH - 1))) >> SH;
    h = (int)((v + (1ll << (kLimb - 1))) >> kLimb);
    l = (int)((unsigned)v - ((unsigned)h << kLimb));
}

// The sums as limbs, in units 2^SH times coarser; rows 0..ROWS-1.
template <int SH, int ROWS = 3> __device__ __forceinline__ FMat fx_round(const FAcc &y)
{
    FMat m;
#pragma unroll
    for (int i = 0; i < ROWS; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            fx_split<SH>(fx_value(y.rh[i][j], y.rl[i][j]), m.rh[i][j], m.rl[i][j]);
            fx_split<SH>(fx_value(y.ih[i][j], y.il[i][j]), m.ih[i][j], m.il[i][j]);
        }
    return m;
}

template <int SH> __device__ __forceinline__ FMat fx_round(const FInt &y)
{
    FMat m;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            fx_split<SH>(y.re[i][j], m.rh[i][j], m.rl[i][j]);
            fx_split<SH>(y.im[i][j], m.ih[i][j], m.il[i][j]);
        }
    return m;
}

// Row 2 of an SU(3) matrix from rows 0 and 1: row2 = conj(row0 x row1).
__device__ __forceinline__ void fx_row2(FMat &u)
{
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int k = (j + 1) % 3, l = (j + 2) % 3;
        long long rh = 0, rl = 0, ih = 0, il = 0;
        fx_mad(rh, rl, u.rh[0][k], u.rl[0][k], u.rh[1][l], u.rl[1][l]);
        fx_mad(rh, rl, -u.ih[0][k], -u.il[0][k], u.ih[1][l], u.il[1][l]);
        fx_mad(rh, rl, -u.rh[0][l], -u.rl[0][l], u.rh[1][k], u.rl[1][k]);
        fx_mad(rh, rl, u.ih[0][l], u.il[0][l], u.ih[1][k], u.il[1][k]);
        fx_mad(ih, il, -u.rh[0][k], -u.rl[0][k], u.ih[1][l], u.il[1][l]);
        fx_mad(ih, il, -u.ih[0][k], -u.il[0][k], u.rh[1][l], u.rl[1][l]);
        fx_mad(ih, il, u.rh[0][l], u.rl[0][l], u.ih[1][k], u.il[1][k]);
        fx_mad(ih, il, u.ih[0][l], u.il[0][l], u.rh[1][k], u.rl[1][k]);
        fx_split<0>(fx_value(rh, rl), u.rh[2][j], u.rl[2][j]);
        fx_split<0>(fx_value(ih, il), u.ih[2][j], u.il[2][j]);
    }
}

// A real scalar of modulus at most 1.
struct FScalar {
    int h, l;
};

inline FScalar fx_scalar(double c)
{
    const long long v = (long long)(c * 288230376151711744.0 + (c < 0 ? -0.5 : 0.5)); // 2^58
    FScalar s;
    s.h = (int)((v + (1ll << (kLimb - 1))) >> kLimb);
    s.l = (int)(v - (long long)s.h * (1ll << kLimb));
    return s;
}

// c m, in the units of m.
__device__ __forceinline__ FInt fx_scaled(const FScalar c, const FMat &m)
{
    FInt r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            long long h = 0, l = 0;
            fx_mad(h, l, c.h, c.l, m.rh[i][j], m.rl[i][j]);
            r.re[i][j] = fx_value(h, l);
            h = l = 0;
            fx_mad(h, l, c.h, c.l, m.ih[i][j], m.il[i][j]);
            r.im[i][j] = fx_value(h, l);
        }
    return r;
}

// y += the sums, in their units.
__device__ __forceinline__ void fx_add(FInt &y, const FAcc &a)
{
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            y.re[i][j] += fx_value(a.rh[i][j], a.rl[i][j]);
            y.im[i][j] += fx_value(a.ih[i][j], a.il[i][j]);
        }
}

// Re tr(a b), in the units of the product.
__device__ __forceinline__ long long fx_re_trace(const FMat &a, const FMat &b)
{
    long long h = 0, l = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            fx_mad(h, l, a.rh[i][k], a.rl[i][k], b.rh[k][i], b.rl[k][i]);
            fx_mad(h, l, -a.ih[i][k], -a.il[i][k], b.ih[k][i], b.il[k][i]);
        }
    return fx_value(h, l);
}

// Rows 0 and 1 of a stored FP64 link as limbs, row 2 rebuilt; a link that is
// not finite or not within 1e-3 of SU(3) is marked.
__device__ __forceinline__ FMat fx_from_rows(const double r[12])
{
    FMat u;
    bool ok = true;
#pragma unroll
    for (int e = 0; e < 6; ++e) {
        const int i = e / 3, j = e % 3;
        const double x = r[2 * e], y = r[2 * e + 1];
        // |x| < 1.5 by its bits (false for a NaN)
        ok = ok && (unsigned)(__double2hiint(x) & 0x7fffffff) < 0x3ff80000u &&
             (unsigned)(__double2hiint(y) & 0x7fffffff) < 0x3ff80000u;
        fx_split<0>(__double2ll_rn(x * 288230376151711744.0), u.rh[i][j], u.rl[i][j]);
        fx_split<0>(__double2ll_rn(y * 288230376151711744.0), u.ih[i][j], u.il[i][j]);
    }
    float n0 = 0.f, n1 = 0.f, cr = 0.f, ci = 0.f;
    constexpr float s = 1.0f / (float)(1 << kLimb);
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float ar = s * (float)u.rh[0][j], ai = s * (float)u.ih[0][j];
        const float br = s * (float)u.rh[1][j], bi = s * (float)u.ih[1][j];
        n0 += ar * ar + ai * ai;
        n1 += br * br + bi * bi;
        cr += ar * br + ai * bi;
        ci += ar * bi - ai * br;
    }
    ok = ok && fabsf(n0 - 1.f) < 1e-3f && fabsf(n1 - 1.f) < 1e-3f && fabsf(cr) < 1e-3f && fabsf(ci) < 1e-3f;
    fx_row2(u);
    if (!ok) u.rh[0][0] = kPoison;
    return u;
}

__device__ __forceinline__ bool fx_poisoned(const FMat &m) { return m.rh[0][0] == kPoison; }

} // namespace lqcd
