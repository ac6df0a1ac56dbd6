// Fixed-point arithmetic for FP64 fields of SU(3) matrices.
//
// GB300 issues 2 FP64 FMAs per clock and SM but 64 integer multiply-adds of
// 32 x 32 + 64 bits (measured: 1.7 and 63.4).  The entries of an SU(3) matrix
// are at most 1 in modulus, so instead of a floating point they can have a
// fixed one: a real x is the 59-bit integer x 2^58 in two signed limbs,
// x 2^58 = h 2^29 + l with -2^28 <= l < 2^28, and a product is
//     x y 2^58 = h h' + (h l' + l h') 2^-29 + l l' 2^-58,
// three multiply-adds into two 64-bit accumulators (the last term, below
// 2^-60, is left out): 21 real FMAs per clock and SM against 2, and 28 with
// complex products in three real ones (FAcc).  Rounding is
// by half a unit of 2^-58, 1.7e-18, where an FP64 result of that size rounds
// by up to 5.5e-17, so sums of products come out more exact than in FP64.
// Sums that pass 1 are kept in coarser units (2^-56 up to 8, 2^-53 up to 64),
// the unit being fixed by the place in the formula.
//
// Overflow: entries of a product of matrices that are unitary to about 1e-3
// are bounded by 1 + 1e-2 through every partial sum (Cauchy-Schwarz).  The
// largest sum is the mixed one of (ar + ai)(br + bi): the high limbs of a row
// add up to sqrt(6) 2^29, the low limbs are at most 2^29, so the two terms of
// one product give at most 4.9 2^58 and six products, the most that share
// accumulators, 29.4 2^58 < 2^63.  Links that are not within 1e-3 of SU(3)
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

// Sums of a matrix of complex products a b in three real ones each (Gauss):
// 1: sum ar br, 2: sum ai bi, 3: sum (ar + ai)(br + bi), so that
// Re = 1 - 2, Im = 3 - 1 - 2; high and mixed sums of each.  In whole numbers
// the cancellation is exact, and no factor is ever negated.
struct FAcc {
    long long h1[3][3], l1[3][3], h2[3][3], l2[3][3], h3[3][3], l3[3][3];
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
        for (int j = 0; j < 3; ++j)
            y.h1[i][j] = y.l1[i][j] = y.h2[i][j] = y.l2[i][j] = y.h3[i][j] = y.l3[i][j] = 0;
}

// x + a b, one instruction.  As a PTX product and sum, which the assembler
// joins: PTX's own mad.wide comes out as a product and a 64-bit addition
// (three instructions) in every other place, and from the C expression the
// compiler may make an unsigned product with corrections.  Where a factor is
// a negated register there is a subtraction all the same, which is why the
// products below have no signs.
__device__ __forceinline__ long long mad_wide(int a, int b, long long x)
{
    asm("{\n\t.reg .s64 t;\n\tmul.wide.s32 t, %1, %2;\n\tadd.s64 %0, %0, t;\n\t}" : "+l"(x) : "r"(a), "r"(b));
    return x;
}

// One real product into a pair of sums.
__device__ __forceinline__ void fx_mad(long long &h, long long &l, int ah, int al, int bh, int bl)
{
    h = mad_wide(ah, bh, h);
    l = mad_wide(ah, bl, l);
    l = mad_wide(al, bh, l);
}

// y += op_a(a) op_b(b), rows 0..ROWS-1; the signs of daggered factors are
// left to fx_value_of (SIGN = -1 for one daggered factor).
template <int FA, int FB, int ROWS = 3>
__device__ __forceinline__ void fx_mul_acc(FAcc &y, const FMat &a, const FMat &b)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int sh[3], sl[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int bi = FB == N ? k : j, bk = FB == N ? j : k;
            sh[j] = FB == N ? b.rh[bi][bk] + b.ih[bi][bk] : b.rh[bi][bk] - b.ih[bi][bk];
            sl[j] = FB == N ? b.rl[bi][bk] + b.il[bi][bk] : b.rl[bi][bk] - b.il[bi][bk];
        }
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            const int ai = FA == N ? i : k, ak = FA == N ? k : i;
            const int arh = a.rh[ai][ak], arl = a.rl[ai][ak], aih = a.ih[ai][ak], ail = a.il[ai][ak];
            const int ash = FA == N ? arh + aih : arh - aih, asl = FA == N ? arl + ail : arl - ail;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int bi = FB == N ? k : j, bk = FB == N ? j : k;
                fx_mad(y.h1[i][j], y.l1[i][j], arh, arl, b.rh[bi][bk], b.rl[bi][bk]);
                fx_mad(y.h2[i][j], y.l2[i][j], aih, ail, b.ih[bi][bk], b.il[bi][bk]);
                fx_mad(y.h3[i][j], y.l3[i][j], ash, asl, sh[j], sl[j]);
            }
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

// Entry (i, j) of the sums, in the units of the high ones; SIGN = -1 where
// one of the factors is daggered.
template <int SIGN>
__device__ __forceinline__ void fx_value_of(const FAcc &y, int i, int j, long long &re, long long &im)
{
    if constexpr (SIGN > 0) {
        re = fx_value(y.h1[i][j] - y.h2[i][j], y.l1[i][j] - y.l2[i][j]);
        im = fx_value(y.h3[i][j] - y.h1[i][j] - y.h2[i][j], y.l3[i][j] - y.l1[i][j] - y.l2[i][j]);
    } else {
        re = fx_value(y.h1[i][j] + y.h2[i][j], y.l1[i][j] + y.l2[i][j]);
        im = fx_value(y.h3[i][j] - y.h1[i][j] + y.h2[i][j], y.l3[i][j] - y.l1[i][j] + y.l2[i][j]);
    }
}

// The sums as limbs, in units 2^SH times coarser; rows 0..ROWS-1.
template <int SH, int SIGN = 1, int ROWS = 3> __device__ __forceinline__ FMat fx_round(const FAcc &y)
{
    FMat m;
#pragma unroll
    for (int i = 0; i < ROWS; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            long long re, im;
            fx_value_of<SIGN>(y, i, j, re, im);
            fx_split<SH>(re, m.rh[i][j], m.rl[i][j]);
            fx_split<SH>(im, m.ih[i][j], m.il[i][j]);
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

// Row 2 of an SU(3) matrix from rows 0 and 1: row2 = conj(row0 x row1), the
// terms of either sign in sums of their own.
__device__ __forceinline__ void fx_row2(FMat &u)
{
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int k = (j + 1) % 3, l = (j + 2) % 3;
        long long ph = 0, pl = 0, mh = 0, ml = 0;
        fx_mad(ph, pl, u.rh[0][k], u.rl[0][k], u.rh[1][l], u.rl[1][l]);
        fx_mad(mh, ml, u.ih[0][k], u.il[0][k], u.ih[1][l], u.il[1][l]);
        fx_mad(mh, ml, u.rh[0][l], u.rl[0][l], u.rh[1][k], u.rl[1][k]);
        fx_mad(ph, pl, u.ih[0][l], u.il[0][l], u.ih[1][k], u.il[1][k]);
        fx_split<0>(fx_value(ph - mh, pl - ml), u.rh[2][j], u.rl[2][j]);
        ph = pl = mh = ml = 0;
        fx_mad(mh, ml, u.rh[0][k], u.rl[0][k], u.ih[1][l], u.il[1][l]);
        fx_mad(mh, ml, u.ih[0][k], u.il[0][k], u.rh[1][l], u.rl[1][l]);
        fx_mad(ph, pl, u.rh[0][l], u.rl[0][l], u.ih[1][k], u.il[1][k]);
        fx_mad(ph, pl, u.ih[0][l], u.il[0][l], u.rh[1][k], u.rl[1][k]);
        fx_split<0>(fx_value(ph - mh, pl - ml), u.ih[2][j], u.il[2][j]);
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

// Re tr(a b), in the units of the product.
__device__ __forceinline__ long long fx_re_trace(const FMat &a, const FMat &b)
{
    long long h = 0, l = 0, mh = 0, ml = 0;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            fx_mad(h, l, a.rh[i][k], a.rl[i][k], b.rh[k][i], b.rl[k][i]);
            fx_mad(mh, ml, a.ih[i][k], a.il[i][k], b.ih[k][i], b.il[k][i]);
        }
    return fx_value(h - mh, l - ml);
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
