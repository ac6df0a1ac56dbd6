// Fixed-point arithmetic for FP64 fields of SU(3) matrices.
//
// GB300 issues 2 FP64 FMAs per clock and SM, but 32 integer multiply-adds of
// 32 x 32 + 64 bits and 128 FP32 FMAs.  The entries of an SU(3) matrix are at
// most 1 in modulus, so instead of a floating point they can have a fixed
// one.  Two forms share the leading part h, a whole number of 2^-30:
//
//   FLimbs   x = (h 2^28 + l) 2^-58, l a signed 28-bit whole number: all
//            sums of products are exact, three multiply-adds per product
//            (h h', h l', l h'; l l' is below 2^-60).  Links, and the few
//            products that the result sees with a weight near 1.
//   FMat     x = (h + l) 2^-30, l in FP32: h h' goes into a 64-bit sum
//            exactly, h l' + l h' into an FP32 sum (the terms are 2^-31 of
//            the product, so its rounding is near 2^-55 of it).  Staples, and
//            the many products under the rectangle and cube coefficients.
//
// Complex products take three whole-number products (Gauss: exact, so the
// cancellation costs nothing, and without signs: a negated factor would make
// a product and a 64-bit subtraction of every multiply-add).  In the second
// form the integer and the FP32 work run on the two halves of the FMA pipe:
// about 400 issue slots per 3x3 product and warp against 1730 (108 FMAs of 16
// clocks) on the FP64 pipe.
//
// Sums that pass 1 are kept in coarser units; the unit is fixed by the place
// in the formula.  High sums wrap modulo 2^64, so only results have to fit:
// entries of products of matrices that are unitary to about 1e-3 are bounded
// by 1 + 1e-2.  Links that are not within 1e-3 of SU(3), or not finite, are
// marked (kPoison) and take the floating-point path.
#pragma once

#include "su3.cuh"

namespace lqcd {

constexpr int kUnit = 30; // entries of links and staples in units of 2^-30

// h of entry (0, 0) of a matrix that has no fixed-point form.
constexpr int kPoison = (int)0x80000000;

struct FMat {
    int rh[3][3];
    float rl[3][3];
    int ih[3][3];
    float il[3][3];
};

struct FLimbs {
    int rh[3][3], rl[3][3], ih[3][3], il[3][3];
};

// High and mixed sums of the three real products of a matrix of complex ones.
struct FLimbAcc {
    long long h1[3][3], l1[3][3], h2[3][3], l2[3][3], h3[3][3], l3[3][3];
};

// Sums of a matrix of complex products a b: whole-number parts of
// 1: sum ar br, 2: sum ai bi, 3: sum (ar + ai)(br + bi), so that
// Re = 1 - 2, Im = 3 - 1 - 2; FP32 parts cr, ci of the real and imaginary one.
struct FAcc {
    long long h1[3][3], h2[3][3], h3[3][3];
    float cr[3][3], ci[3][3];
};

// A sum of products in the units of its place: v + c.
struct FSum {
    long long v;
    float c;
};

__device__ __forceinline__ void fx_zero(FAcc &y)
{
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            y.h1[i][j] = y.h2[i][j] = y.h3[i][j] = 0;
            y.cr[i][j] = y.ci[i][j] = 0.f;
        }
}

// x + a b, one instruction.  As a PTX product and sum, which the assembler
// joins: PTX's own mad.wide comes out as a product and a 64-bit addition
// (three instructions) in every other place, and from the C expression the
// compiler may make an unsigned product with corrections.
__device__ __forceinline__ long long mad_wide(int a, int b, long long x)
{
    asm("{\n\t.reg .s64 t;\n\tmul.wide.s32 t, %1, %2;\n\tadd.s64 %0, %0, t;\n\t}" : "+l"(x) : "r"(a), "r"(b));
    return x;
}

// y += op_a(a) op_b(b), rows 0..ROWS-1 (the sign of the second whole-number
// sum is left to fx_total).
template <int FA, int FB, int ROWS = 3>
__device__ __forceinline__ void fx_mul_acc(FAcc &y, const FMat &a, const FMat &b)
{
    constexpr float SA = FA == N ? 1.f : -1.f, SB = FB == N ? 1.f : -1.f; // signs of the imaginary parts
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int bs[3];
        float br[3], bi[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int p = FB == N ? k : j, q = FB == N ? j : k;
            bs[j] = FB == N ? b.rh[p][q] + b.ih[p][q] : b.rh[p][q] - b.ih[p][q];
            br[j] = (float)b.rh[p][q];
            bi[j] = (float)b.ih[p][q];
        }
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            const int u = FA == N ? i : k, v = FA == N ? k : i;
            const int arh = a.rh[u][v], aih = a.ih[u][v], as = FA == N ? arh + aih : arh - aih;
            const float ar = (float)arh, ai = (float)aih, arl = a.rl[u][v], ail = a.il[u][v];
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int p = FB == N ? k : j, q = FB == N ? j : k;
                y.h1[i][j] = mad_wide(arh, b.rh[p][q], y.h1[i][j]);
                y.h2[i][j] = mad_wide(aih, b.ih[p][q], y.h2[i][j]);
                y.h3[i][j] = mad_wide(as, bs[j], y.h3[i][j]);
                float cr = y.cr[i][j], ci = y.ci[i][j];
                cr = fmaf(ar, b.rl[p][q], cr);
                ci = fmaf(SB * ar, b.il[p][q], ci);
                cr = fmaf(arl, br[j], cr);
                ci = fmaf(SB * arl, bi[j], ci);
                cr = fmaf(-SA * SB * ai, b.il[p][q], cr);
                ci = fmaf(SA * ai, b.rl[p][q], ci);
                cr = fmaf(-SA * SB * ail, bi[j], cr);
                ci = fmaf(SA * ail, br[j], ci);
                y.cr[i][j] = cr;
                y.ci[i][j] = ci;
            }
        }
    }
}

// Entry (i, j) of the sums; SIGN = -1 where one of the factors is daggered.
template <int SIGN> __device__ __forceinline__ void fx_total(const FAcc &y, int i, int j, FSum &re, FSum &im)
{
    if constexpr (SIGN > 0) {
        re.v = y.h1[i][j] - y.h2[i][j];
        im.v = y.h3[i][j] - y.h1[i][j] - y.h2[i][j];
    } else {
        re.v = y.h1[i][j] + y.h2[i][j];
        im.v = y.h3[i][j] - y.h1[i][j] + y.h2[i][j];
    }
    re.c = y.cr[i][j];
    im.c = y.ci[i][j];
}

// A sum in units 2^SH times coarser, as h + l.
template <int SH> __device__ __forceinline__ void fx_split(const FSum s, int &h, float &l)
{
    static_assert(SH >= 2 && SH <= 33, "shift");
    if constexpr (SH == 33) {
        fx_split<32>(FSum{s.v >> 1, 0.5f * s.c}, h, l);
    } else if constexpr (SH == 32) {
        const unsigned lo = (unsigned)s.v;
        h = (int)(s.v >> 32) + (int)(lo >> 31);
        l = fmaf((float)(int)lo, 0x1p-32f, s.c * 0x1p-32f);
    } else {
        constexpr float scale = 1.f / (float)(1ll << SH);
        h = (int)((s.v + (1ll << (SH - 1))) >> SH);
        l = fmaf((float)(int)((unsigned)s.v - ((unsigned)h << SH)), scale, s.c * scale);
    }
}

// All entries, rows 0..ROWS-1.
template <int SH, int SIGN = 1, int ROWS = 3> __device__ __forceinline__ FMat fx_round(const FAcc &y)
{
    FMat m;
#pragma unroll
    for (int i = 0; i < ROWS; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            FSum re, im;
            fx_total<SIGN>(y, i, j, re, im);
            fx_split<SH>(re, m.rh[i][j], m.rl[i][j]);
            fx_split<SH>(im, m.ih[i][j], m.il[i][j]);
        }
    return m;
}

// A real scalar of modulus at most 1, in units of 2^-30.
struct FScalar {
    int h;
    float l;
};

inline FScalar fx_scalar(double c)
{
    const double x = c * 1073741824.0; // 2^30
    FScalar s;
    s.h = (int)(x + (x < 0 ? -0.5 : 0.5));
    s.l = (float)(x - (double)s.h);
    return s;
}

// c x, x = h + l; in units 2^-30 of those of x.
__device__ __forceinline__ FSum fx_scaled(const FScalar c, int h, float l)
{
    return FSum{mad_wide(c.h, h, 0), fmaf((float)c.h, l, c.l * (float)h)};
}

// c m, in the units of m.
__device__ __forceinline__ FMat fx_scaled(const FScalar c, const FMat &m)
{
    FMat r;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            fx_split<kUnit>(fx_scaled(c, m.rh[i][j], m.rl[i][j]), r.rh[i][j], r.rl[i][j]);
            fx_split<kUnit>(fx_scaled(c, m.ih[i][j], m.il[i][j]), r.ih[i][j], r.il[i][j]);
        }
    return r;
}

// Re tr(a b^dag), in the units of the product.
__device__ __forceinline__ FSum fx_re_trace_dag(const FMat &a, const FMat &b)
{
    FSum s{0, 0.f};
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int k = 0; k < 3; ++k) {
            s.v = mad_wide(a.rh[i][k], b.rh[i][k], s.v);
            s.v = mad_wide(a.ih[i][k], b.ih[i][k], s.v);
            s.c = fmaf((float)a.rh[i][k], b.rl[i][k], s.c);
            s.c = fmaf(a.rl[i][k], (float)b.rh[i][k], s.c);
            s.c = fmaf((float)a.ih[i][k], b.il[i][k], s.c);
            s.c = fmaf(a.il[i][k], (float)b.ih[i][k], s.c);
        }
    return s;
}

// ------------------------------------------------------------ whole limbs

__device__ __forceinline__ void fx_zero(FLimbAcc &y)
{
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j)
            y.h1[i][j] = y.l1[i][j] = y.h2[i][j] = y.l2[i][j] = y.h3[i][j] = y.l3[i][j] = 0;
}

// One real product into a high and a mixed sum.
__device__ __forceinline__ void fx_mad(long long &h, long long &l, int ah, int al, int bh, int bl)
{
    h = mad_wide(ah, bh, h);
    l = mad_wide(ah, bl, l);
    l = mad_wide(al, bh, l);
}

// y += op_a(a) op_b(b), rows 0..ROWS-1 (the sign of the second sums is left
// to fx_total).
template <int FA, int FB, int ROWS = 3>
__device__ __forceinline__ void fx_mul_acc(FLimbAcc &y, const FLimbs &a, const FLimbs &b)
{
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        int sh[3], sl[3];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const int p = FB == N ? k : j, q = FB == N ? j : k;
            sh[j] = FB == N ? b.rh[p][q] + b.ih[p][q] : b.rh[p][q] - b.ih[p][q];
            sl[j] = FB == N ? b.rl[p][q] + b.il[p][q] : b.rl[p][q] - b.il[p][q];
        }
#pragma unroll
        for (int i = 0; i < ROWS; ++i) {
            const int u = FA == N ? i : k, v = FA == N ? k : i;
            const int arh = a.rh[u][v], arl = a.rl[u][v], aih = a.ih[u][v], ail = a.il[u][v];
            const int ash = FA == N ? arh + aih : arh - aih, asl = FA == N ? arl + ail : arl - ail;
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                const int p = FB == N ? k : j, q = FB == N ? j : k;
                fx_mad(y.h1[i][j], y.l1[i][j], arh, arl, b.rh[p][q], b.rl[p][q]);
                fx_mad(y.h2[i][j], y.l2[i][j], aih, ail, b.ih[p][q], b.il[p][q]);
                fx_mad(y.h3[i][j], y.l3[i][j], ash, asl, sh[j], sl[j]);
            }
        }
    }
}

// A high and a mixed sum in the units of the high one.
__device__ __forceinline__ long long fx_value(long long h, long long l) { return h + ((l + (1ll << 27)) >> 28); }

// Entry (i, j) of the sums; SIGN = -1 where one of the factors is daggered.
template <int SIGN>
__device__ __forceinline__ void fx_total(const FLimbAcc &y, int i, int j, long long &re, long long &im)
{
    if constexpr (SIGN > 0) {
        re = fx_value(y.h1[i][j] - y.h2[i][j], y.l1[i][j] - y.l2[i][j]);
        im = fx_value(y.h3[i][j] - y.h1[i][j] - y.h2[i][j], y.l3[i][j] - y.l1[i][j] - y.l2[i][j]);
    } else {
        re = fx_value(y.h1[i][j] + y.h2[i][j], y.l1[i][j] + y.l2[i][j]);
        im = fx_value(y.h3[i][j] - y.h1[i][j] + y.h2[i][j], y.l3[i][j] - y.l1[i][j] + y.l2[i][j]);
    }
}

// A whole number v of 2^-(58 + SH) as limbs of 2^-30 and 2^-58 (SH at most 3).
template <int SH> __device__ __forceinline__ void fx_limbs(long long v, int &h, int &l)
{
    h = (int)((v + (1ll << (27 + SH))) >> (28 + SH));
    l = (int)((unsigned)v - ((unsigned)h << (28 + SH)));
    if constexpr (SH > 0) l = (l + (1 << (SH > 0 ? SH - 1 : 0))) >> SH;
}

// The entries of a product (units 2^-60), rows 0..ROWS-1.
template <int SIGN, int ROWS = 3> __device__ __forceinline__ FLimbs fx_round(const FLimbAcc &y)
{
    FLimbs m;
#pragma unroll
    for (int i = 0; i < ROWS; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            long long re, im;
            fx_total<SIGN>(y, i, j, re, im);
            fx_limbs<2>(re, m.rh[i][j], m.rl[i][j]);
            fx_limbs<2>(im, m.ih[i][j], m.il[i][j]);
        }
    return m;
}

// Row 2 of an SU(3) matrix from rows 0 and 1: row2 = conj(row0 x row1), the
// terms of either sign in sums of their own.
__device__ __forceinline__ void fx_row2(FLimbs &u)
{
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const int k = (j + 1) % 3, l = (j + 2) % 3;
        long long ph = 0, pl = 0, mh = 0, ml = 0;
        fx_mad(ph, pl, u.rh[0][k], u.rl[0][k], u.rh[1][l], u.rl[1][l]);
        fx_mad(mh, ml, u.ih[0][k], u.il[0][k], u.ih[1][l], u.il[1][l]);
        fx_mad(mh, ml, u.rh[0][l], u.rl[0][l], u.rh[1][k], u.rl[1][k]);
        fx_mad(ph, pl, u.ih[0][l], u.il[0][l], u.ih[1][k], u.il[1][k]);
        fx_limbs<2>(fx_value(ph - mh, pl - ml), u.rh[2][j], u.rl[2][j]);
        ph = pl = mh = ml = 0;
        fx_mad(mh, ml, u.rh[0][k], u.rl[0][k], u.ih[1][l], u.il[1][l]);
        fx_mad(mh, ml, u.ih[0][k], u.il[0][k], u.rh[1][l], u.rl[1][l]);
        fx_mad(ph, pl, u.rh[0][l], u.rl[0][l], u.ih[1][k], u.il[1][k]);
        fx_mad(ph, pl, u.ih[0][l], u.il[0][l], u.rh[1][k], u.rl[1][k]);
        fx_limbs<2>(fx_value(ph - mh, pl - ml), u.ih[2][j], u.il[2][j]);
    }
}

// The same matrix with an FP32 remainder.
__device__ __forceinline__ FMat fx_remainder(const FLimbs &a)
{
    FMat m;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        m.rh[e / 3][e % 3] = a.rh[e / 3][e % 3];
        m.rl[e / 3][e % 3] = 0x1p-28f * (float)a.rl[e / 3][e % 3];
        m.ih[e / 3][e % 3] = a.ih[e / 3][e % 3];
        m.il[e / 3][e % 3] = 0x1p-28f * (float)a.il[e / 3][e % 3];
    }
    return m;
}

// Re tr(a b): high and mixed sum.
__device__ __forceinline__ long long fx_re_trace(const FLimbs &a, const FLimbs &b)
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

// x 2^-shift in units of 2^-58 for |x| < 2 (shift 0), cut towards zero: 13
// integer operations, where scaling and converting on the FP64 pipe take two
// of its slots of 16 clocks.
// With flip = -1 the negative of it.
__device__ __forceinline__ long long fx_of_double(double x, int shift, int flip = 0)
{
    const int hi = __double2hiint(x);
    const unsigned lo = (unsigned)__double2loint(x);
    const int e = (hi >> 20) & 0x7ff;
    // 53-bit mantissa in units 2^(e - 1075), moved up by 6: the value for e = 1023
    const unsigned long long m = ((unsigned long long)((hi & 0xfffff) | 0x100000) << 32 | lo) << 6;
    const long long v = (long long)(m >> min(1023 - e + shift, 63));
    const long long s = (long long)((hi >> 31) ^ flip);
    return (v ^ s) - s;
}

__device__ __forceinline__ int exponent_of(double x) { return (__double2hiint(x) >> 20) & 0x7ff; }

// Whether rows 0 and 1 are orthonormal to 1e-3.
__device__ __forceinline__ bool fx_near_su3(const FLimbs &u)
{
    float n0 = 0.f, n1 = 0.f, cr = 0.f, ci = 0.f;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const float ar = 0x1p-30f * (float)u.rh[0][j], ai = 0x1p-30f * (float)u.ih[0][j];
        const float br = 0x1p-30f * (float)u.rh[1][j], bi = 0x1p-30f * (float)u.ih[1][j];
        n0 += ar * ar + ai * ai;
        n1 += br * br + bi * bi;
        cr += ar * br + ai * bi;
        ci += ar * bi - ai * br;
    }
    return fabsf(n0 - 1.f) < 1e-3f && fabsf(n1 - 1.f) < 1e-3f && fabsf(cr) < 1e-3f && fabsf(ci) < 1e-3f;
}

// Rows 0 and 1 of a stored FP64 link, row 2 rebuilt; a link that is not
// finite or not within 1e-3 of SU(3) is marked.
__device__ __forceinline__ FLimbs fx_from_rows(const double r[12])
{
    FLimbs u;
    bool ok = true;
#pragma unroll
    for (int e = 0; e < 6; ++e) {
        const int i = e / 3, j = e % 3;
        const double x = r[2 * e], y = r[2 * e + 1];
        // |x| < 1.5 by its bits (false for a NaN)
        ok = ok && (unsigned)(__double2hiint(x) & 0x7fffffff) < 0x3ff80000u &&
             (unsigned)(__double2hiint(y) & 0x7fffffff) < 0x3ff80000u;
        fx_limbs<0>(__double2ll_rn(x * 0x1p58), u.rh[i][j], u.rl[i][j]);
        fx_limbs<0>(__double2ll_rn(y * 0x1p58), u.ih[i][j], u.il[i][j]);
    }
    ok = ok && fx_near_su3(u);
    fx_row2(u);
    if (!ok) u.rh[0][0] = kPoison;
    return u;
}

// Rows 0 and 1 of a stored FP64 link by integer operations (row 2 is not
// set); false where they have no fixed-point form.
__device__ __forceinline__ bool fx_limbs_of_rows(const double r[12], FLimbs &u)
{
    bool ok = true;
#pragma unroll
    for (int e = 0; e < 6; ++e) {
        ok = ok && exponent_of(r[2 * e]) < 1024 && exponent_of(r[2 * e + 1]) < 1024;
        fx_limbs<0>(fx_of_double(r[2 * e], 0), u.rh[e / 3][e % 3], u.rl[e / 3][e % 3]);
        fx_limbs<0>(fx_of_double(r[2 * e + 1], 0), u.ih[e / 3][e % 3], u.il[e / 3][e % 3]);
    }
    return ok && fx_near_su3(u);
}

template <typename M> __device__ __forceinline__ bool fx_poisoned(const M &m) { return m.rh[0][0] == kPoison; }

// Matrices near 1 or near a subgroup of SU(3) have small entries that count by
// themselves, and the fixed point keeps only an absolute precision: at least
// kSmallMost of the 18 reals are below 2^-5, or kSmallSome below 2^-7 (15 of 18
// are small near 1, 12 near diagonal matrices, 9 or 8 near the real ones and an
// SU(2) or U(2) block).
constexpr int kSmallMost = 13, kSmallSome = 8, kSmallMostBits = 5, kSmallSomeBits = 7;

// The number of reals below 2^-BITS.
template <int BITS> __device__ __forceinline__ int fx_small(const FLimbs &u)
{
    constexpr int c = 1 << (kUnit - BITS);
    int n = 0;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        n += (unsigned)(u.rh[e / 3][e % 3] + c) < 2u * c;
        n += (unsigned)(u.ih[e / 3][e % 3] + c) < 2u * c;
    }
    return n;
}

__device__ __forceinline__ bool fx_near_subgroup(const FLimbs &u)
{
    return fx_small<kSmallMostBits>(u) >= kSmallMost || fx_small<kSmallSomeBits>(u) >= kSmallSome;
}

} // namespace lqcd
