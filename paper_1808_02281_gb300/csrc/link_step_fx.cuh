// U <- exp(i Q) U with Gram-Schmidt for FP64 links in the fixed point of
// fixed.cuh.
//
// In floating point a link is about 550 operations on a pipe that issues 2 a
// clock and SM: 9.5 k clocks a warp where the 256 bytes of a link take 385
// from memory.  Here that pipe scales the momenta, converts the change of the
// link, adds it and takes the product of the rows; inputs are taken apart with
// integer operations (a conversion on the FP64 pipe costs as much as an FMA).
//
// With c1 = tr Q^2 / 2, c0 = det Q the series of exp(i Q) is
// f0 + f1 Q + f2 Q^2 (su3.cuh), and what is computed in whole numbers is the
// change of the link,
//     (f0 - 1) U + f1 (Q U) + f2 (Q (Q U)),
// in a unit of its own: with Q = 2^-t Q', Q' scaled to c1 = 1/16 to 1/2, it is
// known to 2^-(57 + t), whatever the size of Q, and is added in FP64 to the link
// as it was stored.  Small entries of links near 1 (or near a subgroup) so keep
// their digits.  Where Q itself is larger, exp(i 2^-s Q) is applied 2^s times.
// rms error of the worst class of entries against extended precision, of its
// own size (U = exp(i w), w and x normal): 0.9 to 1.7e-16 for w from 0 to 0.5
// and x from 1e-12 to 1; in floating point 1.1 to 2.9e-16.
// Components of Q of very different sizes (fx_uneven) and links that are not
// SU(3) to 2^-30 after the step, scales above s = 2 and what is not finite take
// the floating-point step (link_step).
#pragma once

#include "fixed.cuh"

namespace lqcd {

namespace {

// (h 2^28 + l) 2^-58
struct FxS {
    int h, l;
};

__device__ __forceinline__ FxS fxs(long long v)
{
    FxS s;
    fx_limbs<0>(v, s.h, s.l);
    return s;
}

// a b, units 2^-58
__device__ __forceinline__ long long fxs_mul(const FxS a, const FxS b)
{
    long long h = 0, l = 0;
    fx_mad(h, l, a.h, a.l, b.h, b.l);
    return (fx_value(h, l) + 2) >> 2;
}

// 2^58 / n!, n = 3 to 12, as limbs.
constexpr FxS inverse_factorial(int n)
{
    double f = 288230376151711744.0;
    for (int i = 2; i <= n; ++i) f /= (double)i;
    const long long v = (long long)(f + 0.5), h = (v + (1ll << 27)) >> 28;
    return FxS{(int)h, (int)(v - h * (1ll << 28))};
}
__constant__ const FxS kInverseFactorial[10] = {
    inverse_factorial(3), inverse_factorial(4), inverse_factorial(5),  inverse_factorial(6),  inverse_factorial(7),
    inverse_factorial(8), inverse_factorial(9), inverse_factorial(10), inverse_factorial(11), inverse_factorial(12)};

// (f0 - 1) / c0, f1, f2 for c0, c1 in units of 2^-58 (c1 <= 1/2): the forward
// recurrence of exp_i_hermitian, where a_n = c0 d_(n-1) for every n > 2, the
// terms from n = 13 (below 2^-32) in FP32.
__device__ __forceinline__ void fx_exp_coefficients(long long c0, long long c1, long long f[6])
{
    const FxS s0 = fxs(c0), s1 = fxs(c1);
    // n = 1, 2: i Q, -Q^2 / 2
    f[0] = f[1] = f[2] = f[5] = 0; // real and imaginary part of (f0 - 1) / c0, f1r, f2i
    f[3] = 1ll << 58;              // f1i
    f[4] = -(1ll << 57);           // f2r
    // (a, b, d) with the sign of i^n: it turns from odd to even n
    long long a = 0, b = 0, d = -(1ll << 58);
#pragma unroll 1
    for (int m = 0; m < 5; ++m) {
        const auto odd = kInverseFactorial[2 * m], even = kInverseFactorial[2 * m + 1];
        FxS ds = fxs(d);
        f[1] += fxs_mul(odd, ds);
        long long an = fxs_mul(s0, ds), bn = a + fxs_mul(s1, ds);
        d = b;
        a = an;
        b = bn;
        ds = fxs(d);
        f[3] += fxs_mul(odd, fxs(b));
        f[5] += fxs_mul(odd, ds);
        f[0] -= fxs_mul(even, ds);
        an = -fxs_mul(s0, ds);
        bn = -a - fxs_mul(s1, ds);
        d = -b;
        a = an;
        b = bn;
        f[2] += fxs_mul(even, fxs(b));
        f[4] += fxs_mul(even, fxs(d));
    }
    float fa = (float)a, fb = (float)b, fd = (float)d;
    const float g0 = 0x1p-58f * (float)c0, g1 = 0x1p-58f * (float)c1;
    float t[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};
    float ff = 1.f / 479001600.f;
#pragma unroll
    for (int n = 13; n <= 19; ++n) {
        const float sign = n & 1 ? 1.f : -1.f;
        const int o = n & 1;
        ff *= 1.f / (float)n;
        t[0 + o] = fmaf(ff, sign * fd, t[0 + o]);
        const float an = sign * g0 * fd, bn = sign * fmaf(g1, fd, fa), dn = sign * fb;
        fa = an;
        fb = bn;
        fd = dn;
        t[2 + o] = fmaf(ff, fb, t[2 + o]);
        t[4 + o] = fmaf(ff, fd, t[4 + o]);
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) f[i] += (long long)__float2int_rn(t[i]); // below 2^-32: fits 27 bits
}

// Below this exponent field nothing of an exponent shows in a link (2^-900).
constexpr int kLeastExponent = 123;

// Whether the components of x beside a subgroup are below 2^-6 of the largest
// (exponent field em): the four that leave a U(2) block, or any five (of an
// SU(2) block, of real rotations, of diagonal links).  The link step then has to
// keep small ones to a precision of their own.  Of Gaussian momenta it is one
// link in four million: a single one among the last blocks of a small lattice
// costs 18 us.
__device__ __forceinline__ bool fx_uneven(const double x[8], int em)
{
    unsigned m = 0;
#pragma unroll
    for (int a = 0; a < 8; ++a) m |= (em - exponent_of(x[a]) > 6 ? 1u : 0u) << a;
    return __popc(m) >= 5 || (m & 0x78) == 0x78 || (m & 0x1b) == 0x1b || (m & 0x63) == 0x63;
}

// Row i of a b, units 2^-60.
__device__ __forceinline__ void fx_row_mul(const FLimbs &a, int i, const FLimbs &b, long long re[3], long long im[3])
{
    FLimbAcc y; // row 0
#pragma unroll
    for (int j = 0; j < 3; ++j) y.h1[0][j] = y.l1[0][j] = y.h2[0][j] = y.l2[0][j] = y.h3[0][j] = y.l3[0][j] = 0;
#pragma unroll
    for (int k = 0; k < 3; ++k) {
        const int sh = a.rh[i][k] + a.ih[i][k], sl = a.rl[i][k] + a.il[i][k];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            fx_mad(y.h1[0][j], y.l1[0][j], a.rh[i][k], a.rl[i][k], b.rh[k][j], b.rl[k][j]);
            fx_mad(y.h2[0][j], y.l2[0][j], a.ih[i][k], a.il[i][k], b.ih[k][j], b.il[k][j]);
            fx_mad(y.h3[0][j], y.l3[0][j], sh, sl, b.rh[k][j] + b.ih[k][j], b.rl[k][j] + b.il[k][j]);
        }
    }
#pragma unroll
    for (int j = 0; j < 3; ++j) fx_total<1>(y, 0, j, re[j], im[j]);
}

// exp(i sum_a x^a T_a) U with Gram-Schmidt, rows 0 and 1 of both as 12 reals;
// false where it does not apply (r is then unchanged).
__device__ __forceinline__ bool fx_link_step(const double x[8], double r[12])
{
    // x = 2^(k+1) y, the largest |y^a| 1/4 to 1/2 (1/8 where they are many):
    // the products then round to 2^-57 of Q and not of 1
    int em = kLeastExponent;
#pragma unroll
    for (int a = 0; a < 8; ++a) em = max(em, exponent_of(x[a]));
    int k = em - 1022;
    if (k > 2) return false; // also not finite
    if (em > kLeastExponent && fx_uneven(x, em)) return false;
    long long y[8];
    float c1f = 0.f;
#pragma unroll
    for (int a = 0; a < 8; ++a) {
        y[a] = fx_of_double(x[a], k + 1);
        const float t = 0x1p-30f * (float)(int)(y[a] >> 28);
        c1f = fmaf(t, t, c1f);
    }
    if (c1f > 0.5f) {
        ++k;
#pragma unroll
        for (int a = 0; a < 8; ++a) y[a] >>= 1;
    }
    const int s = max(k, 0); // 2^s steps
    if (s > 2) return false;
    const int t = s - k; // of Q 2^-t
    // the link
    FLimbs u;
    {
        if (!fx_limbs_of_rows(r, u)) return false;
        fx_row2(u);
    }
    // Q and its invariants
    FLimbs q;
    FxS m1;                     // imaginary part of f1: limbs, the others with FP32 remainders
    FScalar g0, g1, g2, m0, m2; // f0 - 1, f1, f2: real and imaginary parts
    {
        FxS ys[8];
        long long c1 = 0, l1 = 0;
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            ys[a] = fxs(y[a]);
            fx_mad(c1, l1, ys[a].h, ys[a].l, ys[a].h, ys[a].l);
        }
        c1 = (fx_value(c1, l1) + 2) >> 2;
        const long long w = (long long)(0.57735026918962576451 * 288230376151711744.0); // 2^58 / sqrt(3)
        const FxS ws{(int)((w + (1ll << 27)) >> 28), (int)(w - (((w + (1ll << 27)) >> 28) << 28))};
        const long long z = fxs_mul(ws, ys[7]);
        const FxS d0 = fxs(y[2] + z), d1 = fxs(z - y[2]), d2 = fxs(-2 * z);
        // det Q = d0 d1 d2 + 2 Re(Q01 Q12 Q20) - d0 |Q12|^2 - d1 |Q02|^2 - d2 |Q01|^2,
        // Q01 = y0 - i y1, Q02 = y3 - i y4, Q12 = y5 - i y6
        const auto sq = [&](int i, int j) { return fxs_mul(ys[i], ys[i]) + fxs_mul(ys[j], ys[j]); };
        const long long pr = fxs_mul(ys[0], ys[5]) - fxs_mul(ys[1], ys[6]); // Q01 Q12 = pr - i pi
        const long long pi = fxs_mul(ys[0], ys[6]) + fxs_mul(ys[1], ys[5]);
        long long c0 = fxs_mul(fxs(fxs_mul(d0, d1) - sq(0, 1)), d2) - fxs_mul(d0, fxs(sq(5, 6))) -
                       fxs_mul(d1, fxs(sq(3, 4)));
        c0 += 2 * (fxs_mul(fxs(pr), ys[3]) + fxs_mul(fxs(pi), ys[4]));
        // The change of the link in units of 2^-(58 + t): with the invariants
        // of Q 2^-t, (f0 - 1) 2^t, f1 and f2 2^-t
        long long f[6];
        fx_exp_coefficients(c0 >> min(3 * t, 63), c1 >> min(2 * t, 63), f);
        const FxS c0t = fxs(c0 >> min(2 * t, 63));
        f[0] = fxs_mul(c0t, fxs(f[0]));
        f[1] = fxs_mul(c0t, fxs(f[1]));
        const int down = min(t, 63);
        f[4] >>= down;
        f[5] >>= down;
        const auto scalar = [](long long v) {
            const FxS l = fxs(v);
            return FScalar{l.h, 0x1p-28f * (float)l.l};
        };
        g0 = scalar(f[0]);
        m0 = scalar(f[1]);
        g1 = scalar(f[2]);
        m1 = fxs(f[3]);
        g2 = scalar(f[4]);
        m2 = scalar(f[5]);
        const auto put = [&](int i, int j, const FxS re, const FxS im) {
            q.rh[i][j] = q.rh[j][i] = re.h;
            q.rl[i][j] = q.rl[j][i] = re.l;
            q.ih[i][j] = -im.h;
            q.il[i][j] = -im.l;
            q.ih[j][i] = im.h;
            q.il[j][i] = im.l;
        };
        put(0, 1, ys[0], ys[1]);
        put(0, 2, ys[3], ys[4]);
        put(1, 2, ys[5], ys[6]);
        const FxS dd[3] = {d0, d1, d2};
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            q.rh[i][i] = dd[i].h;
            q.rl[i][i] = dd[i].l;
            q.ih[i][i] = q.il[i][i] = 0;
        }
    }
    long long vr[2][3], vi[2][3]; // rows 0 and 1, units 2^-58
    long long er[2][3], ei[2][3]; // their change, units 2^-(58 + t)
    const int tt = min(t, 62);
    const long long half = (1ll << tt) >> 1;
#pragma unroll 1
    for (int rep = 0;; ++rep) {
        // Q U decides the accuracy of the change: whole limbs
        FLimbs w1;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            long long re[3], im[3];
            fx_row_mul(q, i, u, re, im);
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                fx_limbs<2>(re[j], w1.rh[i][j], w1.rl[i][j]);
                fx_limbs<2>(im[j], w1.ih[i][j], w1.il[i][j]);
            }
        }
        FAcc acc;
        fx_zero(acc);
        fx_mul_acc<N, N, 2>(acc, fx_remainder(q), fx_remainder(w1));
        const FMat w2 = fx_round<kUnit, 1, 2>(acc);
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                FSum re{0, 0.f}, im{0, 0.f};
                const auto add = [](FSum &t, const FScalar c, float sign, int h, float l) {
                    t.v = mad_wide(sign < 0.f ? -c.h : c.h, h, t.v);
                    t.c = fmaf(sign * (float)c.h, l, fmaf(sign * c.l, (float)h, t.c));
                };
                const float url = 0x1p-28f * (float)u.rl[i][j], uil = 0x1p-28f * (float)u.il[i][j];
                const float wrl = 0x1p-28f * (float)w1.rl[i][j], wil = 0x1p-28f * (float)w1.il[i][j];
                add(re, g0, 1.f, u.rh[i][j], url);
                add(re, m0, -1.f, u.ih[i][j], uil);
                add(re, g1, 1.f, w1.rh[i][j], wrl);
                add(re, g2, 1.f, w2.rh[i][j], w2.rl[i][j]);
                add(re, m2, -1.f, w2.ih[i][j], w2.il[i][j]);
                add(im, g0, 1.f, u.ih[i][j], uil);
                add(im, m0, 1.f, u.rh[i][j], url);
                add(im, g1, 1.f, w1.ih[i][j], wil);
                add(im, g2, 1.f, w2.ih[i][j], w2.il[i][j]);
                add(im, m2, 1.f, w2.rh[i][j], w2.rl[i][j]);
                long long lr = 0, li = 0;
                fx_mad(re.v, lr, -m1.h, -m1.l, w1.ih[i][j], w1.il[i][j]);
                fx_mad(im.v, li, m1.h, m1.l, w1.rh[i][j], w1.rl[i][j]);
                er[i][j] = ((fx_value(re.v, lr) + 2) >> 2) + __float2int_rn(0.25f * re.c);
                ei[i][j] = ((fx_value(im.v, li) + 2) >> 2) + __float2int_rn(0.25f * im.c);
                vr[i][j] = mad_wide(u.rh[i][j], 1 << 28, (long long)u.rl[i][j]) + ((er[i][j] + half) >> tt);
                vi[i][j] = mad_wide(u.ih[i][j], 1 << 28, (long long)u.il[i][j]) + ((ei[i][j] + half) >> tt);
            }
        if (rep + 1 >> s) break; // 2^s steps
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                fx_limbs<0>(vr[i][j], u.rh[i][j], u.rl[i][j]);
                fx_limbs<0>(vi[i][j], u.ih[i][j], u.il[i][j]);
            }
        fx_row2(u);
    }
    // Gram-Schmidt to first order in the departures.  Those of the lengths
    // are whole numbers of 2^-60 ...
    const auto departure = [&](int i) {
        long long h = 0, l = 0;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const FxS a = fxs(vr[i][j]), b = fxs(vi[i][j]);
            fx_mad(h, l, a.h, a.l, a.h, a.l);
            fx_mad(h, l, b.h, b.l, b.h, b.l);
        }
        return fx_value(h, l) - (1ll << 60);
    };
    const long long n0 = departure(0), n1 = departure(1);
    if (llabs(n0) >= 1ll << 30 || llabs(n1) >= 1ll << 30) return false;
    // ... and the product of the rows is taken in FP64, as the rows
    // themselves: small entries keep their digits.  One step: the link as it
    // was stored and its change; several: the link as a whole number.
    double v[12];
    const double unit = __hiloint2double((1023 - 58 - (s > 0 ? 0 : t)) << 20, 0);
#pragma unroll
    for (int e = 0; e < 6; ++e) {
        const int i = e / 3, j = e % 3;
        v[2 * e] = fma((double)(s > 0 ? vr[i][j] : er[i][j]), unit, s > 0 ? 0.0 : r[2 * e]);
        v[2 * e + 1] = fma((double)(s > 0 ? vi[i][j] : ei[i][j]), unit, s > 0 ? 0.0 : r[2 * e + 1]);
    }
    double pr = 0.0, pi = 0.0; // <row0, row1> = sum conj(u0) u1
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const double a = v[2 * j], b = v[2 * j + 1], c = v[6 + 2 * j], d = v[7 + 2 * j];
        pr = fma(a, c, fma(b, d, pr));
        pi = fma(a, d, fma(-b, c, pi));
    }
    if (exponent_of(pr) >= 1023 - 30 || exponent_of(pi) >= 1023 - 30) return false;
    const double f0 = -0x1p-61 * (double)(int)n0, f1 = -0x1p-61 * (double)(int)n1;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
        const double a = v[2 * j], b = v[2 * j + 1], c = v[6 + 2 * j], d = v[7 + 2 * j];
        r[6 + 2 * j] = fma(-pr, a, fma(pi, b, fma(f1, c, c)));
        r[7 + 2 * j] = fma(-pr, b, fma(-pi, a, fma(f1, d, d)));
        r[2 * j] = fma(f0, a, a);
        r[2 * j + 1] = fma(f0, b, b);
    }
    return true;
}

} // namespace

} // namespace lqcd
