// U <- exp(i Q) U with Gram-Schmidt for FP64 links in the fixed point of
// fixed.cuh.
//
// In floating point a link is about 550 operations on a pipe that issues 2 a
// clock and SM: 9.5 k clocks a warp where the 256 bytes of a link take 385
// from memory.  Here the FP64 pipe only scales the momenta and converts the
// results; inputs are taken apart with integer operations (a conversion on
// the FP64 pipe costs as much as an FMA).
//
// With c1 = tr Q^2 / 2, c0 = det Q the series of exp(i Q) is
// f0 + f1 Q + f2 Q^2 (su3.cuh), applied as
//     U + (f0 - 1) U + f1 (Q U) + f2 (Q (Q U)),
// so that the rounding of the products is small with Q: they are formed with
// Q scaled by a power of two to c1 = 1/8 to 1/2.  Where Q itself is larger,
// exp(i 2^-s Q) is applied 2^s times.
// The links are unitary to rounding in every molecular-dynamics step, so
// Gram-Schmidt is a first-order correction by the departures, which are exact
// whole numbers below 2^-30; links that depart further, scales above s = 2 and
// what is not finite take the floating-point step (link_step).
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

// f0 - 1, f1, f2 for c0, c1 in units of 2^-58 (c1 <= 1/2): the forward
// recurrence of exp_i_hermitian, the terms from n = 13 (below 2^-32) in FP32.
__device__ __forceinline__ void fx_exp_coefficients(long long c0, long long c1, long long f[6])
{
    const FxS s0 = fxs(c0), s1 = fxs(c1);
    // n = 1, 2: i Q, -Q^2 / 2
    f[0] = f[1] = f[2] = f[5] = 0; // f0r - 1, f0i, f1r, f2i
    f[3] = 1ll << 58;              // f1i
    f[4] = -(1ll << 57);           // f2r
    // (a, b, d) with the sign of i^n: it turns from odd to even n
    long long a = 0, b = 0, d = -(1ll << 58);
#pragma unroll 1
    for (int m = 0; m < 5; ++m) {
        const auto odd = kInverseFactorial[2 * m], even = kInverseFactorial[2 * m + 1];
        FxS ds = fxs(d);
        long long an = fxs_mul(s0, ds), bn = a + fxs_mul(s1, ds);
        d = b;
        a = an;
        b = bn;
        ds = fxs(d);
        f[1] += fxs_mul(odd, fxs(a));
        f[3] += fxs_mul(odd, fxs(b));
        f[5] += fxs_mul(odd, ds);
        an = -fxs_mul(s0, ds);
        bn = -a - fxs_mul(s1, ds);
        d = -b;
        a = an;
        b = bn;
        f[0] += fxs_mul(even, fxs(a));
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
        const float an = sign * g0 * fd, bn = sign * fmaf(g1, fd, fa), dn = sign * fb;
        fa = an;
        fb = bn;
        fd = dn;
        ff *= 1.f / (float)n;
        const int o = n & 1;
        t[0 + o] = fmaf(ff, fa, t[0 + o]);
        t[2 + o] = fmaf(ff, fb, t[2 + o]);
        t[4 + o] = fmaf(ff, fd, t[4 + o]);
    }
#pragma unroll
    for (int i = 0; i < 6; ++i) f[i] += (long long)__float2int_rn(t[i]); // below 2^-32: fits 27 bits
}

// exp(i sum_a x^a T_a) U with Gram-Schmidt, rows 0 and 1 of both as 12 reals;
// false where it does not apply (r is then unchanged).
__device__ __forceinline__ bool fx_link_step(const double x[8], double r[12])
{
    // x = 2^(k+1) y with the entries of sum_a y^a lambda_a near 1 or below:
    // the products then round to 2^-55 of Q and not of 1
    int em = 1010;
#pragma unroll
    for (int a = 0; a < 8; ++a) em = max(em, exponent_of(x[a]));
    int k = em - 1022;
    if (k > 2) return false; // also not finite
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
    // the link
    FLimbs u;
    {
        if (!fx_limbs_of_rows(r, u)) return false;
        fx_row2(u);
    }
    // Q and its invariants
    FMat q;
    FScalar g0, g1, g2, m0, m1, m2; // f0 - 1, f1, f2: real and imaginary parts
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
        // back to the scale of one step: Q 2^(k-s)
        const int t = s - k;
        long long f[6];
        fx_exp_coefficients(c0 >> 3 * t, c1 >> 2 * t, f);
        f[2] >>= t;
        f[3] >>= t;
        f[4] >>= 2 * t;
        f[5] >>= 2 * t;
        const auto scalar = [](long long v) {
            FScalar t;
            int l;
            fx_limbs<0>(v, t.h, l);
            t.l = 0x1p-28f * (float)l;
            return t;
        };
        g0 = scalar(f[0]);
        m0 = scalar(f[1]);
        g1 = scalar(f[2]);
        m1 = scalar(f[3]);
        g2 = scalar(f[4]);
        m2 = scalar(f[5]);
        const auto put = [&](int i, int j, const FxS re, const FxS im) {
            q.rh[i][j] = q.rh[j][i] = re.h;
            q.rl[i][j] = q.rl[j][i] = 0x1p-28f * (float)re.l;
            q.ih[i][j] = -im.h;
            q.il[i][j] = -0x1p-28f * (float)im.l;
            q.ih[j][i] = im.h;
            q.il[j][i] = 0x1p-28f * (float)im.l;
        };
        put(0, 1, ys[0], ys[1]);
        put(0, 2, ys[3], ys[4]);
        put(1, 2, ys[5], ys[6]);
        const FxS dd[3] = {d0, d1, d2};
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            q.rh[i][i] = dd[i].h;
            q.rl[i][i] = 0x1p-28f * (float)dd[i].l;
            q.ih[i][i] = 0;
            q.il[i][i] = 0.f;
        }
    }
    long long vr[2][3], vi[2][3]; // rows 0 and 1, units 2^-58
#pragma unroll 1
    for (int rep = 0;; ++rep) {
        const FMat um = fx_remainder(u);
        FAcc acc;
        fx_zero(acc);
        fx_mul_acc<N, N>(acc, q, um);
        const FMat w1 = fx_round<kUnit>(acc);
        fx_zero(acc);
        fx_mul_acc<N, N, 2>(acc, q, w1);
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
                add(re, g0, 1.f, um.rh[i][j], um.rl[i][j]);
                add(re, m0, -1.f, um.ih[i][j], um.il[i][j]);
                add(re, g1, 1.f, w1.rh[i][j], w1.rl[i][j]);
                add(re, m1, -1.f, w1.ih[i][j], w1.il[i][j]);
                add(re, g2, 1.f, w2.rh[i][j], w2.rl[i][j]);
                add(re, m2, -1.f, w2.ih[i][j], w2.il[i][j]);
                add(im, g0, 1.f, um.ih[i][j], um.il[i][j]);
                add(im, m0, 1.f, um.rh[i][j], um.rl[i][j]);
                add(im, g1, 1.f, w1.ih[i][j], w1.il[i][j]);
                add(im, m1, 1.f, w1.rh[i][j], w1.rl[i][j]);
                add(im, g2, 1.f, w2.ih[i][j], w2.il[i][j]);
                add(im, m2, 1.f, w2.rh[i][j], w2.rl[i][j]);
                vr[i][j] = mad_wide(u.rh[i][j], 1 << 28, (long long)u.rl[i][j]) + ((re.v + 2) >> 2) +
                           __float2int_rn(0.25f * re.c);
                vi[i][j] = mad_wide(u.ih[i][j], 1 << 28, (long long)u.il[i][j]) + ((im.v + 2) >> 2) +
                           __float2int_rn(0.25f * im.c);
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
    // Gram-Schmidt to first order in the departures (units 2^-60)
    const auto limbs = [&](int i) {
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            fx_limbs<0>(vr[i][j], u.rh[i][j], u.rl[i][j]);
            fx_limbs<0>(vi[i][j], u.ih[i][j], u.il[i][j]);
        }
    };
    long long worst = 0;
    const auto normalise = [&](int i) {
        long long h = 0, l = 0;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            fx_mad(h, l, u.rh[i][j], u.rl[i][j], u.rh[i][j], u.rl[i][j]);
            fx_mad(h, l, u.ih[i][j], u.il[i][j], u.ih[i][j], u.il[i][j]);
        }
        const long long d = fx_value(h, l) - (1ll << 60);
        worst = max(worst, llabs(d));
        const int dd = (int)d; // u -= u d / 2
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            vr[i][j] -= mad_wide(u.rh[i][j], dd, 1ll << 32) >> 33;
            vi[i][j] -= mad_wide(u.ih[i][j], dd, 1ll << 32) >> 33;
        }
    };
    limbs(0);
    limbs(1);
    normalise(0);
    limbs(0);
    {
        // <row0, row1> = sum conj(u0) u1
        long long rh = 0, rl = 0, ph = 0, pl = 0, mh = 0, ml = 0;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            fx_mad(rh, rl, u.rh[0][j], u.rl[0][j], u.rh[1][j], u.rl[1][j]);
            fx_mad(rh, rl, u.ih[0][j], u.il[0][j], u.ih[1][j], u.il[1][j]);
            fx_mad(ph, pl, u.rh[0][j], u.rl[0][j], u.ih[1][j], u.il[1][j]);
            fx_mad(mh, ml, u.ih[0][j], u.il[0][j], u.rh[1][j], u.rl[1][j]);
        }
        const long long pr = fx_value(rh, rl), pi = fx_value(ph - mh, pl - ml);
        worst = max(worst, max(llabs(pr), llabs(pi)));
        const int r32 = (int)pr, i32 = (int)pi, n32 = -i32;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            vr[1][j] -= mad_wide(u.rh[0][j], r32, mad_wide(u.ih[0][j], n32, 1ll << 31)) >> 32;
            vi[1][j] -= mad_wide(u.ih[0][j], r32, mad_wide(u.rh[0][j], i32, 1ll << 31)) >> 32;
        }
    }
    limbs(1);
    normalise(1);
    if (worst >= 1ll << 30) return false;
#pragma unroll
    for (int e = 0; e < 6; ++e) {
        r[2 * e] = 0x1p-58 * (double)vr[e / 3][e % 3];
        r[2 * e + 1] = 0x1p-58 * (double)vi[e / 3][e % 3];
    }
    return true;
}

} // namespace

} // namespace lqcd
