// Box-Muller normals for FP32 fields from 53-bit uniforms without the FP64
// pipe: log, square root and cosine in pairs of FP32 numbers (a rounded value
// and its remainder).  The remainder tells whether the FP64 evaluation rounds to
// the same FP32 number; where it may not (one normal in 2900) that is done.  log
// and cos in FP64 are some 80 operations on a pipe that issues 2 a clock and SM;
// these are about 190 instructions on the others.
//
// log: 53-bit u = 2^-k m, m in [0.70, 1.42), 1/m looked up to 8 bits (exactly 1
// next to m = 1, so that log u keeps its relative accuracy there), r = m/c - 1
// exact as a pair, and the series of log(1 + r), |r| < 2^-7.  cos(2 pi u): the
// quadrant and the nearest of 32 angles in it from the leading bits, then the
// addition theorem with the series of the rest (below 0.025).
#pragma once

#include <cmath>
#include <cstdint>

namespace lqcd {

// Logarithm, sine and cosine of a few arguments for the tables, by their
// series (atanh for the logarithm).
constexpr double series_log(double x)
{
    const double t = (x - 1.0) / (x + 1.0), t2 = t * t;
    double s = 0.0, p = t;
    for (int n = 1; n < 60; n += 2, p *= t2) s += p / n;
    return 2.0 * s;
}
constexpr double series_sin(double x, bool cosine)
{
    double s = 0.0, p = cosine ? 1.0 : x;
    for (int n = cosine ? 1 : 2; n < 40; n += 2) {
        s += p;
        p *= -x * x / (n * (n + 1.0));
    }
    return s;
}

struct NormalTables {
    // interval i of m in [1, 2): 1/c, log(1/c) as a pair; c is halved from i = 53
    alignas(16) float log[128][4];
    // angle 2 pi i / 128, i = 0 to 16: cosine and sine as pairs
    alignas(16) float trig[17][4];
    constexpr NormalTables() : log(), trig()
    {
        for (int i = 0; i < 128; ++i) {
            const double c = (1.0 + (i + 0.5) / 128.0) * (i >= 53 ? 0.5 : 1.0);
            double inv = (double)(int)(256.0 / c + 0.5) / 256.0;
            if (i == 0 || i == 127) inv = 1.0;
            const double l = series_log(inv);
            log[i][0] = (float)inv;
            log[i][1] = (float)l;
            log[i][2] = (float)(l - (double)log[i][1]);
            log[i][3] = 0.f;
        }
        for (int i = 0; i <= 16; ++i) {
            const double x = 2.0 * 3.14159265358979323846 * i / 128.0;
            const double c = series_sin(x, true), s = series_sin(x, false);
            trig[i][0] = (float)c;
            trig[i][1] = (float)(c - (double)trig[i][0]);
            trig[i][2] = (float)s;
            trig[i][3] = (float)(s - (double)trig[i][2]);
        }
    }
};

// a b rounded, where a compiler may not make an FMA of the product and a sum.
__host__ __device__ inline float product(float a, float b)
{
#ifdef __CUDA_ARCH__
    return __fmul_rn(a, b);
#else
    return a * b;
#endif
}

// a + b = s + e exactly.
__host__ __device__ inline void two_sum(float a, float b, float &s, float &e)
{
    s = a + b;
    const float t = s - a;
    e += (a - (s - t)) + (b - t);
}

// sqrt(-2 log((w1 + 1) 2^-53)) cos(2 pi w2 2^-53) for 53-bit w1, w2: the FP32
// number, its remainder t, and the square root.
__host__ __device__ inline float normal_of(uint64_t w1, uint64_t w2, const NormalTables &tab, float &t, float &root)
{
    // -log u
    const uint64_t W = w1 + 1;
#ifdef __CUDA_ARCH__
    const int lz = __clzll((long long)W);
#else
    const int lz = __builtin_clzll(W);
#endif
    const uint64_t M = W << lz; // m 2^63, m in [1, 2)
    const int i = (int)(M >> 56) & 127;
    const float half = i >= 53 ? 0.5f : 1.0f;
    const float k = (float)(lz - (i >= 53 ? 11 : 10)); // u = 2^-k m
    const float mh = half * 0x1p-23f * (float)(int)(M >> 40);
    const float ml = half * 0x1p-55f * (float)(uint32_t)(M >> 8);
    const float inv = tab.log[i][0];
    const float p = product(mh, inv);
    float rh = p - 1.f, rl = fmaf(mh, inv, -p) + ml * inv;
    const int64_t D = (int64_t)((1ull << 53) - W); // u = 1 - D 2^-53
    if (D < (1ll << 45)) { // next to 1 (k = 0, inv = 1): r = -D 2^-53 exactly
        const float h = (float)D;
        rh = -0x1p-53f * h;
        rl = -0x1p-53f * (float)(D - (int64_t)h);
    }
    const float q = product(rh, rh), qe = fmaf(rh, rh, -q);
    float lo = 0.f, s;
    two_sum(k * 0x1.62e4p-1f, tab.log[i][1], s, lo); // log 2 to 16 bits: exact times k
    two_sum(s, -rh, s, lo);
    two_sum(s, 0.5f * q, s, lo);
    const float cub = rh * q * fmaf(rh, fmaf(rh, fmaf(rh, -1.f / 6.f, 0.2f), -0.25f), 1.f / 3.f);
    lo += fmaf(k, 0x1.7f7d1cp-20f, tab.log[i][2]) - (cub + (fmaf(rl, q - rh, rl) - 0.5f * qe));
    const float Lh = s + lo, Ll = (s - Lh) + lo;
    // sqrt(2 L)
    const float x = 2.f * Lh;
    t = root = 0.f;
    if (!(x > 0.f)) return 0.f; // u = 1
#ifdef __CUDA_ARCH__
    const float is = rsqrtf(x);
#else
    const float is = 1.f / sqrtf(x);
#endif
    const float sh = product(x, is), sl = 0.5f * is * fmaf(2.f, Ll, fmaf(-sh, sh, x));
    // cos(2 pi v): quadrant j, |f| <= 2^50
    const int j = (int)((w2 + (1ull << 50)) >> 51);
    const int64_t f = (int64_t)w2 - ((int64_t)j << 51);
    const int a = (int)((f + (1ll << 45)) >> 46); // angle 2 pi a / 128, -16 to 16
    const int64_t g = f - ((int64_t)a << 46);      // |g| <= 2^45
    const int gh = (int)((g + (1ll << 21)) >> 22);
    const float fh = (float)gh, fl = (float)(int)(g - ((int64_t)gh << 22));
    constexpr float c1 = 0x1.921fb6p-29f, c2 = -0x1.777a5cp-54f; // 2 pi 2^-31 as a pair
    const float dh = product(fh, c1);
    const float dl = fmaf(fh, c1, -dh) + fmaf(fh, c2, fl * 0x1.921fb6p-51f);
    const float z = product(dh, dh);
    const float ze = fmaf(dh, dh, -z), d3 = product(dh, z); // d^2 = z + ze, d^3 = d3 + d3e (with dl)
    const float d3e = fmaf(dh, z, -d3) + fmaf(dh, ze, 3.f * z * dl);
    constexpr float sixth = 1.f / 6.f, sixth_rest = (float)(1.0 / 6.0 - (double)sixth);
    const float s3 = product(d3, sixth), s3e = fmaf(d3, sixth, -s3) + fmaf(d3, sixth_rest, d3e * sixth);
    const float sl1 = (dl - s3) + fmaf(d3 * z, 1.f / 120.f, -s3e); // sin d = dh + sl1
    const float vh = 0.5f * z; // 1 - cos d as a pair
    const float vl = fmaf(dh, dl, fmaf(z * z, fmaf(z, 1.f / 720.f, -1.f / 24.f), 0.5f * ze));
    const int b = a < 0 ? -a : a;
    const float ch = tab.trig[b][0], cl = tab.trig[b][1];
    const float nh = a < 0 ? -tab.trig[b][2] : tab.trig[b][2], nl = a < 0 ? -tab.trig[b][3] : tab.trig[b][3];
    // cosine (j even): C - S sin d - C (1 - cos d); sine (odd): S + C sin d - S (1 - cos d)
    const bool odd = j & 1;
    const float bh = odd ? nh : ch, bl = odd ? nl : cl, oh = odd ? ch : -nh, ol = odd ? cl : -nl;
    const float ph = product(oh, dh);
    const float pe = fmaf(oh, dh, -ph) + fmaf(oh, sl1, ol * dh);
    float th, tl = 0.f;
    two_sum(bh, ph, th, tl);
    const float qh = product(bh, vh);
    two_sum(th, -qh, th, tl);
    tl += (fmaf(-bl, vh, bl) + pe) - (fmaf(bh, vh, -qh) + bh * vl);
    // quadrants: cos, -sin, -cos, sin
    const float r = product(sh, th);
    const float e = fmaf(sh, th, -r) + fmaf(sh, tl, sl * th);
    const float y = r + e;
    const bool minus = (j + 1) & 2;
    t = (r - y) + e;
    if (minus) t = -t;
    root = sh;
    return minus ? -y : y;
}
__host__ __device__ inline float normal_of(uint64_t w1, uint64_t w2, const NormalTables &tab)
{
    float t, root;
    return normal_of(w1, w2, tab, t, root);
}

// Whether y is what the FP64 evaluation rounds to: no midpoint of two FP32
// numbers lies within the errors of the two.  The pairs are within 0.86 of d
// here (1.4 x 10^9 normals against long double, next to the quadrants and to
// u = 1 among them), FP64 within 2^-50 of the root (2 pi u2 is rounded before
// the cosine).
__host__ __device__ inline bool normal_is_rounded(float y, float t, float root)
{
    const float d = fmaf(0x1p-37f, fabsf(y), 0x1p-40f * root);
    return root > 0.f && y + (t + d) == y && y + (t - d) == y;
}

} // namespace lqcd
