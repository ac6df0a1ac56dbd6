// Planes of 3x3 matrices in the fixed-point forms of fixed.cuh or in FP64, in
// blocks of 32 consecutive sites: 16 bytes for a complex entry (h, l of its real
// and imaginary part, or the two parts), entry e = 3 i + j of site s at
// e*512 + s*16 bytes of the block, plane P of a field at P * plane_bytes.
#pragma once

#include "fixed.cuh"

namespace lqcd {

namespace {


// The word at p: GLOBAL, of read-only global memory.
template <bool GLOBAL> __device__ __forceinline__ int4 fx_word(const int4 *p)
{
    if constexpr (GLOBAL) return __ldg(p);
    else return *p;
}

// The matrix with FP32 remainders whose entries lie S words apart.
template <int S, bool GLOBAL> __device__ __forceinline__ FMat fx_mat_at(const int4 *p)
{
    FMat u;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        const int4 v = fx_word<GLOBAL>(p + e * S);
        u.rh[e / 3][e % 3] = v.x;
        u.rl[e / 3][e % 3] = __int_as_float(v.y);
        u.ih[e / 3][e % 3] = v.z;
        u.il[e / 3][e % 3] = __int_as_float(v.w);
    }
    return u;
}

// The same, or of whole limbs (whole), or (dag) its dagger: the off-diagonal
// entries are then read from their mirrored places.
template <int S, bool GLOBAL> __device__ __forceinline__ FMat fx_form_at(const int4 *p, bool whole, bool dag)
{
    const int o = dag ? 2 * S : 0, m = dag ? -1 : 0, f = dag ? (int)0x80000000 : 0;
    const int4 *up = p + o, *dn = p - o, *up2 = up + o, *dn2 = dn - o;
    const int4 v[9] = {fx_word<GLOBAL>(p),           fx_word<GLOBAL>(up + S),      fx_word<GLOBAL>(up2 + 2 * S),
                       fx_word<GLOBAL>(dn + 3 * S),  fx_word<GLOBAL>(p + 4 * S),   fx_word<GLOBAL>(up + 5 * S),
                       fx_word<GLOBAL>(dn2 + 6 * S), fx_word<GLOBAL>(dn + 7 * S),  fx_word<GLOBAL>(p + 8 * S)};
    FMat u;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        u.rh[e / 3][e % 3] = v[e].x;
        u.ih[e / 3][e % 3] = (v[e].z ^ m) - m;
        u.rl[e / 3][e % 3] = __int_as_float(v[e].y);
        u.il[e / 3][e % 3] = __int_as_float(v[e].w);
    }
    if (whole) {
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            u.rl[e / 3][e % 3] = 0x1p-28f * (float)v[e].y;
            u.il[e / 3][e % 3] = 0x1p-28f * (float)v[e].w;
        }
    }
#pragma unroll
    for (int e = 0; e < 9; ++e)
        u.il[e / 3][e % 3] = __int_as_float(__float_as_int(u.il[e / 3][e % 3]) ^ f);
    return u;
}

struct FxPlanes {
    char *base;
    int64_t plane_bytes;
    static constexpr int LANE = 32 * 16;       // bytes of one entry of 32 sites
    static constexpr int BYTES = 9 * LANE;      // of a matrix of 32 sites
    static constexpr int S = LANE / 16;

    __device__ __forceinline__ char *at(int n) const
    {
        return base + (int64_t)(n >> 5) * BYTES + (n & 31) * 16;
    }

    __device__ __forceinline__ const int4 *ptr(const char *r, int plane) const
    {
        return reinterpret_cast<const int4 *>(r + (int64_t)plane * plane_bytes);
    }

    // A matrix in whole limbs.
    __device__ __forceinline__ FLimbs limbs(const char *r, int plane) const
    {
        const int4 *p = ptr(r, plane);
        FLimbs u;
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const int4 v = __ldg(p + e * S);
            u.rh[e / 3][e % 3] = v.x;
            u.rl[e / 3][e % 3] = v.y;
            u.ih[e / 3][e % 3] = v.z;
            u.il[e / 3][e % 3] = v.w;
        }
        return u;
    }

    // A matrix with an FP32 remainder.
    __device__ __forceinline__ FMat mat(const char *r, int plane) const { return fx_mat_at<S, true>(ptr(r, plane)); }

    // Either of the two (whole: whole limbs), or (dag) its dagger, chosen at run time.
    __device__ __forceinline__ FMat form(const char *r, int plane, bool whole, bool dag) const
    {
        return fx_form_at<S, true>(ptr(r, plane), whole, dag);
    }

    __device__ __forceinline__ void store(char *r, int plane, const FLimbs &u) const
    {
        int4 *p = const_cast<int4 *>(ptr(r, plane));
#pragma unroll
        for (int e = 0; e < 9; ++e)
            p[e * S] = make_int4(u.rh[e / 3][e % 3], u.rl[e / 3][e % 3], u.ih[e / 3][e % 3], u.il[e / 3][e % 3]);
    }

    // A matrix in FP64.
    __device__ __forceinline__ Mat<double> floating(const char *r, int plane) const
    {
        const double2 *p = reinterpret_cast<const double2 *>(ptr(r, plane));
        Mat<double> u;
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const double2 v = __ldg(p + e * S);
            u.re[e / 3][e % 3] = v.x;
            u.im[e / 3][e % 3] = v.y;
        }
        return u;
    }

    __device__ __forceinline__ void store(char *r, int plane, const Mat<double> &u) const
    {
        double2 *p = reinterpret_cast<double2 *>(const_cast<int4 *>(ptr(r, plane)));
#pragma unroll
        for (int e = 0; e < 9; ++e) __stcs(p + e * S, make_double2(u.re[e / 3][e % 3], u.im[e / 3][e % 3]));
    }

    template <bool STREAM> __device__ __forceinline__ void store(char *r, int plane, const FMat &u) const
    {
        int4 *p = const_cast<int4 *>(ptr(r, plane));
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const int4 v = make_int4(u.rh[e / 3][e % 3], __float_as_int(u.rl[e / 3][e % 3]), u.ih[e / 3][e % 3],
                                     __float_as_int(u.il[e / 3][e % 3]));
            if constexpr (STREAM) __stcs(p + e * S, v);
            else p[e * S] = v;
        }
    }
};

// Bytes of a plane of V sites.
inline size_t fx_plane_bytes(int64_t V) { return (size_t)((V + 31) / 32) * FxPlanes::BYTES; }

// Link (n, mu) of an FP64 link field of V sites, in whole limbs.
__device__ __forceinline__ FLimbs fx_load_link(const double *__restrict__ links, int64_t V, int mu, int64_t n)
{
    const double2 *p = reinterpret_cast<const double2 *>(links) + (int64_t)mu * 6 * V + n;
    double r[12];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        const double2 v = __ldg(p + q * V);
        r[2 * q] = v.x;
        r[2 * q + 1] = v.y;
    }
    return fx_from_rows(r);
}

} // namespace

} // namespace lqcd
