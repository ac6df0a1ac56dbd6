// Shared by the two staple-field force translation units (force_sf.cu: FP32,
// force_fx.cu: FP64): storage of the staple planes, 32-bit lattice geometry,
// the traversal of the force pass, block reductions, the work queue of the
// batched launches, and the force of one link from its staples.
#pragma once

#include <mutex>

#include "fx_planes.cuh"
#include "kernels.h"
#include "su3.cuh"

namespace lqcd {

namespace {

constexpr int kBlock = 128; // four warps: the four directions of 32 sites

__host__ __device__ __forceinline__ int64_t padded_sites(int64_t V) { return (V + 31) & ~(int64_t)31; }
__host__ __device__ __forceinline__ int64_t virtual_blocks(int64_t V) { return padded_sites(V) / 32; }

enum { SC_BETA6 = 0, SC_CPL, SC_CRT, SC_CCB, SC_ACT, SC_ACTPL, SC_DT };

template <typename R> __device__ __forceinline__ R scalar(const KernelScalars &s, int i)
{
    if constexpr (sizeof(R) == 4) return s.f[i];
    else return s.d[i];
}

// Storage of the 24 FP32 staple planes: compact (rows 0 and 1, 12 reals, the
// third row rebuilt on load) or full (all 18 reals, nothing rebuilt).  Both
// are cut into blocks of 32 consecutive sites: inside a block, 16-byte lane
// q (3 compact, 4 full) of the staple of site s is at q*512 + s*16 bytes, and
// of full staples the last two reals at 4*512 + s*8 -- 72 bytes a full staple,
// every access 16- or 8-byte aligned, and the lanes of one staple a constant
// 512 bytes apart, so that a staple costs one address computation (plus one
// for the tail).  Plane P starts at P * plane_bytes, plane_bytes = the 32-site
// blocks of the lattice (V rounded up to 32) times the block size.  FP64
// staples have a form of their own (FxPlanes).
// Pass A writes them with evict-first stores: the 3.6 GB (at 32^3x64) would
// otherwise push the links that pass A re-reads out of L2.
constexpr int kStaplePlanes = 24;

struct FullBlock {
    static constexpr int NW = 4;                 // whole 16-byte lanes per staple
    static constexpr int LANE = 32 * 16;         // bytes of one lane of a block
    static constexpr int BYTES = NW * LANE + 32 * 8;
};

inline size_t full_plane_bytes(int64_t V, int precision)
{
    return precision == LQCD_F64 ? fx_plane_bytes(V) : (size_t)((V + 31) / 32) * FullBlock::BYTES;
}

// Compact planes: the first two rows (12 reals) of every staple, the third
// rebuilt on load, in the same 32-site blocks (lane q, q < 3, of site s at
// q*512 + s*16).
struct CompactBlock {
    static constexpr int NW = 3;
    static constexpr int LANE = 32 * 16;
    static constexpr int BYTES = NW * LANE;
};

template <bool FULL> struct Planes;

template <> struct Planes<false> {
    using B = CompactBlock;
    char *base;
    int64_t plane_bytes;
    using Ref = char *;

    __device__ __forceinline__ Ref at(int n) const
    {
        return base + (int64_t)(n >> 5) * B::BYTES + (n & 31) * 16;
    }

    __device__ __forceinline__ Mat<float> load(Ref r, int plane) const
    {
        const float4 *p = reinterpret_cast<const float4 *>(r + (int64_t)plane * plane_bytes);
        float x[12];
#pragma unroll
        for (int q = 0; q < B::NW; ++q) {
            const float4 v = __ldg(p + q * (B::LANE / 16));
            x[4 * q + 0] = v.x;
            x[4 * q + 1] = v.y;
            x[4 * q + 2] = v.z;
            x[4 * q + 3] = v.w;
        }
        Mat<float> u;
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                u.re[i][j] = x[6 * i + 2 * j];
                u.im[i][j] = x[6 * i + 2 * j + 1];
            }
        rebuild_row2(u);
        return u;
    }

    __device__ __forceinline__ void store(Ref r, int plane, const Mat<float> &u) const
    {
        float4 *p = reinterpret_cast<float4 *>(r + (int64_t)plane * plane_bytes);
        float x[12];
#pragma unroll
        for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                x[6 * i + 2 * j] = u.re[i][j];
                x[6 * i + 2 * j + 1] = u.im[i][j];
            }
#pragma unroll
        for (int q = 0; q < B::NW; ++q)
            __stcs(p + q * (B::LANE / 16), make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]));
    }
};

template <> struct Planes<true> {
    using B = FullBlock;
    char *base;          // plane 0
    int64_t plane_bytes;

    // The lane-0 and tail addresses of site n in plane 0.
    struct Ref {
        char *p;
        char *t;
    };

    __device__ __forceinline__ Ref at(int n) const
    {
        char *b = base + (int64_t)(n >> 5) * B::BYTES;
        const int s = n & 31;
        return Ref{b + s * 16, b + B::NW * B::LANE + s * 8};
    }

    __device__ __forceinline__ Mat<float> load(const Ref &r, int plane) const
    {
        const int64_t off = (int64_t)plane * plane_bytes;
        const float4 *p = reinterpret_cast<const float4 *>(r.p + off);
        float x[18];
#pragma unroll
        for (int q = 0; q < B::NW; ++q) {
            const float4 v = __ldg(p + q * (B::LANE / 16));
            x[4 * q + 0] = v.x;
            x[4 * q + 1] = v.y;
            x[4 * q + 2] = v.z;
            x[4 * q + 3] = v.w;
        }
        const float2 t = __ldg(reinterpret_cast<const float2 *>(r.t + off));
        x[16] = t.x;
        x[17] = t.y;
        Mat<float> u;
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                u.re[i][j] = x[2 * (3 * i + j)];
                u.im[i][j] = x[2 * (3 * i + j) + 1];
            }
        return u;
    }

    __device__ __forceinline__ void store(const Ref &r, int plane, const Mat<float> &u) const
    {
        const int64_t off = (int64_t)plane * plane_bytes;
        float4 *p = reinterpret_cast<float4 *>(r.p + off);
        float x[18];
#pragma unroll
        for (int i = 0; i < 3; ++i)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                x[2 * (3 * i + j)] = u.re[i][j];
                x[2 * (3 * i + j) + 1] = u.im[i][j];
            }
#pragma unroll
        for (int q = 0; q < B::NW; ++q)
            __stcs(p + q * (B::LANE / 16), make_float4(x[4 * q], x[4 * q + 1], x[4 * q + 2], x[4 * q + 3]));
        __stcs(reinterpret_cast<float2 *>(r.t + off), make_float2(x[16], x[17]));
    }
};

template <bool FULL> __device__ __forceinline__ Planes<FULL> planes_of(const SfLattice &L)
{
    if constexpr (FULL) {
        return Planes<true>{static_cast<char *>(L.staples), L.plane_bytes};
    } else {
        const int64_t V = (int64_t)L.dims[0] * L.dims[1] * L.dims[2] * L.dims[3];
        return Planes<false>{static_cast<char *>(L.staples),
                                ((V + 31) / 32) * CompactBlock::BYTES};
    }
}

// Lattice geometry in 32-bit arithmetic: the staple-field algorithm runs only
// for V < 2^31 sites (its workspace, 1728 bytes a site in FP32, could not
// hold more), so site indices and neighbour offsets fit an int.
struct G32 {
    int L0, L1, L2, L3;
    int s1, s2, s3, V;
};

__device__ __forceinline__ G32 make_g32(const int dims[4])
{
    G32 g;
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

// Slots of SfLattice::div (the magic of each run-time divisor).
enum { DV_S1, DV_S2, DV_S3, DV_VOL, DV_SLICE, DV_MVOL, DV_MX, DV_MY, DV_NMX, DV_NMY, DV_NBX, DV_NBY };

__device__ __forceinline__ int divi(int n, const DivMagic &d) { return (int)div_by((unsigned)n, d); }

// Coordinates of site n (the divisions by the strides as multiply-highs).
__device__ __forceinline__ Coord coord32(const G32 &g, const DivMagic *dm, int n)
{
    Coord x;
    x.c3 = divi(n, dm[DV_S3]);
    int r = n - x.c3 * g.s3;
    x.c2 = divi(r, dm[DV_S2]);
    r -= x.c2 * g.s2;
    x.c1 = divi(r, dm[DV_S1]);
    x.c0 = r - x.c1 * g.s1;
    return x;
}

__device__ __forceinline__ int index32(const G32 &g, const Coord &x)
{
    return x.c0 + g.s1 * x.c1 + g.s2 * x.c2 + g.s3 * x.c3;
}

// Index offset of the step s * hat(mu) (s = +-1) from a site with
// coordinates x, periodic (the direction picked by a select chain, so that
// nothing is indexed at run time in per-thread storage).
__device__ __forceinline__ int step32(const G32 &g, const Coord &x, int mu, int s)
{
    const int L = pick(mu, g.L0, g.L1, g.L2, g.L3);
    const int c = pick(mu, x.c0, x.c1, x.c2, x.c3);
    const int st = pick(mu, 1, g.s1, g.s2, g.s3);
    if (s > 0) return c + 1 == L ? (1 - L) * st : st;
    return c == 0 ? (L - 1) * st : -st;
}

// Traversal order of pass B: the lattice is cut into spatial blocks of
// bx x by x bz sites that run over all t; blocks one after the other, inside
// a block t-slice by t-slice, inside a slice micro-tiles of mx x my x mz
// sites (x fastest within and between micro-tiles).  The staple planes of
// three neighbouring t-slices of one block then stay in L2 while the block
// is swept, and micro-tiles make y and z neighbours L1 hits.
struct Sweep {
    int bx, by, bz, mx, my, mz;
    int nbx, nby, nmx, nmy, mvol;
    int slice, vol;     // sites per block slice and per block
    const DivMagic *dm; // magic of vol, slice, mvol, mx, my, nmx, nmy, nbx, nby
};

__device__ __forceinline__ Sweep make_sweep(const SfLattice &L, const G32 &g)
{
    Sweep s;
    s.bx = L.sweep[0];
    s.by = L.sweep[1];
    s.bz = L.sweep[2];
    s.mx = L.micro[0];
    s.my = L.micro[1];
    s.mz = L.micro[2];
    s.nbx = L.counts[0];
    s.nby = L.counts[1];
    s.nmx = L.counts[2];
    s.nmy = L.counts[3];
    s.mvol = s.mx * s.my * s.mz;
    s.slice = s.bx * s.by * s.bz;
    s.vol = s.slice * g.L3;
    s.dm = L.div;
    return s;
}

__device__ __forceinline__ Coord swept_site(const Sweep &s, int j)
{
    const DivMagic *dm = s.dm;
    const int blk = divi(j, dm[DV_VOL]);
    const int r = j - blk * s.vol;
    Coord c;
    c.c3 = divi(r, dm[DV_SLICE]);
    const int r2 = r - c.c3 * s.slice;
    const int mt = divi(r2, dm[DV_MVOL]), w = r2 - mt * s.mvol;
    const int wq = divi(w, dm[DV_MX]), xin = w - wq * s.mx;
    const int zin = divi(wq, dm[DV_MY]), yin = wq - zin * s.my;
    const int mq = divi(mt, dm[DV_NMX]), mxi = mt - mq * s.nmx;
    const int mzi = divi(mq, dm[DV_NMY]), myi = mq - mzi * s.nmy;
    const int q = divi(blk, dm[DV_NBX]), bxi = blk - q * s.nbx;
    const int bzi = divi(q, dm[DV_NBY]), byi = q - bzi * s.nby;
    c.c0 = bxi * s.bx + mxi * s.mx + xin;
    c.c1 = byi * s.by + myi * s.my + yin;
    c.c2 = bzi * s.bz + mzi * s.mz + zin;
    return c;
}

// Sum over the block of one double per thread (result in thread 0); the
// trailing barrier lets the caller run it again in the next virtual block.
__device__ __forceinline__ double block_sum(double v)
{
    __shared__ double part[kBlock / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) part[warp] = v;
    __syncthreads();
    double s = 0.0;
    if (warp == 0) {
        s = lane < kBlock / 32 ? part[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    }
    __syncthreads();
    return s;
}

// block_sum over the four warps of row group `row` of a CTA of ROWS groups
// (named barrier 1 + row over its 128 threads; same order of summation).
template <int ROWS> __device__ __forceinline__ double group_sum(double v, int row)
{
    if constexpr (ROWS == 1) {
        return block_sum(v);
    } else {
        __shared__ double part[ROWS * kBlock / 32];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
        const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
        if (lane == 0) part[warp] = v;
        asm volatile("bar.sync %0, %1;" ::"r"(1 + row), "r"(kBlock) : "memory");
        double s = 0.0;
        if ((warp & 3) == 0) {
            s = lane < kBlock / 32 ? part[warp + lane] : 0.0;
#pragma unroll
            for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        }
        asm volatile("bar.sync %0, %1;" ::"r"(1 + row), "r"(kBlock) : "memory");
        return s;
    }
}

// Next virtual block for a persistent CTA of a batched launch, taken from a
// work counter: the blocks in flight stay a contiguous window of the sweep
// (as with hardware block scheduling), which keeps the L2 reuse of the
// traversal; a fixed stride per CTA would let the window spread out.
__device__ __forceinline__ int64_t next_virtual_block(unsigned long long *counter)
{
    __shared__ unsigned long long s_vb;
    if (threadIdx.x == 0) s_vb = atomicAdd(counter, 1ull);
    __syncthreads();
    const int64_t vb = (int64_t)s_vb;
    __syncthreads();
    return vb;
}

// The same queue with the next block claimed (by thread 0) when the current
// one starts and handed to the block when it ends, so that the atomic's
// latency overlaps the current block's work.
__device__ __forceinline__ unsigned long long claim_virtual_block(unsigned long long *counter)
{
    return threadIdx.x == 0 ? atomicAdd(counter, 1ull) : 0ull;
}

__device__ __forceinline__ int64_t publish_virtual_block(unsigned long long claimed)
{
    __shared__ unsigned long long s_vb;
    if (threadIdx.x == 0) s_vb = claimed;
    __syncthreads();
    const int64_t vb = (int64_t)s_vb;
    __syncthreads();
    return vb;
}

// Lattice of a batch that virtual block vb (global numbering) belongs to.
__device__ __forceinline__ int batch_entry(const SfBatch &B, int64_t vb)
{
    int c = 0;
    while (c + 1 < B.n && vb >= B.e[c + 1].vb_begin) ++c;
    return c;
}

// ------------------------------------------ force of a link from its staples

// Products of two SU(3) factors are accumulated as y += s * (a * op(b)) with
// the third row of the product rebuilt from its first two (mul_acc_su3: the
// third row of a is never rebuilt or loaded; FP32, 3.65 against 3.75 ms at
// 32^3x64), or (DIRECT, the floating-point path of single FP64 links) as plain
// products accumulated in full, the sum scaled once.
template <int FB, bool DIRECT, typename R>
__device__ __forceinline__ void acc_su3(Mat<R> &y, const Mat<R> &a, const Mat<R> &b, R s)
{
    if constexpr (DIRECT) mul_acc<N, FB>(y, a, b); // s applied by the caller
    else mul_acc_su3<FB>(y, a, b, s);
}

// Where the staples of a site and of its neighbours are stored: in the
// lattice-wide staple field, the site index itself.
struct LatticeSites {
    const G32 *g;
    const Coord *c;
    int k;
    __device__ __forceinline__ int at0() const { return k; }
    __device__ __forceinline__ int nb(int mu, int s) const { return k + step32(*g, *c, mu, s); }
};

// The staples that start with link(k+rho, d), d = +-nu_d (NEG: minus), t += B_d y:
//   y = [ c_cube sum_{b perp rho, d} S_b(k+d) S^{(d)}_b(k) + c_rect S_d(k+d) A_d^dag ]
// (the orientation of the shared links fixed at compile time, so that each
// sign has one small loop body).
// CLOSE = false: y into t.
template <bool NEG, bool UNROLLQ, bool DIRECT, bool CLOSE = true, typename R, typename SF, typename SI>
__device__ __forceinline__ void d_terms(Mat<R> &t, const R *__restrict__ links,
                                        const SF &sf, const SI &si, const G32 &g,
                                        const Coord &c, int rho, int k, int kp, int id, R c_rt,
                                        R c_cb)
{
    constexpr int FD = NEG ? D : N;
    const int64_t V = g.V;
    const int base = rho * 6;
    const int jd = 2 * id + (NEG ? 1 : 0);
    const int nud = (rho + 1 + id) & 3;
    const int kd = k + step32(g, c, nud, NEG ? -1 : 1); // k + d
    // S^{(d)}_b(k): plane nud*6 + j' at k, or (NEG) its dagger at k - nud = kd
    const auto at_d = sf.at(si.nb(nud, NEG ? -1 : 1));
    const auto at_2 = NEG ? at_d : sf.at(si.at0());
    Mat<R> y;
    set_zero(y);
    // the four signed b perpendicular to rho and d: two directions, two signs
#pragma unroll(UNROLLQ ? 2 : 1)
    for (int q = 0; q < 2; ++q) {
        const int ib = q == 0 ? (id == 0 ? 1 : 0) : (id == 2 ? 1 : 2);
        const int nub = (rho + 1 + ib) & 3;
        const int jp = 2 * ((nub - nud - 1) & 3);
        acc_su3<FD, DIRECT>(y, sf.load(at_d, base + 2 * ib),
                            sf.load(at_2, nud * 6 + jp), c_cb);
        acc_su3<FD, DIRECT>(y, sf.load(at_d, base + 2 * ib + 1),
                            sf.load(at_2, nud * 6 + jp + 1), c_cb);
    }
    Mat<R> r3 = sf.load(at_d, base + jd);
    if constexpr (DIRECT) {
        scale(y, c_cb);
        scale(r3, c_rt);
    }
    if constexpr (!NEG) {
        acc_su3<D, DIRECT>(y, r3, load_link(links, V, nud, k), c_rt); // A_d = U_nud(k)
        if constexpr (CLOSE) mul_acc<N, N>(t, load_link(links, V, nud, kp), y); // B_d = U_nud(k+rho)
    } else {
        acc_su3<N, DIRECT>(y, r3, load_link(links, V, nud, kd), c_rt);  // A_d = U_nud(k-nud)^dag
        if constexpr (CLOSE) mul_acc<D, N>(t, load_link(links, V, nud, kp + (kd - k)), y); // B_d = U_nud(k+rho-nud)^dag
    }
    if constexpr (!CLOSE) t = y;
}

// The plaquettes and the two rectangle chains along rho: t = c_plaq Pl +
// c_rect (F sum_b S_b(k+rho) S_b(k) + sum_b S_b(k) S_b(k-rho) E); tr_pl the
// trace of U Pl for the action.
template <typename R, bool ACTION, bool DIRECT, typename SF, typename SI>
__device__ __forceinline__ void chain_terms(Mat<R> &t, R &tr_pl, const R *__restrict__ links, const SF &sf, const SI &si,
                                            const G32 &g, const Coord &c, int rho, int k, int kp, R c_pl, R c_rt)
{
    const int64_t V = g.V;
    const int km = k + step32(g, c, rho, -1);
    const int base = rho * 6;
    Mat<R> pl, p1, p2;
    set_zero(pl);
    set_zero(p1);
    set_zero(p2);
    const auto at_k = sf.at(si.at0()), at_p = sf.at(si.nb(rho, 1)), at_m = sf.at(si.nb(rho, -1));
#pragma unroll 1
    for (int jj = 0; jj < 6; ++jj) {
        const Mat<R> s = sf.load(at_k, base + jj);
        add_to(pl, s);
        acc_su3<N, DIRECT>(p1, sf.load(at_p, base + jj), s, c_rt);
        mul_acc<N, N>(p2, s, sf.load(at_m, base + jj));
    }
    if constexpr (ACTION) tr_pl = re_trace_mul<N, N>(load_link(links, V, rho, k), pl);
    t = pl;
    scale(t, c_pl);
    if constexpr (DIRECT) scale(p1, c_rt);
    mul_acc<N, N>(t, load_link(links, V, rho, kp), p1);
    scale(p2, c_rt);
    mul_acc<N, N>(t, p2, load_link(links, V, rho, km));
}

// The force from the staple sum t (stored, and/or the momentum step); returns
// the link's share of the action.
template <typename R, bool ACTION>
__device__ __forceinline__ double finish_link(const SfLattice &L, const KernelScalars &sc, const R *__restrict__ links,
                                              int64_t V, int rho, int k, const Mat<R> &t, R tr_pl)
{
    const Mat<R> m = mul<N, N>(load_link(links, V, rho, k), t);
    R f[8];
    ta_components(m, scalar<R>(sc, SC_BETA6), f);
    if (L.force != nullptr) store_algebra(static_cast<R *>(L.force), V, rho, k, f);
    if (L.mom != nullptr) {
        R *mom = static_cast<R *>(L.mom);
        R p[8];
        load_algebra(mom, V, rho, k, p);
        const R dt = scalar<R>(sc, SC_DT);
#pragma unroll
        for (int q = 0; q < 8; ++q) p[q] = fma(dt, f[q], p[q]);
        store_algebra(mom, V, rho, k, p);
    }
    if constexpr (ACTION) {
        const R tr_t = m.re[0][0] + m.re[1][1] + m.re[2][2];
        return (double)(scalar<R>(sc, SC_ACT) - tr_t * R(1.0 / 6.0) - scalar<R>(sc, SC_ACTPL) * tr_pl);
    }
    return 0.0;
}

// Force (and the fused momentum step) on the link (k, rho), k at coordinates
// c, its staples found through si; returns its share of the action.
template <typename R, bool ACTION, bool UNROLLQ, bool DIRECT, typename SF, typename SI>
__device__ __forceinline__ double force_link(const SfLattice &L, const KernelScalars &sc, const G32 &g,
                                             const SF &sf, const SI &si, const Coord &c,
                                             int k, int rho)
{
    const R *__restrict__ links = static_cast<const R *>(L.links);
    const R c_rt = scalar<R>(sc, SC_CRT), c_cb = scalar<R>(sc, SC_CCB);
    const int kp = k + step32(g, c, rho, 1);
    Mat<R> t;
    R tr_pl = R(0);
    chain_terms<R, ACTION, DIRECT>(t, tr_pl, links, sf, si, g, c, rho, k, kp, scalar<R>(sc, SC_CPL), c_rt);
    // cubes and the rectangles along d: positive, then negative d
#pragma unroll 1
    for (int id = 0; id < 3; ++id)
        d_terms<false, UNROLLQ, DIRECT>(t, links, sf, si, g, c, rho, k, kp, id, c_rt, c_cb);
#pragma unroll 1
    for (int id = 0; id < 3; ++id)
        d_terms<true, UNROLLQ, DIRECT>(t, links, sf, si, g, c, rho, k, kp, id, c_rt, c_cb);
    return finish_link<R, ACTION>(L, sc, links, g.V, rho, k, t, tr_pl);
}

// ------------------------------------------------------------- launch sizes

// Lattices of up to this many virtual blocks have a link's sums computed by
// several warps: four in FP32 (force_sf.cu), eight in FP64 (force_fx.cu).
// While there are fewer blocks than SMs a launch lasts as long as one thread's
// chain of products.  Measured, whole | split, force and action: FP32 4^4 24.6
// | 16.7 us, 64 blocks 28.7 | 19.7, 128 26.7 | 22.6, 256 31.8 | 34.0; FP64 8
// blocks 73.7 | 30.8, 64 75.6 | 45.2, 128 75.9 | 72.4, 256 97 | 123.
constexpr int kSplitBlocks = 128;
inline bool split_lattice(int64_t V)
{
    return virtual_blocks(V) <= kSplitBlocks;
}

// FP64 lattices of up to this many virtual blocks have a word for each of what
// the link pass found, which every warp of the later passes reads; on larger
// ones the reads would add up, and a flag is cleared before the pass (a memset
// is 4 us: 4^4 22.7 -> 27.9 us in a graph, with words 24.1).
constexpr int kNearBlocks = 1024;
inline bool near_words(int64_t V) { return virtual_blocks(V) <= kNearBlocks; }

// Sum over a warp of one double per lane (result in lane 0), the order of
// block_sum's first stage.
__device__ __forceinline__ double warp_sum(double v)
{
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    return v;
}

inline unsigned grid_of(int64_t items)
{
    if (items < 1) items = 1;
    if (items > ((int64_t)1 << 30)) items = (int64_t)1 << 30;
    return (unsigned)items;
}

// CTAs of a persistent launch: as many as are resident on the device at
// once (occupancy of the kernel times the SM count, cached per device).
template <typename K> unsigned persistent_grid(K kernel, int slot, int64_t work)
{
    static std::mutex mu;
    static int cached[64][48] = {{0}};
    int dev = 0;
    if (cudaGetDevice(&dev) != cudaSuccess || dev < 0 || dev >= 64) return grid_of(work);
    int resident = 0;
    {
        std::lock_guard<std::mutex> lk(mu);
        if (cached[dev][slot] == 0) {
            int sms = 0, per_sm = 0;
            cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
            cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, kernel, kBlock, 0);
            cached[dev][slot] = (sms > 0 ? sms : 1) * (per_sm > 0 ? per_sm : 1);
        }
        resident = cached[dev][slot];
    }
    return grid_of(work < resident ? work : resident);
}

} // namespace

} // namespace lqcd
