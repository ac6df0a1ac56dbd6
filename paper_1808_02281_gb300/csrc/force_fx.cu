// Gauge force of the one-loop Symanzik action for FP64 fields: the
// staple-field algorithm of force_sf.cu (same formulas, traversal and action)
// in the fixed-point arithmetic of fixed.cuh, three passes:
//   links_fx     the links in fixed point (all three rows), planes 24..27 of the
//                workspace: every link is read about 18 times by the next two
//                passes, so it is converted (and checked) once
//   staples_fx   the 24 plaquette staples of every site
//   force_fx     the force (momentum step, action) of every link
//
// A thread that reads a marked matrix (a link that is not finite or not
// within 1e-3 of SU(3), or a staple of one) computes its staple or force in
// floating point from the stored links instead.
//
// The force of links near 1, or near a subgroup, is made of small entries, and
// whole numbers of 2^-58 keep too little of them: rms error against extended
// precision, of the force's own size (U = exp(i w), w normal, u0 0.87), 1.1 to
// 1.9e-16 for w of 1 to 0.1, 3.4e-16 at 0.05, below that 1.6e-17 / w; in
// floating point 3.1 to 4e-16 for all w.  So where a quarter of the links of 32
// sites, in each direction, are near a subgroup (fx_near_subgroup; or have no
// fixed-point form) the lattice's flag is set and the other two passes run in
// floating point, on planes of FP64 staples: the whole lattice, for warps of
// which some lanes did one and some the other take up to three times as long.
// 24^3x48: 5.5 ms, in floating point 34.3.
#include "async_copy.cuh"
#include "fx_planes.cuh"
#include "sf_common.cuh"

namespace lqcd {

namespace {

constexpr int kLinkPlane = kStaplePlanes; // planes 24..27: the links
__device__ __forceinline__ FxPlanes fx_planes(const SfLattice &L)
{
    return FxPlanes{static_cast<char *>(L.staples), L.plane_bytes};
}

// Coefficients for the fixed-point sums.  With t = c_plaq Pl + c_rect Rc +
// c_cube Cb, z the larger of c_rect, c_cube in modulus and m a quarter of the
// largest that t can be,
//     t / m = pl Pl + z (beta Rc + alpha Cb)
// is at most 4 and every scalar at most 1 in modulus (use_beta: beta is not 1).
struct FxScalars {
    int plh, pll, zh, zl; // pl and z in limbs of 2^-30 and 2^-58
    FScalar alpha, beta;
    int use_beta;
    double m;
    long long tr0; // Re tr(U t) / m of unit links, units 2^-58
};

// x in units of 2^-58, as limbs.
long long limbs_of(double x, int &h, int &l)
{
    const long long v = (long long)(x * 0x1p58);
    h = (int)((v + (1ll << 27)) >> 28);
    l = (int)(v - (long long)h * (1ll << 28));
    return v;
}

FxScalars make_fx_scalars(const KernelScalars &sc)
{
    const double cp = sc.d[SC_CPL], cr = sc.d[SC_CRT], cc = sc.d[SC_CCB];
    const auto mod = [](double x) { return x < 0 ? -x : x; };
    FxScalars f;
    double z, alpha, beta;
    if (mod(cr) >= mod(cc)) {
        z = cr;
        alpha = cr == 0.0 ? 0.0 : cc / cr;
        beta = 1.0;
    } else {
        z = cc;
        alpha = 1.0;
        beta = cr / cc;
    }
    f.m = 1.5 * mod(cp) + 4.5 * mod(cr) + 6.0 * mod(cc);
    if (f.m == 0.0) f.m = 1.0;
    const long long pv = limbs_of(cp / f.m, f.plh, f.pll), zv = limbs_of(z / f.m, f.zh, f.zl);
    f.alpha = fx_scalar(alpha);
    f.beta = fx_scalar(beta);
    f.use_beta = beta != 1.0;
    // with the scalars as rounded, so that unit links have no action at all
    const long double aq = (long double)f.alpha.h + f.alpha.l, bq = (long double)f.beta.h + f.beta.l;
    f.tr0 = (long long)(18.0L * pv + 3.0L * zv * (18.0L * bq + 24.0L * aq) / 1073741824.0L);
    return f;
}

// ------------------------------------------------------------------ links

// Whether the lattice is computed in floating point; for whole warps.
__device__ __forceinline__ bool floating(const SfLattice &L)
{
    if (L.flag == nullptr) return true;
    if (L.near == nullptr) return *L.flag & L.bit;
    const int n = (int)virtual_blocks(make_g32(L.dims).V);
    int any = 0;
    for (int i = (int)(threadIdx.x & 31); i < n; i += 32) any |= L.near[i];
    return __any_sync(0xffffffffu, any);
}

__device__ __forceinline__ void links_block(const SfLattice &L, int V, int vb)
{
    const int mu = (int)(threadIdx.x >> 5);
    const int x = vb * 32 + (int)(threadIdx.x & 31);
    const FLimbs u = fx_load_link(static_cast<const double *>(L.links), V, mu, x < V ? x : V - 1);
    const FxPlanes sf = fx_planes(L);
    if (x < V) sf.store(sf.at(x), kLinkPlane + mu, u);
    const int n = __popc(__ballot_sync(0xffffffffu, fx_poisoned(u) || fx_near_subgroup(u)));
    const int near = __syncthreads_and(n >= 8);
    if (threadIdx.x > 0) return;
    if (L.near != nullptr) L.near[vb] = near;
    else if (near && !(*(volatile unsigned long long *)L.flag & L.bit)) atomicOr(L.flag, L.bit);
}

__global__ void __launch_bounds__(kBlock) links_fx(const __grid_constant__ SfLattice L)
{
    const int V = make_g32(L.dims).V;
    const int nvb = (int)virtual_blocks(V);
    for (int vb = blockIdx.x; vb < nvb; vb += gridDim.x) links_block(L, V, vb);
}

__global__ void __launch_bounds__(kBlock) links_fx_batched(const __grid_constant__ SfBatch B)
{
    for (int64_t vb = next_virtual_block(B.counter + 2); vb < B.total;) {
        const unsigned long long next = claim_virtual_block(B.counter + 2);
        const SfLattice &L = B.e[batch_entry(B, vb)];
        links_block(L, make_g32(L.dims).V, (int)(vb - L.vb_begin));
        vb = publish_virtual_block(next);
    }
}

// ---------------------------------------------------------------- staples

// op_a(a) op_b(b), rows 0 and 1.
template <int FA, int FB> __device__ __forceinline__ FLimbs fx_mul_top2(const FLimbs &a, const FLimbs &b)
{
    FLimbAcc y;
    fx_zero(y);
    fx_mul_acc<FA, FB, 2>(y, a, b);
    return fx_round<FA == FB ? 1 : -1, 2>(y);
}

// Staple plane `plane` of site x in floating point, from the stored links.
__device__ __forceinline__ Mat<double> direct_staple(const double *links, const G32 &g, const Coord &c, int x, int plane)
{
    const int mu = plane / 6, j = plane - 6 * mu, nu = (mu + 1 + (j >> 1)) & 3;
    const int64_t V = g.V;
    const int xm = x + step32(g, c, mu, 1);
    Mat<double> s;
    if ((j & 1) == 0) {
        const int vp = step32(g, c, nu, 1);
        const Mat<double> t = mul<N, D>(load_link(links, V, nu, xm), load_link(links, V, mu, x + vp));
        s = mul_top2<N, D>(t, load_link(links, V, nu, x));
    } else {
        const int vm = step32(g, c, nu, -1);
        const Mat<double> t = mul<D, D>(load_link(links, V, nu, xm + vm), load_link(links, V, mu, x + vm));
        s = mul_top2<N, N>(t, load_link(links, V, nu, x + vm));
    }
    rebuild_row2(s);
    return s;
}

// Staples j0 to j1 - 1 of direction mu at site x in floating point.
__device__ __noinline__ void staples_floating(const SfLattice &L, int x, int mu, int j0, int j1)
{
    const G32 g = make_g32(L.dims);
    const Coord c = coord32(g, L.div, x);
    const FxPlanes sf = fx_planes(L);
#pragma unroll 1
    for (int j = j0; j < j1; ++j)
        sf.store(sf.at(x), mu * 6 + j, direct_staple(static_cast<const double *>(L.links), g, c, x, mu * 6 + j));
}

// Staples j0 to j1 - 1 of each direction.
__device__ __forceinline__ void staples_block(const SfLattice &L, const G32 &g, int vb, int j0, int j1)
{
    const int mu = (int)(threadIdx.x >> 5);
    const int x = vb * 32 + (int)(threadIdx.x & 31);
    const bool fl = floating(L);
    if (x >= g.V) return;
    if (fl) return staples_floating(L, x, mu, j0, j1);
    const Coord c = coord32(g, L.div, x);
    const FxPlanes sf = fx_planes(L);
    const int xm = x + step32(g, c, mu, 1); // x + mu
    char *out = sf.at(x);
#pragma unroll 1
    for (int j = j0; j < j1; ++j) {
        const int nu = (mu + 1 + (j >> 1)) & 3;
        FLimbs s;
        bool bad;
        if ((j & 1) == 0) {
            // b = +nu:  U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
            const FLimbs a = sf.limbs(sf.at(xm), kLinkPlane + nu),
                         b = sf.limbs(sf.at(x + step32(g, c, nu, 1)), kLinkPlane + mu), d = sf.limbs(sf.at(x), kLinkPlane + nu);
            bad = fx_poisoned(a) || fx_poisoned(b) || fx_poisoned(d);
            s = fx_mul_top2<N, D>(fx_mul_top2<N, D>(a, b), d);
        } else {
            // b = -nu:  U_nu(x+mu-nu)^dag U_mu(x-nu)^dag U_nu(x-nu)
            const int vm = step32(g, c, nu, -1);
            const FLimbs a = sf.limbs(sf.at(xm + vm), kLinkPlane + nu), b = sf.limbs(sf.at(x + vm), kLinkPlane + mu),
                         d = sf.limbs(sf.at(x + vm), kLinkPlane + nu);
            bad = fx_poisoned(a) || fx_poisoned(b) || fx_poisoned(d);
            s = fx_mul_top2<N, N>(fx_mul_top2<D, D>(a, b), d);
        }
        fx_row2(s);
        if (bad) s.rh[0][0] = kPoison;
        sf.store<true>(out, mu * 6 + j, fx_remainder(s));
    }
}

__global__ void __launch_bounds__(kBlock) staples_fx(const __grid_constant__ SfLattice L)
{
    const G32 g = make_g32(L.dims);
    const int nvb = (int)virtual_blocks(g.V);
    if (L.split) { // one staple of each direction per block
        const int vb = blockIdx.x / 6, j = blockIdx.x - 6 * vb;
        staples_block(L, g, vb, j, j + 1);
        return;
    }
    for (int vb = blockIdx.x; vb < nvb; vb += gridDim.x) staples_block(L, g, vb, 0, 6);
}

__global__ void __launch_bounds__(kBlock) staples_fx_batched(const __grid_constant__ SfBatch B)
{
    for (int64_t vb = next_virtual_block(B.counter); vb < B.total;) {
        const unsigned long long next = claim_virtual_block(B.counter);
        const SfLattice &L = B.e[batch_entry(B, vb)];
        staples_block(L, make_g32(L.dims), (int)(vb - L.vb_begin), 0, 6);
        vb = publish_virtual_block(next);
    }
}

// ------------------------------------------------------------------ force

// Staples computed from the stored links in floating point.
struct DirectStaples {
    const double *links;
    const G32 *g;
    const DivMagic *div;

    __device__ __forceinline__ int at(int n) const { return n; }

    __device__ Mat<double> load(int x, int plane) const
    {
        return direct_staple(links, *g, coord32(*g, div, x), x, plane);
    }
};

// Staples from FP64 planes.
struct FloatingStaples {
    FxPlanes sf;

    __device__ __forceinline__ const char *at(int n) const { return sf.at(n); }
    __device__ __forceinline__ Mat<double> load(const char *r, int plane) const { return sf.floating(r, plane); }
};

template <bool ACTION>
__device__ __noinline__ double force_link_floating(const SfLattice &L, const KernelScalars &sc, int k, int rho)
{
    const G32 g = make_g32(L.dims);
    const Coord c = coord32(g, L.div, k);
    const LatticeSites si{&g, &c, k};
    const DirectStaples sf{static_cast<const double *>(L.links), &g, L.div};
    return force_link<double, ACTION, false, true>(L, sc, g, sf, si, c, k, rho);
}

// Of a lattice in floating point.
template <bool ACTION>
__device__ __noinline__ double force_link_of_planes(const SfLattice &L, const KernelScalars &sc, int k, int rho)
{
    const G32 g = make_g32(L.dims);
    const Coord c = coord32(g, L.div, k);
    const LatticeSites si{&g, &c, k};
    return force_link<double, ACTION, false, true>(L, sc, g, FloatingStaples{fx_planes(L)}, si, c, k, rho);
}

// Where a group of products (fx_group) of a link reads: its left factors at
// at_a, its right ones at at_b, the link that closes it at at_x.
struct FxGroup {
    const char *at_a, *at_b, *at_x;
    int base, id, nud;
    bool chain, neg;
};

__device__ __forceinline__ FxGroup fx_group_of(const FxPlanes &sf, const G32 &g, const Coord &c, int rho, int k, int grp)
{
    FxGroup r;
    r.base = rho * 6;
    r.chain = grp < 2;
    r.neg = grp >= 5;
    r.id = r.chain ? 0 : (r.neg ? grp - 5 : grp - 2);
    r.nud = r.chain ? rho : (rho + 1 + r.id) & 3;
    const int kp = k + step32(g, c, rho, 1);
    const int dk = step32(g, c, r.nud, r.neg || grp == 1 ? -1 : 1); // k + dk: k+rho, k-rho, k+d
    const char *at_k = sf.at(k), *at_d = sf.at(k + dk);
    r.at_a = grp == 1 ? at_k : at_d;
    r.at_b = r.chain ? (grp == 0 ? at_k : at_d) : (r.neg ? at_d : at_k);
    r.at_x = grp == 1 ? at_d : sf.at(r.neg ? kp + dk : kp);
    return r;
}

// The planes of product q of a group.
__device__ __forceinline__ void fx_product_planes(const FxGroup &r, int rho, int q, int &pa, int &pb)
{
    pa = pb = r.base + q;
    if (!r.chain) {
        const int ib = q < 2 ? (r.id == 0 ? 1 : 0) : (r.id == 2 ? 1 : 2);
        const int nub = (rho + 1 + ib) & 3;
        pa = r.base + 2 * ib + (q & 1);
        pb = r.nud * 6 + 2 * ((nub - r.nud - 1) & 3) + (q & 1);
        if (q == 4) {
            pa = r.base + 2 * r.id + (r.neg ? 1 : 0);
            pb = kLinkPlane + r.nud;
        }
    }
}

// A thread's words of shared memory: the two factors copied ahead and the
// total of the groups.
constexpr int kAheadWords = 18;
constexpr int kForceShared = (kAheadWords + 9) * kBlock * 16; // bytes of a block

// Starts the copy of a matrix; of the factors of product q.
__device__ __forceinline__ void fx_copy(float4 *dst, const FxPlanes &sf, const char *at, int plane)
{
    const float4 *p = reinterpret_cast<const float4 *>(sf.ptr(at, plane));
#pragma unroll
    for (int e = 0; e < 9; ++e) copy_async(dst + e * kBlock, p + e * FxPlanes::S);
}

__device__ __forceinline__ void fx_fetch(float4 *slot, const FxPlanes &sf, const FxGroup &r, int rho, int q)
{
    int pa, pb;
    fx_product_planes(r, rho, q, pa, pb);
    fx_copy(slot, sf, r.at_a, pa);
    fx_copy(slot + 9 * kBlock, sf, r.at_b, pb);
    copies_commit();
}

// Every sum of products that a link closes is a group: group 0
// F sum_b S_b(k+rho) S_b(k), group 1 sum_b S_b(k) S_b(k-rho) E, groups 2..7
// B_d [ alpha sum_{b perp rho, d} S_b(k+d) S^{(d)}_b(k) + beta S_d(k+d) A_d^dag ]
// for the six directions d.  One piece of code for all of them, and not one
// for each group and sign: a product is about 400 instructions, and with
// eleven copies of it the instruction cache missed (1.5 stalled cycles per
// instruction).  z: the nine entries of the sum, units 2^-56.
// AHEAD: every factor is copied into the thread's own words of shared memory
// (slot) while the product before it is computed, over the end of the group
// into the next; the first product of group 0 by the caller.  With 8 warps an
// SM at 255 registers there is nothing else to hide the reads behind: 24^3x48
// 5.90 -> 5.56 ms, 12^3x24 440 -> 409 us (all factors in L1: 5.03).
template <bool AHEAD>
__device__ __forceinline__ void fx_group(longlong2 z[9], bool &bad, const FxPlanes &sf, const FxScalars &fx, const G32 &g,
                                         const Coord &c, int rho, int k, int grp, float4 *slot)
{
    const FxGroup r = fx_group_of(sf, g, c, rho, k, grp);
    FAcc acc;
    fx_zero(acc);
    const int n = r.chain ? 6 : 5;
#pragma unroll 1
    for (int q = 0; q < n; ++q) {
        int pa, pb;
        fx_product_planes(r, rho, q, pa, pb);
        bool dag = r.neg;
        if (!r.chain && q == 4) { // the rectangle along d, onto alpha times the cubes
            const FMat y = fx_round<32>(acc); // up to 4, units 2^-28
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    const FSum re = fx_scaled(fx.alpha, y.rh[i][j], y.rl[i][j]);
                    const FSum im = fx_scaled(fx.alpha, y.ih[i][j], y.il[i][j]);
                    acc.h1[i][j] = 4 * re.v;
                    acc.h2[i][j] = 0;
                    acc.h3[i][j] = 4 * (re.v + im.v);
                    acc.cr[i][j] = 4.f * re.c;
                    acc.ci[i][j] = 4.f * im.c;
                }
            dag = !r.neg;
        }
        FMat a, b;
        if constexpr (AHEAD) {
            copies_wait<0>();
            const int4 *w = reinterpret_cast<const int4 *>(slot);
            a = fx_mat_at<kBlock, false>(w);
            b = fx_form_at<kBlock, false>(w + 9 * kBlock, pb >= kLinkPlane, dag);
            if (q + 1 < n) fx_fetch(slot, sf, r, rho, q + 1);
            else {
                fx_copy(slot, sf, r.at_x, kLinkPlane + r.nud);
                copies_commit();
            }
        } else {
            a = sf.mat(r.at_a, pa);
            b = sf.form(r.at_b, pb, pb >= kLinkPlane, dag);
        }
        bad = bad || fx_poisoned(a) || fx_poisoned(b);
        if (fx.use_beta && q == 4 && !r.chain) a = fx_scaled(fx.beta, a);
        fx_mul_acc<N, N>(acc, a, b);
    }
    FMat y = fx_round<33>(acc); // up to 6, units 2^-27
    if (fx.use_beta && r.chain) y = fx_scaled(fx.beta, y);
    FMat x;
    if constexpr (AHEAD) {
        copies_wait<0>();
        x = fx_form_at<kBlock, false>(reinterpret_cast<const int4 *>(slot), true, r.neg);
        if (grp < 7) fx_fetch(slot, sf, fx_group_of(sf, g, c, rho, k, grp + 1), rho, 0);
    } else {
        x = sf.form(r.at_x, kLinkPlane + r.nud, true, r.neg);
    }
    bad = bad || fx_poisoned(x);
    if (grp == 1) {
        const FMat t = x;
        x = y;
        y = t;
    }
    fx_zero(acc);
    fx_mul_acc<N, N>(acc, x, y);
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        FSum re, im;
        fx_total<1>(acc, e / 3, e % 3, re, im);
        // units 2^-57; the FP32 part in units of 2^-54
        z[e] = make_longlong2((re.v >> 1) + 4ll * __float2int_rn(0.125f * re.c), (im.v >> 1) + 4ll * __float2int_rn(0.125f * im.c));
    }
}

// The force (and the fused momentum step) from the sum z_of(e) of the groups;
// returns the link's share of the action.
template <bool ACTION, typename Z>
__device__ __forceinline__ double fx_finish(const SfLattice &L, const KernelScalars &sc, const FxScalars &fx,
                                            const FxPlanes &sf, int64_t V, int rho, int k, bool bad, const Z &z_of)
{
    const int base = rho * 6;
    const FLimbs u = sf.limbs(sf.at(k), kLinkPlane + rho);
    if (bad || fx_poisoned(u)) return force_link_floating<ACTION>(L, sc, k, rho);

    // The plaquette sum, t / m and U t / m decide the accuracy of the result:
    // whole limbs.
    long long pr[9], pi[9]; // plaquette sum, up to 6, units 2^-58
#pragma unroll
    for (int e = 0; e < 9; ++e) pr[e] = pi[e] = 0;
#pragma unroll 1
    for (int jj = 0; jj < 6; ++jj) {
        const FMat s = sf.mat(sf.at(k), base + jj);
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            pr[e] = mad_wide(s.rh[e / 3][e % 3], 1 << 28, pr[e] + __float2int_rn(0x1p28f * s.rl[e / 3][e % 3]));
            pi[e] = mad_wide(s.ih[e / 3][e % 3], 1 << 28, pi[e] + __float2int_rn(0x1p28f * s.il[e / 3][e % 3]));
        }
    }
    FLimbs t; // t / m, up to 4, units 2^-28 and 2^-56
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        const int i = e / 3, j = e % 3;
        const longlong2 v = z_of(e);
        const auto sum = [&](long long zval, long long p, int &th, int &tl) {
            int zh;
            float zl;
            fx_split<31>(FSum{zval, 0.f}, zh, zl);     // up to 42, units 2^-25
            const int p32 = (int)p;
            const int ph = (int)(p >> 32) + (int)((unsigned)p32 >> 31);
            // in units 2^-60: pl times p = ph 2^32 + p32, and z times the rest
            const long long x = 16 * mad_wide(fx.plh, ph, 0) + (mad_wide(fx.plh, p32, 0) >> 28) +
                                (mad_wide(fx.pll, ph, 0) >> 24) + 32 * mad_wide(fx.zh, zh, 0) +
                                (mad_wide(fx.zl, zh, 0) >> 23) + 16ll * __float2int_rn(2.f * (float)fx.zh * zl);
            const long long y = (x + 8) >> 4;
            th = (int)((y + (1ll << 27)) >> 28);
            tl = (int)((unsigned)y - ((unsigned)th << 28));
        };
        sum(v.x, pr[e], t.rh[i][j], t.rl[i][j]);
        sum(v.y, pi[e], t.ih[i][j], t.il[i][j]);
    }
    FLimbAcc acc;
    fx_zero(acc);
    fx_mul_acc<N, N>(acc, u, t);
    long long re[3][3], im[3][3]; // U t / m, units 2^-58
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) fx_total<1>(acc, i, j, re[i][j], im[i][j]);
    // f = -(beta/6) Im tr(lambda_a U t) (ta_components)
    const double s = -sc.d[SC_BETA6] * fx.m * 0x1p-58;
    double f[8];
    f[0] = s * (double)(im[0][1] + im[1][0]);
    f[1] = s * (double)(re[0][1] - re[1][0]);
    f[2] = s * (double)(im[0][0] - im[1][1]);
    f[3] = s * (double)(im[0][2] + im[2][0]);
    f[4] = s * (double)(re[0][2] - re[2][0]);
    f[5] = s * (double)(im[1][2] + im[2][1]);
    f[6] = s * (double)(re[1][2] - re[2][1]);
    f[7] = s * 0.57735026918962576451 * (double)(im[0][0] + im[1][1] - 2 * im[2][2]);
    if (L.force != nullptr) store_algebra(static_cast<double *>(L.force), V, rho, k, f);
    if (L.mom != nullptr) {
        double *mom = static_cast<double *>(L.mom);
        double p[8];
        load_algebra(mom, V, rho, k, p);
        const double dt = sc.d[SC_DT];
#pragma unroll
        for (int q = 0; q < 8; ++q) p[q] = fma(dt, f[q], p[q]);
        store_algebra(mom, V, rho, k, p);
    }
    if constexpr (ACTION) {
        // the differences from unit links, exact; share = 3 (1.5 c_plaq + 3
        // c_rect + 4 c_cube) - Re tr(U t) / 6 - (c_plaq / 12) Re tr(U Pl)
        const double d_t = (double)(fx.tr0 - (re[0][0] + re[1][1] + re[2][2]));
        FLimbs p; // plaquette sum, units 2^-27 and 2^-55
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            fx_limbs<3>(pr[e], p.rh[e / 3][e % 3], p.rl[e / 3][e % 3]);
            fx_limbs<3>(pi[e], p.ih[e / 3][e % 3], p.il[e / 3][e % 3]);
        }
        const double d_pl = (double)((18ll << 57) - fx_re_trace(u, p));
        return fma(sc.d[SC_ACTPL] * 0x1p-57, d_pl, fx.m * 0x1p-58 / 6.0 * d_t);
    }
    return 0.0;
}

// The four directions of 32 sites, one per warp.  The total of the groups
// stays in shared memory, out of the registers' way.
template <bool ACTION>
__device__ __forceinline__ double fx_force_block(const SfLattice &L, const KernelScalars &sc, const FxScalars &fx,
                                                 const G32 &g, const Sweep &sw, int vb)
{
    extern __shared__ float4 ahead_s[];
    float4 *slot = ahead_s + threadIdx.x;
    longlong2 *zs = reinterpret_cast<longlong2 *>(ahead_s + kAheadWords * kBlock) + threadIdx.x;
    const int rho = (int)(threadIdx.x >> 5);
    const int j = vb * 32 + (int)(threadIdx.x & 31);
    const bool fl = floating(L);
    if (j >= g.V) return 0.0;
    const Coord c = swept_site(sw, j);
    const int k = index32(g, c);
    if (fl) return force_link_of_planes<ACTION>(L, sc, k, rho);
    const FxPlanes sf = fx_planes(L);
    bool bad = false;
    fx_fetch(slot, sf, fx_group_of(sf, g, c, rho, k, 0), rho, 0);
#pragma unroll 1
    for (int grp = 0; grp < 8; ++grp) {
        longlong2 z[9];
        fx_group<true>(z, bad, sf, fx, g, c, rho, k, grp, slot);
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            if (grp > 0) {
                const longlong2 o = zs[e * kBlock];
                z[e].x += o.x;
                z[e].y += o.y;
            }
            zs[e * kBlock] = z[e];
        }
    }
    return fx_finish<ACTION>(L, sc, fx, sf, g.V, rho, k, bad, [&](int e) { return zs[e * kBlock]; });
}

// The partial sums of virtual block vb: four for a split lattice, so that the
// action does not depend on which kernel made them.
__device__ __forceinline__ void fx_store_partials(const SfLattice &L, int vb, double share)
{
    if (L.split) {
        const double s = warp_sum(share);
        if ((threadIdx.x & 31) == 0) L.partials[vb * 4 + (threadIdx.x >> 5)] = s;
    } else {
        const double s = block_sum(share);
        if (threadIdx.x == 0) L.partials[vb] = s;
    }
}

template <bool ACTION>
__global__ void __launch_bounds__(kBlock, 2)
    force_fx(const __grid_constant__ SfLattice L, const __grid_constant__ KernelScalars sc,
             const __grid_constant__ FxScalars fx)
{
    const G32 g = make_g32(L.dims);
    const Sweep sw = make_sweep(L, g);
    const int nvb = (int)virtual_blocks(g.V);
    for (int vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
        const double acc = fx_force_block<ACTION>(L, sc, fx, g, sw, vb);
        if constexpr (ACTION) fx_store_partials(L, vb, acc);
    }
}

// Split lattices: direction rho of 32 sites, a group on each of eight warps,
// the first adding them up (whole numbers: the sum of force_fx to the bit).
constexpr int kSplitBlock = 256;

template <bool ACTION>
__global__ void __launch_bounds__(kSplitBlock, 1)
    force_fx_split(const __grid_constant__ SfLattice L, const __grid_constant__ KernelScalars sc,
                   const __grid_constant__ FxScalars fx)
{
    __shared__ longlong2 z_s[7][9][32];
    __shared__ unsigned bad_s[8];
    const G32 g = make_g32(L.dims);
    const Sweep sw = make_sweep(L, g);
    const int vb = (int)(blockIdx.x >> 2), rho = (int)(blockIdx.x & 3);
    const int grp = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
    const int j = vb * 32 + lane;
    const Coord c = swept_site(sw, j < g.V ? j : g.V - 1);
    const int k = index32(g, c);
    const FxPlanes sf = fx_planes(L);
    if (floating(L)) {
        if (grp > 0) return;
        double share = j < g.V ? force_link_of_planes<ACTION>(L, sc, k, rho) : 0.0;
        if constexpr (ACTION) {
            share = warp_sum(share);
            if (lane == 0) L.partials[vb * 4 + rho] = share;
        }
        return;
    }
    longlong2 z[9];
    bool bad = false;
    fx_group<false>(z, bad, sf, fx, g, c, rho, k, grp, nullptr);
    const unsigned marks = __ballot_sync(0xffffffffu, bad);
    if (lane == 0) bad_s[grp] = marks;
    if (grp > 0) {
#pragma unroll
        for (int e = 0; e < 9; ++e) z_s[grp - 1][e][lane] = z[e];
    }
    __syncthreads();
    if (grp > 0) return;
#pragma unroll
    for (int p = 1; p < 8; ++p) bad = bad || (bad_s[p] >> lane & 1);
#pragma unroll 1
    for (int p = 0; p < 7; ++p)
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const longlong2 o = z_s[p][e][lane];
            z[e].x += o.x;
            z[e].y += o.y;
        }
    double share = 0.0;
    if (j < g.V) share = fx_finish<ACTION>(L, sc, fx, sf, g.V, rho, k, bad, [&](int e) { return z[e]; });
    if constexpr (ACTION) {
        share = warp_sum(share);
        if (lane == 0) L.partials[vb * 4 + rho] = share;
    }
}

template <bool ACTION>
__global__ void __launch_bounds__(kBlock, 2)
    force_fx_batched(const __grid_constant__ SfBatch B, const __grid_constant__ KernelScalars sc,
                     const __grid_constant__ FxScalars fx)
{
    for (int64_t vb = next_virtual_block(B.counter + 1); vb < B.total;) {
        const unsigned long long next = claim_virtual_block(B.counter + 1);
        const SfLattice &L = B.e[batch_entry(B, vb)];
        const G32 g = make_g32(L.dims);
        const int v = (int)(vb - L.vb_begin);
        const double acc = fx_force_block<ACTION>(L, sc, fx, g, make_sweep(L, g), v);
        if constexpr (ACTION) fx_store_partials(L, v, acc);
        vb = publish_virtual_block(next);
    }
}

} // namespace

int fx_planes_count() { return kStaplePlanes + 4; }

cudaError_t launch_fx_passes(const SfLattice &L, const KernelScalars &sc, bool action, cudaStream_t st)
{
    const unsigned grid = grid_of(virtual_blocks((int64_t)L.dims[0] * L.dims[1] * L.dims[2] * L.dims[3]));
    const FxScalars fx = make_fx_scalars(sc);
    cudaError_t e = cudaSuccess;
    if (L.flag != nullptr) { // not in a lean workspace
        if (L.near == nullptr) e = cudaMemsetAsync(L.flag, 0, sizeof *L.flag, st);
        if (e != cudaSuccess) return e;
        links_fx<<<grid, kBlock, 0, st>>>(L);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    staples_fx<<<L.split ? 6 * grid : grid, kBlock, 0, st>>>(L);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (L.split) {
        if (action) force_fx_split<true><<<4 * grid, kSplitBlock, 0, st>>>(L, sc, fx);
        else force_fx_split<false><<<4 * grid, kSplitBlock, 0, st>>>(L, sc, fx);
        return cudaGetLastError();
    }
    const auto k = action ? force_fx<true> : force_fx<false>;
    e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kForceShared);
    if (e != cudaSuccess) return e;
    k<<<grid, kBlock, kForceShared, st>>>(L, sc, fx);
    return cudaGetLastError();
}

cudaError_t launch_fx_passes_batched(const SfBatch &B, const KernelScalars &sc, bool action, cudaStream_t st)
{
    const FxScalars fx = make_fx_scalars(sc);
    cudaError_t e = cudaSuccess;
    if (B.e[0].flag != nullptr) { // not in a lean workspace
        links_fx_batched<<<persistent_grid(links_fx_batched, 0, B.total), kBlock, 0, st>>>(B);
        e = cudaGetLastError();
        if (e != cudaSuccess) return e;
    }
    staples_fx_batched<<<persistent_grid(staples_fx_batched, 1, B.total), kBlock, 0, st>>>(B);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (action) {
        auto k = force_fx_batched<true>;
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kForceShared);
        if (e != cudaSuccess) return e;
        k<<<persistent_grid(k, 2, B.total), kBlock, kForceShared, st>>>(B, sc, fx);
    } else {
        auto k = force_fx_batched<false>;
        e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, kForceShared);
        if (e != cudaSuccess) return e;
        k<<<persistent_grid(k, 3, B.total), kBlock, kForceShared, st>>>(B, sc, fx);
    }
    return cudaGetLastError();
}

} // namespace lqcd
