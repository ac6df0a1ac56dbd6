// Gauge force of the one-loop Symanzik action for FP64 fields: the
// staple-field algorithm of force_sf.cu (same formulas, traversal and action)
// in the fixed-point arithmetic of fixed.cuh, three passes:
//   links_fx     the links as limbs (all three rows), planes 24..27 of the
//                workspace: every link is read about 18 times by the next two
//                passes, so it is converted (and checked) once
//   staples_fx   the 24 plaquette staples of every site
//   force_fx     the force (momentum step, action) of every link
//
// What bounds it.  In FP64 the force is 7.3 k FMA per link on a pipe that
// issues 2 a clock and SM (98 ms at 32^3x64 for the pipe alone); here it is
// three integer multiply-adds each on the pipe that issues 64, and the bytes
// (144 per staple in either form) start to count.
//
// A thread that reads a marked matrix (a link that is not finite or not
// within 1e-3 of SU(3), or a staple of one) computes its staple or force in
// floating point from the stored links instead.
#include "sf_common.cuh"
#include "fixed.cuh"

namespace lqcd {

namespace {

constexpr int kLinkPlane = kStaplePlanes; // planes 24..27: the links
using FxBlock = FullBlock<double>;        // 9 lanes of 16 bytes: one complex entry each

struct FxPlanes {
    char *base;
    int64_t plane_bytes;

    __device__ __forceinline__ char *at(int n) const
    {
        return base + (int64_t)(n >> 5) * FxBlock::BYTES + (n & 31) * 16;
    }

    __device__ __forceinline__ FMat load(const char *r, int plane) const
    {
        const int4 *p = reinterpret_cast<const int4 *>(r + (int64_t)plane * plane_bytes);
        FMat u;
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const int4 v = __ldg(p + e * (FxBlock::LANE / 16));
            u.rh[e / 3][e % 3] = v.x;
            u.rl[e / 3][e % 3] = v.y;
            u.ih[e / 3][e % 3] = v.z;
            u.il[e / 3][e % 3] = v.w;
        }
        return u;
    }

    // The matrix or (dag) its dagger, chosen at run time: the off-diagonal
    // entries are read from their mirrored places.
    __device__ __forceinline__ FMat load_form(const char *r, int plane, bool dag) const
    {
        const int4 *p = reinterpret_cast<const int4 *>(r + (int64_t)plane * plane_bytes);
        constexpr int S = FxBlock::LANE / 16;
        const int o = dag ? 2 * S : 0, m = dag ? -1 : 0;
        const int4 *up = p + o, *dn = p - o, *up2 = up + o, *dn2 = dn - o;
        const int4 v[9] = {__ldg(p),           __ldg(up + S),      __ldg(up2 + 2 * S), __ldg(dn + 3 * S), __ldg(p + 4 * S),
                           __ldg(up + 5 * S),  __ldg(dn2 + 6 * S), __ldg(dn + 7 * S),  __ldg(p + 8 * S)};
        FMat u;
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            u.rh[e / 3][e % 3] = v[e].x;
            u.rl[e / 3][e % 3] = v[e].y;
            u.ih[e / 3][e % 3] = (v[e].z ^ m) - m;
            u.il[e / 3][e % 3] = (v[e].w ^ m) - m;
        }
        return u;
    }

    template <bool STREAM> __device__ __forceinline__ void store(char *r, int plane, const FMat &u) const
    {
        int4 *p = reinterpret_cast<int4 *>(r + (int64_t)plane * plane_bytes);
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const int4 v = make_int4(u.rh[e / 3][e % 3], u.rl[e / 3][e % 3], u.ih[e / 3][e % 3], u.il[e / 3][e % 3]);
            if constexpr (STREAM) __stcs(p + e * (FxBlock::LANE / 16), v);
            else p[e * (FxBlock::LANE / 16)] = v;
        }
    }
};

__device__ __forceinline__ FxPlanes fx_planes(const SfLattice &L)
{
    return FxPlanes{static_cast<char *>(L.staples), L.plane_bytes};
}

// Coefficients for the fixed-point sums.  With t = c_plaq Pl + c_rect Rc +
// c_cube Cb and z the larger of c_rect, c_cube in modulus, m the larger of
// c_plaq, z:
//     t / m = pl Pl + z (beta Rc + alpha Cb),
// every scalar at most 1 in modulus (use_beta: beta is not 1).
struct FxScalars {
    FScalar pl, z, alpha, beta;
    int use_beta;
    double m;
};

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
    f.m = mod(cp) > mod(z) ? mod(cp) : mod(z);
    if (f.m == 0.0) f.m = 1.0;
    f.pl = fx_scalar(cp / f.m);
    f.z = fx_scalar(z / f.m);
    f.alpha = fx_scalar(alpha);
    f.beta = fx_scalar(beta);
    f.use_beta = beta != 1.0;
    return f;
}

// ------------------------------------------------------------------ links

__device__ __forceinline__ void links_block(const SfLattice &L, int V, int vb)
{
    const int mu = (int)(threadIdx.x >> 5);
    const int x = vb * 32 + (int)(threadIdx.x & 31);
    if (x >= V) return;
    const double2 *p = static_cast<const double2 *>(L.links) + (int64_t)mu * 6 * V + x;
    double r[12];
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        const double2 v = __ldg(p + (int64_t)q * V);
        r[2 * q] = v.x;
        r[2 * q + 1] = v.y;
    }
    const FxPlanes sf = fx_planes(L);
    sf.store<false>(sf.at(x), kLinkPlane + mu, fx_from_rows(r));
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

// t <- op_a(a) op_b(b), rows 0 and 1 rounded to 2^-58.
template <int FA, int FB> __device__ __forceinline__ FMat fx_mul_top2(const FMat &a, const FMat &b)
{
    FAcc y;
    fx_zero(y);
    fx_mul_acc<FA, FB, 2>(y, a, b);
    return fx_round<0, FA == FB ? 1 : -1, 2>(y);
}

__device__ __forceinline__ void staples_block(const SfLattice &L, const G32 &g, int vb)
{
    const int mu = (int)(threadIdx.x >> 5);
    const int x = vb * 32 + (int)(threadIdx.x & 31);
    if (x >= g.V) return;
    const Coord c = coord32(g, L.div, x);
    const FxPlanes sf = fx_planes(L);
    const int xm = x + step32(g, c, mu, 1); // x + mu
    char *out = sf.at(x);
#pragma unroll 1
    for (int iv = 0; iv < 3; ++iv) {
        const int nu = (mu + 1 + iv) & 3;
        const int vp = step32(g, c, nu, 1), vm = step32(g, c, nu, -1);
        const int pmu = kLinkPlane + mu, pnu = kLinkPlane + nu;
        {
            // b = +nu:  U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
            const FMat a = sf.load(sf.at(xm), pnu), b = sf.load(sf.at(x + vp), pmu), d = sf.load(sf.at(x), pnu);
            FMat s = fx_mul_top2<N, D>(fx_mul_top2<N, D>(a, b), d);
            fx_row2(s);
            if (fx_poisoned(a) || fx_poisoned(b) || fx_poisoned(d)) s.rh[0][0] = kPoison;
            sf.store<true>(out, mu * 6 + 2 * iv, s);
        }
        {
            // b = -nu:  U_nu(x+mu-nu)^dag U_mu(x-nu)^dag U_nu(x-nu)
            const FMat a = sf.load(sf.at(xm + vm), pnu), b = sf.load(sf.at(x + vm), pmu), d = sf.load(sf.at(x + vm), pnu);
            FMat s = fx_mul_top2<N, N>(fx_mul_top2<D, D>(a, b), d);
            fx_row2(s);
            if (fx_poisoned(a) || fx_poisoned(b) || fx_poisoned(d)) s.rh[0][0] = kPoison;
            sf.store<true>(out, mu * 6 + 2 * iv + 1, s);
        }
    }
}

__global__ void __launch_bounds__(kBlock) staples_fx(const __grid_constant__ SfLattice L)
{
    const G32 g = make_g32(L.dims);
    const int nvb = (int)virtual_blocks(g.V);
    for (int vb = blockIdx.x; vb < nvb; vb += gridDim.x) staples_block(L, g, vb);
}

__global__ void __launch_bounds__(kBlock) staples_fx_batched(const __grid_constant__ SfBatch B)
{
    for (int64_t vb = next_virtual_block(B.counter); vb < B.total;) {
        const unsigned long long next = claim_virtual_block(B.counter);
        const SfLattice &L = B.e[batch_entry(B, vb)];
        staples_block(L, make_g32(L.dims), (int)(vb - L.vb_begin));
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
        const int mu = plane / 6, j = plane - 6 * mu, nu = (mu + 1 + (j >> 1)) & 3;
        const Coord c = coord32(*g, div, x);
        const int64_t V = g->V;
        const int xm = x + step32(*g, c, mu, 1);
        Mat<double> s;
        if ((j & 1) == 0) {
            const int vp = step32(*g, c, nu, 1);
            const Mat<double> t = mul<N, D>(load_link(links, V, nu, xm), load_link(links, V, mu, x + vp));
            s = mul_top2<N, D>(t, load_link(links, V, nu, x));
        } else {
            const int vm = step32(*g, c, nu, -1);
            const Mat<double> t = mul<D, D>(load_link(links, V, nu, xm + vm), load_link(links, V, mu, x + vm));
            s = mul_top2<N, N>(t, load_link(links, V, nu, x + vm));
        }
        rebuild_row2(s);
        return s;
    }
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

// Force (and the fused momentum step) on the link (k, rho); returns its
// share of the action (force_link of sf_common.cuh in fixed point).
//
// Every sum of products that a link closes is a group of one loop: group 0
// F sum_b S_b(k+rho) S_b(k), group 1 sum_b S_b(k) S_b(k-rho) E, groups 2..7
// B_d [ alpha sum_{b perp rho, d} S_b(k+d) S^{(d)}_b(k) + beta S_d(k+d) A_d^dag ]
// for the six directions d.  One loop, and not a piece of code for each group
// and sign: a product is 280 instructions, and with eleven copies of it the
// instruction cache missed (1.5 stalled cycles per instruction).  The sums
// take 108 registers of the 255 that two CTAs per SM leave, so the total z of
// the groups stays in shared memory.
template <bool ACTION>
__device__ __forceinline__ double fx_force_link(const SfLattice &L, const KernelScalars &sc, const FxScalars &fx,
                                                const G32 &g, const Coord &c, int k, int rho)
{
    __shared__ longlong2 z_s[9][kBlock]; // units 2^-56
    longlong2 *z = &z_s[0][threadIdx.x];
    const FxPlanes sf = fx_planes(L);
    const int64_t V = g.V;
    const int kp = k + step32(g, c, rho, 1);
    const int base = rho * 6;
    bool bad = false;

#pragma unroll 1
    for (int grp = 0; grp < 8; ++grp) {
        const bool chain = grp < 2, neg = grp >= 5;
        const int id = chain ? 0 : (neg ? grp - 5 : grp - 2);
        const int nud = chain ? rho : (rho + 1 + id) & 3;
        const int dk = step32(g, c, nud, neg || grp == 1 ? -1 : 1); // k + dk: k+rho, k-rho, k+d
        const char *at_k = sf.at(k), *at_d = sf.at(k + dk);
        const char *at_a = grp == 1 ? at_k : at_d;
        const char *at_b = chain ? (grp == 0 ? at_k : at_d) : (neg ? at_d : at_k);
        FAcc acc;
        fx_zero(acc);
        const int n = chain ? 6 : 5;
#pragma unroll 1
        for (int q = 0; q < n; ++q) {
            int pa = base + q, pb = base + q;
            bool dag = neg;
            if (!chain) {
                const int ib = q < 2 ? (id == 0 ? 1 : 0) : (id == 2 ? 1 : 2);
                const int nub = (rho + 1 + ib) & 3;
                pa = base + 2 * ib + (q & 1);
                pb = nud * 6 + 2 * ((nub - nud - 1) & 3) + (q & 1);
                if (q == 4) { // the rectangle along d, onto alpha times the cubes
                    const FMat y = fx_round<2>(acc); // up to 4, units 2^-56
                    const FInt w = fx_scaled(fx.alpha, y);
                    fx_zero(acc);
#pragma unroll
                    for (int i = 0; i < 3; ++i)
#pragma unroll
                        for (int j = 0; j < 3; ++j) {
                            acc.h1[i][j] = 4 * w.re[i][j];
                            acc.h3[i][j] = 4 * (w.re[i][j] + w.im[i][j]);
                        }
                    pa = base + 2 * id + (neg ? 1 : 0);
                    pb = kLinkPlane + nud;
                    dag = !neg;
                }
            }
            FMat a = sf.load(at_a, pa);
            const FMat b = sf.load_form(at_b, pb, dag);
            bad = bad || fx_poisoned(a) || fx_poisoned(b);
            if (fx.use_beta && q == 4 && !chain) a = fx_round<0>(fx_scaled(fx.beta, a));
            fx_mul_acc<N, N>(acc, a, b);
        }
        FMat y = fx_round<2>(acc);
        if (fx.use_beta && chain) y = fx_round<0>(fx_scaled(fx.beta, y));
        FMat x = sf.load_form(grp == 1 ? at_d : sf.at(neg ? kp + dk : kp), kLinkPlane + nud, neg);
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
            longlong2 s;
            fx_value_of<1>(acc, e / 3, e % 3, s.x, s.y);
            if (grp > 0) {
                const longlong2 o = z[e * kBlock];
                s.x += o.x;
                s.y += o.y;
            }
            z[e * kBlock] = s;
        }
    }

    const FMat u = sf.load(sf.at(k), kLinkPlane + rho);
    bad = bad || fx_poisoned(u);
    if (bad) return force_link_floating<ACTION>(L, sc, k, rho);

    FMat plm; // plaquette sum, units 2^-56
    {
        FInt pl;
#pragma unroll
        for (int e = 0; e < 9; ++e) pl.re[e / 3][e % 3] = pl.im[e / 3][e % 3] = 0;
#pragma unroll 1
        for (int jj = 0; jj < 6; ++jj) {
            const FMat s = sf.load(sf.at(k), base + jj);
#pragma unroll
            for (int i = 0; i < 3; ++i)
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    pl.re[i][j] = mad_wide(s.rh[i][j], 1 << kLimb, pl.re[i][j]) + s.rl[i][j];
                    pl.im[i][j] = mad_wide(s.ih[i][j], 1 << kLimb, pl.im[i][j]) + s.il[i][j];
                }
        }
        plm = fx_round<2>(pl);
    }
    FInt t;
#pragma unroll
    for (int e = 0; e < 9; ++e) {
        const longlong2 s = z[e * kBlock];
        t.re[e / 3][e % 3] = s.x;
        t.im[e / 3][e % 3] = s.y;
    }
    t = fx_scaled(fx.z, fx_round<3>(t)); // units 2^-53
    const FInt tp = fx_scaled(fx.pl, plm);
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            t.re[i][j] += (tp.re[i][j] + 4) >> 3;
            t.im[i][j] += (tp.im[i][j] + 4) >> 3;
        }
    FAcc acc;
    fx_zero(acc);
    fx_mul_acc<N, N>(acc, u, fx_round<0>(t));
    FInt m;
#pragma unroll
    for (int i = 0; i < 3; ++i)
#pragma unroll
        for (int j = 0; j < 3; ++j) fx_value_of<1>(acc, i, j, m.re[i][j], m.im[i][j]);
    // f = -(beta/6) Im tr(lambda_a U t) (ta_components)
    const double s = -sc.d[SC_BETA6] * fx.m * 0x1p-53;
    double f[8];
    f[0] = s * (double)(m.im[0][1] + m.im[1][0]);
    f[1] = s * (double)(m.re[0][1] - m.re[1][0]);
    f[2] = s * (double)(m.im[0][0] - m.im[1][1]);
    f[3] = s * (double)(m.im[0][2] + m.im[2][0]);
    f[4] = s * (double)(m.re[0][2] - m.re[2][0]);
    f[5] = s * (double)(m.im[1][2] + m.im[2][1]);
    f[6] = s * (double)(m.re[1][2] - m.re[2][1]);
    f[7] = s * 0.57735026918962576451 * (double)(m.im[0][0] + m.im[1][1] - 2 * m.im[2][2]);
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
        const double tr_t = (double)(m.re[0][0] + m.re[1][1] + m.re[2][2]);
        const double tr_pl = (double)fx_re_trace(u, plm) * 0x1p-56;
        return fma(-sc.d[SC_ACTPL], tr_pl, fma(-fx.m * 0x1p-53 / 6.0, tr_t, sc.d[SC_ACT]));
    }
    return 0.0;
}

template <bool ACTION>
__device__ __forceinline__ double fx_force_block(const SfLattice &L, const KernelScalars &sc, const FxScalars &fx,
                                                 const G32 &g, const Sweep &sw, int vb)
{
    const int rho = (int)(threadIdx.x >> 5);
    const int j = vb * 32 + (int)(threadIdx.x & 31);
    if (j >= g.V) return 0.0;
    const Coord c = swept_site(sw, j);
    return fx_force_link<ACTION>(L, sc, fx, g, c, index32(g, c), rho);
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
        if constexpr (ACTION) {
            const double s = block_sum(acc);
            if (threadIdx.x == 0) L.partials[vb] = s;
        }
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
        const double acc = fx_force_block<ACTION>(L, sc, fx, g, make_sweep(L, g), (int)(vb - L.vb_begin));
        if constexpr (ACTION) {
            const double s = block_sum(acc);
            if (threadIdx.x == 0) L.partials[vb - L.vb_begin] = s;
        }
        vb = publish_virtual_block(next);
    }
}

} // namespace

int fx_planes_count() { return kStaplePlanes + 4; }

cudaError_t launch_fx_passes(const SfLattice &L, const KernelScalars &sc, bool action, cudaStream_t st)
{
    const unsigned grid = grid_of(virtual_blocks((int64_t)L.dims[0] * L.dims[1] * L.dims[2] * L.dims[3]));
    const FxScalars fx = make_fx_scalars(sc);
    links_fx<<<grid, kBlock, 0, st>>>(L);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    staples_fx<<<grid, kBlock, 0, st>>>(L);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (action) force_fx<true><<<grid, kBlock, 0, st>>>(L, sc, fx);
    else force_fx<false><<<grid, kBlock, 0, st>>>(L, sc, fx);
    return cudaGetLastError();
}

cudaError_t launch_fx_passes_batched(const SfBatch &B, const KernelScalars &sc, bool action, cudaStream_t st)
{
    const FxScalars fx = make_fx_scalars(sc);
    links_fx_batched<<<persistent_grid(links_fx_batched, 0, B.total), kBlock, 0, st>>>(B);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    staples_fx_batched<<<persistent_grid(staples_fx_batched, 1, B.total), kBlock, 0, st>>>(B);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    if (action) {
        auto k = force_fx_batched<true>;
        k<<<persistent_grid(k, 2, B.total), kBlock, 0, st>>>(B, sc, fx);
    } else {
        auto k = force_fx_batched<false>;
        k<<<persistent_grid(k, 3, B.total), kBlock, 0, st>>>(B, sc, fx);
    }
    return cudaGetLastError();
}

} // namespace lqcd
