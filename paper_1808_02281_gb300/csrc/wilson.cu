// Wilson fermion hopping term (Sec. III of the paper): the hopping operator
// calD of Eq. 18_7_17_4 applied to a spinor field, and the hopping-term force
// on every link, -i(B - C)_TA of Eqs. 18_1_29_19 to 18_7_17_30.
//
// Both are HBM-streaming kernels (a few hundred flops per 100-400 bytes), so
// the design is about bytes: spinors and links are read in 16-byte lanes,
// neighbours come from L1/L2 (a time slice of a 32^3 spinor field is 3 MB),
// and every (1 -+ gamma_mu) is applied as a spin projection to two colour
// vectors, so that each link multiplies two colour vectors instead of four.
#include "async_copy.cuh"
#include "fixed.cuh"
#include "sites.cuh"

namespace lqcd {
namespace {

// ------------------------------------------------------------ gamma basis

// Euclidean gamma matrices of the chiral basis, gamma_mu acting along
// direction mu = x, y, z, t.  Each has one non-zero entry per row:
// gamma_mu[alpha][gperm(mu, alpha)] = i^gcode(mu, alpha):
//   gamma_x: columns 3 2 1 0, entries  i  i -i -i
//   gamma_y: columns 3 2 1 0, entries -1  1  1 -1
//   gamma_z: columns 2 3 0 1, entries  i -i -i  i
//   gamma_t: columns 2 3 0 1, entries  1  1  1  1
__host__ __device__ constexpr int gperm(int mu, int alpha) { return mu < 2 ? 3 - alpha : alpha ^ 2; }

__host__ __device__ constexpr int gcode(int mu, int alpha)
{
    return mu == 0   ? (alpha < 2 ? 1 : 3)
           : mu == 1 ? ((alpha == 0 || alpha == 3) ? 2 : 0)
           : mu == 2 ? ((alpha == 0 || alpha == 3) ? 1 : 3)
                     : 0;
}

// (re, im) = i^K (xr + i xi)
template <int K, typename R> __device__ __forceinline__ void times_ipow(R &re, R &im, R xr, R xi)
{
    constexpr int k = K & 3;
    if constexpr (k == 0) {
        re = xr;
        im = xi;
    } else if constexpr (k == 1) {
        re = -xi;
        im = xr;
    } else if constexpr (k == 2) {
        re = -xr;
        im = -xi;
    } else {
        re = xi;
        im = -xr;
    }
}

template <typename R> struct Spinor {
    R re[4][3], im[4][3];
};
// Two colour vectors: the independent rows 0 and 1 of (1 + s gamma_mu) psi.
template <typename R> struct Half {
    R re[2][3], im[2][3];
};

// ------------------------------------------------------------ spinor I/O

template <typename R>
__device__ __forceinline__ Spinor<R> load_spinor(const R *__restrict__ x, int64_t V, int64_t n)
{
    using V4 = typename Vec<R>::type;
    constexpr int W = Vec<R>::W;
    const V4 *p = reinterpret_cast<const V4 *>(x) + n;
    R r[24];
#pragma unroll
    for (int q = 0; q < 24 / W; ++q) {
        const V4 v = __ldg(p + q * V);
        if constexpr (W == 4) {
            r[4 * q + 0] = v.x;
            r[4 * q + 1] = v.y;
            r[4 * q + 2] = v.z;
            r[4 * q + 3] = v.w;
        } else {
            r[2 * q + 0] = v.x;
            r[2 * q + 1] = v.y;
        }
    }
    Spinor<R> s;
#pragma unroll
    for (int al = 0; al < 4; ++al)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            s.re[al][a] = r[2 * (3 * al + a)];
            s.im[al][a] = r[2 * (3 * al + a) + 1];
        }
    return s;
}

template <typename R>
__device__ __forceinline__ void store_spinor(R *__restrict__ x, int64_t V, int64_t n, const Spinor<R> &s)
{
    using V4 = typename Vec<R>::type;
    constexpr int W = Vec<R>::W;
    V4 *p = reinterpret_cast<V4 *>(x) + n;
    R r[24];
#pragma unroll
    for (int al = 0; al < 4; ++al)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            r[2 * (3 * al + a)] = s.re[al][a];
            r[2 * (3 * al + a) + 1] = s.im[al][a];
        }
#pragma unroll
    for (int q = 0; q < 24 / W; ++q) {
        V4 v;
        if constexpr (W == 4) v = make_float4(r[4 * q], r[4 * q + 1], r[4 * q + 2], r[4 * q + 3]);
        else v = make_double2(r[2 * q], r[2 * q + 1]);
        p[q * V] = v;
    }
}

// ------------------------------------------------ spin projection algebra

// Rows 0 and 1 of (1 + S gamma_MU) x.  Rows gperm(MU, 0) and gperm(MU, 1) of
// the same spinor are S i^gcode(MU, gperm) times them (gamma_MU^2 = 1), so
// these two colour vectors carry all of it.
template <int MU, int S, int AL, typename R>
__device__ __forceinline__ void project_row(Half<R> &h, const Spinor<R> &x)
{
    constexpr int p = gperm(MU, AL);
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        R tr, ti;
        times_ipow<gcode(MU, AL) + (S < 0 ? 2 : 0)>(tr, ti, x.re[p][a], x.im[p][a]);
        h.re[AL][a] = x.re[AL][a] + tr;
        h.im[AL][a] = x.im[AL][a] + ti;
    }
}

template <int MU, int S, typename R> __device__ __forceinline__ Half<R> project(const Spinor<R> &x)
{
    Half<R> h;
    project_row<MU, S, 0>(h, x);
    project_row<MU, S, 1>(h, x);
    return h;
}

// acc += (1 + S gamma_MU) applied form of the half spinor g: rows 0, 1 are g,
// row gperm(MU, alpha) is S i^gcode(MU, gperm(MU, alpha)) g_alpha.
template <int MU, int S, typename R>
__device__ __forceinline__ void accumulate(Spinor<R> &acc, const Half<R> &g)
{
#pragma unroll
    for (int a = 0; a < 3; ++a) {
        R tr, ti;
        acc.re[0][a] += g.re[0][a];
        acc.im[0][a] += g.im[0][a];
        acc.re[1][a] += g.re[1][a];
        acc.im[1][a] += g.im[1][a];
        constexpr int p0 = gperm(MU, 0), p1 = gperm(MU, 1);
        times_ipow<gcode(MU, p0) + (S < 0 ? 2 : 0)>(tr, ti, g.re[0][a], g.im[0][a]);
        acc.re[p0][a] += tr;
        acc.im[p0][a] += ti;
        times_ipow<gcode(MU, p1) + (S < 0 ? 2 : 0)>(tr, ti, g.re[1][a], g.im[1][a]);
        acc.re[p1][a] += tr;
        acc.im[p1][a] += ti;
    }
}

// op(u) applied to both colour vectors of h (F = N: u, F = D: u^dagger).
template <int F, typename R> __device__ __forceinline__ Half<R> colour_mul(const Mat<R> &u, const Half<R> &h)
{
    Half<R> r;
#pragma unroll
    for (int al = 0; al < 2; ++al)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            R re = R(0), im = R(0);
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                re = fma(el_re<F>(u, a, b), h.re[al][b], re);
                re = fma(-el_im<F>(u, a, b), h.im[al][b], re);
                im = fma(el_re<F>(u, a, b), h.im[al][b], im);
                im = fma(el_im<F>(u, a, b), h.re[al][b], im);
            }
            r.re[al][a] = re;
            r.im[al][a] = im;
        }
    return r;
}

// m[b][a] += SIGN * sum_alpha p_alpha[b] conj(q_alpha[a]) over the two rows.
template <int SIGN, typename R>
__device__ __forceinline__ void outer_acc(Mat<R> &m, const Half<R> &p, const Half<R> &q)
{
#pragma unroll
    for (int b = 0; b < 3; ++b)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            R re = m.re[b][a], im = m.im[b][a];
#pragma unroll
            for (int al = 0; al < 2; ++al) {
                // p * conj(q) = (pr qr + pi qi) + i (pi qr - pr qi)
                re = fma(R(SIGN) * p.re[al][b], q.re[al][a], re);
                re = fma(R(SIGN) * p.im[al][b], q.im[al][a], re);
                im = fma(R(SIGN) * p.im[al][b], q.re[al][a], im);
                im = fma(-R(SIGN) * p.re[al][b], q.im[al][a], im);
            }
            m.re[b][a] = re;
            m.im[b][a] = im;
        }
}

// ------------------------------------------------------- hopping operator

// acc += (1 - gamma_MU) U_{n,MU} x_{n+MU} + (1 + gamma_MU) U_{n-MU,MU}^dag x_{n-MU}
template <int MU, typename R, typename I>
__device__ __forceinline__ void hop(Spinor<R> &acc, const R *__restrict__ links,
                                    const R *__restrict__ x, const Sites<I> &g, const Coord &c, I n)
{
    const int64_t V = g.V;
    const int64_t nf = n + hop_offset(g, c, MU, 1);
    accumulate<MU, -1>(acc, colour_mul<N>(load_link(links, V, MU, n), project<MU, -1>(load_spinor(x, V, nf))));
    const int64_t nb = n + hop_offset(g, c, MU, -1);
    accumulate<MU, +1>(acc, colour_mul<D>(load_link(links, V, MU, nb), project<MU, +1>(load_spinor(x, V, nb))));
}

// The x hops from the lanes of the same warp, when a warp holds whole x
// rows (the x extent divides 32; lanes n and n +- x are then lanes of one
// row of L0 lanes, with periodic wrap inside the row).  Each lane projects
// its own spinor both ways, keeps (1 - gamma_x) x_n for lane n-1's forward
// hop and applies its own link's dagger to (1 + gamma_x) x_n for lane n+1's
// backward hop (U_{n,x} is the backward link of site n+x), so that lane n
// receives 2 x 12 reals by shuffles instead of loading two neighbour
// spinors and the backward link (15 of the 78 16-byte loads of a site).
template <typename R> __device__ __forceinline__ R shfl_row(R v, int src)
{
    return __shfl_sync(0xffffffffu, v, src);
}

template <typename R> __device__ __forceinline__ Half<R> shfl_half(const Half<R> &h, int src)
{
    Half<R> r;
#pragma unroll
    for (int al = 0; al < 2; ++al)
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            r.re[al][a] = shfl_row(h.re[al][a], src);
            r.im[al][a] = shfl_row(h.im[al][a], src);
        }
    return r;
}

constexpr int kDslashBlock = 128;

// FP32 operator: what bounds it is the latency of HBM and L2 (384 bytes and
// about 1,400 instructions a site), so what counts is bytes in flight.  Loads
// into registers keep one hop of a warp in flight, and each site begins with
// an empty pipe.  Here every thread copies the operands of its hops (a
// neighbour's spinor and a link: nine 16-byte words) asynchronously into its
// own words of shared memory, kRing hops ahead and over the end of a site into
// the next of its sites; no thread reads another's words, so there is no
// barrier, only the thread's own copy groups.  The copies pass L1 by (through
// L1, which the ring leaves little of: 178 us).
// 32^3x64: 159 -> 133 us (5.1 -> 6.1 TB/s of 384 B a site), 32^4: 84 -> 69 us,
// 24^3x48: 55 -> 51 us; below that the launch is what counts.
// A ring of two hops and 4 blocks an SM (147 KB of shared memory, up to 128
// registers): 133 us at 32^3x64; 3 blocks of three hops 131, if it were
// dynamic shared memory (55 KB a block); 5 blocks of two hops at 96
// registers 145, 4 of three hops 144; 64 or 256 threads a block the same; one
// site a thread instead of as many blocks as are resident 139.
constexpr int kRing = 2;
constexpr int kDslashMinBlocks = 4;
constexpr int kHopWords = 9;

// The hops of a site in their order: +-y, +-z, +-t, then +-x.  XSHFL: the x
// hops both come from the site's own spinor and link, by shuffles.  The last
// hop brings the site's own spinor in both forms.
template <bool XSHFL> struct Hops {
    static constexpr int kCount = XSHFL ? 7 : 9;
    static constexpr bool own(int s) { return s == kCount - 1; }
    static constexpr int mu(int s) { return s < 6 ? 1 + s / 2 : 0; }
    static constexpr int sign(int s) { return (s & 1) ? -1 : 1; }
};

// Starts the copies of hop S of site n.
template <bool XSHFL, int S, typename I>
__device__ __forceinline__ void fetch_hop(float4 *slot, const float *__restrict__ x, const float *__restrict__ links,
                                          const Sites<I> &g, const Coord &c, I n)
{
    using H = Hops<XSHFL>;
    constexpr int mu = H::mu(S);
    constexpr bool own = H::own(S);
    const int64_t V = g.V;
    const int64_t m = own ? (int64_t)n : (int64_t)(n + hop_offset(g, c, mu, H::sign(S)));
    const float4 *px = reinterpret_cast<const float4 *>(x) + m;
#pragma unroll
    for (int q = 0; q < 6; ++q) copy_async(slot + q * kDslashBlock, px + q * V);
    if constexpr (XSHFL || !own) {
        const float4 *pu = reinterpret_cast<const float4 *>(links) + (int64_t)mu * 3 * V + (H::sign(S) > 0 ? (int64_t)n : m);
#pragma unroll
        for (int q = 0; q < 3; ++q) copy_async(slot + (6 + q) * kDslashBlock, pu + q * V);
    }
}

__device__ __forceinline__ Spinor<float> slot_spinor(const float4 *slot)
{
    Spinor<float> s;
#pragma unroll
    for (int q = 0; q < 6; ++q) {
        const float4 v = slot[q * kDslashBlock];
        s.re[2 * q / 3][2 * q % 3] = v.x;
        s.im[2 * q / 3][2 * q % 3] = v.y;
        s.re[(2 * q + 1) / 3][(2 * q + 1) % 3] = v.z;
        s.im[(2 * q + 1) / 3][(2 * q + 1) % 3] = v.w;
    }
    return s;
}
__device__ __forceinline__ Mat<float> slot_link(const float4 *slot)
{
    Mat<float> u;
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        const float4 v = slot[(6 + q) * kDslashBlock];
        u.re[2 * q / 3][2 * q % 3] = v.x;
        u.im[2 * q / 3][2 * q % 3] = v.y;
        u.re[(2 * q + 1) / 3][(2 * q + 1) % 3] = v.z;
        u.im[(2 * q + 1) / 3][(2 * q + 1) % 3] = v.w;
    }
    rebuild_row2(u);
    return u;
}

// One thread's pass over its sites: hop S lies in slot S % kRing, and the slots
// turn by kCount from site to site.
template <bool XSHFL, typename I> struct HopRing {
    using H = Hops<XSHFL>;
    float4 *slot[kRing];
    const float *x, *links;
    Coord c, cn; // of this site and of the thread's next
    I n, nn;
    bool more; // there is a next site

    // The copies of hop S, or of hop S - kCount of the next site; always one
    // group, so that copies_wait counts hops.

    template <int S> __device__ __forceinline__ void fetch(const Sites<I> &g)
    {
        if constexpr (S < H::kCount) {
            fetch_hop<XSHFL, S>(slot[S % kRing], x, links, g, c, n);
        } else {
            if (more) fetch_hop<XSHFL, S - H::kCount>(slot[S % kRing], x, links, g, cn, nn);
        }
        copies_commit();
    }

    // acc += hop S (the last: acc = ca x + cb acc), and the copies of hop
    // S + kRing into the slot that is read out.
    template <int S> __device__ __forceinline__ void hop(Spinor<float> &acc, const Sites<I> &g, float ca, float cb)
    {
        constexpr int mu = H::mu(S);
        float4 *const p = slot[S % kRing];
        copies_wait<kRing - 1>();
        if constexpr (!H::own(S)) {
            const Half<float> h = project<mu, -H::sign(S)>(slot_spinor(p));
            const Mat<float> u = slot_link(p);
            fetch<S + kRing>(g);
            accumulate<mu, -H::sign(S)>(acc, colour_mul<(H::sign(S) > 0 ? N : D)>(u, h));
        } else {
            if constexpr (XSHFL) {
                const int lane = (int)(threadIdx.x & 31), m = g.L0 - 1;
                const int up = (lane & ~m) | ((lane + 1) & m), dn = (lane & ~m) | ((lane - 1) & m);
                const Spinor<float> xn = slot_spinor(p);
                const Mat<float> u = slot_link(p);
                const Half<float> fw = shfl_half(project<0, -1>(xn), up);
                const Half<float> bw = shfl_half(colour_mul<D>(u, project<0, +1>(xn)), dn);
                accumulate<0, -1>(acc, colour_mul<N>(u, fw));
                accumulate<0, +1>(acc, bw);
            }
            if (ca != 0.0f) {
                const Spinor<float> xn = slot_spinor(p);
#pragma unroll
                for (int al = 0; al < 4; ++al)
#pragma unroll
                    for (int b = 0; b < 3; ++b) {
                        acc.re[al][b] = fma(ca, xn.re[al][b], cb * acc.re[al][b]);
                        acc.im[al][b] = fma(ca, xn.im[al][b], cb * acc.im[al][b]);
                    }
            } else {
#pragma unroll
                for (int al = 0; al < 4; ++al)
#pragma unroll
                    for (int b = 0; b < 3; ++b) {
                        acc.re[al][b] *= cb;
                        acc.im[al][b] *= cb;
                    }
            }
            fetch<S + kRing>(g);
        }
    }
};

// out_n = ca x_n + cb (calD x)_n in FP32.
template <bool XSHFL, typename I>
__global__ void __launch_bounds__(kDslashBlock, kDslashMinBlocks) wilson_dslash(const __grid_constant__ WilsonArgs a)
{
    using H = Hops<XSHFL>;
    __shared__ float4 ring_s[kRing * kHopWords * kDslashBlock];
    const Sites<I> g = make_sites<I>(a.dims);
    const I step = (I)gridDim.x * blockDim.x;
    HopRing<XSHFL, I> r;
    r.x = static_cast<const float *>(a.x);
    r.links = static_cast<const float *>(a.links);
    r.n = (I)blockIdx.x * blockDim.x + threadIdx.x;
    if (r.n >= g.V) return;
#pragma unroll
    for (int s = 0; s < kRing; ++s) r.slot[s] = ring_s + s * kHopWords * kDslashBlock + threadIdx.x;
    if constexpr (sizeof(I) == 4) r.c = coord_fast(g, a.div, r.n);
    else r.c = coord_in(g, r.n);
    r.more = false;
    r.template fetch<0>(g);
    r.template fetch<1>(g);
    for (;;) {
        Spinor<float> acc;
#pragma unroll
        for (int al = 0; al < 4; ++al)
#pragma unroll
            for (int b = 0; b < 3; ++b) acc.re[al][b] = acc.im[al][b] = 0.0f;
        r.template hop<0>(acc, g, a.fca, a.fcb);
        r.template hop<1>(acc, g, a.fca, a.fcb);
        r.template hop<2>(acc, g, a.fca, a.fcb);
        r.template hop<3>(acc, g, a.fca, a.fcb);
        r.nn = r.n + step;
        r.more = r.nn < g.V;
        if (r.more) {
            if constexpr (sizeof(I) == 4) r.cn = coord_fast(g, a.div, r.nn);
            else r.cn = coord_in(g, r.nn);
        }
        r.template hop<4>(acc, g, a.fca, a.fcb);
        r.template hop<5>(acc, g, a.fca, a.fcb);
        r.template hop<6>(acc, g, a.fca, a.fcb);
        if constexpr (!XSHFL) {
            r.template hop<7>(acc, g, a.fca, a.fcb);
            r.template hop<8>(acc, g, a.fca, a.fcb);
        }
        store_spinor(static_cast<float *>(a.out), (int64_t)g.V, (int64_t)r.n, acc);
        if (!r.more) break;
        r.n = r.nn;
        r.c = r.cn;
        float4 *old[kRing];
#pragma unroll
        for (int s = 0; s < kRing; ++s) old[s] = r.slot[s];
#pragma unroll
        for (int s = 0; s < kRing; ++s) r.slot[s] = old[(s + H::kCount) % kRing];
    }
}

// out_n = ca x_n + cb acc (x not read for ca = 0).
__device__ __forceinline__ void store_dslash(const WilsonArgs &a, const double *__restrict__ x, int64_t V, int64_t n,
                                             Spinor<double> &acc, double ca, double cb)
{
    Spinor<double> xn;
    if (ca != 0.0) xn = load_spinor(x, V, n);
#pragma unroll
    for (int al = 0; al < 4; ++al)
#pragma unroll
        for (int b = 0; b < 3; ++b) {
            acc.re[al][b] *= cb;
            acc.im[al][b] *= cb;
            if (ca != 0.0) {
                acc.re[al][b] = fma(ca, xn.re[al][b], acc.re[al][b]);
                acc.im[al][b] = fma(ca, xn.im[al][b], acc.im[al][b]);
            }
        }
    store_spinor(static_cast<double *>(a.out), V, n, acc);
}

// gcode at run time.
__device__ __forceinline__ int gcode_of(int mu, int alpha)
{
    return mu == 0 ? (alpha < 2 ? 1 : 3) : mu == 1 ? ((alpha == 0 || alpha == 3) ? 2 : 0)
           : mu == 2 ? ((alpha == 0 || alpha == 3) ? 1 : 3) : 0;
}

// --------------------------------------------------- hopping-term force

// B - C on link (k, RHO), both as sums over the two independent spin rows:
//   B = sum_alpha (U chi_alpha) (x) psi_alpha^dag,  chi = (1 - g) X_{k+rho}, psi = (1 - g) Y_k
//   C = sum_alpha xi_alpha (x) (U eta_alpha)^dag,   xi = (1 + g) X_k,      eta = (1 + g) Y_{k+rho}
// (Eqs. 18_1_29_20_2 and 18_1_29_20_3 with (1 -+ g) Hermitian and
// (1 -+ g)^2 = 2 (1 -+ g), so the projector moves onto the other factor and
// the four spin rows fold into two.)
template <int RHO, typename R>
__device__ __forceinline__ Mat<R> b_minus_c(const R *__restrict__ links, const R *__restrict__ X,
                                            const R *__restrict__ Y, int64_t V, int64_t k, int64_t kp)
{
    const Mat<R> u = load_link(links, V, RHO, k);
    Mat<R> m;
    set_zero(m);
    outer_acc<1>(m, colour_mul<N>(u, project<RHO, -1>(load_spinor(X, V, kp))),
                 project<RHO, -1>(load_spinor(Y, V, k)));
    outer_acc<-1>(m, project<RHO, +1>(load_spinor(X, V, k)),
                  colour_mul<N>(u, project<RHO, +1>(load_spinor(Y, V, kp))));
    return m;
}

constexpr int kForceBlock = 128; // 32 sites x 4 directions, one direction per warp

// f = coef h stored and/or applied to the momenta.
__device__ __forceinline__ void finish_force(const WilsonArgs &a, int64_t V, int rho, int64_t k, const double f[8])
{
    if (a.force != nullptr) store_algebra(static_cast<double *>(a.force), V, rho, k, f);
    if (a.mom != nullptr) {
        double *mom = static_cast<double *>(a.mom);
        double p[8];
        load_algebra(mom, V, rho, k, p);
#pragma unroll
        for (int q = 0; q < 8; ++q) p[q] = fma(a.dt, f[q], p[q]);
        store_algebra(mom, V, rho, k, p);
    }
}

// ------------------------------------------ hopping-term force in fixed point

// Two colour vectors in whole limbs of 2^-28 and 2^-56 of their spinor's scale.
struct FHalf {
    int rh[2][3], rl[2][3], ih[2][3], il[2][3];
};

// What the fixed point loses, and how it is seen.  A spinor's reals are known
// to 2^-58 of the largest, so a result made of much smaller ones only (colours
// or spin rows that nothing mixes in: links near 1 or diagonal) would have lost
// its digits.  Such results are themselves small: where a complex one is below
// 2^-kPairBits of the scale of its spinors, or kFewReals of a site's 24 reals
// (a spin row, a colour) or kFewComponents of a force's 8 (a colour) below
// 2^-kRealBits or 2^-kComponentBits, the site or link is computed in floating
// point.  Of normal spinors on normal links that is one in a million: a single
// one among the last blocks of a small lattice costs 20 us.
constexpr int kPairBits = 12, kRealBits = 6, kFewReals = 6, kComponentBits = 7, kFewComponents = 4;

// Exponent field that stands for the scale of a spinor of zeros.
constexpr int kZeroScale = 64;

// Rows 0 and 1 of (1 + s gamma_mu) x_n, mu at run time, over 2^(e - 1022) with
// e the largest exponent field of the spinor's 24 reals; false where that is out
// of range or not finite.
__device__ __forceinline__ bool fx_half(const double *__restrict__ x, int64_t V, int64_t n, int mu, bool minus, FHalf &h,
                                        int &e)
{
    // rows 0, 1 go with rows 3, 2 (mu < 2) or 2, 3; where i^gcode is odd the
    // parts of those are exchanged, by where they are read
    const double2 *p = reinterpret_cast<const double2 *>(x) + n;
    const bool turn = mu == 0 || mu == 2;
    const double *p2 = x + 2 * (n + (mu < 2 ? 9 : 6) * V), *p3 = x + 2 * (n + (mu < 2 ? 6 : 9) * V);
    const int ore = turn ? 1 : 0, oim = 1 - ore;
    double2 v[12];
#pragma unroll
    for (int q = 0; q < 6; ++q) v[q] = __ldg(p + q * V);
#pragma unroll
    for (int q = 0; q < 3; ++q) {
        v[6 + q] = make_double2(__ldg(p2 + 2 * q * V + ore), __ldg(p2 + 2 * q * V + oim));
        v[9 + q] = make_double2(__ldg(p3 + 2 * q * V + ore), __ldg(p3 + 2 * q * V + oim));
    }
    e = 0;
#pragma unroll
    for (int q = 0; q < 12; ++q) e = max(e, max(exponent_of(v[q].x), exponent_of(v[q].y)));
    if (e <= kZeroScale || e > 2040) { // results up to 2^6 of the scale
        if (e != 0) return false;
        bool zero = true; // and no subnormals
#pragma unroll
        for (int q = 0; q < 12; ++q) zero = zero && v[q].x == 0.0 && v[q].y == 0.0;
        if (!zero) return false;
        e = kZeroScale;
    }
    const int shift = e - 1022;
#pragma unroll
    for (int al = 0; al < 2; ++al) {
        // times s i^gcode(mu, al)
        const int code = ((mu == 0 ? 1 : mu == 1 ? (al == 0 ? 2 : 0) : mu == 2 ? (al == 0 ? 1 : 3) : 0) + (minus ? 2 : 0)) & 3;
        const int sr = code == 1 || code == 2 ? -1 : 0, si = code >= 2 ? -1 : 0; // masks of the signs
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const double2 w = v[6 + 3 * al + a], u = v[3 * al + a];
            const long long re = fx_of_double(u.x, shift) + fx_of_double(w.x, shift, sr);
            const long long im = fx_of_double(u.y, shift) + fx_of_double(w.y, shift, si);
            fx_limbs<2>(re, h.rh[al][a], h.rl[al][a]);
            fx_limbs<2>(im, h.ih[al][a], h.il[al][a]);
        }
    }
    return true;
}

// u h (D: u^dagger h) on both colour vectors.
template <int F> __device__ __forceinline__ void fx_colour_sums(const FLimbs &u, const FHalf &h, int al, FLimbAcc &y)
{
#pragma unroll
    for (int a = 0; a < 3; ++a) y.h1[a][0] = y.l1[a][0] = y.h2[a][0] = y.l2[a][0] = y.h3[a][0] = y.l3[a][0] = 0;
#pragma unroll
    for (int b = 0; b < 3; ++b) {
        const int sh = h.rh[al][b] + h.ih[al][b], sl = h.rl[al][b] + h.il[al][b];
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            const int p = F == N ? a : b, q = F == N ? b : a;
            fx_mad(y.h1[a][0], y.l1[a][0], u.rh[p][q], u.rl[p][q], h.rh[al][b], h.rl[al][b]);
            fx_mad(y.h2[a][0], y.l2[a][0], u.ih[p][q], u.il[p][q], h.ih[al][b], h.il[al][b]);
            fx_mad(y.h3[a][0], y.l3[a][0], F == N ? u.rh[p][q] + u.ih[p][q] : u.rh[p][q] - u.ih[p][q],
                   F == N ? u.rl[p][q] + u.il[p][q] : u.rl[p][q] - u.il[p][q], sh, sl);
        }
    }
}

__device__ __forceinline__ void fx_colour_mul(const FLimbs &u, FHalf &h)
{
#pragma unroll
    for (int al = 0; al < 2; ++al) {
        FLimbAcc y; // column 0
        fx_colour_sums<N>(u, h, al, y);
#pragma unroll
        for (int a = 0; a < 3; ++a) {
            long long re, im;
            fx_total<1>(y, a, 0, re, im);
            fx_limbs<2>(re, h.rh[al][a], h.rl[al][a]);
            fx_limbs<2>(im, h.ih[al][a], h.il[al][a]);
        }
    }
}

// The force on one FP64 link.  With N_0 = (U (1 - g) X_{k+rho}) (x) ((1 - g) Y_k)^dag
// and N_1 = (U (1 + g) Y_{k+rho}) (x) ((1 + g) X_k)^dag, spin rows 0 and 1 summed,
// B = N_0 and C = N_1^dag, so h^i = Im tr(lambda_i N_0) + Im tr(lambda_i N_1): one
// loop body for both, the direction at run time, so that the four warps of a
// block run the same code.
//
// In floating point this is 720 operations a link on the FP64 pipe (2 a clock
// and SM) and 108 numbers read.  Here every spinor is a block of whole numbers
// of its own scale, taken apart by integer operations; the FP64 pipe makes the
// 16 components.
__device__ __forceinline__ bool hopping_force_fx(const WilsonArgs &a, int64_t V, int rho, int64_t k, int64_t kp)
{
    __shared__ int4 u_s[9][kForceBlock]; // the link, out of the registers' way
    int4 *us = &u_s[0][threadIdx.x];
    {
        FLimbs u;
        const double2 *p = static_cast<const double2 *>(a.links) + (int64_t)rho * 6 * V + k;
        double r[12];
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const double2 v = __ldg(p + q * V);
            r[2 * q] = v.x;
            r[2 * q + 1] = v.y;
        }
        if (!fx_limbs_of_rows(r, u)) return false;
        fx_row2(u);
#pragma unroll
        for (int e = 0; e < 9; ++e)
            us[e * kForceBlock] = make_int4(u.rh[e / 3][e % 3], u.rl[e / 3][e % 3], u.ih[e / 3][e % 3], u.il[e / 3][e % 3]);
    }
    double f[8] = {0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0};
    int scale = 0; // largest sum of the exponent fields of two spinors
#pragma unroll 1
    for (int t = 0; t < 2; ++t) {
        const double *s0 = static_cast<const double *>(t == 0 ? a.x : a.y), *s1 = static_cast<const double *>(t == 0 ? a.y : a.x);
        FHalf p, q;
        int ep, eq;
        if (!fx_half(s0, V, kp, rho, t == 0, p, ep)) return false;
        {
            FLimbs u;
#pragma unroll
            for (int e = 0; e < 9; ++e) {
                const int4 v = us[e * kForceBlock];
                u.rh[e / 3][e % 3] = v.x;
                u.rl[e / 3][e % 3] = v.y;
                u.ih[e / 3][e % 3] = v.z;
                u.il[e / 3][e % 3] = v.w;
            }
            fx_colour_mul(u, p);
        }
        // a small colour is a small row of the product: a field of such leaves here
        bool thin = false;
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            constexpr unsigned c = 1u << (27 - kComponentBits);
            thin = thin || (p.rh[0][i] + c < 2 * c && p.ih[0][i] + c < 2 * c && p.rh[1][i] + c < 2 * c && p.ih[1][i] + c < 2 * c);
        }
        if (thin && ep > kZeroScale) return false;
        if (!fx_half(s1, V, k, rho, t == 0, q, eq)) return false;
        if (ep > kZeroScale && eq > kZeroScale) scale = max(scale, ep + eq);
        long long re[3][3], im[3][3]; // N, units 2^-56 of the two scales
#pragma unroll
        for (int i = 0; i < 3; ++i) {
            FLimbAcc y; // row 0
#pragma unroll
            for (int j = 0; j < 3; ++j) y.h1[0][j] = y.l1[0][j] = y.h2[0][j] = y.l2[0][j] = y.h3[0][j] = y.l3[0][j] = 0;
#pragma unroll
            for (int al = 0; al < 2; ++al) {
                const int sh = p.rh[al][i] + p.ih[al][i], sl = p.rl[al][i] + p.il[al][i];
#pragma unroll
                for (int j = 0; j < 3; ++j) {
                    fx_mad(y.h1[0][j], y.l1[0][j], p.rh[al][i], p.rl[al][i], q.rh[al][j], q.rl[al][j]);
                    fx_mad(y.h2[0][j], y.l2[0][j], p.ih[al][i], p.il[al][i], q.ih[al][j], q.il[al][j]);
                    fx_mad(y.h3[0][j], y.l3[0][j], sh, sl, q.rh[al][j] - q.ih[al][j], q.rl[al][j] - q.il[al][j]);
                }
            }
#pragma unroll
            for (int j = 0; j < 3; ++j) fx_total<-1>(y, 0, j, re[i][j], im[i][j]);
        }
        // Im tr(lambda_a N) times coef, and one power of two for all scales
        const bool zero = ep <= kZeroScale || eq <= kZeroScale;
        const int power = ep + eq - 2044 - 56;
        if (!zero && (power < -1022 || power > 900 || exponent_of(a.coef) > 1023 + 900)) return false;
        const double s = a.coef, w = zero ? 0.0 : __hiloint2double((power + 1023) << 20, 0);
        f[0] = fma(s * (double)(im[0][1] + im[1][0]), w, f[0]);
        f[1] = fma(s * (double)(re[0][1] - re[1][0]), w, f[1]);
        f[2] = fma(s * (double)(im[0][0] - im[1][1]), w, f[2]);
        f[3] = fma(s * (double)(im[0][2] + im[2][0]), w, f[3]);
        f[4] = fma(s * (double)(re[0][2] - re[2][0]), w, f[4]);
        f[5] = fma(s * (double)(im[1][2] + im[2][1]), w, f[5]);
        f[6] = fma(s * (double)(re[1][2] - re[2][1]), w, f[6]);
        f[7] = fma(s * 0.57735026918962576451 * (double)(im[0][0] + im[1][1] - 2 * im[2][2]), w, f[7]);
    }
    // small results (the diagonal components go together)
    const int top = exponent_of(a.coef) + scale - 2044;
    int reals = 0;
#pragma unroll
    for (int q = 0; q < 8; ++q) reals += exponent_of(f[q]) < top - kComponentBits;
    const auto small = [&](int i, int j) { return max(exponent_of(f[i]), exponent_of(f[j])) < top - kPairBits; };
    if (scale > 0 && (reals >= kFewComponents || small(0, 1) || small(3, 4) || small(5, 6) || small(2, 7))) return false;
    finish_force(a, V, rho, k, f);
    return true;
}

// B - C on link (k, rho), the direction at run time.
template <typename R>
__device__ __forceinline__ Mat<R> b_minus_c(const R *__restrict__ links, const R *__restrict__ X,
                                            const R *__restrict__ Y, int64_t V, int rho, int64_t k, int64_t kp)
{
    switch (rho) {
    case 0: return b_minus_c<0>(links, X, Y, V, k, kp);
    case 1: return b_minus_c<1>(links, X, Y, V, k, kp);
    case 2: return b_minus_c<2>(links, X, Y, V, k, kp);
    default: return b_minus_c<3>(links, X, Y, V, k, kp);
    }
}

// The FP64 force in floating point, for links that hopping_force_fx leaves.
__device__ __noinline__ void hopping_force_floating(const WilsonArgs &a, int64_t V, int rho, int64_t k, int64_t kp)
{
    const Mat<double> m = b_minus_c(static_cast<const double *>(a.links), static_cast<const double *>(a.x),
                                    static_cast<const double *>(a.y), V, rho, k, kp);
    double f[8];
    ta_components(m, -a.coef, f);
    finish_force(a, V, rho, k, f);
}

template <typename I>
__global__ void __launch_bounds__(kForceBlock) wilson_hopping_force(const __grid_constant__ WilsonArgs a)
{
    const Sites<I> g = make_sites<I>(a.dims);
    const float *__restrict__ links = static_cast<const float *>(a.links);
    const float *__restrict__ X = static_cast<const float *>(a.x);
    const float *__restrict__ Y = static_cast<const float *>(a.y);
    const int rho = (int)(threadIdx.x >> 5);
    const I ks = (I)blockIdx.x * 32 + (I)(threadIdx.x & 31);
    if (ks >= g.V) return;
    Coord c;
    if constexpr (sizeof(I) == 4) c = coord_fast(g, a.div, ks);
    else c = coord_in(g, ks);
    const int64_t V = g.V, k = ks, kp = (int64_t)(ks + hop_offset(g, c, rho, 1));
    Mat<float> m;
    switch (rho) {
    case 0: m = b_minus_c<0>(links, X, Y, V, k, kp); break;
    case 1: m = b_minus_c<1>(links, X, Y, V, k, kp); break;
    case 2: m = b_minus_c<2>(links, X, Y, V, k, kp); break;
    default: m = b_minus_c<3>(links, X, Y, V, k, kp); break;
    }
    // f^i = coef * h^i,  h^i = -(tr(i T_i M) + c.c.) = Im tr(lambda_i M)
    float f[8];
    ta_components(m, -a.fcoef, f);
    if (a.force != nullptr) store_algebra(static_cast<float *>(a.force), V, rho, k, f);
    if (a.mom != nullptr) {
        float *mom = static_cast<float *>(a.mom);
        float p[8];
        load_algebra(mom, V, rho, k, p);
        const float dt = a.fdt;
#pragma unroll
        for (int q = 0; q < 8; ++q) p[q] = fma(dt, f[q], p[q]);
        store_algebra(mom, V, rho, k, p);
    }
}

// 4 blocks per SM (128 registers, 236 bytes spilled): 151 us at 20x18x14x30; in
// floating point 431.  What bounds it are three pipes alike: instruction issue,
// the integer half of the FMA pipe and the ALUs would each take about 67 us.
template <typename I>
__global__ void __launch_bounds__(kForceBlock, 4) wilson_hopping_force_fx(const __grid_constant__ WilsonArgs a)
{
    const Sites<I> g = make_sites<I>(a.dims);
    const int rho = (int)(threadIdx.x >> 5);
    const I ks = (I)blockIdx.x * 32 + (I)(threadIdx.x & 31);
    if (ks >= g.V) return;
    Coord c;
    if constexpr (sizeof(I) == 4) c = coord_fast(g, a.div, ks);
    else c = coord_in(g, ks);
    const int64_t V = g.V, k = ks, kp = (int64_t)(ks + hop_offset(g, c, rho, 1));
    if (!hopping_force_fx(a, V, rho, k, kp)) hopping_force_floating(a, V, rho, k, kp);
}

// ------------------------------------------------ hopping operator, FP64

// One site of y = ca x + cb calD x in floating point, for sites that
// dslash_site_fx leaves.
template <typename I>
__device__ __noinline__ void dslash_site_floating(const WilsonArgs &a, const Sites<I> &g, const Coord &c, I n)
{
    const double *__restrict__ links = static_cast<const double *>(a.links);
    const double *__restrict__ x = static_cast<const double *>(a.x);
    Spinor<double> acc;
#pragma unroll
    for (int al = 0; al < 4; ++al)
#pragma unroll
        for (int b = 0; b < 3; ++b) acc.re[al][b] = acc.im[al][b] = 0.0;
    hop<0>(acc, links, x, g, c, n);
    hop<1>(acc, links, x, g, c, n);
    hop<2>(acc, links, x, g, c, n);
    hop<3>(acc, links, x, g, c, n);
    store_dslash(a, x, (int64_t)g.V, (int64_t)n, acc, a.ca, a.cb);
}

// Whether spinor n has a colour or three spin rows below 2^-kRealBits of the
// largest: a site of a field of such is left before any work (1.5 % of the
// time of any other).
__device__ __forceinline__ bool uneven_spinor(const double *__restrict__ x, int64_t V, int64_t n)
{
    const double2 *p = reinterpret_cast<const double2 *>(x) + n;
    int row[4] = {0, 0, 0, 0}, col[3] = {0, 0, 0};
#pragma unroll
    for (int q = 0; q < 12; ++q) {
        const double2 v = __ldg(p + q * V);
        const int e = max(exponent_of(v.x), exponent_of(v.y));
        row[q / 3] = max(row[q / 3], e);
        col[q % 3] = max(col[q % 3], e);
    }
    const int least = max(col[0], max(col[1], col[2])) - kRealBits;
    return min(col[0], min(col[1], col[2])) < least ||
           (row[0] < least) + (row[1] < least) + (row[2] < least) + (row[3] < least) >= 3;
}

// The same in fixed point (hopping_force_fx): the eight hops in one loop, the
// direction and sign at run time; every neighbour's half spinor in its own
// scale, the sum in whole numbers of 2^-56 of the largest scale so far.
template <typename I>
__device__ __forceinline__ bool dslash_site_fx(const WilsonArgs &a, const Sites<I> &g, const Coord &c, I n)
{
    const double *__restrict__ x = static_cast<const double *>(a.x);
    const int64_t V = g.V;
    if (uneven_spinor(x, V, (int64_t)n)) return false;
    long long sr[12], si[12]; // spin rows 0 to 3, colours 0 to 2
#pragma unroll
    for (int q = 0; q < 12; ++q) sr[q] = si[q] = 0;
    int scale = 0; // exponent field of the sum's scale
    // whether a complex result is small, or kFewReals real ones
    const auto small = [&] {
        constexpr int cp = 1 << (24 - kPairBits), cr = 1 << (24 - kRealBits);
        int pairs = 0, reals = 0;
#pragma unroll
        for (int q = 0; q < 12; ++q) {
            const unsigned r = (unsigned)(int)(sr[q] >> 32), i = (unsigned)(int)(si[q] >> 32);
            pairs += r + cp < 2u * cp && i + cp < 2u * cp;
            reals += (r + cr < 2u * cr) + (i + cr < 2u * cr);
        }
        return scale > kZeroScale && (pairs > 0 || reals >= kFewReals);
    };
#pragma unroll 1
    for (int t = 0; t < 8; ++t) {
        const int mu = t >> 1;
        const bool back = t & 1;
        const int64_t nb = n + hop_offset(g, c, mu, back ? -1 : 1);
        FHalf h;
        int e;
        if (!fx_half(x, V, nb, mu, !back, h, e)) return false;
        FLimbs u;
        {
            const double2 *p = static_cast<const double2 *>(a.links) + (int64_t)mu * 6 * V + (back ? nb : (int64_t)n);
            double r[12];
#pragma unroll
            for (int q = 0; q < 6; ++q) {
                const double2 v = __ldg(p + q * V);
                r[2 * q] = v.x;
                r[2 * q + 1] = v.y;
            }
            if (!fx_limbs_of_rows(r, u)) return false;
            fx_row2(u);
        }
        if (e > scale) { // the sum so far in the new scale
            const int d = min(e - scale, 63);
#pragma unroll
            for (int q = 0; q < 12; ++q) {
                sr[q] >>= d;
                si[q] >>= d;
            }
            scale = e;
        }
        const int sh = min(scale - e, 60) + 2;
        const long long half = 1ll << (sh - 1);
#pragma unroll
        for (int al = 0; al < 2; ++al) {
            FLimbAcc y;
            if (back) fx_colour_sums<D>(u, h, al, y);
            else fx_colour_sums<N>(u, h, al, y);
            // rows 0, 1 of the hop, and its rows 2, 3 as s i^gcode times them
            const int p = mu < 2 ? 3 - al : 2 + al; // partner row
            const int code = (gcode_of(mu, p) + (back ? 0 : 2)) & 3;
            const long long mr = code == 1 || code == 2 ? -1 : 0, mi = code >= 2 ? -1 : 0;
#pragma unroll
            for (int b = 0; b < 3; ++b) {
                long long re, im;
                if (back) fx_total<-1>(y, b, 0, re, im);
                else fx_total<1>(y, b, 0, re, im);
                re = (re + half) >> sh;
                im = (im + half) >> sh;
                sr[3 * al + b] += re;
                si[3 * al + b] += im;
                const long long tr = (((code & 1) ? im : re) ^ mr) - mr, ti = (((code & 1) ? re : im) ^ mi) - mi;
                if (mu < 2) {
                    sr[3 * (3 - al) + b] += tr;
                    si[3 * (3 - al) + b] += ti;
                } else {
                    sr[3 * (2 + al) + b] += tr;
                    si[3 * (2 + al) + b] += ti;
                }
            }
        }
    }
    if (small()) return false;
    // 2^-56 of 2^(scale - 1022) by the exponent field, so that cb meets a
    // number of the result's own size
    const auto value = [&](long long v) {
        const double d = (double)v;
        return v == 0 ? 0.0 : __hiloint2double(__double2hiint(d) + (scale - 1022 - 56) * (1 << 20), __double2loint(d));
    };
    Spinor<double> acc;
#pragma unroll
    for (int q = 0; q < 12; ++q) {
        acc.re[q / 3][q % 3] = value(sr[q]);
        acc.im[q / 3][q % 3] = value(si[q]);
    }
    store_dslash(a, x, V, (int64_t)n, acc, a.ca, a.cb);
    return true;
}

// 32^4: 752 us, 20x18x14x30: 136; in floating point 2153 and 353 (what
// uneven_spinor finds 2221).  Error against extended precision 6.0e-17, in
// floating point 9.0e-17.
template <typename I>
__global__ void __launch_bounds__(kDslashBlock, 3) wilson_dslash_fx(const __grid_constant__ WilsonArgs a)
{
    const Sites<I> g = make_sites<I>(a.dims);
    for (I n = (I)blockIdx.x * blockDim.x + threadIdx.x; n < g.V; n += (I)gridDim.x * blockDim.x) {
        Coord c;
        if constexpr (sizeof(I) == 4) c = coord_fast(g, a.div, n);
        else c = coord_in(g, n);
        if (!dslash_site_fx(a, g, c, n)) dslash_site_floating(a, g, c, n);
    }
}

unsigned blocks_for(int64_t items, int per_block)
{
    int64_t b = (items + per_block - 1) / per_block;
    if (b < 1) b = 1;
    if (b > ((int64_t)1 << 30)) b = (int64_t)1 << 30;
    return (unsigned)b;
}

// The launch copy of the arguments: FP32 scalars and the strides' division
// magic filled in.
WilsonArgs launch_args(WilsonArgs a)
{
    stride_magic(a.dims, a.div);
    a.fca = (float)a.ca;
    a.fcb = (float)a.cb;
    a.fcoef = (float)a.coef;
    a.fdt = (float)a.dt;
    return a;
}

} // namespace

cudaError_t launch_wilson_dslash(const WilsonArgs &args, cudaStream_t st)
{
    const WilsonArgs a = launch_args(args);
    const int64_t V = (int64_t)a.dims[0] * a.dims[1] * a.dims[2] * a.dims[3];
    const unsigned grid = blocks_for(V, kDslashBlock);
    const bool i32 = sites_fit_int(V);
    if (a.precision == LQCD_F64) {
        if (i32) wilson_dslash_fx<int><<<grid, kDslashBlock, 0, st>>>(a);
        else wilson_dslash_fx<int64_t><<<grid, kDslashBlock, 0, st>>>(a);
    } else {
        // shuffled x hops need whole x rows in every warp: L0 divides 32 (every
        // warp's first site then starts a row) and V is whole warps.  They save
        // 15 of 78 words a site (0.203 -> 0.184 ms at 32^3x64 when introduced).
        const int L0 = a.dims[0];
        const bool xshfl = L0 <= 32 && (32 % L0) == 0 && V % 32 == 0;
        // as many blocks as are resident, each thread over several sites
        int dev = 0, sms = 0;
        cudaError_t e = cudaGetDevice(&dev);
        if (e == cudaSuccess) e = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
        if (e != cudaSuccess) return e;
        const unsigned resident = grid < (unsigned)(sms * kDslashMinBlocks) ? grid : (unsigned)(sms * kDslashMinBlocks);
        const auto k = i32 ? (xshfl ? wilson_dslash<true, int> : wilson_dslash<false, int>)
                           : (xshfl ? wilson_dslash<true, int64_t> : wilson_dslash<false, int64_t>);
        k<<<resident, kDslashBlock, 0, st>>>(a);
    }
    return cudaGetLastError();
}

cudaError_t launch_wilson_hopping_force(const WilsonArgs &args, cudaStream_t st)
{
    const WilsonArgs a = launch_args(args);
    const int64_t V = (int64_t)a.dims[0] * a.dims[1] * a.dims[2] * a.dims[3];
    const unsigned grid = blocks_for(V, 32);
    const bool i32 = sites_fit_int(V);
    if (a.precision == LQCD_F64) {
        if (i32) wilson_hopping_force_fx<int><<<grid, kForceBlock, 0, st>>>(a);
        else wilson_hopping_force_fx<int64_t><<<grid, kForceBlock, 0, st>>>(a);
    } else {
        if (i32) wilson_hopping_force<int><<<grid, kForceBlock, 0, st>>>(a);
        else wilson_hopping_force<int64_t><<<grid, kForceBlock, 0, st>>>(a);
    }
    return cudaGetLastError();
}

} // namespace lqcd
