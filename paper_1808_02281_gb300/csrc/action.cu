// Gauge action S_G = (beta/3) sum_n sum_{34 loops P} c_P [3 - Re tr P_n]
// (paper Eq. 18_6_4_1, loops of Eq. 18_3_27_30) and the kinetic term
// K = (1/2) sum p^2 of the MD Hamiltonian, as deterministic FP64 reductions:
// every thread sums its sites in double, warps reduce by shuffles, blocks
// write one partial each to the caller's workspace, and one block adds the
// partials in a fixed order.  The grid is a fixed multiple of the SM count,
// so the summation order -- and the result, bit for bit -- is reproducible.
#include <cmath>
#include <mutex>

#include <nvtx3/nvToolsExt.h>

#include "fx_planes.cuh"
#include "sites.cuh"

namespace lqcd {

namespace {

constexpr int kBlock = 256;
constexpr int kActionBlock = 128; // four warps: a quarter of the loops of 32 sites each

// Sum over a block of B threads (result in thread 0).
template <int B> __device__ __forceinline__ double block_sum(double v)
{
    __shared__ double warp_part[B / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) warp_part[warp] = v;
    __syncthreads();
    double s = 0.0;
    if (warp == 0) {
        s = lane < B / 32 ? warp_part[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
    }
    return s; // valid in thread 0
}

// Direction of item i of the direction-major order (i < 4 V).
__device__ __forceinline__ int direction_of(int64_t i, int64_t V)
{
    return (int)(i >= V) + (int)(i >= 2 * V) + (int)(i >= 3 * V);
}

// U_{x,d} for d = +-(mu+1), and x advanced to x + hat(d).
template <typename R>
__device__ __forceinline__ Mat<R> walk(const R *__restrict__ links, const Geom &g, Coord &x, int d)
{
    if (d > 0) {
        const Mat<R> m = load_link(links, g.V, d - 1, index_of(g, x));
        step(g, x, d - 1, 1);
        return m;
    }
    step(g, x, -d - 1, -1);
    return dagger(load_link(links, g.V, -d - 1, index_of(g, x)));
}

// The warp of a site's four that a loop of the table belongs to: plaquettes
// and rectangles to their first (long) direction, cubes to the direction that
// they leave out.
__device__ __forceinline__ int loop_owner(const Loop &lp)
{
    const auto dir = [](int d) { return (d > 0 ? d : -d) - 1; };
    return lp.cls < 2 ? dir(lp.d[0]) : 6 - dir(lp.d[0]) - dir(lp.d[1]) - dir(lp.d[2]);
}

// sum c_P (3 - Re tr P) over the loops of warp w at site n, each walked link
// by link in floating point: for FP64 links without a fixed-point form.
__device__ __noinline__ double walked_loops(const ReduceArgs &a, const LoopTable &tab, int64_t n, int w)
{
    const Geom g = make_geom(a.dims);
    const double *links = static_cast<const double *>(a.links);
    const Coord x0 = coord_of(g, n);
    double acc = 0.0;
    for (int l = 0; l < tab.count; ++l) {
        const Loop &lp = tab.l[l];
        if (loop_owner(lp) != w) continue;
        Coord x = x0;
        // the four cube loops of a site are those of the cube it is the lowest
        // corner of: one with a step down starts from above
        if (lp.cls == 2)
            for (int j = 1; j < 3; ++j)
                if (lp.d[j] < 0) step(g, x, -lp.d[j] - 1, 1);
        Mat<double> m = walk(links, g, x, lp.d[0]);
        for (int j = 1; j < lp.len - 1; ++j) m = mul<N, N>(m, walk(links, g, x, lp.d[j]));
        const double retr = re_trace_mul<N, N>(m, walk(links, g, x, lp.d[lp.len - 1]));
        acc += (lp.cls == 0 ? a.c[0] : (lp.cls == 1 ? a.c[1] : a.c[2])) * (3.0 - retr);
    }
    return acc;
}

// FP32: every loop is the product of its links in their order, as the table
// has it, closed by the trace with the last: the rounding of a site's traces is
// random, and the action of a small lattice carries it (1e-8 and less), so
// another grouping would be another value.  What loops have in common at their
// start is multiplied once (U_mu U_mu of three rectangles, U_mu U_{+-nu} of two
// cubes: 108 products a site of 124).  The loops of 32 sites on four warps:
// plaquettes and rectangles on their first direction's, cubes on the one they
// leave out.  A class's traces in a sum with its rounding errors kept (FP64
// additions, 2 a clock and SM, would take as long as a third of the products).
// 32^3x64: 2834 -> 2104 us, 16^3x32: 211 -> 124, 4^4: 72 -> 20; bound by the
// latency of the links (16 warps an SM at 128 registers) and by the instruction
// cache: with the cubes unrolled over one sign 2143 us, over both 2341, all
// loops unrolled 2694; one product's code for all 2576; 3 blocks an SM 2787.
struct Traces32 {
    float s = 0.f, e = 0.f;
    __device__ __forceinline__ void add(float t)
    {
        const float u = s + t, b = u - s;
        e += (s - (u - b)) + (t - b);
        s = u;
    }
    // 3 n - the sum
    __device__ __forceinline__ double below(int n) const { return (3.0 * n - (double)s) - (double)e; }
};

constexpr int kLoopsMinBlocks = 4;

template <typename I>
__global__ void __launch_bounds__(kActionBlock, kLoopsMinBlocks) action_loops_f32(const __grid_constant__ ReduceArgs a)
{
    using M = Mat<float>;
    const Sites<I> g = make_sites<I>(a.dims);
    const int64_t V = g.V;
    const float *__restrict__ links = static_cast<const float *>(a.links);
    const int w = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
    double acc = 0.0;
    const I nvb = (g.V + 31) / 32;
    for (I vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
        const I n = vb * 32 + lane;
        if (n >= g.V) continue;
        Coord c;
        if constexpr (sizeof(I) == 4) c = coord_fast(g, a.div, n);
        else c = coord_in(g, n);
        const auto link = [&](int mu, I at) { return load_link(links, V, mu, (int64_t)at); };
        const auto off = [&](int mu, int s) { return hop_offset(g, c, mu, s); };
        Traces32 pl, rc, cb;
        const I nw = n + off(w, 1);
#pragma unroll 1
        for (int nu = w + 1; nu < 4; ++nu) {
            const M m = mul<N, D>(mul<N, N>(link(w, n), link(nu, nw)), link(w, n + off(nu, 1)));
            pl.add(re_trace_mul<N, D>(m, link(nu, n)));
        }
        {
            const M ww = mul<N, N>(link(w, n), link(w, nw));
            Coord c1 = c;
            step_up(g, c1, w);
            const I n2w = nw + hop_offset(g, c1, w, 1);
#pragma unroll 1
            for (int j = 1; j < 4; ++j) {
                const int nu = (w + j) & 3;
                const I up = off(nu, 1);
                const M m = mul<N, D>(mul<N, D>(mul<N, N>(ww, link(nu, n2w)), link(w, nw + up)), link(w, n + up));
                rc.add(re_trace_mul<N, D>(m, link(nu, n)));
            }
        }
        {
            const int mu = w == 0 ? 1 : 0, nu = w <= 1 ? 2 : 1, r = w == 3 ? 2 : 3;
            const I om = off(mu, 1);
            // mu, s nu, q r, -mu, -s nu, -q r
#pragma unroll 1
            for (int s = 0; s < 2; ++s) {
                const I on = off(nu, s == 0 ? 1 : -1);
                M p;
                if (s == 0) p = mul<N, N>(link(mu, n), link(nu, n + om));
                else p = mul<N, D>(link(mu, n), link(nu, n + om + on));
#pragma unroll 1
                for (int q = 0; q < 2; ++q) {
                    const I oq = off(r, q == 0 ? 1 : -1);
                    M m;
                    if (q == 0) m = mul<N, N>(p, link(r, n + om + on));
                    else m = mul<N, D>(p, link(r, n + om + on + oq));
                    m = mul<N, D>(m, link(mu, n + on + oq));
                    if (s == 0) m = mul<N, D>(m, link(nu, n + oq));
                    else m = mul<N, N>(m, link(nu, n + on + oq));
                    cb.add(q == 0 ? re_trace_mul<N, D>(m, link(r, n)) : re_trace_mul<N, N>(m, link(r, n + oq)));
                }
            }
        }
        acc += a.c[0] * pl.below(3 - w) + a.c[1] * rc.below(3) + a.c[2] * cb.below(4);
    }
    const double s = block_sum<kActionBlock>(acc);
    if (threadIdx.x == 0) {
        a.partials[blockIdx.x] = s;
        for (int i = blockIdx.x + gridDim.x; i < a.blocks; i += gridDim.x) a.partials[i] = 0.0;
    }
}

// FP64: the fixed point of fixed.cuh (FP32 remainders: their rounding is
// random from loop to loop, 2^-54 of one); the class sums are exact.  Links
// from planes made once per call (PLANES), or converted at each of their 23
// reads: two operations per real on the FP64 pipe, which then bounds the
// kernel, for callers without a workspace for the planes; the same bits.
template <bool PLANES> struct Fixed {
    using M = FMat;
    static constexpr int kMinBlocks = 2, kWords = 9;
    using Word = int4;
    FxPlanes planes;
    const double *links;
    int64_t V;

    __device__ __forceinline__ explicit Fixed(const ReduceArgs &a, int64_t v)
        : planes{static_cast<char *>(a.planes), (v + 31) / 32 * FxPlanes::BYTES},
          links(static_cast<const double *>(a.links)), V(v)
    {
    }
    __device__ __forceinline__ M link(int mu, int64_t n) const
    {
        if constexpr (PLANES) return planes.mat(planes.at(n), mu);
        else return fx_remainder(fx_load_link(links, V, mu, n));
    }
    template <int FB> __device__ __forceinline__ static M mul(const M &x, const M &y)
    {
        FAcc acc;
        fx_zero(acc);
        fx_mul_acc<N, FB>(acc, x, y);
        return fx_round<kUnit, FB == N ? 1 : -1>(acc);
    }
    __device__ __forceinline__ static bool bad(const M &x) { return fx_poisoned(x); }
    __device__ __forceinline__ static void mark(M &x) { x.rh[0][0] = kPoison; }
    template <int STRIDE> __device__ __forceinline__ static void put(Word *p, const M &x)
    {
#pragma unroll
        for (int e = 0; e < 9; ++e)
            p[e * STRIDE] = make_int4(x.rh[e / 3][e % 3], __float_as_int(x.rl[e / 3][e % 3]), x.ih[e / 3][e % 3],
                                      __float_as_int(x.il[e / 3][e % 3]));
    }
    template <int STRIDE> __device__ __forceinline__ static M get(const Word *p)
    {
        M x;
#pragma unroll
        for (int e = 0; e < 9; ++e) {
            const int4 v = p[e * STRIDE];
            x.rh[e / 3][e % 3] = v.x;
            x.rl[e / 3][e % 3] = __int_as_float(v.y);
            x.ih[e / 3][e % 3] = v.z;
            x.il[e / 3][e % 3] = __int_as_float(v.w);
        }
        return x;
    }
    struct Traces {
        long long v = 0; // units 2^-56
        float c = 0.f;
        __device__ __forceinline__ void add(const M &x, const M &y)
        {
            const FSum t = fx_re_trace_dag(x, y); // units 2^-60
            v += (t.v + 8) >> 4;
            c = fmaf(0.0625f, t.c, c);
        }
        __device__ __forceinline__ double below(int n) const
        {
            return ((double)(((3ll * n) << 56) - v) - (double)c) * 0x1p-56;
        }
    };
};

// The loops of 32 sites per block, a quarter of them on each of its four
// warps.  From the corners L_{mu nu}(n) = U_mu(n) U_nu(n+mu), three per warp
// and shared, every loop is the trace of a product X Y^dag of two halves:
//   plaquette            X = L_{mu nu},                  Y = L_{nu mu}
//   rectangle            X = U_mu U_mu(+mu) U_nu(+2mu),  Y = L_{nu mu} U_mu(+mu+nu)
//   cube from n          X = L_{xy} U_z(+x+y),           Y = L_{zy} U_x(+z+y),
// (x, y, z) the three rotations of the directions that warp w leaves out w
// of; and the cube loop that misses n and its opposite corner,
//   X = U_b(+a) U_a(+b)^dag U_c(+b),  Y = U_c(+a) U_a(+c)^dag U_b(+c).
// 80 matrix products and 92 link loads per site against 124 and 192 for the
// loops walked one by one.  Rolled loops: the halves are one piece of code
// for six of a warp's loops, as the instruction cache holds few of the
// fixed-point products.
// 24^3x48 FP64: 24.66 -> 1.81 ms (in floating point, loop by loop, bound by the
// FP64 pipe); 16^3x32: issue 49 %, two blocks of 215 registers an SM.
template <typename P, typename I>
__global__ void __launch_bounds__(kActionBlock, P::kMinBlocks)
    action_loops(const __grid_constant__ ReduceArgs a, const __grid_constant__ LoopTable tab)
{
    using M = typename P::M;
    using Word = typename P::Word;
    extern __shared__ __align__(16) unsigned char smem[];
    const Sites<I> g = make_sites<I>(a.dims);
    const P src(a, (int64_t)g.V);
    const int w = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
    // 12 corners of 32 sites, then one matrix of each thread
    Word *corners = reinterpret_cast<Word *>(smem) + lane;
    Word *own = reinterpret_cast<Word *>(smem) + 12 * P::kWords * 32 + threadIdx.x;
    const auto corner = [&](int mu, int nu) { return corners + (mu * 3 + ((nu - mu) & 3) - 1) * (P::kWords * 32); };
    double acc = 0.0;
    const I nvb = (g.V + 31) / 32;
    for (I vb = blockIdx.x; vb < nvb; vb += gridDim.x) {
        const I site = vb * 32 + lane;
        const I n = site < g.V ? site : g.V - 1;
        Coord c;
        if constexpr (sizeof(I) == 4) c = coord_fast(g, a.div, n);
        else c = coord_in(g, n);
        const auto up = [&](int mu) { return hop_offset(g, c, mu, 1); };
        const I ow = up(w);
        bool bad = false;
        {
            const M u = src.link(w, n);
            bad = P::bad(u);
#pragma unroll 1
            for (int j = 0; j < 4; ++j) {
                const M y = src.link((w + j) & 3, n + ow);
                M p = P::template mul<N>(u, y);
                if (P::bad(u) || P::bad(y)) {
                    P::mark(p);
                    bad = true;
                }
                if (j == 0) P::template put<kActionBlock>(own, p);
                else P::template put<32>(corner(w, (w + j) & 3), p);
            }
        }
        __syncthreads();
        typename P::Traces pl, rc, cb;
#pragma unroll 1
        for (int nu = w + 1; nu < 4; ++nu) {
            const M x = P::template get<32>(corner(w, nu)), y = P::template get<32>(corner(nu, w));
            bad = bad || P::bad(x) || P::bad(y);
            pl.add(x, y);
        }
#pragma unroll 1
        for (int it = 0; it < 6; ++it) {
            // X = A B, Y = C D
            const int x = (w + 1 + it % 3) & 3;
            const int y = it < 3 ? w : (w + 1 + (it + 1) % 3) & 3, z = it < 3 ? w : (w + 1 + (it + 2) % 3) & 3;
            I nb, nd;
            if (it < 3) { // rectangle, x = nu
                Coord c1 = c;
                step_up(g, c1, w);
                nb = n + ow + hop_offset(g, c1, w, 1);
                nd = n + ow + up(x);
            } else {
                nb = n + up(x) + up(y);
                nd = n + up(z) + up(y);
            }
            M h;
            {
                const M A = it < 3 ? P::template get<kActionBlock>(own) : P::template get<32>(corner(x, y));
                const M B = src.link(it < 3 ? x : z, nb);
                bad = bad || P::bad(A) || P::bad(B);
                h = P::template mul<N>(A, B);
            }
            const M C = P::template get<32>(it < 3 ? corner(x, w) : corner(z, y));
            const M E = src.link(it < 3 ? w : x, nd);
            bad = bad || P::bad(C) || P::bad(E);
            const M k = P::template mul<N>(C, E);
            if (it < 3) rc.add(h, k);
            else cb.add(h, k);
        }
        {
            const int da = (w + 1) & 3;
#pragma unroll 1
            for (int h = 0; h < 2; ++h) {
                const int p = (w + (h == 0 ? 2 : 3)) & 3, q = (w + (h == 0 ? 3 : 2)) & 3;
                const M A = src.link(p, n + up(da)), B = src.link(da, n + up(p)), E = src.link(q, n + up(p));
                bad = bad || P::bad(A) || P::bad(B) || P::bad(E);
                const M z = P::template mul<N>(P::template mul<D>(A, B), E);
                if (h == 0) P::template put<kActionBlock>(own, z);
                else cb.add(P::template get<kActionBlock>(own), z);
            }
        }
        if (site < g.V) {
            if (bad) acc += walked_loops(a, tab, (int64_t)n, w);
            else acc += a.c[0] * pl.below(3 - w) + a.c[1] * rc.below(3) + a.c[2] * cb.below(4);
        }
        __syncthreads(); // before the corners of the next sites
    }
    const double s = block_sum<kActionBlock>(acc);
    if (threadIdx.x == 0) {
        a.partials[blockIdx.x] = s;
        for (int i = blockIdx.x + gridDim.x; i < a.blocks; i += gridDim.x) a.partials[i] = 0.0;
    }
}

// The links of FP64 fields as planes with FP32 remainders, for action_loops.
__global__ void __launch_bounds__(kBlock) action_planes(const double *__restrict__ links, FxPlanes planes, int64_t V)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < 4 * V;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int mu = direction_of(i, V);
        const int64_t n = i - mu * V;
        planes.store<false>(planes.at(n), mu, fx_remainder(fx_load_link(links, V, mu, n)));
    }
}

// The same number in FP64.  A conversion takes as long as an FMA on the FP64
// pipe; for normal FP32 numbers it is the exponent moved by integer operations.
__device__ __forceinline__ double widen(float x)
{
    const unsigned u = __float_as_uint(x);
    return __hiloint2double((int)((((u >> 3) & 0x0fffffffu) + 0x38000000u) | (u & 0x80000000u)), (int)(u << 29));
}
__device__ __forceinline__ bool is_normal(float x)
{
    const unsigned e = __float_as_uint(x) & 0x7f800000u;
    return e - 0x00800000u < 0x7f000000u;
}

// Sum of the squares of a link's momenta, the same for the same values in
// either precision: one FP64 operation each where it was three (30 -> 13 us
// at 16^3x32 FP32, that pipe's rate).
template <typename R> __device__ __forceinline__ double sum_of_squares(const R p[8])
{
    double v = 0.0;
    if constexpr (sizeof(R) == 4) {
        bool normal = true;
#pragma unroll
        for (int c = 0; c < 8; ++c) normal = normal && is_normal(p[c]);
        if (normal) {
#pragma unroll
            for (int c = 0; c < 8; ++c) {
                const double x = widen(p[c]);
                v = fma(x, x, v);
            }
            return v;
        }
    }
#pragma unroll
    for (int c = 0; c < 8; ++c) v = fma((double)p[c], (double)p[c], v);
    return v;
}

template <typename R> __global__ void __launch_bounds__(kBlock) kinetic_partials(const ReduceArgs a)
{
    const int64_t V = (int64_t)a.dims[0] * a.dims[1] * a.dims[2] * a.dims[3];
    const R *__restrict__ mom = static_cast<const R *>(a.mom);
    double acc = 0.0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < 4 * V;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int mu = direction_of(i, V);
        R p[8];
        load_algebra(mom, V, mu, i - mu * V, p);
        acc += sum_of_squares(p);
    }
    const double s = block_sum<kBlock>(acc);
    if (threadIdx.x == 0) a.partials[blockIdx.x] = 0.5 * s;
}

// One block of 1024 threads adds the partials in a fixed order and scales
// the total.
constexpr int kFinish = 1024;
__global__ void __launch_bounds__(kFinish) finish_sum(const double *partials, int count,
                                                      double scale, double *out)
{
    __shared__ double warp_part[kFinish / 32];
    double v = 0.0;
    for (int i = threadIdx.x; i < count; i += kFinish) v += partials[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) warp_part[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double s = warp_part[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) *out = scale * s;
    }
}

// Departure of the stored links from SU(3), in FP64 whatever the storage
// precision: with rows r0, r1 stored and r2 = conj(r0 x r1) rebuilt (so r2
// is orthogonal to both and det U = |r2|^2), U^dag U = 1 and det U = 1 hold
// exactly when |r0|^2 = |r1|^2 = 1 and <r0, r1> = 0; the measure is
// max(| |r0|^2 - 1 |, | |r1|^2 - 1 |, |<r0, r1>|, | |r2|^2 - 1 |) over links.
template <typename R> __global__ void __launch_bounds__(kBlock) unitarity_partials(const ReduceArgs a)
{
    const Geom g = make_geom(a.dims);
    const R *__restrict__ links = static_cast<const R *>(a.links);
    double worst = 0.0;
    const int64_t nlinks = 4 * g.V;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nlinks;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int mu = direction_of(i, g.V);
        const int64_t n = i - mu * g.V;
        const Mat<R> u = load_link(links, g.V, mu, n);
        double n0 = 0.0, n1 = 0.0, cr = 0.0, ci = 0.0;
#pragma unroll
        for (int j = 0; j < 3; ++j) {
            const double ar = u.re[0][j], ai = u.im[0][j], br = u.re[1][j], bi = u.im[1][j];
            n0 += ar * ar + ai * ai;
            n1 += br * br + bi * bi;
            cr += ar * br + ai * bi; // <r0, r1> = sum conj(a) b
            ci += ar * bi - ai * br;
        }
        const double c2 = cr * cr + ci * ci;
        const double d = fmax(fmax(fabs(n0 - 1.0), fabs(n1 - 1.0)),
                              fmax(sqrt(c2), fabs(n0 * n1 - c2 - 1.0)));
        worst = fmax(worst, d);
    }
    __shared__ double warp_part[kBlock / 32];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) worst = fmax(worst, __shfl_down_sync(0xffffffffu, worst, o));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) warp_part[warp] = worst;
    __syncthreads();
    if (warp == 0) {
        double m = lane < kBlock / 32 ? warp_part[lane] : 0.0;
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
        if (lane == 0) a.partials[blockIdx.x] = m;
    }
}

__global__ void __launch_bounds__(kFinish) finish_max(const double *partials, int count, double *out)
{
    __shared__ double warp_part[kFinish / 32];
    double v = 0.0;
    for (int i = threadIdx.x; i < count; i += kFinish) v = fmax(v, partials[i]);
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_down_sync(0xffffffffu, v, o));
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) warp_part[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double m = warp_part[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) m = fmax(m, __shfl_down_sync(0xffffffffu, m, o));
        if (lane == 0) *out = m;
    }
}

// Library-held scratch of the allocation-free action entry point: one double
// per reduction block.  4096 doubles = 32 KiB, held by every device that
// loads the library until the process exits.
constexpr int kFixedPartials = 4096;
static __device__ __align__(256) double g_fixed_partials[kFixedPartials];

} // namespace

int reduction_blocks(int device)
{
    static std::mutex mu;
    static int cached[64] = {0};
    if (device < 0 || device >= 64) return 0;
    std::lock_guard<std::mutex> lk(mu);
    if (cached[device] == 0) {
        int sms = 0;
        if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, device) != cudaSuccess ||
            sms <= 0)
            return 0;
        cached[device] = sms * 4;
    }
    return cached[device];
}

template <typename P, typename I> static cudaError_t launch_action_t(const ReduceArgs &a, cudaStream_t st)
{
    constexpr int bytes = (12 * 32 + kActionBlock) * P::kWords * (int)sizeof(typename P::Word);
    if constexpr (bytes > 48 * 1024) {
        const cudaError_t e = cudaFuncSetAttribute(action_loops<P, I>, cudaFuncAttributeMaxDynamicSharedMemorySize, bytes);
        if (e != cudaSuccess) return e;
    }
    // the resident blocks (a.blocks is four per SM)
    const int grid = a.blocks * P::kMinBlocks / 4 > 0 ? a.blocks * P::kMinBlocks / 4 : 1;
    action_loops<P, I><<<grid, kActionBlock, bytes, st>>>(a, loop_table());
    return cudaGetLastError();
}

size_t action_plane_bytes(const int dims[4])
{
    return 4 * fx_plane_bytes((int64_t)dims[0] * dims[1] * dims[2] * dims[3]);
}

cudaError_t launch_action(const ReduceArgs &args, cudaStream_t st)
{
    ReduceArgs a = args;
    stride_magic(a.dims, a.div);
    const int64_t V = (int64_t)a.dims[0] * a.dims[1] * a.dims[2] * a.dims[3];
    const bool i32 = sites_fit_int(V);
    cudaError_t e;
    if (a.precision != LQCD_F64) {
        // the resident blocks, of which a.blocks is four per SM (one partial each)
        if (i32) action_loops_f32<int><<<a.blocks, kActionBlock, 0, st>>>(a);
        else action_loops_f32<int64_t><<<a.blocks, kActionBlock, 0, st>>>(a);
        e = cudaGetLastError();
    } else if (a.planes != nullptr && i32) {
        const FxPlanes p{static_cast<char *>(a.planes), (int64_t)fx_plane_bytes(V)};
        action_planes<<<(unsigned)((4 * V + kBlock - 1) / kBlock), kBlock, 0, st>>>(static_cast<const double *>(a.links), p, V);
        e = cudaGetLastError();
        if (e == cudaSuccess) e = launch_action_t<Fixed<true>, int>(a, st);
    } else {
        e = i32 ? launch_action_t<Fixed<false>, int>(a, st) : launch_action_t<Fixed<false>, int64_t>(a, st);
    }
    if (e != cudaSuccess) return e;
    finish_sum<<<1, kFinish, 0, st>>>(a.partials, a.blocks, a.scale, a.out);
    return cudaGetLastError();
}

cudaError_t launch_finish_sum(const double *partials, int count, double scale, double *out,
                              cudaStream_t st)
{
    finish_sum<<<1, kFinish, 0, st>>>(partials, count, scale, out);
    return cudaGetLastError();
}

cudaError_t launch_kinetic(const ReduceArgs &a, cudaStream_t st)
{
    if (a.precision == LQCD_F64)
        kinetic_partials<double><<<a.blocks, kBlock, 0, st>>>(a);
    else
        kinetic_partials<float><<<a.blocks, kBlock, 0, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    finish_sum<<<1, kFinish, 0, st>>>(a.partials, a.blocks, 1.0, a.out);
    return cudaGetLastError();
}

cudaError_t launch_unitarity(const ReduceArgs &a, cudaStream_t st)
{
    if (a.precision == LQCD_F64)
        unitarity_partials<double><<<a.blocks, kBlock, 0, st>>>(a);
    else
        unitarity_partials<float><<<a.blocks, kBlock, 0, st>>>(a);
    cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    finish_max<<<1, kFinish, 0, st>>>(a.partials, a.blocks, a.out);
    return cudaGetLastError();
}

// The 34 loops of Eq. 18_3_27_30 as direction sequences from n:
// plaquettes (mu, nu, -mu, -nu) for mu < nu, rectangles (mu, mu, nu, -mu,
// -mu, -nu) for mu != nu, cubes (mu, s nu, t r, -mu, -s nu, -t r) for
// mu < nu < r and s, t = +-1.
const LoopTable &loop_table()
{
    static LoopTable tab = [] {
        LoopTable t{};
        int n = 0;
        auto put = [&](int cls, std::initializer_list<int> d) {
            Loop &l = t.l[n++];
            l.cls = (int8_t)cls;
            l.len = (int8_t)d.size();
            int j = 0;
            for (int v : d) l.d[j++] = (int8_t)v;
        };
        for (int mu = 1; mu <= 4; ++mu)
            for (int nu = mu + 1; nu <= 4; ++nu) put(0, {mu, nu, -mu, -nu});
        for (int mu = 1; mu <= 4; ++mu)
            for (int nu = 1; nu <= 4; ++nu)
                if (nu != mu) put(1, {mu, mu, nu, -mu, -mu, -nu});
        for (int mu = 1; mu <= 4; ++mu)
            for (int nu = mu + 1; nu <= 4; ++nu)
                for (int r = nu + 1; r <= 4; ++r)
                    for (int s = 1; s >= -1; s -= 2)
                        for (int q = 1; q >= -1; q -= 2)
                            put(2, {mu, s * nu, q * r, -mu, -s * nu, -q * r});
        t.count = n;
        return t;
    }();
    return tab;
}

namespace {

// Device address of g_fixed_partials on `device`, looked up once per device
// (the device must be current).  Host code cannot use the symbol itself: on
// the host it names a host-side stand-in, not device memory.
cudaError_t fixed_partials_address(int device, double **out)
{
    static std::mutex mu;
    static double *addr[64] = {nullptr};
    if (device < 0 || device >= 64) return cudaErrorInvalidDevice;
    std::lock_guard<std::mutex> lk(mu);
    if (addr[device] == nullptr) {
        void *p = nullptr;
        const cudaError_t e = cudaGetSymbolAddress(&p, g_fixed_partials);
        if (e != cudaSuccess) return e;
        if (p == nullptr) return cudaErrorInvalidSymbol;
        addr[device] = static_cast<double *>(p);
    }
    *out = addr[device];
    return cudaSuccess;
}

} // namespace

} // namespace lqcd

// Allocation-free variant of lqcd_gauge_action (declared in include/lqcd.h):
// the same argument checks and kernels, with the per-block partial sums kept
// in the fixed library-held array above instead of a caller workspace.
extern "C" int lqcd_gauge_action_noalloc(const lqcd_desc *desc, const void *links, double *action,
                                         void *stream)
{
    // NVTX range named after the entry point (no-op without a profiler)
    struct Range {
        Range() { nvtxRangePushA("lqcd_gauge_action_noalloc"); }
        ~Range() { nvtxRangePop(); }
    } const trace_range;
    int s = lqcd::check_desc(desc);
    if (s) return s;
    if ((s = lqcd::check_ptrs({links}))) return s;
    if (action == nullptr) return LQCD_ERR_ARG;
    if (((uintptr_t)action & 7u) != 0) return LQCD_ERR_ALIGN;
    int dev = 0;
    cudaError_t e = cudaGetDevice(&dev);
    if (e != cudaSuccess) return lqcd::cuda_status(e);
    const int blocks = lqcd::reduction_blocks(dev);
    if (blocks <= 0) return lqcd::cuda_status(cudaErrorInvalidDevice);
    if (blocks > lqcd::kFixedPartials) return LQCD_ERR_CAPACITY;
    double *partials = nullptr;
    e = lqcd::fixed_partials_address(dev, &partials);
    if (e != cudaSuccess) return lqcd::cuda_status(e);
    lqcd::ReduceArgs a{};
    for (int i = 0; i < 4; ++i) a.dims[i] = desc->dims[i];
    a.precision = desc->precision;
    a.links = links;
    a.c[0] = desc->c_plaq;
    a.c[1] = desc->c_rect;
    a.c[2] = desc->c_cube;
    a.scale = desc->beta / 3.0;
    a.partials = partials;
    a.blocks = blocks;
    a.out = action;
    return lqcd::cuda_status(lqcd::launch_action(a, static_cast<cudaStream_t>(stream)));
}
