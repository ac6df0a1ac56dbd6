// Molecular-dynamics steps and layout conversions, all streaming kernels
// (one thread per link or per 16-byte lane, grid-stride, coalesced 16-byte
// loads and stores of the structure-of-arrays planes).
//   momentum step  p^a += dt f^a                      (f = -dS/domega, Eq. 18_7_25_1)
//   link step      U <- exp(i dt sum_a p^a T_a) U     (left flow of Eq. 18_1_29_3)
//   links from omega  U = exp(i sum_a omega^a T_a)    (Eq. 18_1_29_3)
//   pack / unpack  full 3x3 complex <-> first two rows
#include "async_copy.cuh"
#include "gaussian.cuh"
#include "kernels.h"
#include "link_step_fx.cuh"
#include "su3.cuh"

namespace lqcd {

namespace {

constexpr int kBlock = 256;

int64_t volume(const int dims[4])
{
    return (int64_t)dims[0] * dims[1] * dims[2] * dims[3];
}

unsigned grid_for(int64_t items, int block = kBlock)
{
    int64_t g = (items + block - 1) / block;
    if (g < 1) g = 1;
    if (g > ((int64_t)1 << 30)) g = (int64_t)1 << 30;
    return (unsigned)g;
}

// Direction of link i of the link-major order (i = mu V + n, i < 4 V): three
// comparisons instead of a 64-bit division.
__device__ __forceinline__ int direction_of(int64_t i, int64_t V)
{
    return (int)(i >= V) + (int)(i >= 2 * V) + (int)(i >= 3 * V);
}

// p += dt f over 16-byte lanes of the algebra planes.
template <typename R>
__global__ void __launch_bounds__(kBlock) update_momenta(typename Vec<R>::type *__restrict__ p,
                                                         const typename Vec<R>::type *__restrict__ f,
                                                         int64_t lanes, R dt)
{
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < lanes;
         i += (int64_t)gridDim.x * blockDim.x) {
        auto a = p[i];
        const auto b = __ldg(f + i);
        if constexpr (Vec<R>::W == 4) {
            a.x = fma(dt, b.x, a.x);
            a.y = fma(dt, b.y, a.y);
            a.z = fma(dt, b.z, a.z);
            a.w = fma(dt, b.w, a.w);
        } else {
            a.x = fma(dt, b.x, a.x);
            a.y = fma(dt, b.y, a.y);
        }
        p[i] = a;
    }
}

// U <- exp(i P) U (FROM_UNIT: U = exp(i P)), rows 0 and 1 only, then
// Gram-Schmidt, for one link; p the components of P, load() gives U.
template <typename R, bool FROM_UNIT, typename Load>
__device__ __forceinline__ void link_step(R *__restrict__ links, const R p[8], int64_t V, int mu, int64_t n, const Load &load)
{
    const Mat<R> e = exp_i_hermitian(algebra_matrix(p));
    Mat<R> u;
    if constexpr (FROM_UNIT) {
        u = e;
    } else {
        const Mat<R> v = load();
#pragma unroll
        for (int r = 0; r < 2; ++r)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                R re = R(0), im = R(0);
#pragma unroll
                for (int k = 0; k < 3; ++k) {
                    re = fma(e.re[r][k], v.re[k][j], re);
                    re = fma(-e.im[r][k], v.im[k][j], re);
                    im = fma(e.re[r][k], v.im[k][j], im);
                    im = fma(e.im[r][k], v.re[k][j], im);
                }
                u.re[r][j] = re;
                u.im[r][j] = im;
            }
    }
    reunitarise(u);
    store_link(links, V, mu, n, u);
}

// The FP64 step in floating point, for links that fx_link_step leaves.
template <bool FROM_UNIT>
__device__ __noinline__ void link_step_floating(double *links, const double *mom, double dt, int64_t V, int mu, int64_t n)
{
    double p[8];
    load_algebra(mom, V, mu, n, p);
#pragma unroll
    for (int c = 0; c < 8; ++c) p[c] *= dt;
    link_step<double, FROM_UNIT>(links, p, V, mu, n, [&] { return load_link(links, V, mu, n); });
}

// The FP64 step of link (n, mu).
template <bool FROM_UNIT>
__device__ __forceinline__ void update_link(double *__restrict__ links, const double *__restrict__ mom, double dt, int64_t V,
                                            int mu, int64_t n)
{
    double p[8];
    load_algebra(mom, V, mu, n, p);
#pragma unroll
    for (int c = 0; c < 8; ++c) p[c] *= dt;
    double2 *u = reinterpret_cast<double2 *>(links) + (int64_t)mu * 6 * V + n;
    double r[12] = {1.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 0.0, 1.0, 0.0, 0.0, 0.0};
    if constexpr (!FROM_UNIT) {
#pragma unroll
        for (int q = 0; q < 6; ++q) {
            const double2 v = u[q * V];
            r[2 * q] = v.x;
            r[2 * q + 1] = v.y;
        }
    }
    if (fx_link_step(p, r)) {
#pragma unroll
        for (int q = 0; q < 6; ++q) u[q * V] = make_double2(r[2 * q], r[2 * q + 1]);
    } else {
        link_step_floating<FROM_UNIT>(links, mom, dt, V, mu, n);
    }
}

// Threads of an FP64 link-step block and resident blocks (18x14x22x36, dt 0.05:
// 200 us with 3 blocks of 128, 203 with 4 of 128, 210 with 2 of 192).
constexpr int kFxStepBlock = 128, kFxStepBlocks = 3;

// The link and algebra planes share the site index.
template <bool FROM_UNIT>
__global__ void __launch_bounds__(kFxStepBlock, kFxStepBlocks)
    update_links_f64(double *__restrict__ links, const double *__restrict__ mom, int64_t V, double dt)
{
    const int64_t nlinks = 4 * V;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nlinks;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int mu = direction_of(i, V);
        update_link<FROM_UNIT>(links, mom, dt, V, mu, i - mu * V);
    }
}

// The link step for the links of a batch of lattices: the persistent CTAs
// walk the concatenated link ranges.
struct LinkBatch {
    int n;
    int64_t total;
    int64_t begin[kMaxBatch + 1]; // first link of each lattice in the concatenation
    int64_t V[kMaxBatch];
    void *links[kMaxBatch];
    const void *mom[kMaxBatch];

    // The lattice of link i of the concatenation, from a near one's number.
    __device__ __forceinline__ int lattice_of(int64_t i, int c) const
    {
        while (c > 0 && i < begin[c]) --c;
        while (c + 1 < n && i >= begin[c + 1]) ++c;
        return c;
    }
};

__global__ void __launch_bounds__(kFxStepBlock, kFxStepBlocks) update_links_f64_batched(const __grid_constant__ LinkBatch B, double dt)
{
    int c = 0;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < B.total;
         i += (int64_t)gridDim.x * blockDim.x) {
        c = B.lattice_of(i, c);
        const int64_t V = B.V[c];
        const int64_t l = i - B.begin[c];
        const int mu = direction_of(l, V);
        update_link<false>(static_cast<double *>(B.links[c]), static_cast<const double *>(B.mom[c]), dt, V, mu, l - mu * V);
    }
}

// FP32 step.  It moves 128 bytes a link and executes about 450 instructions on
// them; loading and computing took turns (217 us at 32^3x64, the bytes alone
// 159, the instructions 136).  A thread passes over many links and copies the
// next one's momentum and link (five words) into shared memory while it
// computes: 209 -> 174 us at 32^3x64, 70 -> 59 at 24^3x48.  4 blocks of 256
// as many as the registers allow; 3: 177, 8 of 128: 175.
constexpr int kStepBlock = 256, kStepBlocks = 4, kStepWords = 5;

// A link: the fields of its lattice, its direction and site.
struct StepLink {
    float *links;
    const float *mom;
    int64_t V, n;
    int mu;
};

// Link i of one lattice, or of the concatenation of a batch.
struct LatticeLinks {
    float *links;
    const float *mom;
    int64_t V;
    __device__ __forceinline__ int64_t total() const { return 4 * V; }
    __device__ __forceinline__ StepLink link(int64_t i, int &) const
    {
        const int mu = direction_of(i, V);
        return {links, mom, V, i - mu * V, mu};
    }
};
struct BatchLinks {
    const LinkBatch &B;
    __device__ __forceinline__ int64_t total() const { return B.total; }
    __device__ __forceinline__ StepLink link(int64_t i, int &c) const
    {
        c = B.lattice_of(i, c);
        const int64_t V = B.V[c], l = i - B.begin[c];
        const int mu = direction_of(l, V);
        return {static_cast<float *>(B.links[c]), static_cast<const float *>(B.mom[c]), V, l - mu * V, mu};
    }
};

template <bool FROM_UNIT> __device__ __forceinline__ void fetch_step(float4 *slot, const StepLink &s)
{
    const float4 *p = reinterpret_cast<const float4 *>(s.mom) + (int64_t)s.mu * 2 * s.V + s.n;
#pragma unroll
    for (int q = 0; q < 2; ++q) copy_async(slot + q * kStepBlock, p + q * s.V);
    if constexpr (!FROM_UNIT) {
        const float4 *u = reinterpret_cast<const float4 *>(s.links) + (int64_t)s.mu * 3 * s.V + s.n;
#pragma unroll
        for (int q = 0; q < 3; ++q) copy_async(slot + (2 + q) * kStepBlock, u + q * s.V);
    }
}

template <bool FROM_UNIT, typename Links> __device__ __forceinline__ void step_links(const Links &links, float dt)
{
    __shared__ float4 ring[2 * kStepWords * kStepBlock];
    const int64_t total = links.total(), step = (int64_t)gridDim.x * kStepBlock;
    int64_t i = blockIdx.x * (int64_t)kStepBlock + threadIdx.x;
    if (i >= total) return;
    float4 *slot = ring + threadIdx.x, *next = slot + kStepWords * kStepBlock;
    int c = 0;
    StepLink s = links.link(i, c);
    fetch_step<FROM_UNIT>(slot, s);
    copies_commit();
    for (;;) {
        i += step;
        StepLink s2 = s;
        if (i < total) {
            s2 = links.link(i, c);
            fetch_step<FROM_UNIT>(next, s2);
        }
        copies_commit();
        copies_wait<1>(); // this link's
        const float4 a = slot[0], b = slot[kStepBlock];
        const float p[8] = {a.x * dt, a.y * dt, a.z * dt, a.w * dt, b.x * dt, b.y * dt, b.z * dt, b.w * dt};
        link_step<float, FROM_UNIT>(s.links, p, s.V, s.mu, s.n, [&] {
            Mat<float> u;
#pragma unroll
            for (int q = 0; q < 3; ++q) {
                const float4 v = slot[(2 + q) * kStepBlock];
                u.re[2 * q / 3][2 * q % 3] = v.x;
                u.im[2 * q / 3][2 * q % 3] = v.y;
                u.re[(2 * q + 1) / 3][(2 * q + 1) % 3] = v.z;
                u.im[(2 * q + 1) / 3][(2 * q + 1) % 3] = v.w;
            }
            rebuild_row2(u);
            return u;
        });
        if (i >= total) break;
        s = s2;
        float4 *const t = slot;
        slot = next;
        next = t;
    }
}

template <bool FROM_UNIT>
__global__ void __launch_bounds__(kStepBlock, kStepBlocks) update_links_f32(float *links, const float *mom, int64_t V, float dt)
{
    step_links<FROM_UNIT>(LatticeLinks{links, mom, V}, dt);
}

__global__ void __launch_bounds__(kStepBlock, kStepBlocks) update_links_f32_batched(const __grid_constant__ LinkBatch B, float dt)
{
    step_links<false>(BatchLinks{B}, dt);
}

// Chain rule through U = exp(X) U0, X = i W, W = omega.T (Eq. 18_1_29_3).
// A change d omega moves U by the left perturbation exp(i delta.T) with
// i delta.T = phi(ad_X)(i d omega.T), phi(z) = (e^z - 1)/z.  The force gives
// the left derivative dS/d delta^b = -f^b, so
//     dS/d omega^a = components of phi(-ad_X)(-i F),   F = f.T,
// since phi(ad_X) is orthogonal-adjoint to phi(-ad_X) on su(3).  Writing the
// series terms as -i H_n with Hermitian H_n:
//     H_0 = F,   H_n = -i [W, H_{n-1}] / (n+1),   A = sum_n H_n,
//     dS/d omega^a = -tr(lambda_a A)  (= -f^a at omega = 0).
// With H_n = h^a T_a and [T_a, T_b] = i f_abc T_c that is
//     h_n = w x h_{n-1} / (n+1),  (w x h)_c = f_abc w_a h_b,  dS/d omega = -sum_n h_n
// on eight components (54 FMAs a term instead of the 252 of two matrix
// products): 719 -> 281 us at 32^3x64 FP32 (issue bound; its 96 bytes a link
// would take 119).
// The series stops once (2 |W|_F)^n / (n+1)!, a bound on |H_n|/|F|, is below
// the working precision.
// r = w x h, v = w / 2, s = sqrt(3) w / 2.
template <typename R>
__device__ __forceinline__ void cross8(const R w[8], const R v[8], const R s[8], const R h[8], R r[8])
{
    const auto add = [&](R &t, const R u[8], int a, int b) { t = fma(u[a - 1], h[b - 1], fma(-u[b - 1], h[a - 1], t)); };
#pragma unroll
    for (int a = 0; a < 8; ++a) r[a] = R(0);
    add(r[0], w, 2, 3);
    add(r[0], v, 4, 7);
    add(r[0], v, 6, 5);
    add(r[1], w, 3, 1);
    add(r[1], v, 4, 6);
    add(r[1], v, 5, 7);
    add(r[2], w, 1, 2);
    add(r[2], v, 4, 5);
    add(r[2], v, 7, 6);
    add(r[3], v, 7, 1);
    add(r[3], v, 6, 2);
    add(r[3], v, 5, 3);
    add(r[3], s, 5, 8);
    add(r[4], v, 1, 6);
    add(r[4], v, 7, 2);
    add(r[4], v, 3, 4);
    add(r[4], s, 8, 4);
    add(r[5], v, 5, 1);
    add(r[5], v, 2, 4);
    add(r[5], v, 3, 7);
    add(r[5], s, 7, 8);
    add(r[6], v, 1, 4);
    add(r[6], v, 2, 5);
    add(r[6], v, 6, 3);
    add(r[6], s, 8, 6);
    add(r[7], s, 4, 5);
    add(r[7], s, 6, 7);
}

// 1 / (n + 1), n = 0 to 40: from a table, a division is 20 instructions.
struct Inverses {
    double d[41];
    float f[41];
    constexpr Inverses() : d(), f()
    {
        for (int n = 0; n <= 40; ++n) {
            d[n] = 1.0 / (double)(n + 1);
            f[n] = (float)d[n];
        }
    }
};
__constant__ const Inverses kInverses{};

template <typename R>
__global__ void __launch_bounds__(kBlock) omega_gradient(const R *__restrict__ omega,
                                                         const R *__restrict__ force,
                                                         R *__restrict__ grad, int64_t V)
{
    constexpr int NMAX = sizeof(R) == 8 ? 40 : 24;
    const R eps = sizeof(R) == 8 ? R(1e-17) : R(1e-9);
    const int64_t nlinks = 4 * V;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nlinks;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int mu = direction_of(i, V);
        const int64_t n = i - mu * V;
        R w[8], h[8], acc[8];
        load_algebra(omega, V, mu, n, w);
        load_algebra(force, V, mu, n, h);
        R ww = R(0);
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            acc[a] = h[a];
            ww = fma(w[a], w[a], ww);
        }
        const R bound = R(2) * sqrt(R(0.5) * ww); // 2 |W|_F
        R v[8], s[8];
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            v[a] = R(0.5) * w[a];
            s[a] = R(0.86602540378443864676) * w[a];
        }
        R est = R(1);
        for (int k = 1; k <= NMAX; ++k) {
            R t[8];
            cross8(w, v, s, h, t);
            R inv;
            if constexpr (sizeof(R) == 8) inv = kInverses.d[k];
            else inv = kInverses.f[k];
#pragma unroll
            for (int a = 0; a < 8; ++a) {
                h[a] = t[a] * inv;
                acc[a] += h[a];
            }
            est *= bound * inv;
            if (est < eps) break;
        }
#pragma unroll
        for (int a = 0; a < 8; ++a) acc[a] = -acc[a];
        store_algebra(grad, V, mu, n, acc);
    }
}

// Real r (0..NR-1) of item (n, mu) of a structure-of-arrays field with NR
// reals per item and W-wide lanes.
template <typename R, int NR>
__device__ __forceinline__ int64_t soa_index(int64_t V, int mu, int64_t n, int r)
{
    constexpr int W = Vec<R>::W;
    return (((int64_t)mu * (NR / W) + r / W) * V + n) * W + r % W;
}

// Precision conversion of a link (NR = 12) or algebra (NR = 8) field; the
// stored reals are converted one by one (FP32 -> FP64 exactly).
template <typename RS, typename RD, int NR>
__global__ void __launch_bounds__(kBlock) convert_field(const RS *__restrict__ src,
                                                        RD *__restrict__ dst, int64_t V)
{
    const int64_t nitems = 4 * V;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nitems;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int mu = direction_of(i, V);
        const int64_t n = i - mu * V;
#pragma unroll
        for (int r = 0; r < NR; ++r)
            dst[soa_index<RD, NR>(V, mu, n, r)] = (RD)src[soa_index<RS, NR>(V, mu, n, r)];
    }
}

// full [V][4][3][3] (re, im) -> compact link layout (rows 0, 1)
template <typename R>
__global__ void __launch_bounds__(kBlock) pack(const R *__restrict__ full, R *__restrict__ links,
                                               int64_t V)
{
    const int64_t nlinks = 4 * V;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nlinks;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int mu = direction_of(i, V);
        const int64_t n = i - mu * V;
        const R *src = full + (n * 4 + mu) * 18;
        Mat<R> u;
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                u.re[r][j] = src[(3 * r + j) * 2];
                u.im[r][j] = src[(3 * r + j) * 2 + 1];
            }
        store_link(links, V, mu, n, u);
    }
}

template <typename R>
__global__ void __launch_bounds__(kBlock) unpack(const R *__restrict__ links, R *__restrict__ full,
                                                 int64_t V)
{
    const int64_t nlinks = 4 * V;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nlinks;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int mu = direction_of(i, V);
        const int64_t n = i - mu * V;
        const Mat<R> u = load_link(links, V, mu, n);
        R *dst = full + (n * 4 + mu) * 18;
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                dst[(3 * r + j) * 2] = u.re[r][j];
                dst[(3 * r + j) * 2 + 1] = u.im[r][j];
            }
    }
}

// Gram-Schmidt of rows 0 and 1 of every stored link in FP64 (row 2 is
// rebuilt on every load), rounded back to the storage precision.
template <typename R> __global__ void __launch_bounds__(kBlock) reunitarise_fp64(R *__restrict__ links, int64_t V)
{
    const int64_t nlinks = 4 * V;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nlinks;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int mu = direction_of(i, V);
        const int64_t n = i - mu * V;
        const Mat<R> u = load_link(links, V, mu, n);
        Mat<double> w;
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                w.re[r][j] = (double)u.re[r][j];
                w.im[r][j] = (double)u.im[r][j];
            }
        reunitarise(w);
        Mat<R> v;
#pragma unroll
        for (int r = 0; r < 3; ++r)
#pragma unroll
            for (int j = 0; j < 3; ++j) {
                v.re[r][j] = (R)w.re[r][j];
                v.im[r][j] = (R)w.im[r][j];
            }
        store_link(links, V, mu, n, v);
    }
}

// Word i of the counter-based SplitMix64 stream `seed` (Steele, Lea & Flood,
// "Fast splittable pseudorandom number generators", OOPSLA 2014):
// mix(seed + (i + 1) * golden gamma) with the published finaliser.
__device__ __forceinline__ uint64_t splitmix_word(uint64_t seed, uint64_t i)
{
    uint64_t z = seed + (i + 1) * 0x9E3779B97F4A7C15ull;
    z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
    z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
    return z ^ (z >> 31);
}

// Standard normal j of stream `seed`: the Box-Muller transform (cosine
// branch) of words 2j and 2j+1 as 53-bit uniforms, u1 in (0, 1], u2 in [0, 1).
__device__ __forceinline__ double gaussian_of(uint64_t seed, uint64_t j)
{
    const uint64_t w1 = splitmix_word(seed, 2 * j), w2 = splitmix_word(seed, 2 * j + 1);
    const double u1 = ((double)(w1 >> 11) + 1.0) * 0x1p-53;
    const double u2 = (double)(w2 >> 11) * 0x1p-53;
    return sqrt(-2.0 * log(u1)) * cos(2.0 * 3.141592653589793 * u2);
}

// The same for FP32 storage, to the bit (gaussian.cuh): 16^3x32 62 us, all by
// the FP64 evaluation 548; 2.7 x 10^9 normals compared.
__device__ const NormalTables kNormalTables{};

__device__ __noinline__ float gaussian_rounded(uint64_t seed, uint64_t j) { return (float)gaussian_of(seed, j); }

__device__ __forceinline__ float gaussian_f32(uint64_t seed, uint64_t j)
{
    float t, root;
    const float y = normal_of(splitmix_word(seed, 2 * j) >> 11, splitmix_word(seed, 2 * j + 1) >> 11, kNormalTables, t, root);
    return normal_is_rounded(y, t, root) ? y : gaussian_rounded(seed, j);
}

// p^a_{n,mu} = normal number (n*4 + mu)*8 + a of the stream.
template <typename R>
__global__ void __launch_bounds__(kBlock) gaussian_momenta(R *__restrict__ mom, int64_t V, uint64_t seed)
{
    const int64_t nlinks = 4 * V;
    for (int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; i < nlinks;
         i += (int64_t)gridDim.x * blockDim.x) {
        const int mu = direction_of(i, V);
        const int64_t n = i - mu * V;
        R p[8];
#pragma unroll
        for (int a = 0; a < 8; ++a) {
            const uint64_t j = (uint64_t)((n * 4 + mu) * 8 + a);
            if constexpr (sizeof(R) == 4) p[a] = gaussian_f32(seed, j);
            else p[a] = gaussian_of(seed, j);
        }
        store_algebra(mom, V, mu, n, p);
    }
}

} // namespace

cudaError_t launch_reunitarise(const MdArgs &a, cudaStream_t st)
{
    const int64_t V = volume(a.dims);
    if (a.precision == LQCD_F64)
        reunitarise_fp64<double><<<grid_for(4 * V), kBlock, 0, st>>>(static_cast<double *>(a.links), V);
    else
        reunitarise_fp64<float><<<grid_for(4 * V), kBlock, 0, st>>>(static_cast<float *>(a.links), V);
    return cudaGetLastError();
}

cudaError_t launch_gaussian_momenta(const MdArgs &a, cudaStream_t st)
{
    const int64_t V = volume(a.dims);
    if (a.precision == LQCD_F64)
        gaussian_momenta<double><<<grid_for(4 * V), kBlock, 0, st>>>(static_cast<double *>(a.mom_out), V, a.seed);
    else
        gaussian_momenta<float><<<grid_for(4 * V), kBlock, 0, st>>>(static_cast<float *>(a.mom_out), V, a.seed);
    return cudaGetLastError();
}

cudaError_t launch_update_momenta(const MdArgs &a, cudaStream_t st)
{
    const int64_t V = volume(a.dims);
    if (a.precision == LQCD_F64) {
        const int64_t lanes = 4 * 8 * V / 2;
        update_momenta<double><<<grid_for(lanes), kBlock, 0, st>>>(
            static_cast<double2 *>(a.mom_out), static_cast<const double2 *>(a.force), lanes, a.dt);
    } else {
        const int64_t lanes = 4 * 8 * V / 4;
        update_momenta<float><<<grid_for(lanes), kBlock, 0, st>>>(
            static_cast<float4 *>(a.mom_out), static_cast<const float4 *>(a.force), lanes,
            (float)a.dt);
    }
    return cudaGetLastError();
}

namespace {

// The blocks of `block` threads for n links, at most `per_sm` on every SM.
unsigned step_grid(int64_t n, int block, int per_sm)
{
    int dev = 0, sms = 1;
    if (cudaGetDevice(&dev) == cudaSuccess) cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    const int64_t blocks = (n + block - 1) / block, cap = (int64_t)(sms > 0 ? sms : 1) * per_sm;
    return (unsigned)(blocks < 1 ? 1 : (blocks < cap ? blocks : cap));
}

template <bool FROM_UNIT> cudaError_t launch_step(const MdArgs &a, double dt, cudaStream_t st)
{
    const int64_t V = volume(a.dims);
    if (a.precision == LQCD_F64)
        update_links_f64<FROM_UNIT><<<grid_for(4 * V, kFxStepBlock), kFxStepBlock, 0, st>>>(
            static_cast<double *>(a.links), static_cast<const double *>(a.mom), V, dt);
    else
        update_links_f32<FROM_UNIT><<<step_grid(4 * V, kStepBlock, kStepBlocks), kStepBlock, 0, st>>>(
            static_cast<float *>(a.links), static_cast<const float *>(a.mom), V, (float)dt);
    return cudaGetLastError();
}

} // namespace

cudaError_t launch_update_links(const MdArgs &a, cudaStream_t st) { return launch_step<false>(a, a.dt, st); }

cudaError_t launch_update_links_batched(int precision, int n, const LinkStepItem *items, double dt,
                                        cudaStream_t st)
{
    if (n < 1 || n > kMaxBatch) return cudaErrorInvalidValue;
    LinkBatch B{};
    B.n = n;
    int64_t pos = 0;
    for (int c = 0; c < n; ++c) {
        B.begin[c] = pos;
        B.V[c] = items[c].V;
        B.links[c] = items[c].links;
        B.mom[c] = items[c].mom;
        pos += 4 * items[c].V;
    }
    B.begin[n] = pos;
    B.total = pos;
    if (precision == LQCD_F64)
        update_links_f64_batched<<<step_grid(pos, kFxStepBlock, 8), kFxStepBlock, 0, st>>>(B, dt);
    else
        update_links_f32_batched<<<step_grid(pos, kStepBlock, kStepBlocks), kStepBlock, 0, st>>>(B, (float)dt);
    return cudaGetLastError();
}

cudaError_t launch_links_from_omega(const MdArgs &a, cudaStream_t st) { return launch_step<true>(a, 1.0, st); }

cudaError_t launch_omega_gradient(const MdArgs &a, cudaStream_t st)
{
    const int64_t V = volume(a.dims);
    if (a.precision == LQCD_F64)
        omega_gradient<double><<<grid_for(4 * V), kBlock, 0, st>>>(
            static_cast<const double *>(a.mom), static_cast<const double *>(a.force),
            static_cast<double *>(a.mom_out), V);
    else
        omega_gradient<float><<<grid_for(4 * V), kBlock, 0, st>>>(
            static_cast<const float *>(a.mom), static_cast<const float *>(a.force),
            static_cast<float *>(a.mom_out), V);
    return cudaGetLastError();
}

template <int NR> static cudaError_t launch_convert_t(const MdArgs &a, int dst_precision,
                                                      cudaStream_t st)
{
    const int64_t V = volume(a.dims);
    const void *src = a.full_in;
    void *dst = a.full_out;
    const unsigned grid = grid_for(4 * V);
    if (a.precision == LQCD_F32 && dst_precision == LQCD_F64)
        convert_field<float, double, NR><<<grid, kBlock, 0, st>>>(static_cast<const float *>(src),
                                                                  static_cast<double *>(dst), V);
    else if (a.precision == LQCD_F64 && dst_precision == LQCD_F32)
        convert_field<double, float, NR><<<grid, kBlock, 0, st>>>(static_cast<const double *>(src),
                                                                  static_cast<float *>(dst), V);
    else if (a.precision == LQCD_F32)
        convert_field<float, float, NR><<<grid, kBlock, 0, st>>>(static_cast<const float *>(src),
                                                                 static_cast<float *>(dst), V);
    else
        convert_field<double, double, NR><<<grid, kBlock, 0, st>>>(
            static_cast<const double *>(src), static_cast<double *>(dst), V);
    return cudaGetLastError();
}

cudaError_t launch_convert(const MdArgs &a, int dst_precision, bool links, cudaStream_t st)
{
    return links ? launch_convert_t<12>(a, dst_precision, st) : launch_convert_t<8>(a, dst_precision, st);
}

cudaError_t launch_pack(const MdArgs &a, cudaStream_t st)
{
    const int64_t V = volume(a.dims);
    if (a.precision == LQCD_F64)
        pack<double><<<grid_for(4 * V), kBlock, 0, st>>>(static_cast<const double *>(a.full_in),
                                                          static_cast<double *>(a.links), V);
    else
        pack<float><<<grid_for(4 * V), kBlock, 0, st>>>(static_cast<const float *>(a.full_in),
                                                         static_cast<float *>(a.links), V);
    return cudaGetLastError();
}

cudaError_t launch_unpack(const MdArgs &a, cudaStream_t st)
{
    const int64_t V = volume(a.dims);
    if (a.precision == LQCD_F64)
        unpack<double><<<grid_for(4 * V), kBlock, 0, st>>>(static_cast<const double *>(a.links),
                                                            static_cast<double *>(a.full_out), V);
    else
        unpack<float><<<grid_for(4 * V), kBlock, 0, st>>>(static_cast<const float *>(a.links),
                                                           static_cast<float *>(a.full_out), V);
    return cudaGetLastError();
}

} // namespace lqcd
