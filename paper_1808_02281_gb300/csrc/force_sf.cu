// Gauge force of the one-loop Symanzik action from plaquette-staple fields
// (paper Sec. II, Eq. 18_7_25_2; loops of Eq. 18_3_27_30), two kernels.
//
// Pass A (staple_fields) stores, for every link (x, mu) and every signed
// direction b perpendicular to mu, the plaquette staple
//     S^{(mu)}_b(x) = link(x+mu, b) U_mu(x+b)^dag link(x, b)^dag
// (the path x+mu -> x+mu+b -> x+b -> x): 24 "directions" per site instead
// of 4.  It is a product of three SU(3) matrices, so it is SU(3): its first
// two rows (which need only two rows of the first product) determine the
// third, conj(row0 x row1).  Planes are stored compact (two rows, the third
// rebuilt on load) or full (all 18 reals; the default schedule).
//
// Pass B (force_from_staples) builds every staple of the link (k, rho) from
// those fields.  With S = S^{(rho)} and A_b = link(k, b), B_b = link(k+rho, b),
// F = U_rho(k+rho), E = U_rho(k-rho), and the unitarity of the links:
//   plaquette            S_b(k)
//   rectangle, link first on the long side    F S_b(k+rho) S_b(k)
//   rectangle, link second on the long side   S_b(k) S_b(k-rho) E
//   rectangle along b    B_b S_b(k+b) A_b^dag
//   cube (a, b)          B_a S_b(k+a) S^{(a)}_b(k),  S^{(-c)}_b(k) = S^{(c)}_b(k-c)^dag
// (each equals the corresponding staple of the path form -- products of the
// same links -- once U U^dag = 1 is used for the link that the two staple
// factors share).  Summed with the loop coefficients and regrouped,
//   t = c_plaq sum_b S_b(k) + c_rect (F sum_b S_b(k+rho) S_b(k) + sum_b S_b(k) S_b(k-rho) E)
//     + sum_d B_d [ c_cube sum_{b perp d} S_b(k+d) S^{(d)}_b(k) + c_rect S_d(k+d) A_d^dag ],
// 51 SU(3) products per link in pass B and 12 (10 stored rows) per link in
// pass A, against 180 for the 48 staples walked one by one.  Every product
// of two SU(3) factors in pass B likewise forms two rows and takes its third
// from them, so the left factor's third row is never needed.
//
// The action comes out of pass B at no extra products: summing
// Re tr(U_{k,rho} t_{k,rho}) over links counts every loop once per link on it
// (L = 4 or 6 times) with its c_P, so with the plaquette staple sum Pl,
//   S_G = (beta/3) sum_links [ 3 (1.5 c_plaq + 3 c_rect + 4 c_cube)
//                              - Re tr(U t)/6 - (c_plaq/12) Re tr(U Pl) ]
// (Eq. 18_6_4_1), each link's share formed in the working precision from its
// two traces and summed in FP64.
//
// Work decomposition.  Both passes run in "virtual blocks" of 128 threads:
// the four warps of a block take the four directions of the same 32 sites
// (the planes around a site are read while they are in L1/L2, and each warp
// reads one plane per instruction, so a quarter-warp covers 8 consecutive
// sites of one 128-byte line).  A single lattice is launched with one CTA per
// virtual block; a batch of lattices of different extents runs as one
// persistent launch whose CTAs take the virtual blocks of all lattices from
// a work counter.  The
// action partial sum of a virtual block is the same in both, so a batched
// result equals the single-lattice result bit for bit.
#include <atomic>
#include <mutex>

#include "sf_common.cuh"

namespace lqcd {

namespace {

// ---------------------------------------------------------------- pass A

// The six staples S^{(mu)}_b, b = +-nu (nu != mu), of the link (x, mu), x
// at coordinates c; stored at staple index sx of sf.
template <typename R, bool FULL>
__device__ __forceinline__ void site_staples(const R *__restrict__ links, const G32 &g, const Coord &c,
                                             int x, int mu, const Planes<FULL> &sf, int sx)
{
    const int64_t V = g.V;
    const int xm = x + step32(g, c, mu, 1); // x + mu
    const auto at = sf.at(sx);
#pragma unroll 1
    for (int iv = 0; iv < 3; ++iv) {
        const int nu = (mu + 1 + iv) & 3;
        const int vp = step32(g, c, nu, 1), vm = step32(g, c, nu, -1);
        // b = +nu:  U_nu(x+mu) U_mu(x+nu)^dag U_nu(x)^dag
        // rows 0 and 1 of each staple (which need rows 0 and 1 of the first
        // product only); a full plane takes its third row from them, the
        // staple being a product of three SU(3) links
        Mat<R> t = mul<N, D>(load_link(links, V, nu, xm), load_link(links, V, mu, x + vp));
        Mat<R> up = mul_top2<N, D>(t, load_link(links, V, nu, x));
        if constexpr (FULL) rebuild_row2(up);
        sf.store(at, mu * 6 + 2 * iv, up);
        // b = -nu:  U_nu(x+mu-nu)^dag U_mu(x-nu)^dag U_nu(x-nu)
        t = mul<D, D>(load_link(links, V, nu, xm + vm), load_link(links, V, mu, x + vm));
        Mat<R> dn = mul_top2<N, N>(t, load_link(links, V, nu, x + vm));
        if constexpr (FULL) rebuild_row2(dn);
        sf.store(at, mu * 6 + 2 * iv + 1, dn);
    }
}

// Staple plane mu*6 + j of site x (site_staples one at a time).
template <typename R, bool FULL>
__device__ __forceinline__ void site_staple(const R *__restrict__ links, const G32 &g, const Coord &c, int x, int mu, int j,
                                            const Planes<FULL> &sf)
{
    const int64_t V = g.V;
    const int nu = (mu + 1 + (j >> 1)) & 3;
    const int xm = x + step32(g, c, mu, 1);
    Mat<R> s;
    if ((j & 1) == 0) {
        const Mat<R> t = mul<N, D>(load_link(links, V, nu, xm), load_link(links, V, mu, x + step32(g, c, nu, 1)));
        s = mul_top2<N, D>(t, load_link(links, V, nu, x));
    } else {
        const int vm = step32(g, c, nu, -1);
        const Mat<R> t = mul<D, D>(load_link(links, V, nu, xm + vm), load_link(links, V, mu, x + vm));
        s = mul_top2<N, N>(t, load_link(links, V, nu, x + vm));
    }
    if constexpr (FULL) rebuild_row2(s);
    sf.store(sf.at(x), mu * 6 + j, s);
}

// The 24 staples of the 32 sites of virtual block vb: thread = (site, mu).
template <typename R, bool FULL>
__device__ __forceinline__ void staples_block(const SfLattice &L, const G32 &g, int vb)
{
    const int mu = (int)(threadIdx.x >> 5);
    const int x = vb * 32 + (int)(threadIdx.x & 31);
    if (x >= g.V) return;
    site_staples<R, FULL>(static_cast<const R *>(L.links), g, coord32(g, L.div, x), x, mu,
                                planes_of<FULL>(L), x);
}

template <typename R, bool FULL>
__global__ void __launch_bounds__(kBlock) staple_fields(const __grid_constant__ SfLattice L)
{
    const G32 g = make_g32(L.dims);
    const int nvb = (int)virtual_blocks(g.V);
    for (int vb = blockIdx.x; vb < nvb; vb += gridDim.x) staples_block<R, FULL>(L, g, vb);
}

// Staples q, q + 4 of each direction (split lattices: a quarter of the work
// of staples_block in a CTA of its own).
template <typename R, bool FULL>
__device__ __forceinline__ void split_staples_block(const SfLattice &L, const G32 &g, int vb, int q)
{
    const int mu = (int)(threadIdx.x >> 5);
    const int x = vb * 32 + (int)(threadIdx.x & 31);
    if (x >= g.V) return;
    const Coord c = coord32(g, L.div, x);
#pragma unroll 1
    for (int j = q; j < 6; j += 4)
        site_staple<R, FULL>(static_cast<const R *>(L.links), g, c, x, mu, j, planes_of<FULL>(L));
}

template <typename R, bool FULL>
__global__ void __launch_bounds__(kBlock) staple_fields_split(const __grid_constant__ SfLattice L)
{
    split_staples_block<R, FULL>(L, make_g32(L.dims), (int)(blockIdx.x >> 2), (int)(blockIdx.x & 3));
}

// The same for a batch of split lattices only.
template <typename R, bool FULL>
__global__ void __launch_bounds__(kBlock) staple_fields_split_batched(const __grid_constant__ SfBatch B)
{
    const SfLattice &L = B.e[batch_entry(B, blockIdx.x)];
    const int v = (int)(blockIdx.x - L.vb_begin);
    split_staples_block<R, FULL>(L, make_g32(L.dims), v >> 2, v & 3);
}

template <typename R, bool FULL>
__global__ void __launch_bounds__(kBlock) staple_fields_batched(const __grid_constant__ SfBatch B)
{
    for (int64_t vb = next_virtual_block(B.counter); vb < B.total;) {
        const unsigned long long next = claim_virtual_block(B.counter);
        const int c = batch_entry(B, vb);
        const SfLattice &L = B.e[c];
        staples_block<R, FULL>(L, make_g32(L.dims), (int)(vb - L.vb_begin));
        vb = publish_virtual_block(next);
    }
}

// ---------------------------------------------------------------- pass B

// Force (and the fused momentum step) on the 128 links of virtual block vb
// of the sweep; returns the thread's share of the action (0 for a padding
// site).
template <typename R, bool ACTION, bool UNROLLQ, bool FULL>
__device__ __forceinline__ double force_block(const SfLattice &L, const KernelScalars &sc,
                                              const G32 &g, const Sweep &sw, int vb)
{
    const int rho = (int)((threadIdx.x >> 5) & 3);
    const int j = vb * 32 + (int)(threadIdx.x & 31);
    if (j >= g.V) return 0.0;
    const Coord c = swept_site(sw, j);
    const int k = index32(g, c);
    const LatticeSites si{&g, &c, k};
    return force_link<R, ACTION, UNROLLQ, false>(L, sc, g, planes_of<FULL>(L), si, c, k, rho);
}

// Split lattices: the links of direction rho of virtual block vb, warp 0 their
// plaquettes and chains, warps 1 to 3 the sums of products that the links +-d
// of one direction close; warp 0 closes them, in force_link's order, so that
// force and action have the bits of force_block.  20 products in a row against
// 51 of a thread.  The action's share goes to partial vb*4 + rho.
template <typename R, bool ACTION>
__device__ __forceinline__ void split_force_block(const SfLattice &L, const KernelScalars &sc, const G32 &g,
                                                  const Sweep &sw, int vb, int rho)
{
    __shared__ R y_s[6][18][32]; // of +d, then of -d
    const int part = (int)(threadIdx.x >> 5), lane = (int)(threadIdx.x & 31);
    const int j = vb * 32 + lane;
    const Coord c = swept_site(sw, j < g.V ? j : g.V - 1);
    const int k = index32(g, c), kp = k + step32(g, c, rho, 1);
    const LatticeSites si{&g, &c, k};
    const auto sf = planes_of<true>(L);
    const R *__restrict__ links = static_cast<const R *>(L.links);
    const R c_rt = scalar<R>(sc, SC_CRT), c_cb = scalar<R>(sc, SC_CCB);
    Mat<R> t;
    R tr_pl = R(0);
    if (part == 0) {
        chain_terms<R, ACTION, false>(t, tr_pl, links, sf, si, g, c, rho, k, kp, scalar<R>(sc, SC_CPL), c_rt);
    } else {
        const auto put = [&](int i, const Mat<R> &y) {
#pragma unroll
            for (int e = 0; e < 9; ++e) {
                y_s[i][2 * e][lane] = y.re[e / 3][e % 3];
                y_s[i][2 * e + 1][lane] = y.im[e / 3][e % 3];
            }
        };
        d_terms<false, false, false, false>(t, links, sf, si, g, c, rho, k, kp, part - 1, c_rt, c_cb);
        put(part - 1, t);
        d_terms<true, false, false, false>(t, links, sf, si, g, c, rho, k, kp, part - 1, c_rt, c_cb);
        put(part + 2, t);
    }
    __syncthreads();
    if (part == 0) {
        const auto get = [&](int i) {
            Mat<R> y;
#pragma unroll
            for (int e = 0; e < 9; ++e) {
                y.re[e / 3][e % 3] = y_s[i][2 * e][lane];
                y.im[e / 3][e % 3] = y_s[i][2 * e + 1][lane];
            }
            return y;
        };
#pragma unroll
        for (int id = 0; id < 3; ++id) mul_acc<N, N>(t, load_link(links, g.V, (rho + 1 + id) & 3, kp), get(id));
#pragma unroll
        for (int id = 0; id < 3; ++id) {
            const int nud = (rho + 1 + id) & 3;
            mul_acc<D, N>(t, load_link(links, g.V, nud, kp + step32(g, c, nud, -1)), get(3 + id));
        }
        double share = 0.0;
        if (j < g.V) share = finish_link<R, ACTION>(L, sc, links, g.V, rho, k, t, tr_pl);
        if constexpr (ACTION) {
            share = warp_sum(share);
            if (lane == 0) L.partials[vb * 4 + rho] = share;
        }
    }
    __syncthreads(); // before y_s is written again
}

template <typename R, bool ACTION>
__global__ void __launch_bounds__(kBlock, 4)
    force_split(const __grid_constant__ SfLattice L, const __grid_constant__ KernelScalars sc)
{
    const G32 g = make_g32(L.dims);
    split_force_block<R, ACTION>(L, sc, g, make_sweep(L, g), (int)(blockIdx.x >> 2), (int)(blockIdx.x & 3));
}

// The same for a batch of split lattices only: a batch with a large lattice
// among them takes the whole blocks for all (with quarter blocks in one kernel
// with whole ones the large lattices took 3 to 6 % longer, and a launch of
// their own is 7 us).
template <typename R, bool ACTION>
__global__ void __launch_bounds__(kBlock, 4)
    force_split_batched(const __grid_constant__ SfBatch B, const __grid_constant__ KernelScalars sc)
{
    const SfLattice &L = B.e[batch_entry(B, blockIdx.x)];
    const G32 g = make_g32(L.dims);
    const int v = (int)(blockIdx.x - L.vb_begin);
    split_force_block<R, ACTION>(L, sc, g, make_sweep(L, g), v >> 2, v & 3);
}

// Resident CTAs per SM the register allocation aims at: 4 (128 registers)
// unless the fused action asks for more registers (3) -- or DENSE forces 4.
template <bool ACTION, bool DENSE> constexpr int min_blocks() { return (ACTION && !DENSE) ? 3 : 4; }

// ROWS > 1: a CTA of ROWS groups of four warps on consecutive virtual
// blocks (y-neighbouring x rows of the sweep), so that the staples of a
// row's +-y neighbours are the own-row staples of another group of the CTA.
template <typename R, bool ACTION, bool UNROLLQ, bool DENSE = false, bool FULL = false, int ROWS = 1>
__global__ void __launch_bounds__(ROWS * kBlock, (min_blocks<ACTION, DENSE>() / ROWS > 0
                                                       ? min_blocks<ACTION, DENSE>() / ROWS
                                                       : 1))
    force_from_staples(const __grid_constant__ SfLattice L, const __grid_constant__ KernelScalars sc)
{
    const G32 g = make_g32(L.dims);
    const Sweep sw = make_sweep(L, g);
    const int nvb = (int)virtual_blocks(g.V);
    const int row = ROWS == 1 ? 0 : (int)(threadIdx.x >> 7);
    for (int vb0 = blockIdx.x * ROWS; vb0 < nvb; vb0 += gridDim.x * ROWS) {
        const int vb = vb0 + row;
        double acc = 0.0;
        if (vb < nvb) acc = force_block<R, ACTION, UNROLLQ, FULL>(L, sc, g, sw, vb);
        if constexpr (ACTION) {
            const double s = group_sum<ROWS>(acc, row);
            if ((threadIdx.x & (kBlock - 1)) == 0 && vb < nvb) L.partials[vb] = s;
        }
    }
}

template <typename R, bool ACTION, bool UNROLLQ, bool DENSE = false, bool FULL = false>
__global__ void __launch_bounds__(kBlock, (min_blocks<ACTION, DENSE>()))
    force_from_staples_batched(const __grid_constant__ SfBatch B,
                               const __grid_constant__ KernelScalars sc)
{
    for (int64_t vb = next_virtual_block(B.counter + 1); vb < B.total;) {
        const unsigned long long next = claim_virtual_block(B.counter + 1);
        const int c = batch_entry(B, vb);
        const SfLattice &L = B.e[c];
        const G32 g = make_g32(L.dims);
        const double acc = force_block<R, ACTION, UNROLLQ, FULL>(
            L, sc, g, make_sweep(L, g), (int)(vb - L.vb_begin));
        if constexpr (ACTION) {
            const int64_t v = vb - L.vb_begin;
            if (L.split) { // the partial sums of force_split
                const double s = warp_sum(acc);
                if ((threadIdx.x & 31) == 0) L.partials[v * 4 + (threadIdx.x >> 5)] = s;
            } else {
                const double s = block_sum(acc);
                if (threadIdx.x == 0) L.partials[v] = s;
            }
        }
        vb = publish_virtual_block(next);
    }
}

// One block per lattice of a batch: its action from its partial sums, in the
// order and grouping of finish_sum, so batched and single results agree.
__global__ void __launch_bounds__(1024) finish_batched(const __grid_constant__ SfBatch B, double scale)
{
    const SfLattice &L = B.e[blockIdx.x];
    if (L.action == nullptr) return;
    const int count = (int)virtual_blocks((int64_t)L.dims[0] * L.dims[1] * L.dims[2] * L.dims[3]) * (L.split ? 4 : 1);
    __shared__ double warp_part[32];
    double v = 0.0;
    for (int i = threadIdx.x; i < count; i += 1024) v += L.partials[i];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
    const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
    if (lane == 0) warp_part[warp] = v;
    __syncthreads();
    if (warp == 0) {
        double s = warp_part[lane];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) s += __shfl_down_sync(0xffffffffu, s, o);
        if (lane == 0) *L.action = scale * s;
    }
}

// Pass-B schedules (same arithmetic, different traversal or occupancy; FP64
// has one kernel, force_fx.cu, and takes only the traversal from these):
//   0  micro-tiles 8x2x2, inner b loop rolled
//   1  micro-tiles 8x2x2, inner b loop unrolled
//   2  x rows (no micro-tiles), inner b loop rolled
//   3  x rows, registers capped for 4 CTAs/SM also with the fused action
//   4  x rows, staple planes stored full (18 reals, no row rebuilt on load),
//      spatial blocks up to 64x8x8 (full planes are 1.5x the bytes per site:
//      smaller blocks keep the sweep's working set in L2; 4.22 against
//      4.45 ms with 64x16x16 at 32^3x64 FP32)
//   5  as 4, registers capped for 4 CTAs/SM
//   6  as 4 with spatial blocks up to 64x16x16
//   7  as 5 in CTAs of two groups of four warps on consecutive virtual
//      blocks: with x extent 32 those are y-neighbouring x rows, and a row's
//      +-y staples are the other group's own staples (L1 hits)
//   8  as 7 with spatial blocks up to 64x16x8
// The process-wide choice per precision is set by lqcd_set_force_variant or
// lqcd_autotune_force; -1 means the default (default_variant).
constexpr int kSfVariants = 9;

// Built-in choice: full staples with the 4-CTA register cap in FP32 (at
// 32^3x64 3.42 ms against 3.45-3.46 ms for the two-row CTAs and 3.64-3.66
// for the others; at 32^4 1.73 against 1.75 ms), the same traversal in FP64.
// The two-row CTAs won (3.54 against 3.67 ms at 32^3x64) while the sweep
// still divided by run-time extents; with multiply-high divisions the
// one-row CTA is ahead.  The dims are kept for shape-dependent choices.
int default_variant(int precision, const int dims[4])
{
    (void)dims;
    return precision == LQCD_F64 ? 4 : 5;
}

bool full_staples(int variant) { return variant >= 4; }

// Slot of a kernel instance in the occupancy cache of persistent_grid:
// kind (0 pass B, 1 pass B capped, 2 pass B full, 3 pass B full capped,
// 4 pass A compact, 5 pass A full) x action x unrolled.
int grid_slot(int kind, bool action, bool unrolled)
{
    return kind * 4 + (action ? 2 : 0) + (unrolled ? 1 : 0);
}

std::atomic<int> g_sf_variant[2] = {{-1}, {-1}};

// Largest divisor of L not above cap.
int block_extent(int L, int cap)
{
    for (int b = cap < L ? cap : L; b > 1; --b)
        if (L % b == 0) return b;
    return 1;
}

void set_traversal(SfLattice &L, int variant)
{
    const int cap_y = (variant == 4 || variant == 5 || variant == 7) ? 8 : 16;
    const int cap_z = (variant >= 4 && variant != 6) ? 8 : 16;
    L.sweep[0] = block_extent(L.dims[0], 64);
    L.sweep[1] = block_extent(L.dims[1], cap_y);
    L.sweep[2] = block_extent(L.dims[2], cap_z);
    if (variant >= 2) {
        L.micro[0] = L.sweep[0];
        L.micro[1] = L.micro[2] = 1;
    } else {
        L.micro[0] = block_extent(L.sweep[0], 8);
        L.micro[1] = L.sweep[1] % 2 == 0 ? 2 : 1;
        L.micro[2] = L.sweep[2] % 2 == 0 ? 2 : 1;
    }
    // the divisors of coord32 and swept_site (all below 2^31: V < 2^31)
    const int *d = L.dims;
    const int64_t slice = (int64_t)L.sweep[0] * L.sweep[1] * L.sweep[2];
    const int64_t dv[12] = {d[0],
                            (int64_t)d[0] * d[1],
                            (int64_t)d[0] * d[1] * d[2],
                            slice * d[3],
                            slice,
                            (int64_t)L.micro[0] * L.micro[1] * L.micro[2],
                            L.micro[0],
                            L.micro[1],
                            L.sweep[0] / L.micro[0],
                            L.sweep[1] / L.micro[1],
                            d[0] / L.sweep[0],
                            d[1] / L.sweep[1]};
    for (int i = 0; i < 12; ++i) L.div[i] = div_magic((unsigned)(dv[i] > 0 ? dv[i] : 1));
    L.counts[0] = (int)dv[DV_NBX];
    L.counts[1] = (int)dv[DV_NBY];
    L.counts[2] = (int)dv[DV_NMX];
    L.counts[3] = (int)dv[DV_NMY];
}

KernelScalars make_scalars(const ForceArgs &a)
{
    KernelScalars k;
    const double sc[7] = {a.beta / 6.0, a.c_plaq, a.c_rect, a.c_cube,
                          3.0 * (1.5 * a.c_plaq + 3.0 * a.c_rect + 4.0 * a.c_cube), a.c_plaq / 12.0,
                          a.dt};
    for (int i = 0; i < 7; ++i) {
        k.d[i] = sc[i];
        k.f[i] = (float)sc[i];
    }
    return k;
}

int resolve_variant(const ForceArgs &a)
{
    if (a.variant >= 0 && a.variant < kSfVariants) return a.variant;
    const int p = a.precision == LQCD_F64 ? 1 : 0;
    const int v = g_sf_variant[p].load();
    return v < 0 ? default_variant(a.precision, a.dims) : v;
}

template <bool ACTION>
cudaError_t launch_pass_b(const SfLattice &L, const KernelScalars &sc, int variant, cudaStream_t st)
{
    const int64_t V = (int64_t)L.dims[0] * L.dims[1] * L.dims[2] * L.dims[3];
    const unsigned grid = grid_of(virtual_blocks(V));
    if (variant == 1) force_from_staples<float, ACTION, true><<<grid, kBlock, 0, st>>>(L, sc);
    else if (variant == 3) force_from_staples<float, ACTION, false, true><<<grid, kBlock, 0, st>>>(L, sc);
    else if (variant == 4 || variant == 6)
        force_from_staples<float, ACTION, false, false, true><<<grid, kBlock, 0, st>>>(L, sc);
    else if (variant == 5)
        force_from_staples<float, ACTION, false, true, true><<<grid, kBlock, 0, st>>>(L, sc);
    else if (variant >= 7)
        force_from_staples<float, ACTION, false, true, true, 2>
            <<<grid_of((virtual_blocks(V) + 1) / 2), 2 * kBlock, 0, st>>>(L, sc);
    else force_from_staples<float, ACTION, false><<<grid, kBlock, 0, st>>>(L, sc);
    return cudaGetLastError();
}

template <bool ACTION>
cudaError_t launch_pass_b_batched(const SfBatch &B, const KernelScalars &sc, int variant,
                                  cudaStream_t st)
{
    if (variant == 1) {
        auto k = force_from_staples_batched<float, ACTION, true>;
        k<<<persistent_grid(k, grid_slot(0, ACTION, true), B.total), kBlock, 0, st>>>(B, sc);
    } else if (variant == 3) {
        auto k = force_from_staples_batched<float, ACTION, false, true>;
        k<<<persistent_grid(k, grid_slot(1, ACTION, false), B.total), kBlock, 0, st>>>(B, sc);
    } else if (variant == 4 || variant == 6) {
        auto k = force_from_staples_batched<float, ACTION, false, false, true>;
        k<<<persistent_grid(k, grid_slot(2, ACTION, false), B.total), kBlock, 0, st>>>(B, sc);
    } else if (variant == 5 || variant >= 7) {
        auto k = force_from_staples_batched<float, ACTION, false, true, true>;
        k<<<persistent_grid(k, grid_slot(3, ACTION, false), B.total), kBlock, 0, st>>>(B, sc);
    } else {
        auto k = force_from_staples_batched<float, ACTION, false>;
        k<<<persistent_grid(k, grid_slot(0, ACTION, false), B.total), kBlock, 0, st>>>(B, sc);
    }
    return cudaGetLastError();
}

size_t round_up256(size_t b) { return (b + 255) & ~(size_t)255; }

cudaError_t launch_passes(const SfLattice &L, const KernelScalars &sc, int variant, bool action, cudaStream_t st)
{
    const unsigned grid = grid_of(virtual_blocks((int64_t)L.dims[0] * L.dims[1] * L.dims[2] * L.dims[3]));
    if (L.split) {
        staple_fields_split<float, true><<<4 * grid, kBlock, 0, st>>>(L);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        if (action) force_split<float, true><<<4 * grid, kBlock, 0, st>>>(L, sc);
        else force_split<float, false><<<4 * grid, kBlock, 0, st>>>(L, sc);
        return cudaGetLastError();
    }
    if (full_staples(variant)) staple_fields<float, true><<<grid, kBlock, 0, st>>>(L);
    else staple_fields<float, false><<<grid, kBlock, 0, st>>>(L);
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return action ? launch_pass_b<true>(L, sc, variant, st) : launch_pass_b<false>(L, sc, variant, st);
}

cudaError_t launch_passes_batched(const SfBatch &B, const KernelScalars &sc, int variant, bool action, cudaStream_t st)
{
    SfBatch quarters = B; // blocks of a quarter each
    quarters.total = 0;
    bool all_split = true;
    for (int c = 0; c < B.n; ++c) {
        const int *d = B.e[c].dims;
        quarters.e[c].vb_begin = quarters.total;
        quarters.total += 4 * virtual_blocks((int64_t)d[0] * d[1] * d[2] * d[3]);
        all_split = all_split && B.e[c].split;
    }
    if (all_split) {
        staple_fields_split_batched<float, true><<<grid_of(quarters.total), kBlock, 0, st>>>(quarters);
        const cudaError_t e = cudaGetLastError();
        if (e != cudaSuccess) return e;
        if (action) force_split_batched<float, true><<<grid_of(quarters.total), kBlock, 0, st>>>(quarters, sc);
        else force_split_batched<float, false><<<grid_of(quarters.total), kBlock, 0, st>>>(quarters, sc);
        return cudaGetLastError();
    }
    if (full_staples(variant)) {
        auto ka = staple_fields_batched<float, true>;
        ka<<<persistent_grid(ka, grid_slot(5, false, false), B.total), kBlock, 0, st>>>(B);
    } else {
        auto ka = staple_fields_batched<float, false>;
        ka<<<persistent_grid(ka, grid_slot(4, false, false), B.total), kBlock, 0, st>>>(B);
    }
    const cudaError_t e = cudaGetLastError();
    if (e != cudaSuccess) return e;
    return action ? launch_pass_b_batched<true>(B, sc, variant, st) : launch_pass_b_batched<false>(B, sc, variant, st);
}

} // namespace

// FP32: room for the 24 planes in the larger (full, 18-real, in blocks of 32
// sites) of the two storage forms, so that every schedule fits the same
// workspace.  FP64: the 24 planes, the 4 planes of the links in limbs, 256 bytes
// for the flag, and the words of small lattices.
size_t staple_field_bytes(const int dims[4], int precision, bool lean)
{
    const int64_t V = (int64_t)dims[0] * dims[1] * dims[2] * dims[3];
    const bool fixed = precision == LQCD_F64 && !lean;
    return round_up256((fixed ? fx_planes_count() : kStaplePlanes) * full_plane_bytes(V, precision)) +
           (fixed ? 256 + (near_words(V) ? round_up256(virtual_blocks(V) * sizeof(int)) : 0) : 0);
}

bool staple_fields_supported(const int dims[4])
{
    return (int64_t)dims[0] * dims[1] * dims[2] * dims[3] < ((int64_t)1 << 31);
}

int staple_force_partials(const int dims[4], bool lean)
{
    const int64_t V = (int64_t)dims[0] * dims[1] * dims[2] * dims[3];
    return (int)virtual_blocks(V) * (split_lattice(V) && !lean ? 4 : 1);
}

cudaError_t launch_force_staple_fields(const ForceArgs &a, cudaStream_t st)
{
    const int variant = resolve_variant(a);
    const int64_t V = (int64_t)a.dims[0] * a.dims[1] * a.dims[2] * a.dims[3];
    SfLattice L{};
    for (int i = 0; i < 4; ++i) L.dims[i] = a.dims[i];
    set_traversal(L, variant);
    L.plane_bytes = (int64_t)full_plane_bytes(V, a.precision);
    L.split = split_lattice(V) && !a.lean && (a.precision == LQCD_F64 || full_staples(variant));
    L.links = a.links;
    L.staples = a.staples;
    L.force = a.force;
    L.mom = a.mom;
    L.partials = a.partials;
    L.action = a.action;
    const KernelScalars sc = make_scalars(a);
    const bool action = a.action != nullptr;
    if (a.precision == LQCD_F64 && !a.lean) {
        L.flag = reinterpret_cast<unsigned long long *>(static_cast<char *>(a.staples) + fx_planes_count() * L.plane_bytes);
        L.bit = 1;
        if (near_words(V)) L.near = reinterpret_cast<int *>(L.flag + 32);
    }
    const cudaError_t e = a.precision == LQCD_F64 ? launch_fx_passes(L, sc, action, st)
                                                  : launch_passes(L, sc, variant, action, st);
    if (e != cudaSuccess || !action) return e;
    return launch_finish_sum(a.partials, (int)virtual_blocks(V) * (L.split ? 4 : 1), a.beta / 3.0, a.action, st);
}

cudaError_t launch_force_staple_fields_batched(const ForceArgs &a, int n, const SfLattice *items,
                                               unsigned long long *counter, cudaStream_t st)
{
    if (n < 1 || n > kMaxBatch) return cudaErrorInvalidValue;
    const int variant = resolve_variant(a);
    SfBatch B{};
    B.n = n;
    B.counter = counter;
    bool any_action = false;
    for (int c = 0; c < n; ++c) {
        const int *d = items[c].dims;
        const int64_t V = (int64_t)d[0] * d[1] * d[2] * d[3];
        B.e[c] = items[c];
        set_traversal(B.e[c], variant);
        B.e[c].plane_bytes = (int64_t)full_plane_bytes(V, a.precision);
        B.e[c].split = split_lattice(V) && !a.lean && (a.precision == LQCD_F64 || full_staples(variant));
        if (!a.lean) {
            B.e[c].flag = counter + 3;
            B.e[c].bit = 1ull << c;
        }
        B.e[c].vb_begin = B.total;
        B.total += virtual_blocks(V);
        any_action = any_action || B.e[c].action != nullptr;
    }
    const KernelScalars sc = make_scalars(a);
    cudaError_t e = cudaMemsetAsync(counter, 0, 4 * sizeof(unsigned long long), st);
    if (e != cudaSuccess) return e;
    e = a.precision == LQCD_F64 ? launch_fx_passes_batched(B, sc, any_action, st)
                                : launch_passes_batched(B, sc, variant, any_action, st);
    if (e != cudaSuccess || !any_action) return e;
    finish_batched<<<n, 1024, 0, st>>>(B, a.beta / 3.0);
    return cudaGetLastError();
}

int staple_force_variants() { return kSfVariants; }

int staple_force_variant(int precision, const int dims[4])
{
    const int p = precision == LQCD_F64 ? 1 : 0;
    const int v = g_sf_variant[p].load();
    return v < 0 ? default_variant(precision, dims) : v;
}

void set_staple_force_variant(int precision, int variant)
{
    g_sf_variant[precision == LQCD_F64 ? 1 : 0].store(variant);
}

} // namespace lqcd
