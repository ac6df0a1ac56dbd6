"""Workloads of the framework as a user's program runs them, with their exact values.

Every case goes through the public entry points of ``paper_1808_02281_gb300``
(``lqcd``, ``hmc``, ``autograd``).  ``listed()`` gives the standing cases,
``draw(rng)`` more of the same ranges; ``prepare`` makes what a program holds
before the call (links, momenta, spinors, the workspace it keeps), ``run``
makes one pass, ``work`` counts the bytes and flops that a pass cannot do
without and ``exact`` recomputes the outputs in 64 bits with plain torch, the
loops walked link by link (no unitarity used, nothing of the framework).

Inputs are synthetic: links U = exp(i w_a T_a) with w_a ~ N(0, sigma^2),
Gaussian momenta and spinors, all drawn from the seed on the GPU.
"""
import math

import numpy as np
import torch

from paper_1808_02281_gb300 import autograd, hmc, lqcd

BETA, KAPPA, DT = 6.0, 0.1315, 0.05


def _case(name, kind, dims, prec, sigma=0.3, u0=0.87, store="mom"):
    """store: whether a force pass stores the force or steps the momenta with it."""
    return {"name": name, "kind": kind, "dims": dims, "prec": prec, "sigma": sigma, "u0": u0, "store": store}


def listed():
    return [
        # force and action of the smallest lattice of the correctness workloads:
        # launches and latency
        _case("force_4x4x4x4_f64", "force", "4x4x4x4", "f64", 0.5, 0.87, "force"),
        # odd extents, a few tens of thousands of sites: rows that fill no warp
        _case("force_15x13x11x21_f32", "force", "15x13x11x21", "f32", 0.3, 0.87, "force"),
        # force and action in double precision: the runs that the
        # single-precision ones are checked against
        _case("force_24x24x24x48_f64", "force", "24x24x24x48", "f64", 0.3, 0.87, "force"),
        # the production MD momentum step: single precision, larger than L2
        _case("force_32x32x32x64_f32", "force", "32x32x32x64", "f32", 0.3, 0.87),
        # the FP64 action of the Metropolis test
        _case("action_24x24x24x48_f64", "action", "24x24x24x48", "f64", 0.3, 0.87),
        # the MD link step, production size and precision
        _case("links_32x32x32x64_f32", "links", "32x32x32x64", "f32", 0.3, 0.87),
        # the MD link step of a double-precision run on a lattice of odd rows
        _case("links_18x14x22x36_f64", "links", "18x14x22x36", "f64", 0.3, 0.87),
        # the differentiable action: forward and backward
        _case("grad_32x32x32x64_f32", "grad", "32x32x32x64", "f32", 0.3, 0.87),
        # one MD step (momenta, then links) of 16 lattices of uneven sizes
        _case("batch_step_f32", "batch", "8x8x8x8*4,12x12x12x24*4,16x16x16x32*4,24x24x24x48*4",
              "f32", 0.3, 0.87),
        # an HMC trajectory: momentum refresh, H in FP64, 5 Omelyan steps, H
        _case("hmc_16x16x16x32_f32", "hmc", "16x16x16x32", "f32", 0.15, 0.86),
        # the Wilson operator inside a solver: y = x - kappa calD x
        _case("dslash_32x32x32x64_f32", "dslash", "32x32x32x64", "f32", 0.3, 0.87),
        # the fermion force's momentum step in double precision, ragged rows
        _case("hopping_20x18x14x30_f64", "hopping", "20x18x14x30", "f64", 0.3, 0.87),
    ]


# kind: largest number of sites that is drawn, per precision
_LIMIT = {"force": (1 << 21, 24 * 24 * 24 * 48), "action": (1 << 21, 24 * 24 * 24 * 48),
          "links": (1 << 21, 1 << 20), "grad": (1 << 20, 1 << 17), "batch": (1 << 20, 1 << 17),
          "hmc": (16 * 16 * 16 * 32, 8 * 8 * 8 * 16), "dslash": (1 << 21, 1 << 20),
          "hopping": (1 << 21, 1 << 20)}


def _draw_dims(rng, most, least=64):
    """Extents 2..64, their product spread over the logarithm of least..most."""
    want = least * (most / least) ** rng.random()
    for _ in range(1000):
        mean = want ** 0.25
        d = [max(2, min(64, int(round(mean * 2.0 ** rng.uniform(-0.8, 0.8))))) for _ in range(4)]
        v = d[0] * d[1] * d[2] * d[3]
        if least <= v <= most and want / 2 <= v <= want * 2:
            return "x".join(map(str, d)), v
    return "4x4x4x4", 256


def draw(rng):
    kind = rng.choice(["force", "force", "force", "action", "links", "grad", "batch", "hmc",
                       "dslash", "hopping"])
    prec = rng.choice(["f32", "f32", "f64"])
    most = _LIMIT[kind][prec == "f64"]
    if kind == "batch":
        parts, left = [], most
        for _ in range(rng.randint(2, 8)):
            dims, v = _draw_dims(rng, max(128, left // 2))
            times = rng.randint(1, 2)
            if times * v <= left:
                parts.append("%s*%d" % (dims, times))
                left -= times * v
        dims = ",".join(parts) or "4x4x4x4*2"
    else:
        dims = _draw_dims(rng, most)[0]
    return {"kind": kind, "dims": dims, "prec": prec, "sigma": round(rng.uniform(0.1, 0.5), 3),
            "u0": round(rng.uniform(0.84, 0.95), 3), "store": rng.choice(["mom", "force"])}


# ------------------------------------------------- plain torch algebra
# A field of 3x3 matrices is a complex tensor [3, 3, Lt, Lz, Ly, Lx], a spinor
# field [4, 3, Lt, Lz, Ly, Lx]; direction mu = 0..3 is x, y, z, t.

def _mm(a, b):
    r = a[:, 0, None] * b[None, 0]
    for k in (1, 2):
        r.addcmul_(a[:, k, None], b[None, k])
    return r


def _dag(a):
    return a.transpose(0, 1).conj().resolve_conj()


def _sh(a, mu, s=1):
    """The field at n + s mu."""
    return torch.roll(a, -s, dims=a.dim() - 1 - mu)


def _generators(p):
    """sum_a p^a T_a, T_a = lambda_a / 2 (Gell-Mann), p real [8, ...]."""
    h, q = p / 2, p[7] / math.sqrt(12.0)
    z = torch.zeros_like(q)
    c = torch.complex
    return torch.stack([
        torch.stack([c(h[2] + q, z), c(h[0], -h[1]), c(h[3], -h[4])]),
        torch.stack([c(h[0], h[1]), c(q - h[2], z), c(h[5], -h[6])]),
        torch.stack([c(h[3], h[4]), c(h[5], h[6]), c(-2 * q, z)])])


def _exp_i(q, terms=16, halvings=3):
    """exp(i q) by the Taylor series of exp(i q / 2^halvings), squared back."""
    x = q * (1j / 2 ** halvings)
    one = torch.zeros_like(x)
    for i in range(3):
        one[i, i] = 1
    r = one + x / terms
    for k in range(terms - 1, 0, -1):
        r = _mm(x, r).div_(k).add_(one)
    for _ in range(halvings):
        r = _mm(r, r)
    return r


def _third(a, b):
    return torch.stack([a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2],
                        a[0] * b[1] - a[1] * b[0]]).conj().resolve_conj()


def _unitary(u):
    """Gram-Schmidt of rows 0 and 1, row 2 = conj(row 0 x row 1)."""
    a, b = u[0], u[1]
    a = a / a.abs().square().sum(0).sqrt()
    b = b - (a.conj() * b).sum(0) * a
    b = b / b.abs().square().sum(0).sqrt()
    return torch.stack([a, b, _third(a, b)])


def _to_rows(x, W):
    """Real [rows, V] -> the framework's lanes [rows / W, V, W]."""
    return x.reshape(x.shape[0] // W, W, -1).transpose(1, 2).contiguous()


def _from_rows(x):
    """[rows / W, V, W] -> real [rows, V]."""
    return x.transpose(1, 2).reshape(x.shape[0] * x.shape[2], -1)


def _reals(x, n):
    """Complex [..., *sites] -> real [n, V], real and imaginary part of each entry in turn."""
    return torch.view_as_real(x.reshape(n // 2, -1)).transpose(1, 2).reshape(n, -1)


def _complexes(x):
    return torch.complex(x[0::2].contiguous(), x[1::2].contiguous())


def _read_links(links, dims):
    """The stored links [4, 12/W, V, W] as four complex128 fields, row 2 rebuilt."""
    out = []
    for mu in range(4):
        two = _complexes(_from_rows(links[mu]).double()).reshape(2, 3, *dims[::-1])
        out.append(torch.stack([two[0], two[1], _third(two[0], two[1])]))
    return out


def _read_algebra(f, dims):
    return [_from_rows(f[mu]).double().reshape(8, *dims[::-1]) for mu in range(4)]


def _read_spinor(x, dims):
    return _complexes(_from_rows(x).double()).reshape(4, 3, *dims[::-1])


def _links_out(U, W):
    return torch.stack([_to_rows(_reals(u[:2], 12), W) for u in U])


def _algebra_out(f, W):
    return torch.stack([_to_rows(x.reshape(8, -1), W) for x in f])


def _signed(U, nu, s):
    """The link from n to n + s nu."""
    return U[nu] if s > 0 else _dag(_sh(U[nu], nu, -1))


def _staple_sums(U, rho):
    """Sums of the 6 plaquette, 18 rectangle and 24 cube staples of the links along rho."""
    Ud = _dag(U[rho])
    dirs = [(nu, s) for nu in range(4) if nu != rho for s in (1, -1)]
    A = {b: _signed(U, *b) for b in dirs}
    B = {b: _sh(A[b], rho) for b in dirs}
    M = {b: _mm(B[b], _sh(Ud, *b)) for b in dirs}
    plaq = rect = first = second = cube = 0
    for b in dirs:
        Ad = _dag(A[b])
        S = _mm(M[b], Ad)
        Nb = _mm(_sh(Ud, *b), Ad)
        plaq = plaq + S
        first = first + _mm(_sh(M[b], rho), Nb)
        second = second + _mm(M[b], _sh(Nb, rho, -1))
        rect = rect + _mm(_mm(B[b], _sh(S, *b)), Ad)
    rect = rect + _mm(_sh(U[rho], rho), first) + _mm(second, _sh(U[rho], rho, -1))
    for a in dirs:
        inner = 0
        for b in dirs:
            if b[0] != a[0]:
                inner = inner + _mm(_sh(M[b], *a), _dag(_mm(A[b], _sh(A[a], *b))))
        cube = cube + _mm(B[a], inner)
    return plaq, rect, cube


def _components(m, s):
    """-s Im tr(lambda_a m), a = 1..8."""
    return torch.stack([-s * (m[0, 1] + m[1, 0]).imag, -s * (m[0, 1] - m[1, 0]).real,
                        -s * (m[0, 0] - m[1, 1]).imag, -s * (m[0, 2] + m[2, 0]).imag,
                        -s * (m[0, 2] - m[2, 0]).real, -s * (m[1, 2] + m[2, 1]).imag,
                        -s * (m[1, 2] - m[2, 1]).real,
                        -s / math.sqrt(3.0) * (m[0, 0] + m[1, 1] - 2 * m[2, 2]).imag])


def _retr(m):
    return float((m[0, 0] + m[1, 1] + m[2, 2]).real.sum())


def _force_and_action(U, lat):
    """(force as four [8, ...] fields, action)."""
    V = U[0][0, 0].numel()
    f, S = [], 0.0
    for rho in range(4):
        pl, rc, cb = (_mm(U[rho], t) for t in _staple_sums(U, rho))
        # per link: 6 plaquettes / 4, 18 rectangles / 6, 24 cubes / 6 of its own
        S += lat.c_plaq * (4.5 * V - _retr(pl) / 4) + lat.c_rect * (9.0 * V - _retr(rc) / 6) \
            + lat.c_cube * (12.0 * V - _retr(cb) / 6)
        f.append(_components(lat.c_plaq * pl + lat.c_rect * rc + lat.c_cube * cb, lat.beta / 6))
    return f, lat.beta / 3 * S


def _link_step(U, p, dt):
    return [_unitary(_mm(_exp_i(_generators(dt * p[mu])), U[mu])) for mu in range(4)]


# gamma_mu[row][column] = entry, directions x, y, z, t
_GAMMA = [[(3, 1j), (2, 1j), (1, -1j), (0, -1j)], [(3, -1), (2, 1), (1, 1), (0, -1)],
          [(2, 1j), (3, -1j), (0, -1j), (1, 1j)], [(2, 1), (3, 1), (0, 1), (1, 1)]]


def _project(x, mu, s):
    """(1 + s gamma_mu) x."""
    return torch.stack([x[a] + s * v * x[c] for a, (c, v) in enumerate(_GAMMA[mu])])


def _colour(u, x):
    """u x on the colour index of every spin row."""
    return (u[None] * x[:, None]).sum(2)


# ----------------------------------------------------------- the cases

def _lat(case):
    dims = case["dims"].split(",")[0].split("*")[0]
    dims = tuple(int(d) for d in dims.split("x"))
    return lqcd.Lattice.symanzik(dims, BETA, case["u0"], case["prec"])


def _batch_dims(case):
    out = []
    for part in case["dims"].split(","):
        dims, times = part.split("*")
        out += [tuple(int(d) for d in dims.split("x"))] * int(times)
    return out


def _draw_links(lat, sigma, gen):
    """Random links, rows orthonormal to the stored precision."""
    out = []
    for _ in range(4):
        p = sigma * torch.randn((8, lat.V), generator=gen, device="cuda", dtype=lat.dtype)
        u = _unitary(_exp_i(_generators(p), terms=6, halvings=1))
        out.append(_to_rows(_reals(u[:2], 12), lat.W))
    return torch.stack(out)


def _normal(shape, lat, gen, sigma=1.0):
    return sigma * torch.randn(shape, generator=gen, device="cuda", dtype=lat.dtype)


def prepare(case, seed):
    kind, lat = case["kind"], _lat(case)
    gen = torch.Generator(device="cuda")
    gen.manual_seed(int(seed))
    st = {"kind": kind, "lat": lat}
    if kind == "batch":
        dims = _batch_dims(case)
        lats = [lat.with_(dims=d) for d in dims]
        st["bs"] = hmc.BatchState.create(lat, dims, [_draw_links(x, case["sigma"], gen) for x in lats],
                                         [_normal(x.algebra_shape, x, gen) for x in lats])
        return st
    st["links"] = _draw_links(lat, case["sigma"], gen)
    if kind in ("force", "links", "hopping", "hmc"):
        st["mom"] = _normal(lat.algebra_shape, lat, gen)
    if kind == "force" and case["store"] == "force":
        st["force"], st["mom"] = torch.empty_like(st["mom"]), None
    if kind in ("force", "action", "hmc"):   # an MD program's one workspace
        st["ws"] = lqcd.make_workspace(lat)
    if kind == "force":
        st["S"] = torch.empty((), dtype=torch.float64, device="cuda")
    if kind == "hmc":
        st["seed"] = 1000 + int(seed)
    if kind == "grad":
        st["omega"] = _normal(lat.algebra_shape, lat, gen, 0.1).requires_grad_()
    if kind in ("dslash", "hopping"):
        st["x"] = _normal(lat.spinor_shape, lat, gen)
        st["y"] = _normal(lat.spinor_shape, lat, gen)
    return st


HMC_DT, HMC_STEPS = 0.05, 5


def run(st):
    kind, lat = st["kind"], st["lat"]
    if kind == "force":   # f, or p += dt f, and S
        out = lqcd.md_force_step(lat, st["links"], force=st.get("force"), mom=st["mom"], dt=DT,
                                 action=st["S"], workspace=st["ws"])
        return [t for t in out if t is not None]
    if kind == "action":
        return [lqcd.gauge_action(lat, st["links"], workspace=st["ws"])]
    if kind == "links":   # U <- exp(i dt p.T) U
        return [lqcd.md_update_links(lat, st["links"], st["mom"], DT)]
    if kind == "grad":
        S = autograd.symanzik_action(st["omega"], st["links"], lat)
        g, = torch.autograd.grad(S, st["omega"])
        return [S.detach(), g]
    if kind == "batch":
        bs = st["bs"]
        hmc.batch_kick(bs, DT)
        hmc.batch_drift(bs, DT)
        return [bs.links, bs.mom]
    if kind == "hmc":     # the links before the trajectory are kept for a rejection
        md = hmc.MDState(lat, st["links"].clone(), st["mom"], st["ws"])
        lqcd.gaussian_momenta(lat, st["seed"], out=md.mom)
        H0 = hmc.hamiltonian(md, "f64")
        hmc.omelyan(md, HMC_DT, HMC_STEPS)
        return [H0, hmc.hamiltonian(md, "f64"), md.links, md.mom]
    if kind == "dslash":
        return [lqcd.wilson_dslash(lat, st["links"], st["x"], 1.0, -KAPPA, out=st["y"])]
    # hopping: p += dt f
    lqcd.wilson_hopping_force(lat, st["links"], st["x"], st["y"], KAPPA, mom=st["mom"], dt=DT)
    return [st["mom"]]


# products of 3x3 complex matrices (198 flops) per link of a force: 12 for
# the six plaquette staples, 6 + 2 for the rectangles along the link, 36 for
# the cubes and the other rectangles, 1 for U t; per site of an action: 16
# two-link corners and 28 closed loops, then 34 traces (36 flops)
_FORCE_FLOPS, _ACTION_FLOPS = 57 * 198, 44 * 198 + 34 * 36
# exponential, two thirds of a product, Gram-Schmidt; series of the chain
# rule through the exponential
_LINK_FLOPS, _SERIES_FLOPS = 900, 8 * 2 * 198


def work(case):
    kind, R = case["kind"], 4 if case["prec"] == "f32" else 8
    if kind == "batch":
        links = 4 * sum(math.prod(d) for d in _batch_dims(case))
    else:
        links = 4 * _lat(case).V
    if kind == "force":    # read U; write f, or read p and write it
        return {"bytes": links * (20 if case["store"] == "force" else 28) * R, "flops": links * _FORCE_FLOPS}
    if kind == "action":   # read U
        return {"bytes": links * 12 * R, "flops": links / 4 * _ACTION_FLOPS}
    if kind == "links":    # read U, p; write U
        return {"bytes": links * 32 * R, "flops": links * _LINK_FLOPS}
    if kind == "grad":     # read U0, omega; write the gradient
        return {"bytes": links * 28 * R, "flops": links * (_FORCE_FLOPS + _ACTION_FLOPS / 4 + _LINK_FLOPS
                                                           + _SERIES_FLOPS)}
    if kind == "batch":    # the momentum step, then the link step
        return {"bytes": links * 60 * R, "flops": links * (_FORCE_FLOPS + _LINK_FLOPS)}
    if kind == "hmc":      # 11 momentum steps, 10 link steps, two Hamiltonians, the refresh
        return {"bytes": links * R * (11 * 28 + 10 * 32 + 2 * 20 + 8),
                "flops": links * (11 * _FORCE_FLOPS + 10 * _LINK_FLOPS + 2 * _ACTION_FLOPS / 4)}
    if kind == "dslash":   # read x, four links; write y
        return {"bytes": links * 24 * R, "flops": links / 4 * 1392}
    return {"bytes": links * 40 * R, "flops": links * 600}


def _normals(seed, count):
    """Box-Muller normals of the SplitMix64 stream `seed`."""
    with np.errstate(over="ignore"):
        z = np.uint64(seed) + np.arange(1, 2 * count + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        z = (z ^ (z >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        z = (z ^ (z >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        z = z ^ (z >> np.uint64(31))
    u = (z >> np.uint64(11)).astype(np.float64)
    return np.sqrt(-2.0 * np.log((u[0::2] + 1.0) * 2.0 ** -53)) * np.cos(2.0 * np.pi * u[1::2] * 2.0 ** -53)


def _kinetic(p):
    return 0.5 * sum(float(x.square().sum()) for x in p)


def exact(case, seed):
    st = prepare(case, seed)
    kind, lat = case["kind"], st["lat"]
    dims, W = lat.dims, lat.W
    if kind == "batch":
        links, mom = [], []
        for d, u, p in zip(st["bs"].dims, st["bs"].links, st["bs"].mom):
            U, P = _read_links(u, d), _read_algebra(p, d)
            P = [a + DT * b for a, b in zip(P, _force_and_action(U, lat)[0])]
            links.append(_links_out(_link_step(U, P, DT), W))
            mom.append(_algebra_out(P, W))
        return [links, mom]
    U = _read_links(st["links"], dims)
    if kind == "force":
        f, S = _force_and_action(U, lat)
        if st["mom"] is not None:
            f = [a + DT * b for a, b in zip(_read_algebra(st["mom"], dims), f)]
        return [_algebra_out(f, W), torch.tensor(S, dtype=torch.float64)]
    if kind == "action":
        return [torch.tensor(_force_and_action(U, lat)[1], dtype=torch.float64)]
    if kind == "links":
        return [_links_out(_link_step(U, _read_algebra(st["mom"], dims), DT), W)]
    if kind == "grad":
        om = _read_algebra(st["omega"].detach(), dims)
        f, S = _force_and_action(_link_step(U, om, 1.0), lat)
        grad = []
        for mu in range(4):   # dS/domega = -(sum_n (-ad_X)^n / (n+1)! f), X = i omega.T
            w, h = _generators(om[mu]), _generators(f[mu])
            acc = h.clone()
            for n in range(1, 25):
                h = (_mm(w, h) - _mm(h, w)) * (-1j / (n + 1))
                acc = acc + h
            # acc = sum_a g_a T_a is Hermitian: tr(lambda_a acc) = -Im tr(lambda_a (-i) acc)
            grad.append(-_components(acc * -1j, 1.0))
        return [torch.tensor(S, dtype=torch.float64), _algebra_out(grad, W)]
    if kind == "hmc":
        V = lat.V
        p = torch.from_numpy(_normals(st["seed"], V * 32).reshape(V, 4, 8)).cuda()
        p = [p[:, mu].t().reshape(8, *dims[::-1]) for mu in range(4)]
        lam = 0.1931833275037836

        def kick(c):
            return [a + c * b for a, b in zip(p, _force_and_action(U, lat)[0])]
        H0 = _kinetic(p) + _force_and_action(U, lat)[1]
        p = kick(lam * HMC_DT)
        for i in range(HMC_STEPS):
            U = _link_step(U, p, HMC_DT / 2)
            p = kick((1 - 2 * lam) * HMC_DT)
            U = _link_step(U, p, HMC_DT / 2)
            p = kick((2 if i < HMC_STEPS - 1 else 1) * lam * HMC_DT)
        H1 = _kinetic(p) + _force_and_action(U, lat)[1]
        return [H0, H1, _links_out(U, W), _algebra_out(p, W)]
    x = _read_spinor(st["x"], dims)
    if kind == "dslash":
        acc = 0
        for mu in range(4):
            back = _sh(_dag(U[mu]), mu, -1)
            acc = acc + _colour(U[mu], _project(_sh(x, mu), mu, -1))
            acc = acc + _colour(back, _project(_sh(x, mu, -1), mu, 1))
        return [_to_rows(_reals(x - KAPPA * acc, 24), W)]
    y, p = _read_spinor(st["y"], dims), _read_algebra(st["mom"], dims)
    for mu in range(4):
        u = U[mu]
        m = (_colour(u, _project(_sh(x, mu), mu, -1))[:, :, None] * y[:, None].conj()).sum(0) \
            - (x[:, :, None] * _colour(u, _project(_sh(y, mu), mu, 1))[:, None].conj()).sum(0)
        p[mu] = p[mu] + DT * _components(m, -KAPPA)
    return [_algebra_out(p, W)]
