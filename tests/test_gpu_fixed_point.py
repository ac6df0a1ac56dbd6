"""FP64 force and action on links without a fixed-point form (not within 1e-3
of SU(3), or not finite): the links and loops that read one are computed in
floating point, everything else in fixed point, and neither shows.

References: the staple-field formulas of the force written out in numpy (they
use U U^dag = 1, so for such links they differ from the walked staples), and
the oracle's action, which walks the loops."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1808_02281_gb300 import build as B
from paper_1808_02281_gb300 import lqcd, synth
from tests import helpers as H

pytestmark = pytest.mark.gpu

# sum of up to 48 products of a few matrices of entries near 1, each rounded
# to 1.1e-16: 1e-13 of the largest entry is a wide margin
TOL = 1e-13


@pytest.fixture(scope="module", autouse=True)
def _library():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()


def _third(U):
    U = U.copy()
    U[..., 2, :] = np.conj(np.cross(U[..., 0, :], U[..., 1, :]))
    return U


def _dag(a):
    return np.conj(np.swapaxes(a, -1, -2))


def _force(U, dims, beta, c):
    """f[V, 4, 8] from the staple fields, U [V, 4, 3, 3] with row 2 rebuilt."""
    grid = U.reshape(*dims[::-1], 4, 3, 3)
    link = [grid[..., mu, :, :] for mu in range(4)]
    sh = lambda a, mu, s: np.roll(a, -s, axis=3 - mu)  # noqa: E731
    S = {}
    for mu in range(4):
        for nu in range(4):
            if nu == mu:
                continue
            S[mu, nu, 1] = _third(sh(link[nu], mu, 1) @ _dag(sh(link[mu], nu, 1)) @ _dag(link[nu]))
            dn = sh(link[nu], nu, -1)
            S[mu, nu, -1] = _third(_dag(sh(dn, mu, 1)) @ _dag(sh(link[mu], nu, -1)) @ dn)
    out = np.empty((*dims[::-1], 4, 8))
    for rho in range(4):
        dirs = [(nu, s) for nu in range(4) if nu != rho for s in (1, -1)]
        pl = sum(S[(rho, *b)] for b in dirs)
        p1 = sum(sh(S[(rho, *b)], rho, 1) @ S[(rho, *b)] for b in dirs)
        p2 = sum(S[(rho, *b)] @ sh(S[(rho, *b)], rho, -1) for b in dirs)
        t = c[0] * pl + c[1] * (sh(link[rho], rho, 1) @ p1 + p2 @ sh(link[rho], rho, -1))
        for d, s in dirs:
            A = link[d] if s > 0 else _dag(sh(link[d], d, -1))
            y = c[1] * sh(S[rho, d, s], d, s) @ _dag(A)
            for b in dirs:
                if b[0] != d:
                    second = S[(d, *b)] if s > 0 else _dag(sh(S[(d, *b)], d, -1))
                    y = y + c[2] * sh(S[(rho, *b)], d, s) @ second
            t = t + sh(A, rho, 1) @ y
        m = beta / 6 * (link[rho] @ t)
        out[..., rho, :] = -np.einsum("aij,...ji->...a", H.gell_mann(), m).imag
    return out.reshape(-1, 4, 8)


def _links(lat, U):
    return lqcd.pack_links(lat, lqcd.full_to_device(lat, U))


@pytest.mark.parametrize("u0", [0.87, 1.0])  # u0 = 1: no cube term
@pytest.mark.parametrize("scaled", [(), (0,), (3, 17, 41)])
@pytest.mark.parametrize("dims", [(4, 4, 2, 3), (3, 2, 5, 4)])
def test_scaled_links(dims, scaled, u0):
    lat = lqcd.Lattice.symanzik(dims, 6.0, u0, "f64")
    U = O.links_from_omega(synth.omega(dims, 0.4, 3)).reshape(lat.V, 4, 3, 3)
    for i in scaled:  # rows scaled by 1.01: outside of 1e-3
        U[i // 4, i % 4, :2] *= 1.01
    U = _third(U)
    c = O.coefficients(u0)
    links = _links(lat, U)
    force = lqcd.empty_algebra(lat)
    S = torch.empty((), dtype=torch.float64, device="cuda")
    lqcd.md_force_step(lat, links, force=force, action=S)
    ref = _force(U, dims, 6.0, c)
    assert np.abs(lqcd.algebra_from_device(force) - ref).max() <= TOL * np.abs(ref).max()
    want = O.gauge_action(dims, U, 6.0, c)
    whole = lqcd.make_workspace(lat)   # room for the link planes, or not: the same bits
    a = float(lqcd.gauge_action(lat, links, workspace=whole).item())
    assert a == float(lqcd.gauge_action(lat, links).item())
    assert abs(a - want) <= TOL * abs(want)
    if not scaled:
        assert abs(float(S.item()) - want) <= TOL * abs(want)


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_links_that_are_not_finite(value):
    """The force of every link whose staples read the entry is not finite, as
    with the walked staples; the others are what they were."""
    dims = (6, 5, 4, 6)
    lat = lqcd.Lattice.symanzik(dims, 6.0, 0.87, "f64", force_algo=lqcd.FORCE_STAPLE_FIELDS)
    links = lqcd.links_from_omega(lat, lqcd.algebra_to_device(lat, synth.omega(dims, 0.3, 1)))
    clean = lqcd.algebra_from_device(lqcd.gauge_force(lat, links))
    links[1, 2, 77, 0] = value
    f = lqcd.algebra_from_device(lqcd.gauge_force(lat, links))
    paths = lqcd.algebra_from_device(lqcd.gauge_force(lat.with_(force_algo=lqcd.FORCE_PATHS), links))
    bad = ~np.isfinite(paths).all(-1)
    assert bad.any() and not bad.all()
    assert (~np.isfinite(f).all(-1) >= bad).all()
    fine = np.isfinite(f).all(-1)
    assert np.array_equal(f[fine], clean[fine])
    assert not np.isfinite(float(lqcd.gauge_action(lat, links).item()))


@pytest.mark.parametrize("coef", [(1.0, 0.0, 0.0), (0.0, 1.0, 0.0), (0.0, 0.0, 1.0), (0.2, -0.1, 0.7), (-1.0, 1e-9, 1e3),
                                  (0.0, 0.0, 0.0)])
def test_any_coefficients(coef):
    """The scalars of the fixed-point sums for any sizes and signs."""
    dims = (3, 4, 5, 2)
    lat = lqcd.Lattice(dims, "f64", 6.0, *coef, force_algo=lqcd.FORCE_STAPLE_FIELDS)
    omega = synth.omega(dims, 0.5, 2)
    links = lqcd.links_from_omega(lat, lqcd.algebra_to_device(lat, omega))
    force = lqcd.empty_algebra(lat)
    S = torch.empty((), dtype=torch.float64, device="cuda")
    lqcd.md_force_step(lat, links, force=force, action=S)
    U = O.links_from_omega(omega)
    ref = O.gauge_force(dims, U, 6.0, np.array(coef))
    want = O.gauge_action(dims, U, 6.0, np.array(coef))
    assert np.abs(lqcd.algebra_from_device(force) - ref).max() <= 1e-12 * np.abs(ref).max()
    assert abs(float(S.item()) - want) <= 1e-12 * abs(want)
    assert abs(float(lqcd.gauge_action(lat, links).item()) - want) <= 1e-12 * abs(want)


@pytest.mark.parametrize("scale_x, scale_y", [(1.0, 1.0), (1e-200, 1e200), (3e140, 2e-90), (0.0, 1.0)])
@pytest.mark.parametrize("scaled", [(), (5, 6)])
def test_hopping_force_scales(scale_x, scale_y, scaled):
    """FP64 hopping-term force of spinors of any size, entries of very
    different sizes among them, and of links without a fixed-point form."""
    dims = (3, 4, 2, 5)
    lat = lqcd.Lattice.symanzik(dims, 6.0, 0.87, "f64")
    U = O.links_from_omega(synth.omega(dims, 0.4, 3)).reshape(lat.V, 4, 3, 3)
    for i in scaled:
        U[i // 4, i % 4, :2] *= 1.01
    U = _third(U)
    X, Y = (synth.spinor(dims, s) for s in (11, 12))
    X[::7] *= 1e-9
    Y[:, 2] *= 1e-5
    X, Y = (s[..., 0] + 1j * s[..., 1] for s in (X * scale_x, Y * scale_y))
    f = lqcd.algebra_from_device(lqcd.wilson_hopping_force(lat, _links(lat, U), lqcd.spinor_to_device(lat, X),
                                                           lqcd.spinor_to_device(lat, Y), coef=0.5))
    ref = O.wilson_hopping_force(dims, U, X, Y, 0.5)
    # each link's force against the size of the spinors it is made of
    size = np.abs(ref).max(-1, keepdims=True) + 1e-300
    big = np.abs(f - ref).max(-1, keepdims=True) / size
    assert (big[np.broadcast_to(size > 1e-290, big.shape)] <= 1e-11).all()
    if scale_x == 0.0:
        assert not f.any()


@pytest.mark.parametrize("dt", [0.05, 0.6, 3.0, 40.0])
@pytest.mark.parametrize("scaled", [(), (0, 9)])
def test_link_step_sizes(dt, scaled):
    """FP64 link step from small to large exponents (the step is then made 2^s
    times, or in floating point) and on links that depart from SU(3)."""
    dims = (3, 4, 2, 5)
    lat = lqcd.Lattice.symanzik(dims, 6.0, 0.87, "f64")
    U = O.links_from_omega(synth.omega(dims, 0.4, 3)).reshape(lat.V, 4, 3, 3)
    for i in scaled:
        U[i // 4, i % 4, 0] *= 1.0 + 1e-6
        U[i // 4, i % 4, 1] += 1e-4 * U[i // 4, i % 4, 0]
    U = _third(U)
    p = synth.momenta(dims, 4)
    p[::3] *= 1e-6
    links = _links(lat, U)
    lqcd.md_update_links(lat, links, lqcd.algebra_to_device(lat, p), dt)
    got = lqcd.full_from_device(lqcd.unpack_links(lat, links))
    # exponents up to about 10 dt: their rounding is that of the angle
    assert np.abs(got - O.md_update_links(U, p, dt)).max() <= 1e-13 * max(1.0, 10 * dt)


@pytest.mark.parametrize("scale", [1.0, 1e-250, 1e200])
@pytest.mark.parametrize("scaled", [(), (5, 6)])
@pytest.mark.parametrize("dims", [(3, 4, 2, 5), (1, 2, 7, 3)])
def test_hopping_operator_scales(dims, scale, scaled):
    """FP64 hopping operator of spinors whose sizes change by many orders from
    site to site (each neighbour has its own scale), zeros among them, and of
    links without a fixed-point form."""
    lat = lqcd.Lattice.symanzik(dims, 6.0, 0.87, "f64")
    U = O.links_from_omega(synth.omega(dims, 0.4, 3)).reshape(lat.V, 4, 3, 3)
    for i in scaled:
        U[i // 4, i % 4, :2] *= 1.01
    U = _third(U)
    x = synth.spinor(dims, 11)
    x = (x[..., 0] + 1j * x[..., 1]) * scale
    x[1::5] *= 1e-12
    x[2::7] = 0.0
    x[3::11] *= 1e25
    got = lqcd.spinor_from_device(lqcd.wilson_dslash(lat, _links(lat, U), lqcd.spinor_to_device(lat, x), 1.0, -0.13))
    ref = x - 0.13 * O.wilson_hopping(dims, U, x)
    # every site against the largest of the nine spinors it is made of: 8 hops,
    # a few roundings each
    grid = np.abs(x).max((1, 2)).reshape(dims[::-1])
    near = np.max([grid] + [np.roll(grid, s, axis) for axis in range(4) for s in (1, -1)], axis=0).reshape(-1)
    assert (np.abs(got - ref).max((1, 2)) <= 2e-15 * near).all()
    zero = torch.zeros(lat.spinor_shape, dtype=torch.float64, device="cuda")
    assert not lqcd.wilson_dslash(lat, _links(lat, U), zero, 0.0, 1.0).any()
