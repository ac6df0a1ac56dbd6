"""FP64 calls on fields with entries of very different sizes: links near 1 or
near a subgroup of SU(3), steps of any size, spinors whose components differ
by many orders.  Errors are taken against the size of the entries themselves,
class by class, not against the largest of the field.

References from the stored FP64 inputs: the link steps in long double (80 or
128 bits), the others in floating point, which keeps small entries."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1808_02281_gb300 import build as B
from paper_1808_02281_gb300 import lqcd, synth
from tests import helpers as H
from tests.test_gpu_fixed_point import _force as staple_force, _third as _third64

pytestmark = pytest.mark.gpu

DIMS = (3, 4, 2, 5)
LD, CLD = np.longdouble, np.clongdouble


@pytest.fixture(scope="module", autouse=True)
def _library():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()


def _mm(a, b):
    return (a[..., :, :, None] * b[..., None, :, :]).sum(-2)


def _exp(omega):
    """exp(i omega.T), T_a = lambda_a / 2, by its series with 6 squarings."""
    lam = H.gell_mann().astype(CLD)
    lam[7] = np.diag([1, 1, -2]) / np.sqrt(LD(3))
    x = np.einsum("...a,aij->...ij", omega.astype(LD), lam) * CLD(1j) / 128
    one = np.broadcast_to(np.eye(3, dtype=CLD), x.shape)
    r = one + x / 24
    for k in range(23, 0, -1):
        r = _mm(x, r) / LD(k) + one
    for _ in range(6):
        r = _mm(r, r)
    return r


def _third(U):
    U = U.astype(CLD)
    U[..., 2, :] = np.conj(np.cross(U[..., 0, :], U[..., 1, :]))
    return U


def _gram_schmidt(U):
    a, b = U[..., 0, :], U[..., 1, :]
    a = a / np.sqrt((a * a.conj()).real.sum(-1, keepdims=True))
    b = b - (a.conj() * b).sum(-1, keepdims=True) * a
    b = b / np.sqrt((b * b.conj()).real.sum(-1, keepdims=True))
    return np.stack([a, b], -2)


def _omega(kind, sigma, seed):
    """Normal components of size sigma; with a kind, those of the subgroup of
    size 0.5 (diagonal links, an SU(2) block, the three U(2) blocks, real rotations)."""
    o = synth.momenta(DIMS, seed) * sigma
    for a in {"": (), "ab": (2, 7), "su2": (0, 1, 2), "u2": (0, 1, 2, 7), "u2b": (2, 3, 4, 7), "u2c": (2, 5, 6, 7),
              "so3": (1, 4, 6)}[kind]:
        o[..., a] = synth.momenta(DIMS, seed + 50)[..., a] * 0.5
    return o


def _links(lat, U):
    return lqcd.pack_links(lat, lqcd.full_to_device(lat, U))


def _rows(links):
    """Rows 0, 1 of the stored links [4, 6, V, 2] as [V, 4, 2, 3]."""
    x = links.cpu().numpy().transpose(2, 0, 1, 3)
    return (x[..., 0] + 1j * x[..., 1]).reshape(x.shape[0], 4, 2, 3)


def _check_classes(got, want, tol):
    """Every real of the trailing axes against the largest of its kind in the field."""
    for part in (np.real, np.imag) if np.iscomplexobj(want) else (np.asarray,):
        g, w = part(got).astype(LD), part(want)
        size = np.abs(w).max(0)
        assert (np.abs(g - w).max(0) <= tol * size + 1e-300).all(), (np.abs(g - w).max(0) / (size + 1e-300)).max()


# A floating-point step is some 30 roundings of 1.1e-16; the fixed-point one
# a few.  4e-15 of the largest entry of a class holds for both.
@pytest.mark.parametrize("kind, sigma, step", [
    ("", 0.3, 1e-6), ("", 1e-2, 0.05), ("", 1e-2, 1e-2), ("", 1e-4, 1e-4), ("", 1e-8, 1e-8), ("", 1e-8, 1e-3), ("", 1e-3, 1e-12),
    ("", 0.0, 1e-12), ("", 0.0, 1e-18), ("", 0.0, 1e-200), ("", 1e-8, 0.6), ("ab", 1e-8, 0.05), ("ab", 1e-8, 1e-9),
    ("su2", 1e-8, 1e-9), ("so3", 1e-8, 1e-6)])
def test_link_step_of_small_entries(kind, sigma, step):
    lat = lqcd.Lattice.symanzik(DIMS, 6.0, 0.87, "f64")
    links = _links(lat, _exp(_omega(kind, sigma, 3)).astype(complex))
    U = _third(np.concatenate([_rows(links), np.zeros((lat.V, 4, 1, 3))], -2))
    p = synth.momenta(DIMS, 4)
    lqcd.md_update_links(lat, links, lqcd.algebra_to_device(lat, p), step)
    want = _gram_schmidt(_mm(_exp(p * step), U)[..., :2, :])  # p dt in FP64, as the step takes it
    _check_classes(_rows(links), want, 4e-15)


@pytest.mark.parametrize("kind", ["", "ab", "su2", "u2", "u2b", "u2c", "so3"])
@pytest.mark.parametrize("sigma", [1.0, 0.05, 1e-3, 1e-8, 1e-16, 1e-30])
def test_links_from_small_omega(kind, sigma):
    """Also exponents of a subgroup with small components beside it."""
    lat = lqcd.Lattice.symanzik(DIMS, 6.0, 0.87, "f64")
    omega = _omega(kind, sigma, 7)
    links = lqcd.links_from_omega(lat, lqcd.algebra_to_device(lat, omega))
    _check_classes(_rows(links), _gram_schmidt(_exp(omega)[..., :2, :]), 4e-15)


def _field(dims, kind, sigma, seed):
    V = int(np.prod(dims))
    o = synth.momenta(dims, seed) * sigma
    for a in {"ab": (2, 7), "u2": (0, 1, 2, 7), "so3": (1, 4, 6)}.get(kind, ()):
        o[..., a] = synth.momenta(dims, seed + 50)[..., a] * 0.5
    if kind in ("scaled", "block", "temporal"):
        o = synth.momenta(dims, seed + 50) * 0.4
    if kind == "block":       # 32 sites of small links in a field of large ones
        o[32:64] = synth.momenta(dims, seed)[32:64] * sigma
    U = _third64(O.links_from_omega(o).reshape(V, 4, 3, 3))
    if kind == "scaled":      # no link within 1e-3 of SU(3)
        U = _third64(U * 1.01)
    if kind == "temporal":    # one direction of unit links
        U[:, 3] = np.eye(3)
    return U


# (16, 8, 8, 5) is above the size up to which a link's sums are split over warps.
# Up to some 1000 roundings of terms of the size of the force: 1e-14 of the
# largest of a component.  Fields that are not small: 1e-13 of the largest of all.
@pytest.mark.parametrize("dims", [(3, 4, 2, 5), (16, 8, 8, 5)])
@pytest.mark.parametrize("kind, sigma", [("", 0.0), ("", 1e-2), ("", 1e-4), ("", 1e-8), ("", 1e-20), ("ab", 1e-8), ("u2", 1e-6),
                                         ("so3", 1e-8), ("scaled", 0.0), ("block", 1e-8), ("temporal", 0.0)])
def test_force_of_small_entries(dims, kind, sigma):
    lat = lqcd.Lattice.symanzik(dims, 6.0, 0.87, "f64", force_algo=lqcd.FORCE_STAPLE_FIELDS)
    U = _field(dims, kind, sigma, 5)
    links = _links(lat, U)
    want = staple_force(U, dims, 6.0, O.coefficients(0.87))
    p = synth.momenta(dims, 6) * (sigma or 1.0)
    mom, force, S = lqcd.algebra_to_device(lat, p), lqcd.empty_algebra(lat), torch.empty((), dtype=torch.float64, device="cuda")
    lqcd.md_force_step(lat, links, force=force, mom=mom, dt=0.5, action=S)
    got = lqcd.algebra_from_device(force)
    if kind in ("scaled", "block", "temporal"):
        assert np.abs(got - want).max() <= 1e-13 * np.abs(want).max()
    else:
        _check_classes(got, want, 1e-14)
    q = p + 0.5 * got
    assert np.abs(lqcd.algebra_from_device(mom) - q).max() <= 2.3e-16 * np.abs(q).max()
    if kind != "scaled":   # 34 loops a site, each to 1e-15, under the prefactor 2
        want = O.gauge_action(dims, U, 6.0, O.coefficients(0.87))
        assert abs(float(S.item()) - want) <= 68e-15 * lat.V
    # in a batch with a lattice of large links: the same bits, and those of the other too
    other = lat.with_(dims=(5, 4, 3, 4))
    big = lqcd.links_from_omega(other, lqcd.algebra_to_device(other, synth.omega(other.dims, 0.4, 8)))
    fs, actions = [lqcd.empty_algebra(lat), lqcd.empty_algebra(other)], torch.empty(2, dtype=torch.float64, device="cuda")
    lqcd.md_force_step_batched(lat, [dims, other.dims], [links, big], force=fs, actions=actions)
    assert torch.equal(fs[0], force) and float(actions[0]) == float(S)
    assert torch.equal(fs[1], lqcd.gauge_force(other, big))


# Of a spinor: the colour, the spin rows, the complex entries or the parts that
# are small, by a factor eps
SMALL = {"colour": lambda x, e: x.__setitem__((slice(None), slice(None), 1), x[:, :, 1] * e),
         "colours": lambda x, e: x.__setitem__((slice(None), slice(None), 2), x[:, :, 2] * e * e) or
         x.__setitem__((slice(None), slice(None), 0), x[:, :, 0] * e),
         "rows": lambda x, e: x.__setitem__((slice(None), slice(1, None)), x[:, 1:] * e),
         "row": lambda x, e: x.__setitem__((slice(None), 2), x[:, 2] * e),
         "point": lambda x, e: x.__setitem__(slice(1, None), x[1:] * e) or x.__setitem__((0, slice(1, None)), x[0, 1:] * e),
         "entry": lambda x, e: x.__setitem__((slice(None), slice(1, None), 0), x[:, 1:, 0] * e),
         "parts": lambda x, e: x.imag.__imul__(e)}


def _gammas():
    g = np.zeros((4, 4, 4), complex)
    for mu, (cols, vals) in enumerate([((3, 2, 1, 0), (1j, 1j, -1j, -1j)), ((3, 2, 1, 0), (-1, 1, 1, -1)),
                                       ((2, 3, 0, 1), (1j, -1j, -1j, 1j)), ((2, 3, 0, 1), (1, 1, 1, 1))]):
        g[mu, range(4), cols] = vals
    return g


def _sizes(dims, U, X, Y):
    """Sums of the moduli of the terms of each real or complex result: of
    calD X, of the hopping-term force of X and Y."""
    g, grid = np.abs(_gammas()), dims[::-1]
    sh = lambda a, mu, s: np.roll(a.reshape(*grid, *a.shape[1:]), -s, axis=3 - mu).reshape(a.shape)  # noqa: E731
    m = lambda a: np.abs(a.real) + np.abs(a.imag)  # noqa: E731
    out, force = 0, np.zeros((len(X), 4, 8))
    lam = np.abs(H.gell_mann())
    for mu in range(4):
        u, P = m(U[:, mu]), np.eye(4) + g[mu]
        out = out + np.einsum("st,nab,ntb->nsa", P, u, sh(m(X), mu, 1))
        out = out + sh(np.einsum("st,nba,ntb->nsa", P, u, m(X)), mu, -1)
        uX, uY = (np.einsum("st,nab,ntb->nsa", P, u, sh(m(a), mu, 1)) for a in (X, Y))
        N = np.einsum("nsa,nsb->nab", uX, m(Y)) + np.einsum("nsa,nsb->nab", uY, m(X))
        force[:, mu] = np.einsum("iab,nba->ni", lam, N + N.transpose(0, 2, 1))
    return out, force


# A result against the sum of the moduli of its terms: 1e-14 of it, some 100
# roundings, or the 2^-55 of the scale to which the fixed point knows results that
# are above 2^-7 of it (7e-15).
@pytest.mark.parametrize("eps", [1e-3, 1e-9, 1e-30])
@pytest.mark.parametrize("kind", sorted(SMALL))
@pytest.mark.parametrize("sigma", [0.0, 0.4])
def test_wilson_of_uneven_spinors(kind, sigma, eps):
    lat = lqcd.Lattice.symanzik(DIMS, 6.0, 0.87, "f64")
    U = _third64(O.links_from_omega(synth.momenta(DIMS, 3) * sigma).reshape(lat.V, 4, 3, 3))
    X, Y = (s[..., 0] + 1j * s[..., 1] for s in (synth.spinor(DIMS, 11), synth.spinor(DIMS, 12)))
    for s in (X, Y):
        SMALL[kind](s, eps)
    links, x, y = _links(lat, U), lqcd.spinor_to_device(lat, X), lqcd.spinor_to_device(lat, Y)
    size, fsize = _sizes(DIMS, U, X, Y)
    got = lqcd.spinor_from_device(lqcd.wilson_dslash(lat, links, x, 0.0, 0.7))
    assert (np.abs(got - 0.7 * O.wilson_hopping(DIMS, U, X)) <= 1e-14 * size).all()
    f = lqcd.algebra_from_device(lqcd.wilson_hopping_force(lat, links, x, y, coef=0.7))
    assert (np.abs(f - O.wilson_hopping_force(DIMS, U, X, Y, 0.7)) <= 1e-14 * fsize).all()


# Scaling a spinor by a power of two scales its results by it, to the bit, as
# long as they are normal numbers: 2^-955 is next to the smallest scale of the
# fixed point, and the coefficients are small.
@pytest.mark.parametrize("px, py", [(-955, 955), (940, -900), (-300, -300), (-955, 100), (870, 40)])
@pytest.mark.parametrize("coef", [0.7, 0.7 * 2.0 ** -20])
def test_wilson_scales_with_the_spinors(coef, px, py):
    lat = lqcd.Lattice.symanzik(DIMS, 6.0, 0.87, "f64")
    U = O.links_from_omega(synth.momenta(DIMS, 3) * 0.4).reshape(lat.V, 4, 3, 3)
    links = _links(lat, U)
    x, y = (lqcd.spinor_to_device(lat, synth.spinor(DIMS, s)) for s in (11, 12))
    sx, sy = x * 2.0 ** px, y * 2.0 ** py
    want = lqcd.wilson_dslash(lat, links, x, 0.0, coef)
    assert torch.equal(lqcd.wilson_dslash(lat, links, sx, 0.0, coef), want * 2.0 ** px)
    want = lqcd.wilson_hopping_force(lat, links, x, y, coef=coef)
    assert torch.equal(lqcd.wilson_hopping_force(lat, links, sx, sy, coef=coef), want * 2.0 ** (px + py))


@pytest.mark.parametrize("algo", [lqcd.FORCE_STAPLE_FIELDS, lqcd.FORCE_PATHS])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_what_a_link_that_is_not_finite_reaches(value, algo):
    """The links that may read it, found from the formulas; every other link
    has the force that it had, to the bit."""
    dims = (6, 5, 4, 6)
    lat = lqcd.Lattice.symanzik(dims, 6.0, 0.87, "f64", force_algo=algo)
    links = lqcd.links_from_omega(lat, lqcd.algebra_to_device(lat, synth.omega(dims, 0.3, 1)))
    clean = lqcd.algebra_from_device(lqcd.gauge_force(lat, links))
    U = lqcd.full_from_device(lqcd.unpack_links(lat, links))
    links[1, 2, 77, 0] = value
    U[77, 1] = np.nan
    with np.errstate(invalid="ignore"):
        reach = ~np.isfinite(staple_force(U, dims, 6.0, O.coefficients(0.87))).all(-1)
    assert 40 < reach.sum() < reach.size // 2
    f = lqcd.algebra_from_device(lqcd.gauge_force(lat, links))
    assert np.isfinite(f[~reach]).all() and np.array_equal(f[~reach], clean[~reach])
    assert not np.isfinite(f[reach]).all(-1).any()


def test_hopping_force_of_a_large_coefficient():
    """A coefficient of 2^990 and spinors that make up for it."""
    lat = lqcd.Lattice.symanzik(DIMS, 6.0, 0.87, "f64")
    links = _links(lat, O.links_from_omega(synth.momenta(DIMS, 3) * 0.4).reshape(lat.V, 4, 3, 3))
    x, y = (lqcd.spinor_to_device(lat, synth.spinor(DIMS, s)) for s in (11, 12))
    want = lqcd.wilson_hopping_force(lat, links, x, y, coef=0.7)
    got = lqcd.wilson_hopping_force(lat, links, x * 2.0 ** -500, y * 2.0 ** -490, coef=0.7 * 2.0 ** 990)
    assert (got - want).abs().max() <= 1e-14 * want.abs().max()
