"""The staple-field force in the least workspace that it takes: 24 planes of 18
reals a site, sites rounded up to 32, and one double per 32 sites."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1808_02281_gb300 import build as B
from paper_1808_02281_gb300 import hmc, lqcd, synth

pytestmark = pytest.mark.gpu

DIMS = [(3, 2, 2, 3), (4, 4, 4, 6), (17, 8, 8, 4)]  # two whose sums are split over warps in a larger one
TOL = {"f64": 1e-12, "f32": 2e-5}


@pytest.fixture(scope="module", autouse=True)
def _library():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()


def _least(dims, prec):
    blocks = (int(np.prod(dims)) + 31) // 32
    up = lambda b: (b + 255) // 256 * 256  # noqa: E731
    return up(24 * 18 * (8 if prec == "f64" else 4) * 32 * blocks) + up(8 * blocks)


def _guarded(n):
    """A workspace of n bytes, and the bytes behind it."""
    buf = torch.full((n + 4096,), 0x5a, dtype=torch.uint8, device="cuda")
    return buf[:n], buf[n:]


@pytest.mark.parametrize("algo", [lqcd.FORCE_AUTO, lqcd.FORCE_STAPLE_FIELDS])
@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("dims", DIMS)
def test_least_workspace(dims, prec, algo):
    lat = lqcd.Lattice.symanzik(dims, 6.0, 0.87, prec, force_algo=algo)
    n = max(_least(dims, prec), lqcd.reduction_workspace().numel())  # AUTO's action without staple fields takes that
    omega = synth.omega(dims, 0.3, 5)
    links = lqcd.links_from_omega(lat, lqcd.algebra_to_device(lat, omega))
    f, S = lqcd.empty_algebra(lat), torch.empty((), dtype=torch.float64, device="cuda")
    ws, behind = _guarded(n)
    lqcd.md_force_step(lat, links, force=f, action=S, workspace=ws)
    U, c = O.links_from_omega(omega), O.coefficients(0.87)
    ref, want = O.gauge_force(dims, U, 6.0, c), O.gauge_action(dims, U, 6.0, c)
    assert np.abs(lqcd.algebra_from_device(f) - ref).max() <= TOL[prec] * np.abs(ref).max()
    assert abs(float(S) - want) <= TOL[prec] * abs(want)
    assert (behind == 0x5a).all()
    # the staple fields, and not another algorithm
    assert torch.equal(f, lqcd.gauge_force(lat.with_(force_algo=lqcd.FORCE_STAPLE_FIELDS), links, workspace=ws))
    assert not torch.equal(f, lqcd.gauge_force(lat.with_(force_algo=lqcd.FORCE_FACTORED), links))
    best, times = lqcd.autotune_force(lat, links, reps=1, workspace=ws)
    lqcd.set_force_variant(lat, -1)
    assert len(times) == lqcd.force_variant_count(lat) and (behind == 0x5a).all()
    if algo == lqcd.FORCE_STAPLE_FIELDS:
        with pytest.raises(RuntimeError):
            lqcd.gauge_force(lat, links, workspace=ws[:_least(dims, prec) - 256])


@pytest.mark.parametrize("prec", ["f64", "f32"])
def test_least_batch_workspace(prec):
    bs = hmc.initial_batch(DIMS, prec, seed=7)
    n = sum(_least(d, prec) for d in bs.dims) + 256
    actions = torch.empty(len(DIMS), dtype=torch.float64, device="cuda")
    force = [lqcd.empty_algebra(bs.params.with_(dims=d)) for d in bs.dims]
    ws, behind = _guarded(n)
    lqcd.md_force_step_batched(bs.params, bs.dims, bs.links, force=force, actions=actions, workspace=ws)
    assert (behind == 0x5a).all()
    for c, d in enumerate(bs.dims):
        lat = bs.params.with_(dims=d, force_algo=lqcd.FORCE_STAPLE_FIELDS)
        f, S = lqcd.empty_algebra(lat), torch.empty((), dtype=torch.float64, device="cuda")
        one, _ = _guarded(max(_least(d, prec), lqcd.reduction_workspace().numel()))
        lqcd.md_force_step(lat, bs.links[c], force=f, action=S, workspace=one[:_least(d, prec)])
        assert torch.equal(f, force[c]) and float(S) == float(actions[c]), d
    with pytest.raises(RuntimeError):
        lqcd.md_force_step_batched(bs.params, bs.dims, bs.links, force=force, actions=actions, workspace=ws[:n - 256])


def test_recommended_workspace_fits_the_device():
    """Above 240 GB the least workspace is the recommended one."""
    for dims, planes in (((96, 96, 96, 64), 28), ((96, 96, 96, 72), 24)):
        lat = lqcd.Lattice.symanzik(dims, 6.0, 0.87, "f64")
        per_site = lqcd.workspace_bytes(lat) / lat.V
        assert planes * 144 <= per_site < planes * 144 + 1
