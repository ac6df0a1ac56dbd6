"""Small lattices, whose link sums are split over several warps: around the
size where that starts, for every extent parity, alone and in batches (all
split, or mixed with larger ones)."""
import numpy as np
import pytest
import torch

from oracle import oracle as O
from paper_1808_02281_gb300 import build as B
from paper_1808_02281_gb300 import hmc, lqcd, synth

pytestmark = pytest.mark.gpu

# 32 sites are a block; lattices of up to 128 blocks are split
SIZES = [(1, 1, 1, 1), (2, 2, 2, 4), (3, 1, 11, 1), (7, 3, 5, 9), (16, 8, 4, 4), (17, 8, 15, 1), (16, 8, 8, 4), (13, 9, 7, 5), (13, 9, 9, 4)]
TOL = {"f64": 1e-12, "f32": 2e-5}


@pytest.fixture(scope="module", autouse=True)
def _library():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("dims", SIZES)
def test_force_and_action(dims, prec):
    lat = lqcd.Lattice.symanzik(dims, 6.0, 0.87, prec, force_algo=lqcd.FORCE_STAPLE_FIELDS)
    omega = synth.omega(dims, 0.3, 5)
    links = lqcd.links_from_omega(lat, lqcd.algebra_to_device(lat, omega))
    force, S = lqcd.empty_algebra(lat), torch.empty((), dtype=torch.float64, device="cuda")
    p = synth.momenta(dims, 6)
    mom = lqcd.algebra_to_device(lat, p)
    lqcd.md_force_step(lat, links, force=force, mom=mom, dt=0.1, action=S)
    U, c = O.links_from_omega(omega), O.coefficients(0.87)
    f, want = O.gauge_force(dims, U, 6.0, c), O.gauge_action(dims, U, 6.0, c)
    assert np.abs(lqcd.algebra_from_device(force) - f).max() <= TOL[prec] * np.abs(f).max()
    assert abs(float(S.item()) - want) <= TOL[prec] * abs(want)
    q = O.md_update_momenta(p, f, 0.1)
    assert np.abs(lqcd.algebra_from_device(mom) - q).max() <= TOL[prec] * np.abs(q).max()
    again = lqcd.gauge_force(lat, links)   # without the action and the momenta
    assert torch.equal(again, force)


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("dims_list", [SIZES[:6], SIZES[2:5] + [(17, 8, 8, 2)], [(20, 8, 12, 6), (4, 4, 4, 4)]])
def test_batches_equal_single(dims_list, prec):
    bs = hmc.initial_batch(dims_list, prec, seed=7)
    actions = torch.empty(len(dims_list), dtype=torch.float64, device="cuda")
    force = [lqcd.empty_algebra(bs.params.with_(dims=d)) for d in bs.dims]
    lqcd.md_force_step_batched(bs.params, bs.dims, bs.links, force=force, actions=actions, workspace=bs.workspace)
    for c, d in enumerate(bs.dims):
        lat = bs.params.with_(dims=d)
        f, S = lqcd.empty_algebra(lat), torch.empty((), dtype=torch.float64, device="cuda")
        lqcd.md_force_step(lat, bs.links[c], force=f, action=S)
        assert torch.equal(f, force[c]), d
        assert float(S) == float(actions[c]), d


@pytest.mark.parametrize("prec", ["f64", "f32"])
@pytest.mark.parametrize("tile", [(4, 4, 4, 4), (2, 3, 4, 5)])
def test_split_has_the_bits_of_the_whole(tile, prec):
    """Links that repeat with period `tile` on a lattice that is not split: every
    copy has the force of the split lattice of one tile, to the bit, and the
    action is the tile's times the copies (sums in FP64: 1e-13)."""
    times = (2, 2, 4, 4) if tile[0] == 4 else (4, 4, 4, 4)
    big = tuple(a * b for a, b in zip(tile, times))
    small, large = (lqcd.Lattice.symanzik(d, 6.0, 0.87, prec, force_algo=lqcd.FORCE_STAPLE_FIELDS) for d in (tile, big))
    grids = np.indices(big[::-1])  # t, z, y, x
    n = np.zeros(big[::-1], dtype=np.int64)
    for g, d in zip(grids, tile[::-1]):
        n = n * d + g % d
    at = torch.from_numpy(n.reshape(-1)).cuda()
    links = lqcd.links_from_omega(small, lqcd.algebra_to_device(small, synth.omega(tile, 0.4, 9)))
    copies = lqcd.pack_links(large, lqcd.unpack_links(small, links)[at].contiguous())
    out = []
    for lat, U in ((small, links), (large, copies)):
        S = torch.empty((), dtype=torch.float64, device="cuda")
        force = lqcd.empty_algebra(lat)
        lqcd.md_force_step(lat, U, force=force, action=S)
        out.append((lqcd.algebra_from_device(force), float(S.item())))
    (f, s), (f_copies, s_copies) = out
    assert (f_copies.reshape(large.V, -1) == f.reshape(small.V, -1)[n.reshape(-1)]).all()
    assert abs(s_copies - s * large.V / small.V) <= 1e-13 * abs(s_copies)
