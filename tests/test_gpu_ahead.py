"""The FP32 hopping operator and link step where a thread passes over several
sites or links: lattices above the number of resident threads, whole and
ragged, against the FP64 kernels of the same fields.

Tolerance of the operator: with M the largest spinor component, a hop is a projection (2 M, one
rounding), three complex products with a row of an SU(3) link (sum at most
2 sqrt(3) M, six fused operations, the third row six roundings more) and an
addition to a sum of at most 8 hops: 8 hops of 13 roundings of 3.5 M and 8
additions to at most 28 M, 590 M of 2^-24.  Of the link step: of entries of at
most 1, dt p (|dt p| below 2, three roundings of it), the exponential (its
squarings, 20 roundings), a product (12 roundings of partial sums up to sqrt(3))
and the Gram-Schmidt step (16): 60 of 2^-24.
"""
import numpy as np
import pytest
import torch

from paper_1808_02281_gb300 import build as B
from paper_1808_02281_gb300 import lqcd, synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()


@pytest.mark.parametrize("dims", [(32, 16, 16, 16), (18, 18, 18, 19), (16, 10, 30, 41), (64, 12, 13, 17), (1, 400, 20, 25)])
def test_operator_over_several_sites_a_thread(dims):
    lat, ref = lqcd.Lattice(dims, "f32"), lqcd.Lattice(dims, "f64")
    omega = lqcd.algebra_to_device(lat, synth.omega(dims, 0.4, 5))
    U = lqcd.links_from_omega(lat, omega)
    U64 = lqcd.convert_links(lat, U, "f64")
    x = synth.spinor(dims, 17)
    X = lqcd.spinor_to_device(lat, x)
    X64 = lqcd.spinor_to_device(ref, lqcd.spinor_from_device(X))
    tol = 590 * 2.0**-24 * float(X.abs().max())
    for ca, cb in ((0.0, 1.0), (1.0, -0.1315)):
        got = lqcd.spinor_from_device(lqcd.wilson_dslash(lat, U, X, ca, cb))
        want = lqcd.spinor_from_device(lqcd.wilson_dslash(ref, U64, X64, ca, cb))
        assert np.abs(got - want).max() <= tol


def _random_step(dims, seed):
    lat = lqcd.Lattice(dims, "f32")
    U = lqcd.links_from_omega(lat, lqcd.algebra_to_device(lat, synth.omega(dims, 0.4, seed)))
    return lat, U, lqcd.algebra_to_device(lat, synth.omega(dims, 1.0, seed + 1))


@pytest.mark.parametrize("dims", [(16, 16, 16, 10), (15, 13, 11, 21), (7, 9, 40, 31), (1, 401, 20, 11)])
def test_link_step_over_several_links_a_thread(dims):
    lat, U, p = _random_step(dims, 3)
    ref = lqcd.Lattice(dims, "f64")
    U64, p64 = lqcd.convert_links(lat, U, "f64"), lqcd.convert_algebra(lat, p, "f64")
    for _ in range(2):
        lqcd.md_update_links(lat, U, p, 0.25)
        lqcd.md_update_links(ref, U64, p64, 0.25)
        err = (lqcd.convert_links(lat, U, "f64") - U64).abs().max()
        assert float(err) <= 60 * 2.0**-24
        U64 = lqcd.convert_links(lat, U, "f64")


def test_batched_link_step_over_several_links_a_thread():
    dims = [(15, 13, 11, 21), (3, 4, 5, 6), (1, 1, 1, 1), (16, 16, 16, 10), (2, 3, 2, 1)]
    fields = [_random_step(d, 7 + i) for i, d in enumerate(dims)]
    links = [U.clone() for _, U, _ in fields]
    lqcd.md_update_links_batched(fields[0][0], dims, links, [p for _, _, p in fields], 0.25)
    for (lat, U, p), got in zip(fields, links):
        lqcd.md_update_links(lat, U, p, 0.25)
        assert torch.equal(got, U)
