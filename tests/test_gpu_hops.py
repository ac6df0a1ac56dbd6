"""The FP32 hopping operator where a thread passes over several sites: lattices
above the number of resident threads, with x hops by shuffles and without,
whole and ragged, against the FP64 operator of the same links and spinors.

Tolerance: with M the largest spinor component, a hop is a projection (2 M, one
rounding), three complex products with a row of an SU(3) link (sum at most
2 sqrt(3) M, six fused operations, the third row six roundings more) and an
addition to a sum of at most 8 hops: 8 hops of 13 roundings of 3.5 M and 8
additions to at most 28 M, 590 M of 2^-24.
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
