"""FP32 momenta are the FP64 ones rounded once, whatever computes them."""
import numpy as np
import pytest
import torch

from paper_1808_02281_gb300 import build as B
from paper_1808_02281_gb300 import lqcd

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _library():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    B.build()


@pytest.mark.parametrize("seed", [1, 77, 2 ** 63 + 5])
@pytest.mark.parametrize("dims", [(3, 2, 5, 1), (16, 16, 16, 32)])
def test_single_precision_rounds_double(dims, seed):
    single, double = (lqcd.gaussian_momenta(lqcd.Lattice(dims, p), seed) for p in ("f32", "f64"))
    want = lqcd.algebra_from_device(double).astype(np.float32)
    assert np.array_equal(lqcd.algebra_from_device(single).astype(np.float32), want)
