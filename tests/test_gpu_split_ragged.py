"""The general split residual from digits in global memory (n > 1024) at sizes
with ragged output tiles and a remainder in k: exact on inputs whose products
and sums are exact in FP64 (see test_gpu_split_residual.py)."""
import numpy as np
import pytest
import torch

from gpu_util import dev_cm, host_cm

pytestmark = pytest.mark.gpu

mp = pytest.importorskip("paper_2607_12430_gb300")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    mp.lib()


@pytest.mark.parametrize("n", [1025, 1027, 1087, 1151, 1279, 1500])
def test_exact_on_dyadic_inputs(n):
    g = np.random.default_rng(n)
    X = g.integers(-1023, 1024, size=(n, n)) / 1024.0
    X = (2.0 ** g.integers(0, 2, size=n))[:, None] * X * (2.0 ** g.integers(0, 2, size=n))[None, :]
    XX = X @ X
    A = XX + g.integers(-255, 256, size=(n, n)) / 2.0 ** 20
    R = A - XX
    Rs, ns = mp.step_residual_split(dev_cm(A, torch.float64), dev_cm(X, torch.float64), n, e=0)
    assert np.array_equal(host_cm(Rs, n), R.astype(np.float32))
    assert ns == pytest.approx(np.linalg.norm(R), rel=1e-14)
