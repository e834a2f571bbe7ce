"""The tridiagonal reduction held in one thread block, at the edges of its
range: ragged warps (31 to 33 rows), the largest order it takes (224 in FP32,
96 in FP64) and the first that goes to a launch per column, and matrices whose
columns need no reflector (diagonal, tridiagonal, a repeated eigenvalue).

Tolerance: that of the decomposition's own test, 100 n u."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import U32, U64, dev_cm, host_cm

pytestmark = pytest.mark.gpu

mp = pytest.importorskip("paper_2607_12430_gb300")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    mp.lib()


def _check(A, fp64):
    n = A.shape[0]
    e = oracle.scale_exponent(A)
    As = A * 4.0 ** -e
    u = U64 if fp64 else U32
    Asr = As if fp64 else As.astype(np.float32)
    V, lam = mp.step_syevd(dev_cm(Asr, torch.float64 if fp64 else torch.float32), n, fp64=fp64)
    V = host_cm(V, n).astype(np.float64)
    lam = lam.cpu().numpy().astype(np.float64)
    nrm = np.linalg.norm(As)
    assert np.linalg.norm(V.T @ V - np.eye(n)) <= 100 * n * u
    assert np.linalg.norm((V * lam[None, :]) @ V.T - As) <= 100 * n * u * nrm
    assert np.abs(np.sort(lam) - np.linalg.eigvalsh(As)).max() <= 100 * n * u * nrm


@pytest.mark.parametrize("fp64,n", [(f, n) for f in (False, True) for n in (3, 4, 31, 32, 33, 34, 63, 65, 66, 95, 96, 97)]
                         + [(False, n) for n in (98, 127, 129, 160, 191, 193, 223, 224, 225)])
def test_sizes(n, fp64):
    A, _, _ = synth.spd_case(n, -1.0, 1.0, seed=8100 + n)
    _check(A, fp64)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("form", ["diagonal", "tridiagonal", "repeated", "arrow"])
def test_structured(form, fp64):
    n = 70
    d = 1.0 + np.arange(n) / 7.0
    if form == "diagonal":
        A = np.diag(d)
    elif form == "tridiagonal":
        A = np.diag(d + 2) + np.diag(np.full(n - 1, 0.5), 1) + np.diag(np.full(n - 1, 0.5), -1)
    elif form == "repeated":
        w = np.cos(np.arange(n))[:, None]
        A = 2.0 * np.eye(n) + w @ w.T / n
    else:
        A = np.diag(d + 3)
        A[0, 1:] = A[1:, 0] = 1.0 / n
    _check(A, fp64)
