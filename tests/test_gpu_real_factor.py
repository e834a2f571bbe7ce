"""The factor that the FP32 general path computes for a real matrix: A_s = Q T
Q^H by the real QR iteration, through the Schur step, in each of the forms of
its chase (blocks of one warp, matrix resident in shared memory, cooperative,
with more than 32 helpers).

Bounds: every entry of Q takes on the order of n reflections of random
rounding errors, so ||Q^H Q - I||_F grows like n u and the backward error like
sqrt(n) u ||A||_F.  The constants are about twice those of the kernels compiled
for the CPU (3.2 to 3.9 n u and 6.4 to 6.9 sqrt(n) u for n = 25 .. 400), so that
a lost digit or a window with a few wrong entries fails.  Two runs agree bit for
bit: every summation order is fixed, so they can differ only where threads
race."""
import numpy as np
import pytest
import torch

import synth
from gpu_util import U32, dev_cm, host_cm

pytestmark = pytest.mark.gpu

mp = pytest.importorskip("paper_2607_12430_gb300")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    mp.lib()


def factor_errors(A, T, Q):
    """||A - Q T Q^H||_F / ||A||_F and ||Q^H Q - I||_F in FP64."""
    T, Q = T.astype(np.complex128), Q.astype(np.complex128)
    assert np.all(np.tril(T, -1) == 0)
    return (np.linalg.norm(Q @ T @ Q.conj().T - A) / np.linalg.norm(A),
            np.linalg.norm(Q.conj().T @ Q - np.eye(A.shape[0])))


def schur32(A):
    T = dev_cm(A.astype(np.complex64), torch.complex64)
    Q = mp.step_schur(T, A.shape[0])
    return host_cm(T, A.shape[0]), host_cm(Q, A.shape[0])


@pytest.mark.parametrize("n", [2, 24, 25, 81, 130, 224, 225, 300, 512, 1100])
def test_factor(n):
    A = synth.shifted_gaussian(n, 3.0, seed=8500 + n).astype(np.float32).astype(np.float64)
    T, Q = schur32(A)
    back, orth = factor_errors(A, T, Q)
    assert back <= 14 * np.sqrt(n) * U32
    assert orth <= 8 * n * U32
    T2, Q2 = schur32(A)
    assert np.array_equal(T, T2) and np.array_equal(Q, Q2)


@pytest.mark.parametrize("helpers", [0, 1, 24])
def test_staged_and_cooperative_factors(helpers):
    n = 300
    A = synth.shifted_gaussian(n, 3.0, seed=8600).astype(np.float32).astype(np.float64)
    saved = mp.get_tuning()
    try:
        mp.set_tuning([{"n_max": 1 << 20, "blks": 32, "qr_helpers": helpers, "batched": 1, "spd_precision": 0}])
        T, Q = schur32(A)
    finally:
        mp.set_tuning(saved)
    back, orth = factor_errors(A, T, Q)
    assert back <= 14 * np.sqrt(n) * U32 and orth <= 8 * n * U32


@pytest.mark.parametrize("n", [130, 200, 224, 300, 512, 1100])
def test_reflectors_are_orthogonal_to_one_rounding(n):
    """tau agrees with the rounded v of each reflector, so its own rounding is
    what is left of P^T P - I: 4.1 to 5.0 sqrt(n) u and 2.7 to 3.2 n u with the
    kernels compiled for the CPU (5.9 to 7.7 and 3.4 to 4.3 with tau = |d| / ||x||
    as it came)."""
    A = synth.shifted_gaussian(n, 3.0, seed=8550 + n).astype(np.float32).astype(np.float64)
    back, orth = factor_errors(A, *schur32(A))
    assert back <= 5.6 * np.sqrt(n) * U32 and orth <= 3.4 * n * U32
