"""The real multishift QR iteration of the FP32 general path: the initial
iterate X_0 = Re(Q S Q^H) (steps = 0) against the FP64 oracle at the sizes
where the iteration changes form -- the single-warp blocks (n <= 24), the
window block (81), the matrix resident in shared memory (n <= 224), the staged
and the cooperative chase above -- and on matrices that need exceptional
shifts or deflate at once.

Tolerance: Q T Q^H = A_s to 50 n u ||A|| (the bound of the Schur step's own
test) moves the square root by at most that times 1 / (2 min Re sqrt(lambda))
<= 1/2 and ||A|| / ||X|| < 2 on these matrices, and the triangular square root
and the products add 100 n u: 150 n u in all."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import U32

pytestmark = pytest.mark.gpu

mp = pytest.importorskip("paper_2607_12430_gb300")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    mp.lib()


def _x0(A):
    X, info = mp.sqrtm_mixed(torch.from_numpy(A).cuda(), kind=mp.KIND_GENERAL, steps=0)
    assert info["status"] == 0
    return X.cpu().numpy()


def _close(X, A):
    n = A.shape[0]
    return oracle.rel_err(X, oracle.sqrtm_schur(A)) <= 150 * n * U32


@pytest.mark.parametrize("n", [1, 2, 3, 23, 24, 25, 26, 31, 50, 80, 81, 82, 83, 113, 130, 223, 224, 225, 226, 257, 330])
def test_initial_iterate(n):
    A = synth.shifted_gaussian(n, 3.0, seed=7100 + n)
    assert _close(_x0(A), A)


@pytest.mark.parametrize("helpers", [0, 1, 3, 24])
@pytest.mark.parametrize("n", [225, 300])
def test_staged_and_cooperative_chase(n, helpers):
    A = synth.shifted_gaussian(n, 3.0, seed=7200 + n)
    saved = mp.get_tuning()
    try:
        mp.set_tuning([{"n_max": 1 << 20, "blks": 32, "qr_helpers": helpers, "batched": 1, "spd_precision": 0}])
        X = _x0(A)
    finally:
        mp.set_tuning(saved)
    assert _close(X, A)


@pytest.mark.parametrize("n", [40, 97, 240])
def test_exceptional_shifts_and_early_deflation(n):
    cyc = np.asfortranarray(3.0 * np.eye(n) + np.roll(np.eye(n), 1, axis=0))  # equal moduli: shifts at the diagonal stall
    assert _close(_x0(cyc), cyc)
    tri = np.triu(synth.shifted_gaussian(n, 3.0, seed=7300 + n))  # deflates without a sweep
    assert _close(_x0(np.asfortranarray(tri)), tri)
    two = synth.shifted_gaussian(n, 3.0, seed=7400 + n)  # two decoupled blocks
    two[n // 2:, :n // 2] = 0.0
    assert _close(_x0(two), two)


def test_batch_of_every_size_class():
    ns = [1, 2, 17, 24, 25, 63, 64, 65, 96, 128, 129, 200, 224, 225, 256]
    As = [synth.shifted_gaussian(n, 3.0, seed=7500 + n) for n in ns]
    Xs, st = mp.sqrtm_mixed_batched([torch.from_numpy(A).cuda() for A in As], kind=mp.KIND_GENERAL, steps=0)
    assert st == [0] * len(ns)
    for X, A in zip(Xs, As):
        assert _close(X.cpu().numpy(), A), A.shape
