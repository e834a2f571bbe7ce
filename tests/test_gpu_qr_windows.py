"""The complex QR iteration with one CTA per matrix (complex input and the
FP64 method below n = 256, and the Schur step) at the sizes where one window
covers its whole active block, which leaves no update outside it between one
window's rotation log and the next one's: the factors of complex matrices
reproduce A_s to 50 n u ||A|| (the bound of the Schur step's own test) and are
the same, bit for bit, in every run -- each thread's work and every summation
order are fixed, so two runs can differ only where threads race."""
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


def _crandom(n, seed):
    g = np.random.default_rng(seed)
    return 3.0 * np.eye(n) + (g.standard_normal((n, n)) + 1j * g.standard_normal((n, n))) / np.sqrt(2 * n)


@pytest.mark.parametrize("fp64", [False, True])
@pytest.mark.parametrize("n", [25, 26, 30, 40, 50, 60, 81, 100, 150, 255])
def test_factors_hold_and_repeat(n, fp64):
    u, dt = (U64, torch.complex128) if fp64 else (U32, torch.complex64)
    for seed in range(6):
        A = _crandom(n, 8100 + 10 * n + seed)
        A = A if fp64 else A.astype(np.complex64).astype(np.complex128)
        first = None
        for _ in range(8):
            T = dev_cm(A, dt)
            Q = mp.step_schur(T, n, fp64=fp64)
            Th, Qh = host_cm(T, n), host_cm(Q, n)
            if first is None:
                first = Th, Qh
                T2, Q2 = Th.astype(np.complex128), Qh.astype(np.complex128)
                assert np.all(np.tril(T2, -1) == 0)
                assert np.linalg.norm(Q2.conj().T @ Q2 - np.eye(n)) <= 50 * n * u
                assert np.linalg.norm(Q2 @ T2 @ Q2.conj().T - A) <= 50 * n * u * np.linalg.norm(A)
            assert np.array_equal(Th, first[0]) and np.array_equal(Qh, first[1])


@pytest.mark.parametrize("n", [25, 40, 60, 100, 200])
def test_plain_fp64_method(n):
    for seed in range(8):
        A = synth.shifted_gaussian(n, 3.0, seed=8300 + 10 * n + seed)
        X, info = mp.sqrtm_schur_fp64(torch.from_numpy(A).cuda(), kind=mp.KIND_GENERAL)
        assert info["status"] == 0
        assert oracle.rel_err(X.cpu().numpy(), oracle.sqrtm_schur(A)) <= 1e-12


@pytest.mark.parametrize("n,shift", [(25, 3.0), (28, 3.0), (32, 48.707), (33, 3.0), (34, 17.727), (35, 6.425), (35, 14.2),
                                     (36, 3.0), (40, 3.0), (64, 20.0)])
def test_rotations_of_vanishing_entries(n, shift):
    # shift I + a cycle: where a shift meets an eigenvalue exactly, the first
    # entry of a rotation is subnormal and its phase needs scaling
    A = shift * np.eye(n) + np.roll(np.eye(n), 1, axis=0)
    X, info = mp.sqrtm_mixed_complex(torch.from_numpy(A.T.astype(np.complex128).copy()).cuda())
    assert info["status"] == 0
    assert oracle.rel_err(X.cpu().numpy().T, oracle.sqrtm_schur(A)) <= 1e-12
