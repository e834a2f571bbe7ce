"""Real matrices whose eigenvalues lie close together against their distance
from zero: the QR iteration does not see a translation, so s I + B takes about
as many sweeps as B, and its factors are as accurate.

Work of the chase (reflectors times the size of the active block): an
eigenvalue pair takes about four double-shift sweeps in ordinary practice, over
n / 2 pairs and an active block that shrinks linearly 4 (n / 2) n^2 / 3 = 2 n^3 /
3; three times that is allowed.  With shifts that do not resolve the spectrum
whole sweeps go by without a deflation, which takes several times more or ends at
the iteration cap.  Factors: the
bounds of the Schur step's test of ordinary spectra."""
import numpy as np
import pytest
import torch

import oracle
from gpu_util import U32
from test_gpu_real_factor import factor_errors, schur32

pytestmark = pytest.mark.gpu

mp = pytest.importorskip("paper_2607_12430_gb300")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    mp.lib()


def _matrix(kind, n):
    g = np.random.default_rng(8700 + n)
    G = g.standard_normal((n, n))
    name, p = kind
    if name == "gauss":
        A = p * np.eye(n) + G / np.sqrt(n)
    elif name == "sym":
        A = np.eye(n) + p * (G + G.T) / 2
    else:
        P = g.random((n, n))
        A = p * np.eye(n) + P / P.sum(axis=1, keepdims=True)
    return A.astype(np.float32).astype(np.float64)


KINDS = [("gauss", 3.0), ("gauss", 30.0), ("gauss", 300.0), ("gauss", 3000.0), ("sym", 1e-3), ("sym", 1e-5),
         ("sym", 1e-7), ("stochastic", 10.0)]


@pytest.mark.parametrize("kind", KINDS, ids=str)
@pytest.mark.parametrize("n", [23, 25, 63, 65, 127, 129, 223, 225, 330, 520])
def test_factor_and_sweeps(kind, n):
    A = _matrix(kind, n)
    back, orth = factor_errors(A, *schur32(A))
    assert back <= 14 * np.sqrt(n) * U32 and orth <= 8 * n * U32
    X, info = mp.sqrtm_mixed(torch.from_numpy(A).cuda(), kind=mp.KIND_GENERAL)
    assert info["status"] == 0
    assert oracle.rel_err(X.cpu().numpy() @ X.cpu().numpy(), A) <= 1e-12
    assert info["schur_work"] <= 2 * n ** 3


@pytest.mark.parametrize("n", [25, 50, 130, 224, 300])
def test_graded_matrix(n):
    """Entries that grow by 10 orders of magnitude from the lower left to the
    upper right corner: the largest entry says nothing about the spectrum."""
    i = np.arange(n)
    A = _matrix(("gauss", 3.0), n) * 10.0 ** (10.0 * (i[None, :] - i[:, None]) / n)
    back, orth = factor_errors(A.astype(np.float32).astype(np.float64), *schur32(A))
    assert back <= 14 * np.sqrt(n) * U32 and orth <= 8 * n * U32


def test_batch_of_narrow_spectra():
    As = [_matrix(k, n) for n in (25, 64, 101, 128, 200, 225, 256) for k in KINDS]
    Xs, st = mp.sqrtm_mixed_batched([torch.from_numpy(A).cuda() for A in As], kind=mp.KIND_GENERAL)
    assert st == [0] * len(As)
    for X, A in zip(Xs, As):
        X = X.cpu().numpy()
        assert oracle.rel_err(X @ X, A) <= 1e-12


@pytest.mark.parametrize("p", [1e-10, 1e-18, 1e-22, 1e-26])
@pytest.mark.parametrize("n", [30, 50, 130, 224, 300])
def test_block_far_below_the_scale(n, p):
    """Two decoupled blocks, one of them p times the other in either order: the
    reflectors that start its sweeps and the shifts of its last rows are made
    of products of its entries, p^2.  The small block is upper Hessenberg
    already, so that the reduction does not square it.  Each block's factor
    holds to the bounds of a matrix of its own."""
    k = n // 2
    for first in (False, True):
        g = np.random.default_rng(8900 + n)
        A = np.zeros((n, n))
        big = slice(k, n) if first else slice(0, k)
        small = slice(0, k) if first else slice(k, n)
        m = A[small, small].shape[0]
        A[big, big] = 3.0 * np.eye(n - m) + g.standard_normal((n - m, n - m)) / np.sqrt(n - m)
        A[small, small] = p * np.triu(3.0 * np.eye(m) + g.standard_normal((m, m)) / np.sqrt(m), -1)
        A = A.astype(np.float32).astype(np.float64)
        T, Q = schur32(A)
        for b in (big, small):
            back, orth = factor_errors(A[b, b], T[b, b], Q[b, b])
            assert back <= 14 * np.sqrt(n) * U32 and orth <= 8 * n * U32
