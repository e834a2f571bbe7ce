"""The residual of small and middling matrices from exact digit products formed
in the product's own kernel: sizes at the edges of its 128 x 64 tiles, of the
64 entries of k a step takes and of the 128 between two drains, and of its
range (33 .. 1024); the FP64 products it falls back to where the digits would
lose accuracy (graded rows and columns) and for entries that are not finite.

Tolerance: that of the larger sizes' test, n u (|X| |X|)_ij on either side of
the comparison plus the FP32 rounding of the result."""
import numpy as np
import pytest
import torch

import oracle
import synth
from gpu_util import U64, dev_cm, host_cm

pytestmark = pytest.mark.gpu

mp = pytest.importorskip("paper_2607_12430_gb300")


@pytest.fixture(scope="module", autouse=True)
def _lib():
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    mp.lib()


@pytest.mark.parametrize("n", [1, 2, 17, 32, 33, 47, 63, 64, 65, 80, 97, 127, 128, 129, 191, 192, 193, 255, 256, 257, 385,
                               1023, 1024, 1025])
def test_residual(n):
    g = np.random.default_rng(9100 + n)
    X = g.standard_normal((n, n)) / np.sqrt(n) + 2.0 * np.eye(n)
    X[:, n // 2] *= 2.0 ** -40  # one small column, one zero row
    X[n // 3, :] = 0.0
    A = X @ X + g.standard_normal((n, n)) * 1e-13
    ref = oracle.residual(A, X)[0] / 16.0
    bound = 2 * n * U64 * (np.abs(X) @ np.abs(X)) / 16.0 + 2.0 ** -24 * np.abs(ref)
    R, nrm = mp.step_residual_split(dev_cm(A, torch.float64), dev_cm(X, torch.float64), n, e=2)
    R = host_cm(R, n).astype(np.float64)
    assert np.all(np.abs(R - ref) <= 2 * bound)
    assert nrm == pytest.approx(np.linalg.norm(R), rel=1e-6)


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
@pytest.mark.parametrize("n", [40, 150])
def test_entries_that_are_not_finite(n, bad):
    X = np.eye(n) + 0.01 * np.cos(np.arange(n * n)).reshape(n, n)
    X[n - 2, 3] = bad
    R, nrm = mp.step_residual_split(dev_cm(X, torch.float64), dev_cm(X, torch.float64), n, e=0)
    R = host_cm(R, n)
    assert not np.isfinite(nrm)
    assert not np.isfinite(R[n - 2, :]).any() and not np.isfinite(R[:, 3]).any()
    ok = np.ones((n, n), bool)
    ok[n - 2, :] = ok[:, 3] = False
    assert np.isfinite(R[ok]).all()


def _graded(n):
    g = np.random.default_rng(n)
    d = 10.0 ** g.uniform(-3, 3, n)
    return d[:, None] * synth.shifted_gaussian(n, 3.0, seed=n) / d[None, :]


def _residuals(X):
    n = X.shape[0]
    g = np.random.default_rng(n + 1)
    A = X @ X * (1 + 1e-13 * g.standard_normal((n, n)))
    Ad, Xd = dev_cm(A, torch.float64), dev_cm(X, torch.float64)
    Rs, Rf = mp.step_residual_split(Ad, Xd, n, e=1)[0], mp.step_residual(Ad, Xd, n, e=1)[0]
    return host_cm(Rs, n).astype(np.float64), host_cm(Rf, n).astype(np.float64)


@pytest.mark.parametrize("n", [33, 64])
def test_one_graded_tile_takes_fp64_products(n):
    Rs, Rf = _residuals(_graded(n))
    assert np.array_equal(Rs, Rf)  # the same products in the same order


@pytest.mark.parametrize("n", [70, 130, 200, 400])
def test_graded_matrices_keep_fp64_accuracy(n):
    # some tiles with FP64 products, some with digits: together within the
    # FP64 product's bound in norm
    X = _graded(n)
    Rs, Rf = _residuals(X)
    assert np.linalg.norm(Rs - Rf) <= 2 * n * U64 * np.linalg.norm(np.abs(X) @ np.abs(X)) / 4 + 2.0 ** -23 * np.linalg.norm(Rf)


def test_batch():
    As = [torch.from_numpy(synth.shifted_gaussian(n, 3.0, seed=n)).cuda() for n in (200, 129, 64, 33, 32, 20)]
    X1, s1 = mp.sqrtm_mixed_batched(As, kind=mp.KIND_GENERAL, steps=3)
    X2, s2 = mp.sqrtm_mixed_batched(As, kind=mp.KIND_GENERAL, steps=3, precision=mp.PREC_RESID_FP64)
    assert s1 == [0] * 6 and s2 == [0] * 6
    assert torch.equal(X1[4], X2[4]) and torch.equal(X1[5], X2[5])  # n <= 32: FP64 products
    for x, y in zip(X1, X2):
        assert oracle.rel_err(x.cpu().numpy(), y.cpu().numpy()) <= 1e-13


@pytest.mark.parametrize("n", [33, 64, 65, 129, 200])
def test_complex_and_cube_root(n):
    # two corrections from digit products and from FP64 products: both within
    # rounding of the root
    A = synth.shifted_gaussian(n, 3.0, seed=n)
    for f, M in ((mp.sqrtm_mixed_complex, A + 1j * synth.shifted_gaussian(n, 0.0, seed=n + 1)), (mp.cbrtm_mixed, A)):
        Md = torch.from_numpy(M).cuda()
        X1, i1 = f(Md, steps=3)
        X2, i2 = f(Md, steps=3, precision=mp.PREC_RESID_FP64)
        assert i1["status"] == 0 and i2["status"] == 0
        X1, X2 = X1.cpu().numpy(), X2.cpu().numpy()
        assert np.linalg.norm(X1 - X2) <= 1e-13 * np.linalg.norm(X2)


@pytest.mark.parametrize("n", [33, 48, 64, 65, 128, 129, 200, 257, 385, 512, 641, 1000])
def test_every_tile_with_fp64_products(n):
    # X X far above A: no tile takes the digits, and the columns of a tile are
    # shared by 4 or 2 CTAs or one's own: the same products in the same order
    g = np.random.default_rng(n)
    X, A = g.standard_normal((n, n)), 1e-8 * g.standard_normal((n, n))
    Ad, Xd = dev_cm(A, torch.float64), dev_cm(X, torch.float64)
    (Rs, rs), (Rf, rf) = mp.step_residual_split(Ad, Xd, n, e=1), mp.step_residual(Ad, Xd, n, e=1)
    assert np.array_equal(host_cm(Rs, n), host_cm(Rf, n))
    assert rs == pytest.approx(rf, rel=n * n * U64)


def test_batch_with_fp64_tiles():
    # few members, so that a tile has several CTAs; moderately graded
    As = []
    for n in (200, 129, 70, 33, 30):
        d = 10.0 ** np.random.default_rng(n).uniform(-1, 1, n)
        As.append(torch.from_numpy(d[:, None] * synth.shifted_gaussian(n, 3.0, seed=n) / d[None, :]).cuda())
    for sel in (As, As[2:], As[4:]):
        X1, s1 = mp.sqrtm_mixed_batched(sel, kind=mp.KIND_GENERAL, steps=3)
        X2, s2 = mp.sqrtm_mixed_batched(sel, kind=mp.KIND_GENERAL, steps=3, precision=mp.PREC_RESID_FP64)
        assert s1 == [0] * len(sel) and s2 == s1
        for x, y in zip(X1, X2):
            assert oracle.rel_err(x.cpu().numpy(), y.cpu().numpy()) <= 1e-12
