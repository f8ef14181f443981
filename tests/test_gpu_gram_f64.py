"""The FP64 Gram from digit products on the tensor cores (spmesl_gram with
SPMESL_FP64) at the edges of its tiles, K blocks and accumulation lengths,
against an extended-precision sum, and on the columns that it does not scale."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2203_15031_gb300 as sp  # noqa: E402

# relative to sqrt(S_jj S_kk): the roundings of W, of 1/n and of the scaling (2^-53 each) and
# what the digits leave out (below 2^-53)
BAR = 4.0 * 2.0 ** -53


def _exact(X):
    Z = X.astype(np.longdouble)
    return (Z.T @ Z) / np.longdouble(X.shape[0])


def _gram(X, ldx=None, lds=None):
    n, p = X.shape
    ldx, lds = ldx or p, lds or p
    Xd = torch.full((n, ldx), float("nan"), dtype=torch.float64, device="cuda")
    Xd[:, :p] = torch.from_numpy(X).cuda()
    S = torch.full((p, lds), 7.0, dtype=torch.float64, device="cuda")
    nb = sp.spmesl_gram_workspace_bytes(n, p, sp.FP64)
    keep, ws = sp._workspace(nb, Xd.device)
    assert sp.spmesl_gram(Xd, n, p, ldx, sp.FP64, 0, S, lds, ws, nb) == sp.SPMESL_OK
    torch.cuda.synchronize()
    del keep
    S = S.cpu().numpy()
    assert (S[:, p:] == 7.0).all()
    return S[:, :p]


@pytest.mark.parametrize("p", [1, 2, 63, 64, 65, 127, 128, 129, 200])
@pytest.mark.parametrize("n", [1, 31, 64, 65, 255, 256, 257, 520])
def test_edges(n, p):
    rng = np.random.default_rng(1000 * n + p)
    X = rng.standard_normal((n, p)) * np.exp(rng.uniform(-30, 30, p))[None, :]
    if p > 2:
        X[:, 2] = 1000.0 + X[:, 2] / np.abs(X[:, 2]).max()      # one sign, nearly constant
    R = _exact(X)
    d = np.sqrt(np.diag(R))
    for ldx, lds in ((p, p), (p + 3, p + 5)):
        S = _gram(X, ldx, lds)
        assert np.array_equal(S, S.T)
        assert float(np.max(np.abs(S - R) / np.outer(d, d))) <= BAR


def test_columns_that_are_not_scaled():
    rng = np.random.default_rng(5)
    X = rng.standard_normal((100, 140))
    X[:, 3] *= 1e200
    X[:, 5] *= 1e-310
    X[:, 7] = 0.0
    X[4, 9] = np.inf
    X[6, 130] = np.nan
    S = _gram(X)
    with np.errstate(all="ignore"):
        R = X.T @ X / 100
    assert np.array_equal(np.isfinite(S), np.isfinite(R))
    assert np.array_equal(np.isnan(S), np.isnan(R))
    ok = np.isfinite(R)
    ok[[3, 5], :] = ok[:, [3, 5]] = False
    d = np.sqrt(np.diag(np.where(np.isfinite(R), R, 0.0)))
    assert np.max(np.abs(S[ok] - R[ok]) - 1e-14 * np.outer(d, d)[ok]) <= 0.0
    # FP64 sums in sample order: within n roundings of the products' absolute sum
    for j in (3, 5):
        fin = np.isfinite(R[j])
        A = np.abs(X[:, [j]]).T @ np.abs(X[:, fin]) / 100
        assert (np.abs(S[j][fin] - R[j][fin]) <= 200 * 2.0 ** -53 * A[0] + 1e-322).all()


@pytest.mark.parametrize("center", [False, True])
def test_batch_equals_single(center):
    rng = np.random.default_rng(9)
    Xs = [torch.from_numpy(rng.standard_normal((n, p)) + 0.3).cuda()
          for n, p in ((40, 30), (257, 129), (64, 64), (300, 65))]
    lams = [0.6] * len(Xs)
    bt = sp.Batch(list(zip(Xs, lams)), precision="fp64", tol=1e-8, center=center)
    bt.run()
    bt.result()
    for i, X in enumerate(Xs):
        T, s, _ = sp.fit(sp.gram(X, precision="fp64", center=center), 0.6, tol=1e-8,
                         precision="fp64")
        assert torch.equal(bt.Theta[i], T) and torch.equal(bt.sigma[i], s)
