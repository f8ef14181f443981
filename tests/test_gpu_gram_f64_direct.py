"""Columns that the FP64 Gram does not scale, over several tiles and accumulations:
their entries are the FP64 sums in sample order, the others are left as they are."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2203_15031_gb300 as sp  # noqa: E402


def _data(n, p, seed):
    return torch.from_numpy(np.random.default_rng(seed).standard_normal((n, p))).cuda()


# p = 1700 has more tiles than the part has SMs; the columns sit at the edges of tiles and warps
@pytest.mark.parametrize("n,p,cols", [
    (1, 1, [0]), (17, 65, [64]), (300, 140, [0, 31, 32, 63, 64, 127, 128, 139]),
    (520, 257, [5, 256]), (600, 1700, [3, 127, 128, 1000, 1699]), (300, 200, list(range(200))),
    (70, 130, list(range(0, 130, 2))), (65, 96, list(range(40, 90))), (64, 33, [32]), (129, 5000, [2500]),
])
@pytest.mark.parametrize("center", [False, True])
def test_unscaled_columns(n, p, cols, center):
    Y = _data(n, p, 10 * n + p) + (0.25 if center else 0.0)
    X = Y.clone()
    X[:, cols] *= 2.0 ** -480                     # beyond the exponents that are scaled; exact
    S = sp.gram(X, precision="fp64", center=center)
    assert torch.equal(S, S.T)
    R = sp.gram(Y, precision="fp64", center=center)
    f = torch.ones(p, dtype=torch.float64, device="cuda")
    f[cols] = 2.0 ** 480
    S = S * f[:, None] * f[None, :]
    rest = torch.ones(p, dtype=torch.bool, device="cuda")
    rest[cols] = False
    assert torch.equal(S[rest][:, rest], R[rest][:, rest])
    # a sum of n terms: n roundings of it, two of 1/n and the means' on either side
    d = torch.sqrt(R.diagonal()).clamp(min=2.0 ** -40)
    assert float((S - R).abs().div(d[:, None] * d[None, :]).max()) <= (n + 8) * 2.0 ** -53


def test_order_of_the_sums():
    """One chain of fused multiply-adds from the first sample to the last."""
    n, p = 70, 3
    X = torch.zeros((n, p), dtype=torch.float64)
    X[:, 0] = torch.from_numpy(np.random.default_rng(2).standard_normal(n)) * 2.0 ** -480
    X[0, 1], X[1, 1], X[2, 1] = 2.0 ** 60, 1.0, -2.0 ** 60
    X[:3, 0] = 2.0 ** -480
    S = sp.gram(X.cuda(), precision="fp64").cpu()
    # (2^60 + 1) rounds to 2^60, minus 2^60 is 0: the 1 is lost in this order only
    assert float(S[0, 1]) == 0.0 and float(S[1, 0]) == 0.0
    acc = 0.0
    for x in X[:, 0].tolist():
        acc = float(np.longdouble(acc) + np.longdouble(x) * np.longdouble(x))
    assert abs(float(S[0, 0]) - acc * (1.0 / n)) <= 2 * np.spacing(acc / n)


@pytest.mark.parametrize("center", [False, True])
def test_batch_equals_single(center):
    Xs = [_data(n, p, n + p) for n, p in ((40, 30), (520, 129), (300, 65))]
    for X in Xs:
        X[:, 7] *= 2.0 ** -450
    bt = sp.Batch([(X, 0.6) for X in Xs], precision="fp64", tol=1e-8, center=center)
    bt.run()
    bt.result()
    for i, X in enumerate(Xs):
        T, s, _ = sp.fit(sp.gram(X, precision="fp64", center=center), 0.6, tol=1e-8, precision="fp64")
        assert torch.equal(bt.Theta[i], T) and torch.equal(bt.sigma[i], s)
