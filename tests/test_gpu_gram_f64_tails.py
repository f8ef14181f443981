"""The FP64 Gram on columns with tails: no further from the exact entries than
FP64 sums in sample order are."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2203_15031_gb300 as sp  # noqa: E402

P = 70


def _columns(kind, n):
    rng = np.random.default_rng(n + len(kind))
    z = rng.standard_normal((n, P))
    if kind == "t2":
        return rng.standard_t(2, (n, P))
    if kind == "t5":
        return rng.standard_t(5, (n, P))
    if kind == "cauchy":
        return rng.standard_cauchy((n, P))
    if kind == "laplace":
        return rng.laplace(size=(n, P)) * np.exp(rng.uniform(-3, 3, P))
    if kind.startswith("lognormal"):
        return np.exp(float(kind[9:]) * z)
    if kind.startswith("outlier"):                     # in one column
        z[n // 2, 0] *= float(kind[7:])
        return z
    if kind == "regimes":                              # two scales that do not meet
        z[: n // 2, ::2] *= 1e-9
        z[n // 2:, 1::2] *= 1e-9
        return z
    return z


def _exact_and_sums(X):
    """The entries in long double, and as one chain of FP64 fused multiply-adds."""
    W = X.astype(np.longdouble)
    acc = np.zeros((P, P))
    R = np.zeros((P, P), dtype=np.longdouble)
    for i in range(X.shape[0]):
        prod = np.outer(W[i], W[i])
        R += prod
        acc = (acc.astype(np.longdouble) + prod).astype(np.float64)
    n = X.shape[0]
    return R / np.longdouble(n), acc * (1.0 / n)


# a CPU restatement of both gives 0.6 and less for the ratio from n = 30 on; a column whose
# entries are FP64 sums gives 1 exactly
@pytest.mark.parametrize("kind", ["normal", "t5", "t2", "cauchy", "laplace", "lognormal1", "lognormal3",
                                  "outlier30", "outlier1e3", "outlier1e6", "regimes"])
@pytest.mark.parametrize("n", [30, 250, 1000])
def test_no_further_than_sums(kind, n):
    X = _columns(kind, n)
    R, F = _exact_and_sums(X)
    S = sp.gram(torch.from_numpy(X).cuda(), precision="fp64").cpu().numpy()
    assert np.array_equal(S, S.T)
    d = np.sqrt(np.diag(R))
    off = ~np.eye(P, dtype=bool)
    e = ((S - R) / np.outer(d, d)).astype(np.float64)
    f = ((F - R) / np.outer(d, d)).astype(np.float64)
    rms = lambda v: float(np.sqrt(np.mean(v * v)))  # noqa: E731
    assert rms(e[off]) <= rms(f[off])
    # column 0 (the outlier's), against its own entries
    e0, f0 = ((A[0, 1:] - R[0, 1:]).astype(np.float64) for A in (S, F))
    assert rms(e0) <= rms(f0)
