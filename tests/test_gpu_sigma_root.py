"""The returned sigma is the square root of Eq. (14)'s quadratic form to the last bits,
in single fits and in batches, by the lazy and the block solver."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2203_15031_gb300 as sp  # noqa: E402


def _q(S, B):
    """sigma_j^2 in long double from the returned coefficients (S with unit diagonal)."""
    S, B = S.astype(np.longdouble), B.astype(np.longdouble)
    return np.diag(S) - 2 * np.einsum("kj,kj->j", S, B) + np.einsum("kj,kl,lj->j", B, S, B)


# lam 0.05 gives most columns more than 32 coefficients (the block solver)
@pytest.mark.parametrize("lam", [0.5, 0.05])
@pytest.mark.parametrize("prec", ["fp32", "fp64"])
@pytest.mark.parametrize("maxit", [1000, 2])
def test_sigma_is_the_root(lam, prec, maxit):
    rng = np.random.default_rng(1)
    X = rng.standard_normal((200, 90))
    X[:, 1:] += 0.6 * X[:, :-1]
    S = X.T @ X / 200
    d = 1.0 / np.sqrt(np.diag(S))
    S = S * d[:, None] * d[None, :]
    S = (S + S.T) / 2
    np.fill_diagonal(S, 1.0)
    S = S.astype(np.float32).astype(np.float64)
    Sd = torch.from_numpy(S).to(torch.float32 if prec == "fp32" else torch.float64).cuda()
    T, sig, st, B = sp.fit(Sd, lam, tol=1e-5, maxit=maxit, precision=prec, return_B=True)
    B = B.cpu().numpy().T                                     # B[k, j]: coefficient of x_k in regression j
    if not (np.abs(_q(S, B) - sig.cpu().numpy().astype(np.longdouble) ** 2) < 1e-3).all():
        B = B.T
    q = _q(S, B)
    # 90^2 products: their sum's rounding relative to q, halved by the root, and one unit of the root
    bar = (90 * 2.0 ** -53 * 8 / q + 2.0 ** -52)
    err = np.abs(sig.cpu().numpy() / np.sqrt(q) - 1)
    assert (err <= bar).all()
    # a step of the root left out would show as 2^-48: the median over the columns is well below
    assert float(np.median(err)) <= 2.0 ** -51
    if maxit == 1000:
        bt = sp.Batch([(Sd, lam)], kind="S", tol=1e-5, maxit=maxit, precision=prec)
        bt.run()
        bt.result()
        assert torch.equal(bt.sigma[0], sig) and torch.equal(bt.Theta[0], T)
