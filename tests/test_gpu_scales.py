"""Unstandardised FP32 fits at scales where entries of S are denormal or huge, and
coefficient rows longer than their lists (dense rows)."""
from __future__ import annotations

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2203_15031_gb300 as sp  # noqa: E402


def _S(p, n, seed):
    X = np.random.default_rng(seed).standard_normal((n, p))
    X[:, 1:] += 0.5 * X[:, :-1]
    return X.T @ X / n


# 2^-120: a variance is 7e-37 and small covariances are denormal; 2^-129: all of S is; 2^110: 1e33
@pytest.mark.parametrize("e", [-129, -120, 0, 110])
def test_unstandardised_scales(e):
    p, lam = 60, 0.4
    S = (_S(p, 80, 5) * 2.0 ** e).astype(np.float32)
    assert np.isfinite(S).all() and (e > -120 or np.abs(S)[S != 0].min() < 1.2e-38)
    l0 = lam * 2.0 ** (e / 2)                     # sigma lambda0 scales as S does
    Sd = torch.from_numpy(S).cuda()
    # sigma's tolerance is absolute, so a tiny sigma ends after its second step and a huge one
    # at its fixed point or the cap; the oracle stops by the same rules
    kw = dict(tol=1e-5, maxit=60, standardize=False)
    ref = oracle.spmesl(S.astype(np.float64), l0, **kw)
    kw["precision"] = "fp32"
    T, sig, _ = sp.fit(Sd, l0, **kw)
    T, sig = T.cpu().numpy(), sig.cpu().numpy()
    # coefficients to the tolerance and FP32 (2^-20 where S is denormal), a dozen of them a column
    np.testing.assert_allclose(sig, ref["sigma"], rtol=1e-3)
    assert np.max(np.abs(T - ref["Theta"])) <= 1e-2 * np.max(np.abs(ref["Theta"]))


def test_rows_beyond_the_lists():
    """More than 1024 coefficients in a row: the row stays dense for Theta, the export and the
    diagnostics."""
    p, n, lam = 2300, 9000, 2e-3
    g = torch.Generator(device="cuda").manual_seed(3)
    X = torch.randn((n, p), generator=g, device="cuda", dtype=torch.float64)
    S = X.T @ X / n
    d = S.diagonal().rsqrt()
    S = (S * d[:, None] * d[None, :]).float()
    S = (S + S.T) / 2
    S.fill_diagonal_(1.0)
    T, sig, st, B = sp.fit(S, lam, tol=1e-6, maxit=300, precision="fp32", return_B=True, diagnostics=True)
    nz = (B != 0).sum(1)
    assert int(nz.max()) > 1024 and st["nnz_B"] == int(nz.sum())
    W = S.double()
    viol = 0.0
    for M in (B, B.T):                             # either orientation of the export
        G = W - W @ M
        lk = lam * sig[None, :]
        v = torch.where(M != 0, (G - lk * torch.sign(M)).abs(), (G.abs() - lk).clamp(min=0))
        v.fill_diagonal_(0.0)
        viol = float(v.max()) if M is B else min(viol, float(v.max()))
    # tol times the row sums of |S| that a last sweep can leave, and FP32 gradients of ~2000 terms
    assert viol <= 1e-6 * 2300 * 0.02 + 2300 * 2.0 ** -24 * 0.02 + 1e-5
    assert st["kkt_viol"] * lam <= 2 * viol + 1e-6
    assert torch.equal(T, T.T)
    # Theta's entries are nonzero where both regressions of the pair have a coefficient
    off = ~torch.eye(p, dtype=torch.bool, device="cuda")
    assert torch.equal((T != 0) & off, (B != 0) & (B.T != 0) & off)
