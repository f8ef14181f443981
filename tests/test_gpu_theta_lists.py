"""Theta and B from coefficient lists: supports on both sides of what a row of
B^T holds as a list (half its padded length), odd sizes, and a Theta that starts
on an 8-byte boundary, against the FP64 oracle and the eager form's dense rows."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
from checks import compare_theta

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2203_15031_gb300 as sp  # noqa: E402


@pytest.mark.parametrize("p", [2, 17, 33, 40, 65, 130, 257])
@pytest.mark.parametrize("lam", [0.4, 0.02])
def test_lists_and_dense_rows(p, lam):
    # S of an AR(1)-like process with a common factor: a small penalty keeps most coefficients
    rng = np.random.default_rng(p)
    X = rng.standard_normal((4 * p, p)) + 0.5 * rng.standard_normal((4 * p, 1))
    S = X.T @ X / (4 * p)
    Sd = torch.from_numpy(S).cuda()
    T, s, st, B = sp.fit(Sd, lam, tol=1e-10, precision="fp64", return_B=True)
    Te, se, _, Be = sp.fit(Sd, lam, tol=1e-10, precision="fp64", return_B=True,
                           gradient=sp.GRADIENT_EAGER)
    assert st["nnz_B"] == int((B != 0).sum())
    if lam < 0.1 and p > 33:
        ldp = (p + 31) // 32 * 32
        assert int((B != 0).sum(0).max()) > ldp // 2            # some rows are dense
    ref = oracle.spmesl(S, lam, tol=1e-12, maxit=1000)
    # the FP64 path's parity bar
    assert compare_theta(T.cpu().numpy(), ref["Theta"], ref["B"], ref["sigma"], rel=1e-6)["ok"]
    assert float((T - Te).abs().max()) <= 1e-6 * float(Te.abs().max())
    assert float((B - Be).abs().max()) <= 1e-6 * max(1.0, float(Be.abs().max()))


@pytest.mark.parametrize("p", [31, 32, 129])
def test_theta_on_an_8_byte_boundary(p):
    rng = np.random.default_rng(p)
    X = torch.from_numpy(rng.standard_normal((60, p)).astype(np.float32)).cuda()
    S = sp.gram(X)
    want, sw, _ = sp.fit(S, 0.5)
    buf = torch.full((p * p + 3,), float("nan"), dtype=torch.float64, device="cuda")
    sg = torch.empty(p, dtype=torch.float64, device="cuda")
    nb = sp.spmesl_fit_workspace_bytes(p, sp.FP32)
    keep, ws = sp._workspace(nb, S.device)
    assert sp.spmesl_fit(S, 60, p, 0.5, 1e-6, 1000, None, buf[1:], sg, sp.Stats(), ws, nb) == 0
    assert torch.equal(buf[1:1 + p * p].view(p, p), want) and torch.equal(sg, sw)
    assert torch.isnan(buf[0]) and torch.isnan(buf[1 + p * p:]).all()
    del keep
