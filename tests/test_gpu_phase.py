"""The active-set phase at the edges of its slots (one coordinate per lane up to
32, two up to 64, the sweep beyond), in both working precisions, against the
FP64 oracle: a star-shaped covariance whose first column has a support of
exactly m coordinates."""
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

# the parity bars of the other fits: FP32 1e-4, FP64 1e-7 of max |Theta|
BAR = {"fp32": 1e-4, "fp64": 1e-7}


@pytest.mark.parametrize("m", [1, 2, 3, 31, 32, 33, 63, 64, 65])
@pytest.mark.parametrize("prec,tol", [("fp32", 1e-6), ("fp64", 1e-10)])
@pytest.mark.parametrize("standardize", [True, False])
def test_support_of_exactly_m(m, prec, tol, standardize):
    p = 140
    rng = np.random.default_rng(m)
    S = np.eye(p)
    w = (0.06 + 0.04 * rng.random(m)) * rng.choice([-1.0, 1.0], m)
    at = 1 + rng.permutation(p - 1)[:m]
    S[0, at] = S[at, 0] = w
    # neighbours weakly correlated in pairs, so that moves interact
    for a, b in zip(at[::2], at[1::2]):
        S[a, b] = S[b, a] = 0.02
    S = S.astype(np.float32 if prec == "fp32" else np.float64)
    lam = 0.03
    Th, sg, st, B = sp.fit(torch.from_numpy(S).cuda(), lam, tol=tol, precision=prec, return_B=True,
                           standardize=standardize)
    assert st["status"] == sp.SPMESL_OK
    assert int((B[:, 0] != 0).sum()) == m
    ref = oracle.spmesl(S.astype(np.float64), lam, tol=1e-12, maxit=1000, standardize=standardize)
    res = compare_theta(Th.cpu().numpy(), ref["Theta"], ref["B"], ref["sigma"], rel=BAR[prec])
    assert res["ok"], res
