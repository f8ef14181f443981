"""The block solver's refreshes that leave chunks of the gradient out, over sizes
around the chunk (128 coordinates), every column cold (routed by heat) or warm
(handed over), against the FP64 oracle."""
from __future__ import annotations

import numpy as np
import pytest

import oracle
import synth
from checks import compare_theta

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2203_15031_gb300 as sp  # noqa: E402

# the parity bars of the other fits
BAR = {"fp32": 1e-4, "fp64": 1e-7}


@pytest.mark.parametrize("p", [127, 129, 257, 1100])
@pytest.mark.parametrize("kind", ["hub_scaled", "er"])
@pytest.mark.parametrize("prec,tol", [("fp32", 1e-6), ("fp64", 1e-10)])
@pytest.mark.parametrize("route", [dict(heavy_min_p=1, heavy_heat=1), dict(handover=1)])
def test_refreshes_by_chunk(p, kind, prec, tol, route):
    prob = synth.make_problem(kind, p, 150, p, dtype=np.float64)
    S = oracle.gram(prob.X)
    T, s, st = sp.fit(torch.from_numpy(S.astype(np.float32 if prec == "fp32" else np.float64)).cuda(),
                      prob.lambda0, tol=tol, precision=prec, **route)
    assert st["status"] == sp.SPMESL_OK and st["block_columns"] >= 10
    ref = oracle.spmesl(S, prob.lambda0, tol=1e-11, maxit=1000)
    res = compare_theta(T.cpu().numpy(), ref["Theta"], ref["B"], ref["sigma"], rel=BAR[prec])
    assert res["ok"], res


def test_an_indefinite_matrix_is_refused():
    """Coefficients that grow beyond FP32 end at the sigma floor, not as NaN in Theta."""
    X = np.random.default_rng(0).standard_normal((60, 40))
    A = X.T @ X / 60
    A[0, 1] = A[1, 0] = 5.0
    A[2, 3] = A[3, 2] = -4.0
    with pytest.raises(sp.SpmeslError):
        sp.fit(torch.from_numpy(A.astype(np.float32)).cuda(), 0.1, maxit=30)
