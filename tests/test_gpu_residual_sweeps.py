"""The sweeps of the residual form are those of Algorithm 1 coordinate by
coordinate: with the iterations capped, the last iterate is the oracle's.
Common factors and a chunk's worth of coordinates make a support coordinate's
move carry coordinates at zero of its own chunk past the threshold."""
from __future__ import annotations

import numpy as np
import pytest

import oracle

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2203_15031_gb300 as sp  # noqa: E402


@pytest.mark.parametrize("p,n,f", [(64, 60, 0.8), (128, 80, 1.0), (150, 60, 0.7), (300, 60, 0.7)])
@pytest.mark.parametrize("maxit", [2, 3, 4, 6])
@pytest.mark.parametrize("standardize", [True, False])
def test_capped_iterates(p, n, f, maxit, standardize):
    rng = np.random.default_rng(0)
    F = rng.standard_normal((n, 4))
    X = rng.standard_normal((n, p)) + f * F @ rng.standard_normal((4, p))
    lam = np.sqrt(2.0 * np.log(p) / n)
    T, sig, st = sp.fit_residual(torch.from_numpy(X).cuda(), lam, tol=1e-10, maxit=maxit,
                                 precision="fp64", standardize=standardize)
    ref = oracle.spmesl(oracle.gram(X), lam, tol=1e-10, maxit=maxit, standardize=standardize)
    assert st["status"] == sp.SPMESL_NOT_CONVERGED
    assert st["inner_sweeps"] == int(ref["sweeps"].sum())
    # the two forms' rounding (1e-14 in a CPU restatement); an entry late by a sweep shows as 1e-3
    assert np.max(np.abs(T.cpu().numpy() - ref["Theta"])) <= 1e-10 * np.max(np.abs(ref["Theta"]))
    np.testing.assert_allclose(sig.cpu().numpy(), ref["sigma"], rtol=1e-10)
