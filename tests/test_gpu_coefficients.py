"""spmesl_fit_coefficients behind a fit whose status nobody has read: a refused
fit (non-finite S, or a variance that is not positive) leaves B as it is,
whatever the workspace held before."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2203_15031_gb300 as sp  # noqa: E402


def _fit_then_coefficients(S, prec, **kw):
    """The two calls queued one after the other, with no status read between."""
    p = S.shape[0]
    opts = sp.spmesl_default_opts()
    opts.precision = prec
    for k, v in kw.items():
        setattr(opts, k, v)
    nb = sp.spmesl_fit_workspace_bytes(p, prec)
    keep = torch.full((nb + 256,), 0x7f, dtype=torch.uint8, device=S.device)
    ws = keep.data_ptr() + (-keep.data_ptr()) % 256
    Theta = torch.full((p, p), 3.0, dtype=torch.float64, device=S.device)
    sigma = torch.full((p,), 4.0, dtype=torch.float64, device=S.device)
    B = torch.full((p, p), 7.25, dtype=torch.float64, device=S.device)
    assert sp.spmesl_fit(S, 0, p, 0.4, 1e-6, 100, opts, Theta, sigma, None, ws, nb) == sp.SPMESL_OK
    assert sp.spmesl_fit_coefficients(ws, p, prec, B) == sp.SPMESL_OK
    rc = sp.spmesl_fit_result(ws, p, prec, sp.Stats())
    del keep
    return rc, Theta, B


def _data(p, n, prec):
    X = np.random.default_rng(p).standard_normal((n, p))
    X[:, 1:] += 0.6 * X[:, :-1]
    S = X.T @ X / n
    return torch.from_numpy(S.astype(np.float64 if prec == sp.FP64 else np.float32)).cuda()


# below and above the size from which the columns are ordered by heat (more columns than
# resident warps), and with columns routed by heat
@pytest.mark.parametrize("p,kw", [
    (2, {}), (40, {}), (40, dict(gradient=sp.GRADIENT_EAGER)), (40, dict(inner_rule=sp.INNER_JOINT)),
    (130, dict(heavy_min_p=1, heavy_heat=2)), (2600, {}), (2600, dict(heavy_min_p=2000)),
])
@pytest.mark.parametrize("prec", [sp.FP32, sp.FP64])
@pytest.mark.parametrize("bad", ["nan", "variance"])
def test_refused_fit_leaves_b(p, kw, prec, bad):
    S = _data(p, 60, prec)
    if bad == "nan":
        S[p - 1, 0] = S[0, p - 1] = float("nan")
    else:
        S[p - 1, p - 1] = 0.0
    rc, Theta, B = _fit_then_coefficients(S, prec, **kw)
    assert rc == sp.SPMESL_ENONFINITE
    assert bool((B == 7.25).all()) and bool((Theta == 3.0).all())


@pytest.mark.parametrize("p", [40, 2600])
@pytest.mark.parametrize("prec", [sp.FP32, sp.FP64])
def test_solved_fit_exports(p, prec):
    S = _data(p, 60, prec)
    rc, Theta, B = _fit_then_coefficients(S, prec)
    assert rc == sp.SPMESL_OK
    T, s, st, B2 = sp.fit(S, 0.4, tol=1e-6, maxit=100, precision=prec, return_B=True)
    assert torch.equal(B, B2) and torch.equal(Theta, T) and bool((B.diagonal() == 0).all())
