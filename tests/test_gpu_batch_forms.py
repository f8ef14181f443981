"""The lazy solver's two residencies in batches (by the number of columns and whether the
fits are of like sizes) give the single fits' bits on either side of the lines."""
from __future__ import annotations

import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2203_15031_gb300 as sp  # noqa: E402


# on 152 SMs like fits change at 34048 columns, unlike ones (the largest with 1.5 times the
# mean column's chunks) at 109440; the SM count of another part only moves the lines
@pytest.mark.parametrize("sizes", [
    [500] * 60, [500] * 72, [100] * 360, [1100, 120] + [250] * 300, [1100, 120] + [250] * 450,
])
def test_equal_to_single_fits(sizes):
    g = torch.Generator(device="cuda").manual_seed(len(sizes))
    S = []
    for p in sizes:
        X = torch.randn((80, p), generator=g, device="cuda")
        X[:, 1:] += 0.5 * X[:, :-1].clone()
        S.append(X.T @ X / 80)
    bt = sp.Batch([(s, 0.45) for s in S], kind="S", precision="fp32", tol=1e-6)
    bt.run()
    bt.result()
    for i in {0, 1, 2, len(sizes) // 2, len(sizes) - 1}:
        T, sig, _ = sp.fit(S[i], 0.45, tol=1e-6, precision="fp32")
        assert torch.equal(bt.Theta[i], T) and torch.equal(bt.sigma[i], sig)
    bt.close()
