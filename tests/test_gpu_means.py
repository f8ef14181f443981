"""Column means in sample groups, through the centred Gram of every precision
and single against batched fits, at sample counts around the eight groups."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2203_15031_gb300 as sp  # noqa: E402

# relative to sqrt(S_jj S_kk) of the centred data: the Gram bars of the precisions (FP32
# 2e-6 sqrt(n), split BF16 2e-5, FP64 1e-13), and for FP32 data the mean rounded to
# FP32: 2^-24 |mean| per sample, here 2^-24 * 3 / sd on each side
MEAN = 3.0


@pytest.mark.parametrize("p", [1, 31, 32, 33, 65])
@pytest.mark.parametrize("n", [2, 7, 8, 9, 15, 16, 17, 100])
def test_centred_gram(n, p):
    rng = np.random.default_rng(n * 100 + p)
    X = rng.standard_normal((n, p)) + MEAN
    for prec, bar in (("fp64", 1e-13), ("fp32", 2e-6 * n ** 0.5), ("mixed", 2e-5)):
        Xp = X if prec == "fp64" else X.astype(np.float32)
        Z = Xp.astype(np.float64)
        Z = Z - Z.mean(0)
        R = Z.T @ Z / n
        d = np.sqrt(np.diag(R))
        S = sp.gram(torch.from_numpy(Xp).cuda(), precision=prec, center=True).cpu().numpy()
        slack = 0.0 if prec == "fp64" else 2 * 2.0 ** -23 * MEAN / d.min()
        assert np.max(np.abs(S - R) / np.outer(d, d)) <= bar + slack


@pytest.mark.parametrize("prec", ["fp32", "mixed", "fp64"])
def test_batch_equals_single_centred(prec):
    rng = np.random.default_rng(1)
    Xs = [torch.from_numpy((rng.standard_normal((n, p)) + MEAN)
                           .astype(np.float64 if prec == "fp64" else np.float32)).cuda()
          for n, p in ((41, 30), (100, 129), (64, 33))]
    bt = sp.Batch([(x, 0.6) for x in Xs], precision=prec, center=True)
    bt.run()
    bt.result()
    for i, x in enumerate(Xs):
        T, s, _ = sp.fit(sp.gram(x, precision=prec, center=True), 0.6, precision=prec)
        assert torch.equal(bt.Theta[i], T) and torch.equal(bt.sigma[i], s)
