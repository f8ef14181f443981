"""The FP32 Gram at the edges of its two tile shapes, with and without 16-byte
rows of X and S: every entry is one chain of FP32 fused multiply-adds in sample
order, so a host restatement of that chain gives the same bits."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2203_15031_gb300 as sp  # noqa: E402


def _chain(X, rows, cols):
    """fma chains of S[rows][:, cols] on the host.  The product of two FP32 values is exact
    in FP64; the FP64 sum is rounded to odd before FP32, so that the two roundings are one."""
    acc = np.zeros((len(rows), len(cols)), dtype=np.float32)
    for x in X:
        prod = x[rows].astype(np.float64)[:, None] * x[cols].astype(np.float64)[None, :]
        a = acc.astype(np.float64)
        s = a + prod
        b = s - a
        err = (a - (s - b)) + (prod - b)                       # exact error of the sum
        bits = s.view(np.int64)
        away = (err != 0) & ((bits & 1) == 0)
        step = np.where((err > 0) == (s > 0), 1, -1)
        s = np.where(away, (bits + step).view(np.float64), s)
        acc = s.astype(np.float32)
    return acc * np.float32(1.0 / X.shape[0])


@pytest.mark.parametrize("p,ldx,lds", [(1, 1, 1), (63, 63, 63), (64, 64, 64), (65, 68, 65),
                                       (200, 200, 200), (1921, 1921, 1921), (2688, 2688, 2688),
                                       (2689, 2689, 2689), (2692, 2696, 2693), (2820, 2820, 2820)])
@pytest.mark.parametrize("n", [1, 8, 17, 40])
def test_same_bits_as_the_chain(p, ldx, lds, n):
    rng = np.random.default_rng(p + n)
    X = rng.standard_normal((n, p)).astype(np.float32)
    Xd = torch.full((n, ldx), float("nan"), device="cuda")
    Xd[:, :p] = torch.from_numpy(X).cuda()
    S = torch.full((p, lds), 7.0, device="cuda")
    nb = sp.spmesl_gram_workspace_bytes(n, p, sp.FP32)
    keep, ws = sp._workspace(nb, S.device)
    assert sp.spmesl_gram(Xd, n, p, ldx, sp.FP32, 0, S, lds, ws, nb) == sp.SPMESL_OK
    torch.cuda.synchronize()
    del keep
    S = S.cpu().numpy()
    assert (S[:, p:] == 7.0).all()
    S = S[:, :p]
    assert np.array_equal(S, S.T)
    edge = [0, 31, 32, 63, 64, 65, 127, 128, 129, 1023, 1024, 2687, 2688, p - 2, p - 1]
    at = np.array(sorted({e for e in edge if 0 <= e < p}))
    assert np.array_equal(S[np.ix_(at, at)], _chain(X, at, at))
    cols = np.arange(0, p, max(1, p // 40))
    assert np.array_equal(S[np.ix_(at, cols)], _chain(X, at, cols))
