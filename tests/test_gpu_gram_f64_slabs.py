"""The FP64 Gram of tall data, whose digits are formed a slab of 4096 samples at a time."""
from __future__ import annotations

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

import paper_2203_15031_gb300 as sp  # noqa: E402


def _data(n, p, seed, shift=0.0):
    return torch.from_numpy(np.random.default_rng(seed).standard_normal((n, p)) + shift).cuda()


def _gram(X, center=False):
    """spmesl_gram in a workspace of exactly the stated size, the rest of it watched."""
    n, p = X.shape
    nb = sp.spmesl_gram_workspace_bytes(n, p, sp.FP64)
    keep = torch.full((nb + 512,), 0x7f, dtype=torch.uint8, device="cuda")
    ws = keep.data_ptr() + (-keep.data_ptr()) % 256
    S = torch.full((p, p), 5.0, dtype=torch.float64, device="cuda")
    assert sp.spmesl_gram(X, n, p, p, sp.FP64, int(center), S, p, ws, nb) == sp.SPMESL_OK
    torch.cuda.synchronize()
    tail = keep[ws - keep.data_ptr() + nb:]
    assert bool((tail == 0x7f).all())
    return S


@pytest.mark.parametrize("n", [4095, 4096, 4097, 8192, 8255, 12289])
@pytest.mark.parametrize("p", [1, 65, 200])
@pytest.mark.parametrize("center", [False, True])
def test_slabs(n, p, center):
    X = _data(n, p, n + p, 0.25)
    X[:, 0] *= 2.0 ** 200
    S = _gram(X, center)
    assert torch.equal(S, S.T)
    Z = X - (X.mean(0) if center else 0.0)
    R = sum((Z[i:i + 64].T @ Z[i:i + 64] for i in range(0, n, 64))) / n
    d = torch.sqrt(R.diagonal())
    # blocks of 64 products and n / 64 additions of them in R, n / 256 in S; the centred data
    # differ by the roundings of the mean
    bar = (64 + n / 64 + n / 256 + 8) * 2.0 ** -53 + (n / 4) * 2.0 ** -53 * center
    assert float((S - R).abs().div(d[:, None] * d[None, :]).max()) <= bar


def test_slabs_equal_their_sums():
    """Integers: every sum is exact, so the slabs add up to the bit."""
    n, p = 10000, 130
    rng = np.random.default_rng(4)
    X = torch.from_numpy(rng.integers(-1000, 1001, (n, p)).astype(np.float64)).cuda()
    X[:, 7] *= 2.0 ** -480                             # a column that is not scaled
    R = X.clone()
    R[:, 7] *= 2.0 ** 480
    R = (R.T @ R).cpu()                                # below 2^53: exact in any order
    f = torch.ones(p, dtype=torch.float64)
    f[7] = 2.0 ** -480
    assert torch.equal(_gram(X).cpu(), R * f[:, None] * f[None, :] * (1.0 / n))


def test_small_samples_counted_over_the_slabs():
    """A column that breaks the rule on small samples only in its last slab."""
    n, p = 9000, 66
    X = _data(n, p, 3)
    X[4096:, 5] *= 2.0 ** -20
    S = _gram(X)
    acc = np.zeros(p)
    W = X.cpu().numpy()
    ld = W.astype(np.longdouble)
    for i in range(n):                                 # the FP64 sums in sample order
        acc = (acc.astype(np.longdouble) + ld[i, 5] * ld[i]).astype(np.float64)
    assert np.array_equal(S[5].cpu().numpy(), acc * (1.0 / n))


def test_batch_equals_single():
    Xs = [_data(n, p, n) for n, p in ((60, 40), (4096, 30), (4160, 129), (9000, 65))]
    Xs[3][:, 7] *= 2.0 ** -450
    bt = sp.Batch([(X, 0.3) for X in Xs], precision="fp64", tol=1e-8)
    bt.run()
    bt.result()
    for i, X in enumerate(Xs):
        T, s, _ = sp.fit(sp.gram(X, precision="fp64"), 0.3, tol=1e-8, precision="fp64")
        assert torch.equal(bt.Theta[i], T) and torch.equal(bt.sigma[i], s)


def test_workspace_is_bounded():
    at = sp.spmesl_gram_workspace_bytes
    assert at(10 ** 6, 2000, sp.FP64) == at(4096, 2000, sp.FP64) <= 2000 * 14 * 4096 + 2000 * 64
