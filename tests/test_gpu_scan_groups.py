"""The grouped quiet scans of the lazy solver: the number of chunks around the
group sizes, columns whose sweeps move coordinates in any chunk of a group, and
both occupancy forms of the batch kernel, against the FP64 oracle and the same
fits alone."""
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


@pytest.mark.parametrize("p", [127, 128, 129, 256, 257, 384, 385, 512, 513, 640, 769])
@pytest.mark.parametrize("prec,tol", [("fp32", 1e-6), ("fp64", 1e-10)])
def test_chunks_around_the_groups(p, prec, tol):
    prob = synth.make_problem("hub_scaled", p, 120, p, dtype=np.float64)
    S = oracle.gram(prob.X)
    T, s, st = sp.fit(torch.from_numpy(S.astype(np.float32 if prec == "fp32" else np.float64)).cuda(),
                      prob.lambda0, tol=tol, precision=prec)
    assert st["status"] == sp.SPMESL_OK
    ref = oracle.spmesl(S, prob.lambda0, tol=1e-11, maxit=1000)
    res = compare_theta(T.cpu().numpy(), ref["Theta"], ref["B"], ref["sigma"], rel=BAR[prec])
    assert res["ok"], res


def test_both_occupancy_forms_equal_single_fits():
    """Enough columns for the three-block form of the FP32 batch kernel (20 a resident warp),
    and the same fits in a batch small enough for the two-block form."""
    warps = torch.cuda.get_device_properties(0).multi_processor_count * 16
    Xs = [torch.from_numpy(synth.make_problem(k, p, 60, 40 + p).X).cuda()
          for k, p in (("ar1", 300), ("hub_scaled", 257), ("er", 500))]
    copies = 20 * warps // sum(x.shape[1] for x in Xs) + 1
    lam = 0.5
    big = sp.Batch([(x, lam) for _ in range(copies) for x in Xs])
    small = sp.Batch([(x, lam) for x in Xs])
    assert sum(x.shape[1] for x in Xs) * copies > 20 * warps
    big.run()
    small.run()
    big.result()
    small.result()
    for i, x in enumerate(Xs):
        T, s, _ = sp.fit(sp.gram(x), lam)
        for k in (0, copies - 1):
            assert torch.equal(big.Theta[k * len(Xs) + i], T)
        assert torch.equal(small.Theta[i], T) and torch.equal(small.sigma[i], s)
