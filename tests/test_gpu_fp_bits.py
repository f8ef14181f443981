"""The bit-level FP64 helpers of the column solvers themselves (not a restatement of
them), in a small kernel compiled here against their header."""
from __future__ import annotations

import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

torch = pytest.importorskip("torch")
if not torch.cuda.is_available():
    pytest.skip("needs a CUDA device", allow_module_level=True)

from paper_2203_15031_gb300 import _build  # noqa: E402

SOURCE = r"""
#include "cd_device.cuh"
using namespace spmesl;
__global__ void k(const float* f, const double* a, const double* b, const double* c, double* wide,
                  double* soft, float* bound, double* root, int* flags, int n) {
    const int i = blockIdx.x * blockDim.x + threadIdx.x;
    if (i >= n) return;
    wide[i] = exact_double(f[i]);
    soft[i] = soft_std(a[i], c[i]);
    bound[i] = key_bound<double>(abs_key(a[i]));
    root[i] = sqrt_last(c[i], sqrt_heron(c[i]));
    flags[i] = (below(a[i], c[i]) ? 1 : 0) | (abs_above(a[i], c[i]) ? 2 : 0) |
               (may_be_floored(b[i], c[i]) ? 4 : 0) | (differs(a[i], b[i]) ? 8 : 0);
}
extern "C" int run(const float* f, const double* a, const double* b, const double* c, double* wide,
                   double* soft, float* bound, double* root, int* flags, int n) {
    k<<<(n + 255) / 256, 256>>>(f, a, b, c, wide, soft, bound, root, flags, n);
    const cudaError_t e = cudaDeviceSynchronize();
    return e != cudaSuccess ? (int)e : (int)cudaGetLastError();
}
"""


@pytest.fixture(scope="module")
def results(tmp_path_factory):
    d = tmp_path_factory.mktemp("bits")
    (d / "probe.cu").write_text(SOURCE)
    so = d / "probe.so"
    subprocess.run([_build.nvcc(), *_build.ARCH, *_build.FLAGS, "-shared", str(d / "probe.cu"), "-o", str(so)],
                   check=True, capture_output=True)
    rng = np.random.default_rng(0)
    n = 1 << 18
    f = rng.integers(0, 1 << 32, n, dtype=np.uint64).astype(np.uint32).view(np.float32)
    special = np.array([0.0, -0.0, 2.0 ** -126, -(2.0 ** -149), 2.0 ** -127, np.inf, -np.inf, np.nan, 3.4028234e38],
                       np.float32)
    f[: special.size] = special
    # positive scales c over the whole range; a near c and of any size; b around 1e-12 c
    c = np.ldexp(1.0 + rng.random(n), rng.integers(-1060, 1000, n))
    a = c * np.where(rng.random(n) < 0.5, 1.0 + rng.integers(-3, 4, n) * 2.0 ** -52, 10.0 ** rng.uniform(-3, 3, n))
    a *= rng.choice([-1.0, 1.0], n)
    with np.errstate(under="ignore"):
        b = 1e-12 * c * np.where(rng.random(n) < 0.5, 1.0 + rng.integers(-3, 4, n) * 2.0 ** -52,
                                 10.0 ** rng.uniform(-4, 4, n))
    odd = np.array([np.nan, -np.nan, np.inf, -np.inf, 0.0, -0.0, 5e-324, -5e-324, -1.0])
    b[: 9 * 1000] = np.repeat(odd, 1000)
    b[9000:10000] = a[9000:10000]
    a[-2:] = 0.0, -0.0
    dev = [torch.from_numpy(v).cuda() for v in (f, a, b, c)]
    out = [torch.empty(n, dtype=t, device="cuda") for t in (torch.float64, torch.float64, torch.float32,
                                                            torch.float64, torch.int32)]
    torch.cuda.synchronize()
    rc = ctypes.CDLL(str(so)).run(*(ctypes.c_void_p(t.data_ptr()) for t in dev + out), n)
    assert rc == 0
    return (f, a, b, c), [t.cpu().numpy() for t in out]


def test_widening(results):
    (f, _, _, _), (wide, *_) = results
    with np.errstate(invalid="ignore"):
        assert np.array_equal(wide, f.astype(np.float64), equal_nan=True)
    assert np.array_equal(np.signbit(wide[~np.isnan(wide)]), np.signbit(f[~np.isnan(f)]))


def test_compares(results):
    (_, a, b, c), (*_, flags) = results
    assert np.array_equal((flags & 1) != 0, np.abs(a) < c)
    assert np.array_equal((flags & 2) != 0, np.abs(a) > c)
    assert np.array_equal((flags & 8) != 0, a.view(np.int64) != b.view(np.int64))


def test_floor_screen(results):
    (_, _, b, c), (*_, flags) = results
    with np.errstate(invalid="ignore"):
        floored = ~(b > 1e-12 * c)
    assert floored.any() and not floored.all()
    assert ((flags & 4) != 0)[floored].all()
    sure = (flags & 4) == 0
    assert sure.any() and (b[sure] > 1e-12 * c[sure]).all()


def test_soft_threshold_and_bound(results):
    (_, a, _, c), (_, soft, bound, _, _) = results
    ref = np.where(np.abs(a) > c, a - np.copysign(c, a), 0.0)
    assert np.array_equal(soft, ref)
    fits = np.abs(a) < 1e38
    assert (bound[fits].astype(np.float64) >= np.abs(a[fits])).all()
    # one unit of the upper word, and of a float (or of the smallest one)
    assert (bound[fits] <= np.abs(a[fits]) * (1 + 2.0 ** -19) * (1 + 2.0 ** -22) + 2.0 ** -148).all()


def test_square_root(results):
    (_, _, _, c), (_, _, _, root, _) = results
    # the last step corrects an error of 2^-47 by a factor right to 2^-23: its own rounding is left
    assert (np.abs(root - np.sqrt(c)) <= np.spacing(np.sqrt(c))).all()
