"""Host restatements of the solvers' integer forms of FP64 operations (CPU): the
conversion of FP32 values, the tests of |d| < tol and cand > 0, and the upper-word
screen of the sigma floor, each against the FP64 operation itself."""
from __future__ import annotations

import numpy as np


def exact_double(x):
    u = x.view(np.uint32)
    m = u & np.uint32(0x7fffffff)
    direct = (m - np.uint32(0x00800000) >= np.uint32(0x7f000000)) & (m != 0)
    hi = (u & np.uint32(0x80000000)) | np.where(m != 0, (m >> np.uint32(3)) + np.uint32(0x38000000), np.uint32(0))
    bits = (hi.astype(np.uint64) << np.uint64(32)) | (u << np.uint32(29)).astype(np.uint64)
    return np.where(direct, x.astype(np.float64), bits.view(np.float64))


def test_exact_double_of_every_kind_of_float():
    rng = np.random.default_rng(0)
    u = rng.integers(0, 1 << 32, 1 << 20, dtype=np.uint64).astype(np.uint32)
    x = np.concatenate([u.view(np.float32),
                        np.array([0.0, -0.0, 1.0, -1.0, 2.0 ** -126, 2.0 ** -149, -(2.0 ** -127), np.inf,
                                  -np.inf, np.nan, 3.4028234e38], np.float32)])
    with np.errstate(invalid="ignore"):
        assert np.array_equal(exact_double(x), x.astype(np.float64), equal_nan=True)


def test_below_and_sign_on_the_bits():
    rng = np.random.default_rng(1)
    d = np.concatenate([rng.standard_normal(10000) * 10.0 ** rng.uniform(-12, 2, 10000),
                        np.array([0.0, -0.0, 1e-6, -1e-6, np.nextafter(1e-6, 0), np.inf])])
    for tol in (1e-6, 1e-8, 1e-300):
        a = d.view(np.int64) & np.int64(0x7fffffffffffffff)
        assert np.array_equal(a < np.float64(tol).view(np.int64), np.abs(d) < tol)
    assert np.array_equal(d.view(np.int64) > 0, d > 0)


def test_the_floor_screen_keeps_every_floored_value():
    """Every q <= 1e-12 S_jj passes the upper-word screen (which sends it to the exact test)."""
    rng = np.random.default_rng(2)
    sjj = np.concatenate([1.0 + 1e-6 * rng.standard_normal(20000), 10.0 ** rng.uniform(-8, 8, 20000)])
    f = np.concatenate([rng.uniform(0, 1, 39000), np.full(1000, 1.0)])
    q = 1e-12 * sjj * f
    q[::7] *= -1.0
    hi = lambda v: (v.view(np.int64) >> 32).astype(np.int32)  # noqa: E731
    assert (hi(q) <= np.maximum(hi(sjj) - (39 << 20), 1 << 20)).all()
    tiny = np.exp2(-rng.uniform(900, 1020, 20000))       # S_jj of raw FP64 data
    assert (hi(1e-12 * tiny) <= np.maximum(hi(tiny) - (39 << 20), 1 << 20)).all()
    # and values well above the floor do not reach the exact test
    assert not (hi(sjj * 2.0 ** -37) <= hi(sjj) - (39 << 20)).any()
