"""Arithmetic rules of the marker kernels, restated in numpy with their roundings
and checked over the ranges that they are used for."""
import numpy as np
import pytest


@pytest.mark.parametrize("n", [4, 5, 7, 33, 128, 403, 2000, 8192, 65536, 999983])
def test_wrapped_index(n):
    """i - floor(fl(i) fl(1/n)) n with one correction is i mod n for |i| <= 1e7"""
    rng = np.random.default_rng(n)
    i = np.unique(np.concatenate([rng.integers(-10**7, 10**7, 200000), np.arange(-5 * n, 5 * n, max(1, n // 50)),
                                  [k * n + d for k in (-10**7 // n, -1, 0, 1, 10**7 // n - 1) for d in (-1, 0, 1)]]))
    i = i[np.abs(i) <= 10**7].astype(np.int64)
    q = np.floor(i.astype(np.float32) * np.float32(1.0 / n)).astype(np.int64)
    r = i - q * n
    r = np.where(r < 0, r + n, np.where(r >= n, r - n, r))
    assert np.array_equal(r, i % n)


def test_draw_thresholds():
    """k 2^-53 < t and > t for FP32 thresholds, decided on integers, against FP64"""
    rng = np.random.default_rng(1)
    t = np.concatenate([rng.uniform(-1e-5, 1.1, 3000), 10.0 ** rng.uniform(-12, 0, 3000), [0.0, -1e-5, 1.0]]).astype(np.float32)
    for d in (0, 1, -1, 7, -7):
        k = np.clip(np.floor(t.astype(np.float64) * 2.0**53).astype(np.int64) + d, 0, 2**53 - 1)
        u = k.astype(np.float64) * 2.0**-53
        s = t.astype(np.float64) * 2.0**53  # exact in FP32 too: a power of two
        below = (t > 0) & (k < np.ceil(s).astype(np.int64))
        above = ~(t >= 0) | (k > np.floor(s).astype(np.int64))
        assert np.array_equal(below, u < t.astype(np.float64))
        assert np.array_equal(above, u > t.astype(np.float64))
