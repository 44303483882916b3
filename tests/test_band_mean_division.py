"""The division of the coarse costs' window sum by its tap count (band features): one multiplication by the rounded
reciprocal and one residual step is the correctly rounded FP32 quotient, for every significand and every tap count."""

import numpy as np
import pytest


def _fma(a, b, c):
    """fl32(a b + c) of FP32 arrays.  The product is exact in float64 (48 bits); the sum's rounding error there decides
    the rounding to FP32 where the float64 sum lies halfway between two FP32 values."""
    p, c = a.astype(np.float64) * b.astype(np.float64), c.astype(np.float64)
    s = p + c
    t = s - p
    err = (p - (s - t)) + (c - t)
    half = (s.view(np.int64) & ((1 << 29) - 1)) == (1 << 28)
    s = np.where(half & (err > 0), np.nextafter(s, np.inf), np.where(half & (err < 0), np.nextafter(s, -np.inf), s))
    return s.astype(np.float32)


@pytest.mark.parametrize("taps", [1, 3, 5, 9, 15, 25])
def test_reciprocal_and_one_residual_step_round_correctly(taps):
    """Windows are clipped 5 x 5: counts a b with a, b in 1..5.  The others (2, 4, 6, 8, 10, 12, 16, 20) are these
    times a power of two, by which every step below scales exactly, as it does with the exponent of the sum."""
    assert {a * b for a in range(1, 6) for b in range(1, 6)} <= {t << k for t in (1, 3, 5, 9, 15, 25) for k in range(5)}
    n = np.float32(taps)
    r = np.float32(1.0) / n
    for lo in range(1 << 23, 1 << 24, 1 << 21):
        s = np.arange(lo, lo + (1 << 21), dtype=np.int64).astype(np.float32)
        d = s * r
        v = _fma(_fma(-d, np.broadcast_to(n, s.shape), s), np.broadcast_to(r, s.shape), d)
        assert np.array_equal(v, s / n)


def test_fma_emulation_rounds_once():
    """Products whose sum with c lies halfway between two FP32 values but for a term beyond float64."""
    one, tiny = np.float32(1.0), np.float32(2.0 ** -60)
    a = np.array([1.0 + 2.0 ** -23, 1.0 + 2.0 ** -23], np.float32)
    half = np.array([2.0 ** -24, 2.0 ** -24], np.float32)
    assert np.array_equal(_fma(half, np.array([one, one]), a), np.float32([1.0 + 2.0 ** -22] * 2))   # a tie: to even
    b = np.array([2.0 ** -24 * (1 + 2.0 ** -23), 2.0 ** -24 * (1 - 2.0 ** -23)], np.float32)
    assert np.array_equal(_fma(b, np.array([one, one]), np.float32([1.0, 1.0])), np.float32([1.0 + 2.0 ** -23, 1.0]))
    x = _fma(np.float32([2.0 ** -30, -(2.0 ** -30)]), np.array([tiny, tiny]), np.float32([1.0, 1.0]))
    assert np.array_equal(x, np.float32([1.0, 1.0]))
