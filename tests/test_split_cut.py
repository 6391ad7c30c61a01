"""The cut of an FP64 value into six slices (the slab kernels of psi and of the
operators), restated in NumPy: the leading slice comes off in FP64, what is left
is held by two floats truncated to 24 bits, the other slices are cut in FP32.

Bound: half a unit of the last slice (2^-41 for |x| < 2^8, kLead = 8), plus what
truncating a value below 1/2 to 48 bits can add (2^-49).  Cutting the rounded
float-float form of x itself breaks it.
"""
import numpy as np
import pytest

F = np.float32
S = 6


def top24(x):
    """The double x truncated to a 24-bit significand, as a float32 (0 below 2^-126)."""
    b = x.view(np.uint64) & np.uint64(0xFFFFFFFFE0000000)
    y = b.view(np.float64)
    return np.where(np.abs(y) < 2.0 ** -126, 0.0, y).astype(np.float32)


def cut_pair(h, l, n):
    out = []
    for _ in range(n):
        q = np.rint(h)
        r = (h - q).astype(F)
        s = (r + l).astype(F)
        l = ((l - (s - r)) * F(256)).astype(F)
        h = (s * F(256)).astype(F)
        out.append(q.astype(np.float64))
    return out


def cut_fp64(x):
    m = 6755399441055744.0  # 1.5 * 2^52
    q = (x + m) - m
    r = x - q
    h = top24(r)
    l = top24(r - h.astype(np.float64))
    return [q] + cut_pair(F(256) * h, F(256) * l, S - 1)


def left_over(qs, x):
    """x less its slices, exactly (each step stays within 53 bits)."""
    for i, q in enumerate(qs):
        x = x - q * 2.0 ** (-8 * i)
    return x


@pytest.mark.parametrize("scale", [256.0, 1.0, 2.0 ** -20])
def test_six_slices_of_an_fp64_value(scale):
    rng = np.random.default_rng(5)
    x = rng.uniform(-1, 1, 200_000) * scale
    x[:4] = [0.0, np.nextafter(256.0, 0), -np.nextafter(256.0, 0), 0.5]
    qs = cut_fp64(x)
    assert np.abs(qs[0]).max() <= 256 and max(np.abs(q).max() for q in qs[1:]) <= 128
    assert np.abs(left_over(qs, x)).max() <= 2.0 ** -41 + 2.0 ** -49
    if scale == 256.0:  # the form this replaces
        h = x.astype(F)
        l = (x - h.astype(np.float64)).astype(F)
        assert np.abs(left_over(cut_pair(h, l, S), x)).max() > 1.2 * 2.0 ** -41
