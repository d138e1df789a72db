"""The coverage sweep's row intervals, modelled in the kernel's arithmetic
(float32 roots perturbed by their error bound, 32- and 64-bit integers)
against the plain definition: sample column i at i h is covered by a point at
x in a row at distance f exactly when (i h - x)^2 + f^2 <= R^2."""
import math

import numpy as np
import pytest

F = np.float32
PERTURB = [1.0 - 2.0 ** -23, 1.0, 1.0 + 2.0 ** -23]   # the approximate root's error


def root(v, e):
    return F(math.sqrt(float(F(v))) * e)


def isqrt_narrow(B, e):
    w = int(F(root(B, e) * F(1.0 + 2.0 ** -21)))
    return w - 1 if w * w > B else w


def isqrt_wide(B, e):
    f = root(B, e)
    w0 = int(f)
    r = B - w0 * w0
    w = max(w0 + math.floor(F(F(r) / F(F(2.0) * max(f, F(1.0))))), 0)
    if w * w > B:
        w -= 1
    elif (w + 1) ** 2 <= B:
        w += 1
    return w


def half_width(R, f, x, s, narrow, e):
    if narrow:
        return isqrt_narrow(R * R - f * f, e)
    w = root(F(F(R - f) * F(R + f)), e)
    wl, wh = max(int(F(w * F(1.0 - 2.0 ** -20))) - 1, 0), int(F(w * F(1.0 + 2.0 ** -20))) + 1
    if ((x + wl) >> s) != ((x + wh) >> s) or ((wl - x) >> s) != ((wh - x) >> s):
        return isqrt_wide(R * R - f * f, e)
    return wl


@pytest.mark.parametrize("e", PERTURB)
def test_roots_are_floors(e):
    rng = np.random.default_rng(3)
    for w in [0, 1, 2, 3, 46339, 46340] + [int(v) for v in rng.integers(1, 46341, 3000)]:
        for B in (w * w - 1, w * w, w * w + 1, w * w + 2 * w):
            if 0 <= B < 2 ** 31:
                assert isqrt_narrow(B, e) == math.isqrt(B)
    for w in [0, 1, 2, 46341, 2 ** 29] + [int(2 ** v) for v in rng.uniform(0, 29, 5000)]:
        for B in (w * w - 1, w * w, w * w + 1, w * w + 2 * w):
            if 0 <= B <= 2 ** 58:
                assert isqrt_wide(B, e) == math.isqrt(B)


@pytest.mark.parametrize("e", PERTURB)
def test_columns_equal_the_definition(e):
    """Every zoom and radius class, points at random and with a sample at
    exactly R, R + 1 and R - 1 units (3-4-5 and axis-parallel)."""
    rng = np.random.default_rng(4)
    for _ in range(4000):
        s = int(rng.integers(3, 24))
        r16 = int(rng.choice([1, 5, 8, 16, 32, 35, 47, 1024]))
        R = r16 << (s - 3 if s >= 3 else 0)          # h = ps / 2: R = r16 ps / 16
        f = int(rng.integers(0, R + 1))
        x = int(rng.integers(-(4 << s), 4 << s))
        if R % 5 == 0 and rng.random() < 0.5:
            f, x = 3 * R // 5, 4 * R // 5 + int(rng.integers(-1, 2))
        elif rng.random() < 0.3:
            f, x = 0, R + int(rng.integers(-1, 2))
        w = half_width(R, f, x, s, R <= 46340, e)
        lo, hi = -((w - x) >> s), (x + w) >> s
        t = math.isqrt(R * R - f * f)                # |i h - x| <= t
        want = (-((t - x) // (1 << s)), (x + t) // (1 << s))
        assert (lo, hi) == want or (lo > hi and want[0] > want[1])
