"""The fill's crossing columns and row parities, modelled in the kernel's
arithmetic (float32 estimates, 64-bit remainders, 32-bit words) against
Algorithm 2's ray test: half-open straddle in y, crossing strictly to the
right, odd count inside."""
import numpy as np
import pytest

F = np.float32


def clampf(v, lo, hi):
    return int(max(min(F(v), F(hi)), F(lo)))


def crossing_end(s, hw, lx, ly, ex, ey, y, lo, hi, e):
    N = ex * (y - ly) + lx * ey
    assert abs(N) <= 2 ** 62
    inv = F(F(F(1) / F(ey)) * F(1 + e)) * F(2.0 ** -s)
    lo, hi = lo - hw, hi - hw
    t = clampf(F(N) * inv, lo, hi)
    d = N - (t << s) * ey
    t = clampf(F(t) + np.ceil(F(d) * inv), lo, hi)
    d = N - (t << s) * ey
    assert abs(d) < 2 ** 63
    if d > 0:
        t += 1
    elif d <= -(ey << s):
        t -= 1
    return max(min(t, hi), lo) + hw


@pytest.mark.parametrize("e", [-2.0 ** -22, 0.0, 2.0 ** -22])
def test_crossing_end(e):
    """Edges from a unit to the grid's width, through samples exactly too."""
    rng = np.random.default_rng(1)
    for _ in range(20_000):
        s = int(rng.integers(3, 24))
        hw = int(rng.choice([32, 128, 256]))
        h, lim = 1 << s, 2 ** 31 - 1
        size = int(2.0 ** rng.uniform(0, 31))
        y = int(rng.integers(-16, 16)) * h
        below = int(rng.integers(0, size))
        ly, ey = y - below, below + 1 + int(rng.integers(0, max(size - below, 1)))
        ex = int(rng.integers(-size, size + 1))
        lx = int(rng.integers(-hw - 9, hw + 9)) * h - ex * below // ey + int(rng.integers(-1, 2))
        if max(abs(lx), abs(lx + ex), abs(ly), abs(ly + ey)) > lim or ey > lim:
            continue
        lo = int(rng.integers(0, 2 * hw))
        hi = int(rng.integers(lo, 2 * hw + 1))
        # column c is crossed when its sample lies strictly left of the crossing
        N = ex * (y - ly) + lx * ey
        want = min(max(-((-N) // (h * ey)) + hw, lo), hi)
        assert crossing_end(s, hw, lx, ly, ex, ey, y, lo, hi, e) == want


def test_parity_of_a_row():
    """A word's suffix XOR with the carry of the words after it: the parity of
    the crossings beyond each column."""
    rng = np.random.default_rng(2)
    for _ in range(2000):
        width = 32 * int(rng.integers(1, 17))
        clo, chi = sorted(int(v) for v in rng.integers(0, width, 2))
        ends = rng.integers(clo, chi + 2, int(rng.integers(0, 40)))
        words = [0] * 18
        for t in ends:
            if t > clo:
                words[t >> 5] ^= 1 << (t & 31)
        got, carry = set(), 0
        for k in range((chi + 1) >> 5, (clo >> 5) - 1, -1):
            d = sfx = words[k]
            for n in (1, 2, 4, 8, 16):
                sfx ^= sfx >> n
            f = (sfx ^ d ^ carry) & 0xffffffff
            carry ^= 0xffffffff if sfx & 1 else 0
            if k == clo >> 5:
                f &= (0xffffffff << (clo & 31)) & 0xffffffff
            if k < width // 32:
                got |= {32 * k + b for b in range(32) if (f >> b) & 1}
        want = {c for c in range(clo, chi + 1) if np.count_nonzero(ends > c) % 2}
        assert got == want
