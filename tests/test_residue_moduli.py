"""The residue kernels' arithmetic modulo m, restated in exact integers for every value they can meet.

An accumulator value c is an integer of magnitude at most 2^24.  The drain forms k = fl(c * fl(1/m)) rounded to an
integer (the fused multiply-add with 1.5 * 2^23 rounds once, to nearest even) and t = c - m k, exact.  The first
modulus of a pair stores t + 128 in a byte, so its t has to lie in [-128, 127]; a second one, or the last, lone
modulus, keeps t in FP32.  The images take c in [0, 2^22) and need |t| <= 128, the bound of the exact FP32 sums.
"""
import os
import re

import numpy as np
import pytest

SRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2512_01055_gb300", "csrc",
                   "tc_rns.cu")
MODULI = [int(x) for x in re.search(r"MODULI\[RL\] = \{([^}]*)\}", open(SRC).read()).group(1).split(",")]


def residue(c, m):
    """t of the int64 array c: k = round-half-even(c * I / 2^s) with I / 2^s = fl32(1/m)."""
    mant, ex = np.frexp(np.float32(1) / np.float32(m))
    i, s = int(float(mant) * 2 ** 24), 24 - int(ex)
    p = c * i
    q, r, half = p >> s, p & ((1 << s) - 1), 1 << (s - 1)
    return c - m * (q + ((r > half) | ((r == half) & ((q & 1) == 1))))


def test_moduli_are_pairwise_coprime():
    for a in range(len(MODULI)):
        for b in range(a):
            assert np.gcd(MODULI[a], MODULI[b]) == 1


@pytest.mark.parametrize("l", range(len(MODULI)))
def test_residue_fits_where_it_is_kept(l):
    m, packed = MODULI[l], l % 2 == 0 and l + 1 < len(MODULI)
    lo, hi = (-128, 127) if packed else (-m // 2 - 1, m // 2 + 1)
    top, step = 1 << 24, 1 << 21
    for c0 in range(-top, top + 1, step):
        t = residue(np.arange(c0, min(c0 + step, top + 1), dtype=np.int64), m)
        assert lo <= t.min() and t.max() <= hi, (m, c0, t.min(), t.max())
    t = residue(np.arange(1 << 22, dtype=np.int64), m)
    assert np.abs(t).max() <= 128
