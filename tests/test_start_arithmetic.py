"""The 32-bit start of a sieving prime (neg_mod_low): (-b) mod p from the words
of b and of the Barrett reciprocal, replayed in 32-bit integers against the
definition -- over magnitudes of b up to 2^63, p up to its limit, and b at and
around multiples of p, where a short quotient shows."""
import random

import pytest

M32 = (1 << 32) - 1
P_MAX = M32 // 5


def neg_mod_low(b, p):
    m = ((1 << 64) - 1) // p
    bh, bl, mh, ml = b >> 32, b & M32, m >> 32, m & M32
    q = (bh * mh + (bh * ml >> 32) + (bl * mh >> 32)) & M32
    assert (b // p - q) & M32 <= 4
    r = (bl - q * p) & M32
    for s in (2 * p, 2 * p, p):
        r = min(r, (r - s) & M32)
    return p - r if r else 0


@pytest.mark.parametrize("p_bits", [2, 6, 10, 16, 20, 24, 28, 30])
@pytest.mark.parametrize("b_bits", [6, 20, 32, 33, 50, 62, 63])
def test_neg_mod_low(p_bits, b_bits):
    rng = random.Random(64 * p_bits + b_bits)
    for _ in range(400):
        p = min(rng.randrange(1 << (p_bits - 1), 1 << p_bits) | 1, P_MAX)
        if p < 3:
            p = 3
        b = rng.randrange(1 << (b_bits - 1), 1 << b_bits)
        c = b // p * p
        for x in (b, c, c - 1, c + 1, c + p - 1):
            if 0 < x < 1 << 63:
                assert neg_mod_low(x, p) == -x % p, (x, p)


def test_limit_matches_the_kernels():
    import os
    root = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
    with open(os.path.join(root, "paper_2603_02621_gb300", "csrc", "gb_internal.cuh")) as f:
        assert f"kLowModMax = {P_MAX}u" in f.read()
