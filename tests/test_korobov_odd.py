"""Korobov<r,r> in the odd form of the separable families, its integer steps in exact arithmetic."""
import math
import random
from fractions import Fraction as Fr

import pytest

M = (1 << 64) - 1


def mulhi_trunc(a, b):
    al, ah, bl, bh = a & 0xFFFFFFFF, a >> 32, b & 0xFFFFFFFF, b >> 32
    return (ah * bh + ((ah * bl) >> 32) + ((al * bh) >> 32)) & M


def sqhi_trunc(a):
    al, ah = a & 0xFFFFFFFF, a >> 32
    return (ah * ah + (((ah * al) >> 32) << 1)) & M


def odd_map(X, r):
    """(phi 2^64, w 2^64)"""
    low = 0 if X >> 63 else M
    A = ((X << 1) & M) ^ low
    W = M ^ sqhi_trunc(A)
    q = (1 << 62) - 4 + (W >> 3)
    if r >= 2:
        W2 = sqhi_trunc(W)
        if r == 2:
            q += (W2 >> 4) + (W2 >> 5)
        else:
            p1 = (3 << 59) + (W >> 4) + (W >> 6)
            if r == 4:
                p1 += mulhi_trunc(W2, 35 << 55)
            if r >= 5:
                p2 = (35 << 55) + mulhi_trunc(W, 63 << 54)
                if r == 6:
                    p2 += mulhi_trunc(W2, 231 << 52)
                p1 += mulhi_trunc(p2, W2)
            q += mulhi_trunc(p1, W2)
    assert q <= M
    h = mulhi_trunc(A, q)
    assert h < 1 << 62           # |s| q < 1: phi does not wrap
    return (((h << 1) ^ low) + (1 << 63)) & M, W


@pytest.mark.parametrize("r", [1, 2, 3, 4, 5, 6])
def test_error_bound(r):
    """q: 4 units of 2^-62 taken off, at most 3 for each truncated product and one for each
    shift (9 at most in all for r <= 4, 13 above), W off by 2 units; |s| q another 3 units and
    the doubling: below 2 (4 + 13 + 3) 2^-63 = 20 2^-62 of phi."""
    rng = random.Random(r)
    edge = [0, 1, 2, 3, (1 << 63) - 1, 1 << 63, (1 << 63) + 1, M, M - 1, 1 << 62, 3 << 62]
    cases = edge + [rng.getrandbits(64) for _ in range(400)]
    for k in range(64):
        cases += [1 << k, M ^ (1 << k), rng.getrandbits(64) >> k, M ^ (rng.getrandbits(64) >> k),
                  (1 << 63) + (rng.getrandbits(63) >> k), (1 << 63) - (rng.getrandbits(63) >> k) - 1]
    for X in cases:
        F, W = odd_map(X, r)
        x = Fr(X, 1 << 64)
        v = min(x, 1 - x)
        phi = v ** (r + 1) * sum(math.comb(r + k, k) * (1 - v) ** k for k in range(r + 1))
        exact = phi if x <= Fr(1, 2) else 1 - phi
        assert abs(Fr(F, 1 << 64) - exact) <= Fr(20, 1 << 62)
        assert -1 <= W - 4 * x * (1 - x) * (1 << 64) <= 4
