"""The separable families' asymmetric Korobov map: its integer steps in exact arithmetic (range, error
bound, mean error), and the sums it serves at the orders with the fewest fraction bits."""
import math
import random
from fractions import Fraction as Fr

import numpy as np
import pytest

M = (1 << 64) - 1
ORDERS = [(a, b) for a in range(1, 7) for b in range(1, 7) if a != b]


def mulhi_trunc(a, b):
    al, ah, bl, bh = a & 0xFFFFFFFF, a >> 32, b & 0xFFFFFFFF, b >> 32
    return (ah * bh + ((ah * bl) >> 32) + ((al * bh) >> 32)) & M


def phi(X, r0, r1):
    kf = 63 - int(math.log2(math.comb(r0 + r1 + 1, max(r0, r1))))
    P = math.comb(r0 + r1, r1) << kf
    for k in range(r1 - 1, -1, -1):
        P = mulhi_trunc(P, M ^ X) + (math.comb(r0 + k, k) << kf)
        assert P <= M
    pw = X
    for _ in range(r0):
        pw = mulhi_trunc(pw, X)
    top = mulhi_trunc(pw, P)
    assert top < 1 << kf
    return top << (64 - kf), kf


def exact(X, r0, r1):
    u = Fr(X, 1 << 64)
    return u ** (r0 + 1) * sum(math.comb(r0 + k, k) * (1 - u) ** k for k in range(r1 + 1))


@pytest.mark.parametrize("r0,r1", ORDERS)
def test_range_and_error(r0, r1):
    """Each high product is under 3 units low.  Horner's errors (units of 2^-kf) are scaled by
    u^(r0+1) <= 1 and by the (1 - u) that follow, the power's (2^-64) by P < 2^(64 - kf); the last
    product 3 more."""
    rng = random.Random(10 * r0 + r1)
    ends = [0, 1, M, M - 1, 1 << 63, (1 << 63) - 1]
    for X in ends + [rng.getrandbits(64) >> rng.choice([0, 0, 1, 9, 40]) for _ in range(200)] + \
            [M ^ (rng.getrandbits(64) >> rng.choice([1, 9, 40])) for _ in range(100)]:
        F, kf = phi(X, r0, r1)
        err = exact(X, r0, r1) - Fr(F, 1 << 64)
        assert 0 <= err <= Fr(4 * (r0 + r1 + 1), 1 << kf)


@pytest.mark.parametrize("r0,r1", ORDERS)
def test_mean_error(r0, r1):
    """A high product is 1.25 units low on average: the last one, Horner's last one, and the ones
    before it scaled by a (1 - u) each, all times u^(r0+1); together below 3 units of 2^-kf."""
    rng = random.Random(100 * r0 + r1)
    errs = []
    for _ in range(2000):
        X = rng.getrandbits(64)
        F, kf = phi(X, r0, r1)
        errs.append(float((exact(X, r0, r1) - Fr(F, 1 << 64)) * 2 ** kf))
    assert 0 <= np.mean(errs) <= 3


@pytest.mark.gpu
@pytest.mark.parametrize("r0,r1", [(5, 6), (6, 5), (4, 6), (1, 3)])
@pytest.mark.parametrize("fam", [1, 2, 3, 4, 5, 6])
def test_sums(fam, r0, r1):
    """sum c = 6, d = 4: the exponent or base takes at most 6 times the map's 4 (r0 + r1 + 1) units of
    2^-kf, the integrand's own power and the weight some 40 roundings."""
    import torch

    import oracle as O
    import paper_1811_11720_gb300 as q
    d, n, m = 4, 10007, 16
    c = np.linspace(1.0, 1.5, d)
    c, w = 6.0 * c / c.sum(), np.array([0.9, 0.9, 0.3, 0.6])
    D = q.make_shifts(3, m, d)
    z = [1, 76, 306, 400]
    out = q.integrate_device(q.Integrand.genz(fam, c, w), n, z, torch.from_numpy(D.astype(np.int64)).cuda(),
                             ("korobov", r0, r1))
    s = out[1].cpu().numpy()[:2 * m].reshape(m, 2).sum(1)
    o = O.shift_sums(O.genz(fam, c, w), ("korobov", r0, r1), n, z, D)
    kf = 63 - int(math.log2(math.comb(r0 + r1 + 1, max(r0, r1))))
    tol = (d + 1) * 6 * 4 * (r0 + r1 + 1) * 2.0 ** -kf + 40 * 2.0 ** -53
    assert np.all(np.abs(s - o["re"].sum(1)) <= tol * o["abs"])
