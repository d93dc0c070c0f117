"""The asymmetric Korobov map in integer fixed point with run-time orders: its integer steps
restated in exact arithmetic against the Beta integral, and on the GPU against the oracle."""
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


def phi_fixed(X, r0, r1):
    """(phi 2^64 of this half, whether the half is the lower one) as the kernel forms it."""
    deg = max(r0, r1)
    kf = 63 - int(math.log2(math.comb(r0 + r1 + 1, deg)))
    lo = X < 1 << 63
    V = X if lo else M ^ X
    a, b = (r0, r1) if lo else (r1, r0)
    c = [math.comb(a + k, k) << kf if k <= b else 0 for k in range(deg + 1)]
    P = c[deg]
    for k in range(deg - 1, -1, -1):
        P = mulhi_trunc(P, M ^ V) + c[k]
        assert P <= M
    pw = V
    for _ in range(a):
        pw = mulhi_trunc(pw, V)
    F = mulhi_trunc(pw, P) << (64 - kf)
    assert F <= M
    return F, lo, kf, deg


@pytest.mark.parametrize("r0,r1", ORDERS)
def test_phi_error_bound(r0, r1):
    """Each of the deg products of P and of the power is at most 3 units low (W too by one),
    P's error times v^(r+1) <= 1/4, the power's times P <= 2^(64 - kf), the last product 3
    units of 2^-kf and its dropped bits one more."""
    rng = random.Random(100 * r0 + r1)
    for _ in range(300):
        X = rng.getrandbits(64) >> rng.choice([0, 0, 0, 1, 4, 20, 40])
        X = rng.choice([X, M ^ X])
        F, lo, kf, deg = phi_fixed(X, r0, r1)
        u = Fr(X, 1 << 64) if lo else 1 - Fr(X, 1 << 64)
        a, b = (r0, r1) if lo else (r1, r0)
        exact = u ** (a + 1) * sum(math.comb(a + k, k) * (1 - u) ** k for k in range(b + 1))
        assert abs(Fr(F, 1 << 64) - exact) <= Fr(4 * deg + 4 * deg + 4, 1 << kf)


@pytest.mark.gpu
@pytest.mark.parametrize("r0,r1", ORDERS)
def test_sums_against_the_oracle(r0, r1):
    import torch

    import oracle as O
    import paper_1811_11720_gb300 as q
    import workloads as W
    tab = q.GenvecTable.load()
    dev = torch.device("cuda:0")
    n = 4691
    for i, (fam, d, m, fit) in enumerate([(1, 3, 32, False), (2, 5, 20, False), (3, 10, 10, False),
                                          (4, 16, 8, False), (5, 4, 2, False), (6, 2, 50, False),
                                          (3, 1, 1, False), (4, 6, 33, True), ("sector", 8, 16, False),
                                          ("sector", 5, 32, True), ("feynman", 5, 16, False)]):
        D = q.make_shifts(7 * i + r0, m, d)
        z = tab.z_for(n)[:d] if d <= 10 else np.arange(1, d + 1) * 97 % n
        if fam == "sector":
            fl = W.sector_like(i, d, 60, 90)
            f, fo = q.Integrand.polynomial(fl), O.from_feynman(fl)
        elif fam == "feynman":
            fl = W.feynman_regular(i, beta=0.6)
            f, fo = q.Integrand.polynomial(fl), O.feynman_complex(fl)
        else:
            c, w = W.genz_params(fam, d, i)
            f, fo = q.Integrand.genz(fam, c, w), O.genz(fam, c, w)
        p = W.fit_params_example(d, i) if fit else None
        out = q.integrate_device(f, n, z, torch.from_numpy(D.astype(np.int64)).to(dev),
                                 ("korobov", r0, r1), None if p is None else torch.from_numpy(p).to(dev)) \
            if m >= 2 else None
        if out is None:   # one shift has no error: the sums alone
            r = q.rule(n, z, torch.from_numpy(D.astype(np.int64)).to(dev), ("korobov", r0, r1))
            ws = torch.empty(q.sums_workspace_bytes(r, False, 0, n), dtype=torch.uint8, device=dev)
            out = (None, q.sums(f.device_struct(dev), r, 0, n, ws,
                                torch.zeros(2, dtype=torch.float64, device=dev)))
        s = out[1].cpu().numpy()
        o = O.shift_sums(fo, ("korobov", r0, r1), n, z, D, fitp=p)
        got = s[:2 * m].reshape(m, 2).sum(1)
        want = o["re"].sum(1)
        assert np.all(np.abs(got - want) <= 1e-12 * o["abs"]), (fam, d, m)
        if fam == "feynman":
            got, want = s[2 * m:4 * m].reshape(m, 2).sum(1), o["im"].sum(1)
            assert np.all(np.abs(got - want) <= 1e-12 * o["abs"])


@pytest.mark.parametrize("r0,r1", ORDERS)
def test_phi_on_the_whole_interval(r0, r1):
    """The separable families' form: one polynomial on [0, 1], below 1.  The Horner products and
    the r0 + 1 powers are at most 3 units of 2^-kf low each (the powers' losses are scaled by
    u < 1), W one unit of 2^-64: at most 4 (r0 + r1 + 1) units."""
    rng = random.Random(10 * r0 + r1)
    deg = max(r0, r1)
    kf = 63 - int(math.log2(math.comb(r0 + r1 + 1, deg)))
    for X in [0, 1, M, M - 1, 1 << 63] + [rng.getrandbits(64) >> rng.choice([0, 0, 1, 9, 40]) for _ in range(200)] + \
             [M ^ (rng.getrandbits(64) >> rng.choice([1, 9, 40])) for _ in range(100)]:
        P = math.comb(r0 + r1, r1) << kf
        for k in range(r1 - 1, -1, -1):
            P = mulhi_trunc(P, M ^ X) + (math.comb(r0 + k, k) << kf)
            assert P <= M
        pw = mulhi_trunc(X, P)
        for _ in range(r0):
            pw = mulhi_trunc(pw, X)
        assert pw < 1 << kf
        u = Fr(X, 1 << 64)
        exact = u ** (r0 + 1) * sum(math.comb(r0 + k, k) * (1 - u) ** k for k in range(r1 + 1))
        assert 0 <= exact - Fr(pw, 1 << kf) <= Fr(4 * (r0 + r1 + 1), 1 << kf)
