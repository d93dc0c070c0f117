"""The PolySingular map on the integer pipe: its steps in exact arithmetic against the formula, and
fitted sums on the GPU against the oracle, on both sides of the form's guards."""
import math
import random
from fractions import Fraction as Fr

import numpy as np
import pytest

import workloads as W

M = (1 << 64) - 1


def mulhi_trunc(a, b):
    al, ah, bl, bh = a & 0xFFFFFFFF, a >> 32, b & 0xFFFFFFFF, b >> 32
    return (ah * bh + ((ah * bl) >> 32) + ((al * bh) >> 32)) & M


def smulhi_x(c, X):
    h = (mulhi_trunc(c & M, X) - (X if c < 0 else 0)) & M
    return h - (1 << 64) if h >> 63 else h


def recip_fixed(m, rng):
    """2^127 / m; the single-precision estimate with any error it may have"""
    mh, ml = m >> 32, m & 0xFFFFFFFF
    rel = rng.uniform(-1, 1) * 2 ** -21.6
    r0 = int((Fr(1 << 63) / mh) * (1 - Fr(1, 1 << 21)) * (1 + Fr(rel)))
    assert 0 < r0 < 1 << 32
    E = (1 << 63) - 1 - (mh * r0 + ((ml * r0) >> 32))
    assert 0 < E < 1 << 43
    e22 = E >> 20
    E2 = E + ((e22 * e22) >> 23)
    R = (r0 << 32) + ((r0 * (E2 & 0xFFFFFFFF)) >> 31) + ((r0 * (E2 >> 32)) << 1)
    assert R <= M
    return R


def norm(v):
    """a positive double as m 2^(e - 64), m in [2^63, 2^64)"""
    f, e = math.frexp(v)
    return int(Fr(f) * (1 << 64)), e


def test_reciprocal():
    rng = random.Random(2)
    for _ in range(3000):
        m = (1 << 63) + (rng.getrandbits(63) >> rng.choice([0, 0, 1, 20, 62]))
        err = 1 - Fr(recip_fixed(m, rng) * m, 1 << 127)
        assert 0 <= err <= Fr(1, 1 << 59)


@pytest.mark.parametrize("seed", range(8))
def test_map_and_derivative(seed):
    """p: three or fewer truncated products of 2^60- and 2^62-scale factors for each term, v off
    by 2^-59 relatively and its scale, times coefficients below 7: under 2^6 7 units of 2^-60 and
    the 2^-58 scale's own, below 2^-50.  p' likewise at 2^em, with coefficients summing to M."""
    rng = random.Random(seed)
    for a in W.fit_params_example(4, seed) if seed < 6 else [[1.0006, -0.0006, 0.01, 0.008, 0.9, 0.05],
                                                            [1023.0, -1022.0, 0.3, 0.001, 0.6, 0.1]]:
        a0, b, a2, a3, a4, a5 = float(a[0]), -float(a[1]), abs(float(a[2])), abs(float(a[3])), float(a[4]), float(a[5])
        a6 = 1.0 - a2 - a3 - a4 - a5
        k2, k3 = a2 * a0 / (a0 - 1), a3 * (1 + b) / b
        Mx = k2 + k3 + abs(a4) + 2 * abs(a5) + 3 * abs(a6)
        assert Mx < 64
        fx = lambda v, s: round(Fr(v) * Fr(2) ** s)  # noqa: E731
        k0, k1 = math.floor(math.log2(a0)) + 1, math.floor(math.log2(1 + b)) + 1
        em = 61 - math.floor(math.log2(Mx))
        c0, ec0 = norm(a0 - 1)
        cb, ecb = norm(b)

        def ratio(D, c, s):
            assert (1 << 43) <= D <= M
            lz = 64 - D.bit_length()
            assert lz < 32 and s - lz >= 0
            return mulhi_trunc(c, recip_fixed(D << lz, rng)) >> (s - lz)
        for X in [0, 1, M, M - 1, 1 << 63] + [rng.getrandbits(64) >> rng.choice([0, 0, 3, 30]) for _ in range(60)] + \
                [M ^ (rng.getrandbits(64) >> rng.choice([1, 5, 30])) for _ in range(20)]:
            x = Fr(X, 1 << 64)
            v0 = ratio(fx(a0, 64 - k0) - (X >> k0), c0, k0 - ec0 + 1)
            v1 = ratio(fx(b, 64 - k1) + (X >> k1), cb, k1 - ecb + 1)
            assert v0 <= 1 << 62 and v1 <= 1 << 62
            q = smulhi_x(smulhi_x(smulhi_x(fx(a6, 60), X) + fx(a5, 60), X) + fx(a4, 60), X) >> 2
            q += mulhi_trunc(mulhi_trunc(X, v0), fx(a2, 60)) + mulhi_trunc((1 << 62) - v1, fx(a3 * (1 + b), 60))
            sq = lambda v: mulhi_trunc(v, v) << 3  # noqa: E731
            dp = smulhi_x(smulhi_x(fx(3 * a6, em), X) + fx(2 * a5, em), X) + fx(a4, em) + \
                mulhi_trunc(sq(v0), fx(k2, em + 1)) + mulhi_trunc(sq(v1), fx(k3, em + 1))
            A = [Fr(v) for v in (a0, -b, a2, a3, a4, a5, a6)]
            p = A[2] * x * (A[0] - 1) / (A[0] - x) + A[3] * x * (A[1] - 1) / (A[1] - x) + x * (A[4] + x * (A[5] + x * A[6]))
            d = A[2] * A[0] * (A[0] - 1) / (A[0] - x) ** 2 + A[3] * A[1] * (A[1] - 1) / (A[1] - x) ** 2 + A[4] + \
                2 * A[5] * x + 3 * A[6] * x * x
            assert abs(Fr(q, 1 << 58) - p) < Fr(1, 1 << 50)
            assert abs(Fr(dp) / Fr(2) ** em - d) < Fr(Mx) * Fr(1, 1 << 50)


@pytest.mark.gpu
@pytest.mark.parametrize("fit", ["example", "sharp", "wide", "not monotone", "steep"])
@pytest.mark.parametrize("family,d", [("sector", 3), ("sector", 5), ("sector", 8), ("feynman", 4), ("feynman", 5)])
def test_fitted_sums_against_the_oracle(family, d, fit):
    import torch

    import oracle as O
    import paper_1811_11720_gb300 as q
    tab = q.GenvecTable.load()
    fl = W.sector_like(d, d, 100, 150) if family == "sector" else W.feynman_regular(d, d=d, beta=0.6)
    fo = O.from_feynman(fl) if family == "sector" else O.feynman_complex(fl)
    p = W.fit_params_example(d, 5)
    if fit == "sharp":
        p[:, 0], p[:, 1] = 1.001, -0.001       # the fit's bounds
        p[:, 2:4] = 0.004
    if fit == "wide":
        p[:, 0], p[:, 1] = 900.0, -700.0
    if fit == "steep":
        p[0, 0], p[0, 2] = 1.001, 0.3          # p' up to 300: the FP64 form
    if fit == "not monotone":                  # p' < 0 near 1 in one dimension, p above 1 there
        p[0, 2:] = [0.0, 0.0, 1.2, 0.5]
    n, m = 4691, 16
    z, D = tab.z_for(n)[:d], q.make_shifts(d, m, d)
    for tr in (("korobov", 3), ("korobov", 1), ("korobov", 2, 3), ("baker",), ("none",)):
        out = q.integrate_device(q.Integrand.polynomial(fl), n, z,
                                 torch.from_numpy(D.astype(np.int64)).cuda(), tr, torch.from_numpy(p).cuda())
        s = out[1].cpu().numpy()
        o = O.shift_sums(fo, tr, n, z, D, fitp=p)
        parts = [(s[:2 * m], o["re"])] + ([(s[2 * m:], o["im"])] if family == "feynman" else [])
        for got, want in parts:
            err = np.abs(got.reshape(m, 2).sum(1) - want.sum(1)) / o["abs"]
            if fit == "not monotone" and family == "sector":
                assert np.isfinite(got).all()   # F stays at the cube's face where p leaves it
            else:
                assert err.max() <= 1e-12, tr
