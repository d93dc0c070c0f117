"""The complex family with its values at z in fixed point: the integer steps in exact arithmetic,
and the GPU against the oracle on both sides of the form's guard."""
import itertools
import math
import random
from fractions import Fraction as Fr

import numpy as np
import pytest

import workloads as W

M = (1 << 64) - 1


def digits(v):
    """v = h 2^32 + l with signed 32-bit l"""
    lo = v & 0xFFFFFFFF
    lo -= (lo >> 31) << 32
    h = (v - lo) >> 32
    assert -(1 << 31) <= h < 1 << 31
    return h, lo


def dot(pairs, split=False):
    """sum a b 2^-64 as the kernel forms it; its 32-bit sums must hold"""
    wide = cross2 = 0
    pairs = list(pairs)
    cross = len(pairs)
    for a, b in pairs:
        (ah, al), (bh, bl) = digits(a), digits(b)
        wide += ah * bh
        cross += (ah * bl) >> 32
        cross2 += (al * bh) >> 32
    parts = (cross, cross2) if split else (cross + cross2,)
    assert all(-(1 << 31) <= p < 1 << 31 for p in parts) and abs(wide) < 1 << 63
    return wide + cross + cross2


def mulhi_trunc(a, b):
    al, ah, bl, bh = a & 0xFFFFFFFF, a >> 32, b & 0xFFFFFFFF, b >> 32
    return (ah * bh + ((ah * bl) >> 32) + ((al * bh) >> 32)) & M


def smulhi_x(c, X):
    h = mulhi_trunc(c & M, X) - (X if c < 0 else 0)
    h &= M
    return h - (1 << 64) if h >> 63 else h


def test_digit_dot():
    rng = random.Random(1)
    for _ in range(2000):
        pairs = [tuple(rng.choice([-1, 1]) * (rng.getrandbits(61) >> rng.choice([0, 1, 20, 60])) for _ in range(2))
                 for _ in range(rng.randint(1, 3))]
        err = Fr(sum(a * b for a, b in pairs), 1 << 64) - dot(pairs)
        assert abs(err) <= Fr(5, 4) * len(pairs)


@pytest.mark.parametrize("d", [3, 5, 6])
def test_values_at_the_deformed_point(d):
    """F(z) and U(z) as the kernel forms them against exact rationals.  A product is off by at
    most 5/4 units, taken 8 times for those with x, a coefficient by half a unit: below 10.5 N
    units for F(x), N <= 84; a unit is at most 2^-60 of the
    coefficients' sum, itself at most 16 |c0|.  The terms at y: fewer than 3 N units of at most
    2^-56 of bounds up to 64 |c0|.  In all below 2^13 2^-60 16 + 2^9 2^-56 64 = 2^-41 + 2^-41."""
    rng = random.Random(d)
    for trial in range(6):
        fl = W.feynman_regular(trial, d=d, beta=rng.choice([0.6, 0.95]), lam=rng.choice([0.5, 1.0]))
        lam = Fr(fl.lam)

        def by_factors(p):
            t = {}
            for c, e in zip(p.coef, p.exps):
                key = tuple(k for k in range(d) for _ in range(int(e[k])))
                t[key] = t.get(key, 0.0) + float(c)
            return t
        tf, tu = by_factors(fl.F), by_factors(fl.U)
        pairs = list(itertools.combinations_with_replacement(range(d), 2))
        triples = list(itertools.combinations_with_replacement(range(d), 3))
        # fully symmetric tensors: 6 F3 and F2, U2
        f1 = [tf.get((i,), 0.0) for i in range(d)]
        u1 = [tu.get((i,), 0.0) for i in range(d)]

        def second(t, i, j):
            c = t.get((min(i, j), max(i, j)), 0.0)
            return c if i == j else 0.5 * c

        def third(i, j, k):
            key = tuple(sorted((i, j, k)))
            same = len(set(key))
            return tf.get(key, 0.0) * {1: 6.0, 2: 2.0, 3: 1.0}[same]
        R = range(d)
        G = max(abs(f1[i]) + sum(2 * abs(second(tf, i, j)) + 0.5 * sum(abs(third(i, j, k)) for k in R)
                                 for j in R) for i in R)
        Hm = max(2 * abs(second(tf, i, j)) + sum(abs(third(i, j, k)) for k in R) for i in R for j in R)
        GU = max(abs(u1[i]) + 2 * sum(abs(second(tu, i, j)) for j in R) for i in R)
        lg = lambda v: math.floor(math.log2(v))  # noqa: E731
        c0 = abs(tf[()])
        sv, svu = 60 - lg(sum(map(abs, tf.values()))), 60 - lg(sum(map(abs, tu.values())))
        s3 = 60 - lg(sum(abs(tf.get(t, 0.0)) for t in triples))
        s2u = 60 - lg(sum(abs(tu.get(t, 0.0)) for t in pairs))
        sg, sh, sgu = 60 - lg(G), 60 - lg(Hm), 60 - lg(GU)
        fx = lambda v, s: round(Fr(v) * Fr(2) ** s)  # noqa: E731
        for _ in range(8):
            X = [rng.getrandbits(64) >> rng.choice([0, 0, 0, 1, 5, 40]) for _ in R]
            if rng.random() < 0.2:
                X[0] = 0
            if rng.random() < 0.2:
                X[-1] = M
            x = [Fr(v, 1 << 64) for v in X]
            xs = [v >> 3 for v in X]
            h2 = [[fx(2 * second(tf, i, j), sh) for j in R] for i in R]
            H = [[h2[i][j] + 8 * dot((fx(third(i, j, k), sh), xs[k]) for k in R) for j in R] for i in R]
            Y, gq, gy, gUy = [], [], 0, 0
            for i in R:
                v = dot((((H[i][j] >> 1) + (h2[i][j] >> 1), xs[j]) for j in R), split=True)
                e = sg - sh + 3
                gq.append(fx(f1[i], sg) + (v << e if e >= 0 else v >> -e))
                Y.append(smulhi_x(gq[i], (mulhi_trunc(X[i], M ^ X[i]) << 2) & M))
                gU = fx(u1[i], sgu) + 8 * dot((fx(2 * second(tu, i, j), sgu), xs[j]) for j in R)
                assert max(abs(gq[i]), abs(Y[i]), abs(gU)) <= 1 << 61
                gy += dot([(gq[i], Y[i])])
                gUy += dot([(gU, Y[i])])

            def nested(c, s, v, shift, deg, start=()):
                t = fx(c.get(start, 0.0), s) if len(start) >= deg[0] else 0
                if len(start) < deg[1]:
                    t += dot((nested(c, s, v, shift, deg, start + (k,)), v[k])
                             for k in range(start[-1] if start else 0, d)) << shift
                return t
            Fq = nested(tf, sv, xs, 3, (0, 3))
            Uq = nested(tu, svu, xs, 3, (0, 2))
            cF = nested(tf, s3, Y, 0, (3, 3))
            qU = nested(tu, s2u, Y, 0, (2, 2))
            yHy = dot(((dot([(H[i][i], Y[i])]) + 2 * dot(((H[i][j], Y[j]) for j in range(i + 1, d)), split=True), Y[i])
                       for i in R), split=True)
            gy, sy = max(gy, 0), sg + 2
            p2 = lambda e: Fr(2) ** e  # noqa: E731
            Fz = (Fq * p2(-sv) - lam ** 2 / 2 * yHy * p2(-(sh + 2 * sy - 128)),
                  lam ** 3 * cF * p2(-(s3 + 3 * (sy - 64))) - lam * gy * p2(-(sg + sy - 64)))
            Uz = (Uq * p2(-svu) - lam ** 2 * qU * p2(-(s2u + 2 * (sy - 64))),
                  -lam * gUy * p2(-(sgu + sy - 64)))

            def val(t, pt):
                return sum(Fr(c) * math.prod(pt[k] for k in key) for key, c in t.items())

            def grad(t, k):
                return sum(Fr(c) * key.count(k) * math.prod([x[v] for n, v in enumerate(key) if n != key.index(k)])
                           for key, c in t.items() if k in key)
            yv = [-lam * x[k] * (1 - x[k]) * grad(tf, k) for k in R]

            def cval(t):
                re = im = Fr(0)
                for key, c in t.items():
                    a, b = Fr(c), Fr(0)
                    for k in key:
                        a, b = a * x[k] - b * yv[k], a * yv[k] + b * x[k]
                    re, im = re + a, im + b
                return re, im
            for got, want, unit in ((Fz, cval(tf), c0), (Uz, cval(tu), sum(map(abs, tu.values())))):
                for u, v in zip(got, want):
                    assert abs(u - v) <= Fr(unit) * Fr(1, 1 << 40)


@pytest.mark.gpu
@pytest.mark.parametrize("d", [3, 4, 5, 6])
@pytest.mark.parametrize("what", ["smooth", "sign change", "large lambda", "no constant", "fit", "powers", "b = 64 c0"])
def test_sums_against_the_oracle(d, what):
    import torch

    import oracle as O
    import paper_1811_11720_gb300 as q
    tab = q.GenvecTable.load()
    fl = W.feynman_regular(d, d=d, beta=0.95 if what == "sign change" else 0.6,
                           lam=4.0 if what == "large lambda" else 1.0)
    if what == "no constant":      # F(x) near a corner is far below its coefficients
        keep = fl.F.exps.sum(1) > 0
        fl.F.coef = np.abs(fl.F.coef[keep])
        fl.F.exps = fl.F.exps[keep]
    if what == "b = 64 c0":        # coefficients too large beside the constant term
        fl.F.coef[0] = 1.0 / 6.0
    if what == "powers":
        fl.a, fl.b = 1.5, 1.75
    n, m = 4691, 16
    z, D = tab.z_for(n)[:d], q.make_shifts(d, m, d)
    p = W.fit_params_example(d, 2) if what == "fit" else None
    dev = torch.device("cuda:0")
    for tr in (("korobov", 3), ("baker",), ("korobov", 2, 1)):
        out = q.integrate_device(q.Integrand.polynomial(fl), n, z,
                                 torch.from_numpy(D.astype(np.int64)).to(dev), tr,
                                 None if p is None else torch.from_numpy(p).to(dev))
        s = out[1].cpu().numpy()
        o = O.shift_sums(O.feynman_complex(fl), tr, n, z, D, fitp=p)
        for part, want in ((s[:2 * m], o["re"]), (s[2 * m:], o["im"])):
            assert np.all(np.abs(part.reshape(m, 2).sum(1) - want.sum(1)) <= 1e-12 * o["abs"]), tr
        assert int(out[2][1].item()) == o["signfail"]
