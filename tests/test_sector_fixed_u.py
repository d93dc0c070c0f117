"""The real sector family with both polynomials in fixed point: the integer steps in exact
arithmetic (error bound with the truncation compensated), and the GPU against the oracle over
dimensions, degrees, fits (one that leaves the cube among them) and the guards' other sides."""
import math
import random
from fractions import Fraction as Fr

import numpy as np
import pytest

M = (1 << 64) - 1


def mulhi_trunc(a, b):
    al, ah, bl, bh = a & 0xFFFFFFFF, a >> 32, b & 0xFFFFFFFF, b >> 32
    return (ah * bh + ((ah * bl) >> 32) + ((al * bh) >> 32)) & M


@pytest.mark.parametrize("d", [3, 5, 8])
def test_dense_quadratic_error_bound(d):
    """At most 3 units a product and half a unit a coefficient low, the compensation at most
    as much high; every partial sum below 2^63 and a half."""
    rng = random.Random(d)
    n1, n2 = d, d * (d + 1) // 2
    comp = int(1.25 * (n1 + 0.5 * n2))
    for _ in range(50):
        c = [rng.random() * rng.choice([0, 1, 1]) for _ in range((d + 1) * (d + 2) // 2)]
        c[0] += 1e-3
        s = 62 - math.floor(math.log2(sum(c)))
        C = [round(Fr(v) * 2 ** s) for v in c]
        C[-1] += comp
        X = [rng.getrandbits(64) >> rng.choice([0, 0, 1, 8, 30]) for _ in range(d)]
        x = [Fr(v, 1 << 64) for v in X]
        F, exact, idx = 0, Fr(0), 0
        for a in range(d):
            t = 0
            for b in range(a, d):
                t += mulhi_trunc(C[idx], X[b])
                exact += Fr(c[idx]) * x[a] * x[b]
                idx += 1
            t += C[idx]
            exact += Fr(c[idx]) * x[a]
            idx += 1
            F += mulhi_trunc(X[a], t)
        F += C[idx]
        exact += Fr(c[idx])
        assert F < 1 << 63
        err = Fr(F) - exact * 2 ** s
        assert -3.5 * (n1 + n2) - 1 <= err <= comp + 0.5 * (n1 + n2) + 1


def _poly(rng, d, degree, terms, const):
    import workloads as W
    e = np.vstack([W.all_monomials(d, k) for k in range(0 if const else 1, degree + 1)])
    e = e[rng.integers(0, len(e), terms)]
    c = rng.uniform(0, 1, terms)
    if const:
        e[0], c[0] = 0, 0.5
    return W.Polynomial(c, e.astype(np.int32))


@pytest.mark.gpu
@pytest.mark.parametrize("fit", ["none", "inside", "outside"])
@pytest.mark.parametrize("d,du,df,nu,nf,change", [
    (1, 2, 2, 30, 30, None), (2, 2, 3, 60, 60, None), (3, 3, 2, 200, 100, None), (4, 2, 3, 200, 300, None),
    (7, 3, 3, 512, 512, None), (8, 2, 3, 200, 400, None), (8, 2, 3, 10, 400, None), (11, 2, 3, 400, 500, None),
    (16, 2, 2, 512, 512, None), (5, 2, 3, 100, 200, "negative u"), (5, 2, 3, 100, 200, "negative f"),
    (5, 2, 3, 100, 200, "a = 2"), (5, 2, 3, 100, 200, "b = 2")])
def test_sums_against_the_oracle(d, du, df, nu, nf, change, fit):
    import torch

    import oracle as O
    import paper_1811_11720_gb300 as q
    import workloads as W
    rng = np.random.default_rng(1000 * d + nu)
    U, F = _poly(rng, d, du, nu, False), _poly(rng, d, df, nf, True)
    if change == "negative u":
        U.coef[3] = -0.25
    if change == "negative f":
        F.coef[3] = -1e-3
    fl = W.FeynmanLike(U, F, 2.0 if change == "a = 2" else 1.0, 2.0 if change == "b = 2" else 2.5, 0.0, d)
    n, m = 1021, 16
    z = np.arange(1, d + 1) * 76 % n
    D = q.make_shifts(d, m, d)
    p = None
    if fit != "none":
        p = W.fit_params_example(d, 3)
    if fit == "outside":   # p(x) = x (a4 + x (a5 + x a6)): above 1 inside the interval
        p[:, 2:] = 0.0
        p[:, 4], p[:, 5] = 1.5, 1.0
    dev = torch.device("cuda:0")
    out = q.integrate_device(q.Integrand.polynomial(fl), n, z, torch.from_numpy(D.astype(np.int64)).to(dev),
                             ("korobov", 3), None if p is None else torch.from_numpy(p).to(dev))
    s = out[1].cpu().numpy()[:2 * m].reshape(m, 2).sum(1)
    o = O.shift_sums(O.from_feynman(fl), ("korobov", 3), n, z, D, fitp=p)
    if fit == "outside":   # F in fixed point stays at the cube's face: the call runs, and finite
        assert np.isfinite(s).all()
    else:
        assert np.all(np.abs(s - o["re"].sum(1)) <= 1e-12 * o["abs"])
