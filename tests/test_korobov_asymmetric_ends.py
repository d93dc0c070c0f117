"""Integrands that live at one end of the cube under the asymmetric Korobov map, whose coordinate has
to be relative there: sharp corner and C0 peaks on both sides of the limit on their coefficients,
and polynomials with nothing to bound them away from zero."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu

N, M = 20011, 16
# What FP64 itself leaves: x to a few units of 2^-53 near 0 times its power (at most 14 times 7), and
# the alternating sums of the map's coefficients, up to 60 units of 2^-54 of values down to 0.03
# (orders 6 and 1) where the two halves meet.
TOL = 1e-13


def _errors(f, fo, tr, d, fit=None):
    import torch

    import paper_1811_11720_gb300 as q
    z = [1, 76, 306, 400, 17, 19][:d]
    D = q.make_shifts(d, M, d)
    out = q.integrate_device(f, N, z, torch.from_numpy(D.astype(np.int64)).cuda(), tr,
                             None if fit is None else torch.from_numpy(fit).cuda())
    s = out[1].cpu().numpy()
    o = O.shift_sums(fo, tr, N, z, D, fitp=fit)
    parts = [(s[:2 * M], o["re"])] + ([(s[2 * M:4 * M], o["im"])] if f.is_complex else [])
    return max(np.max(np.abs(a.reshape(M, 2).sum(1) - b.sum(1)) / o["abs"]) for a, b in parts)


@pytest.mark.parametrize("tr", [("korobov", 1, 3), ("korobov", 3, 1), ("korobov", 2, 5), ("korobov", 6, 1),
                                ("korobov", 5, 6)])
@pytest.mark.parametrize("fit", [False, True])
@pytest.mark.parametrize("d", [1, 2, 5])
@pytest.mark.parametrize("fam", [3, 5])
@pytest.mark.parametrize("csum", [31.0, 32.0, 1e3, 1e6, 1e8])
def test_sharp_peak_at_the_origin(fam, csum, d, tr, fit):
    import paper_1811_11720_gb300 as q
    c = np.linspace(1.0, 1.5, d)
    c, w = csum * c / c.sum(), np.zeros(d)
    p = W.fit_params_example(d, 2) if fit else None
    if fam == 5 and csum > 1e3 and d > 1:
        pytest.skip("no sample near the origin: exp(-s) for s in the hundreds, where the rounding of s alone is 1e-13")
    assert _errors(q.Integrand.genz(fam, c, w), O.genz(fam, c, w), tr, d, p) <= TOL


def _poly(rows, coef):
    return W.Polynomial(np.array(coef, float), np.array(rows, np.int32))


@pytest.mark.parametrize("tr", [("korobov", 1, 3), ("korobov", 3, 1), ("korobov", 2, 5)])
@pytest.mark.parametrize("b", [0.5, 1.5, 2.5])
@pytest.mark.parametrize("kind", ["sector, no constant", "sector, U in the denominator", "complex, no constant"])
def test_polynomials_singular_at_the_origin(kind, b, tr):
    import paper_1811_11720_gb300 as q
    d = 3
    e1, e2 = W.all_monomials(d, 1), W.all_monomials(d, 2)
    lin, quad = _poly(e1, [0.5, 0.75, 1.0]), _poly(e2, np.linspace(0.1, 1, len(e2)))
    many = _poly(np.vstack([np.zeros((1, d), np.int32)] + [e1, e2] * 8), np.linspace(0.5, 1.0, 1 + 8 * (len(e1) + len(e2))))
    if kind == "sector, no constant":
        fl = W.FeynmanLike(quad, lin, 1.0, b, 0.0, d)
        e = _errors(q.Integrand.polynomial(fl), O.from_feynman(fl), tr, d)
    elif kind == "sector, U in the denominator":
        fl = W.FeynmanLike(lin, many, -b, 1.5, 0.0, d)
        e = _errors(q.Integrand.polynomial(fl), O.from_feynman(fl), tr, d)
    else:
        fl = W.FeynmanLike(quad, _poly(np.vstack([e1, e2]), [0.5, 0.75, 1.0] + [0.25] * len(e2)), 1.0, b, 0.1, d)
        e = _errors(q.Integrand.polynomial(fl), O.feynman_complex(fl), tr, d)
    assert e <= TOL
