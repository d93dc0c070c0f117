"""Sector integrands whose F^-b sits in the corner where U vanishes: U from fixed point only where its
error is small against U itself, through every map, fitted and not, compiled-in and run-time
dimensions."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


def _integrand(d, degu, degf, ratio, b):
    rng = np.random.default_rng(100 * d + 10 * degu + degf)
    eu = W.all_monomials(d, degu)
    ef = np.vstack([W.all_monomials(d, k) for k in range(1, degf + 1)])
    nterm = 120
    cf = rng.uniform(0, 1, nterm)
    U = W.Polynomial(rng.uniform(0, 1, nterm), eu[rng.integers(0, len(eu), nterm)].astype(np.int32))
    F = W.Polynomial(np.concatenate([[ratio * cf.sum()], cf]),
                     np.vstack([np.zeros((1, d), np.int32), ef[rng.integers(0, len(ef), nterm)]]).astype(np.int32))
    return W.FeynmanLike(U, F, 1.0, b, 0.0, d)


@pytest.mark.parametrize("tr", [("none",), ("baker",), ("korobov", 3), ("korobov", 1, 4), ("korobov", 6, 5), ("korobov", 8)])
@pytest.mark.parametrize("ratio,b", [(0.1, 2.5), (1e-2, 4.5), (1e-3, 8.5), (5e-4, 15.5)])
@pytest.mark.parametrize("d,degu,degf", [(2, 2, 1), (3, 2, 1), (3, 3, 1), (4, 2, 3), (5, 3, 1), (8, 2, 1), (8, 2, 3), (10, 2, 2)])
def test_sums(d, degu, degf, ratio, b, tr):
    import torch

    import paper_1811_11720_gb300 as q
    n, m = 4691, 16
    z = [1, 76, 306, 400, 17, 19, 23, 29, 31, 37][:d]
    D = q.make_shifts(d, m, d)
    fl = _integrand(d, degu, degf, ratio, b)
    # F and U within 2^-42 of themselves, F to the power b, and the coordinates' own absolute error
    # (4 units of 2^-58) where F^-b sits, x ~ c0 / (b B)
    tol = (b + 1) * 2.0 ** -42 + 3 * 2.0 ** -56 * b / ratio
    for fit in (None, W.fit_params_example(d, 3)):
        out = q.integrate_device(q.Integrand.polynomial(fl), n, z, torch.from_numpy(D.astype(np.int64)).cuda(), tr,
                                 None if fit is None else torch.from_numpy(fit).cuda())
        s = out[1].cpu().numpy()[:2 * m].reshape(m, 2).sum(1)
        o = O.shift_sums(O.from_feynman(fl), tr, n, z, D, fitp=fit)
        assert np.all(np.abs(s - o["re"].sum(1)) <= tol * o["abs"]), (fit is not None)
