"""Sector integrands under a fit map that leaves the unit interval: the value there is the
integrand's own, U^a F^-b at p(x) outside the cube, as the oracle has it."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tr", [("none",), ("korobov", 3), ("korobov", 2, 3)])
@pytest.mark.parametrize("which", ["one dimension", "all"])
@pytest.mark.parametrize("d,nu,nf,b", [(2, 30, 60, 2.5), (3, 100, 150, 2.5), (5, 100, 200, 2.5), (8, 200, 400, 2.5),
                                       (5, 100, 200, 2.0), (11, 400, 500, 2.5)])
def test_outside_the_cube(d, nu, nf, b, which, tr):
    import torch

    import paper_1811_11720_gb300 as q
    fl = W.sector_like(d, d, nu, nf, b=b)
    p = W.fit_params_example(d, 5)
    rows = slice(0, 1) if which == "one dimension" else slice(None)
    p[rows, 2:4], p[rows, 4], p[rows, 5] = 0.0, 1.5, 1.0   # p(x) = x (1.5 + x (1 - 1.5 x)): up to 1.3
    n, m = 1021, 16
    z = np.arange(1, d + 1) * 76 % n
    D = q.make_shifts(d, m, d)
    out = q.integrate_device(q.Integrand.polynomial(fl), n, z, torch.from_numpy(D.astype(np.int64)).cuda(), tr,
                             torch.from_numpy(p).cuda())
    s = out[1].cpu().numpy()[:2 * m].reshape(m, 2).sum(1)
    o = O.shift_sums(O.from_feynman(fl), tr, n, z, D, fitp=p)
    assert np.all(np.abs(s - o["re"].sum(1)) <= 1e-12 * o["abs"])
