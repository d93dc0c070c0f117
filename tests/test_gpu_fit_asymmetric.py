"""Steep fit maps over the asymmetric Korobov maps with the fewest fraction bits: the coordinate's
absolute error times the fit's slope has to leave both polynomial families within the contract."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("tr", [("korobov", 6, 5), ("korobov", 5, 6), ("korobov", 1, 6), ("korobov", 6, 1)])
@pytest.mark.parametrize("steep", ["at 0", "at 1", "both"])
@pytest.mark.parametrize("fam,d,b", [("sector", 3, 2.5), ("sector", 5, 8.5), ("feynman", 3, 2.5), ("feynman", 5, 8.5)])
def test_sums(fam, d, b, steep, tr):
    import torch

    import paper_1811_11720_gb300 as q
    fl = W.sector_like(d, d, 60, 90, b=b) if fam == "sector" else W.feynman_regular(d, d=d, beta=0.6, b=b)
    fo = O.from_feynman(fl) if fam == "sector" else O.feynman_complex(fl)
    p = W.fit_params_example(d, 5)
    if steep != "at 1":
        p[:, 1], p[:, 3] = -0.002, 0.11    # p'(0) ~ 55
    if steep != "at 0":
        p[:, 0], p[:, 2] = 1.01, 0.3       # p'(1) ~ 30
    if steep == "both":
        p[:, 2], p[:, 3] = 0.15, 0.07      # p'(0) ~ 35, p'(1) ~ 15
    n, m = 4691, 16
    z = [1, 76, 306, 400, 17][:d]
    D = q.make_shifts(d, m, d)
    out = q.integrate_device(q.Integrand.polynomial(fl), n, z, torch.from_numpy(D.astype(np.int64)).cuda(), tr,
                             torch.from_numpy(p).cuda())
    s = out[1].cpu().numpy()
    o = O.shift_sums(fo, tr, n, z, D, fitp=p)
    worst = 0.0
    for got, want in [(s[:2 * m], o["re"])] + ([(s[2 * m:4 * m], o["im"])] if fam == "feynman" else []):
        worst = max(worst, np.max(np.abs(got.reshape(m, 2).sum(1) - want.sum(1)) / o["abs"]))
    assert worst <= 1e-12
