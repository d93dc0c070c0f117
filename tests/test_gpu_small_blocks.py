"""Batches whose blocks have fewer threads than the integrand has dimensions (one or two streams of
one to three shifts): every family that batches, through the fixed-point forms and the FP64 ones."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


def _integrand(q, fam, d):
    if fam == "sector":
        fl = W.sector_like(d, d, 40, 60)
        return q.Integrand.polynomial(fl), O.from_feynman(fl)
    if fam == "feynman":
        fl = W.feynman_regular(d, d=d, beta=0.6)
        return q.Integrand.polynomial(fl), O.feynman_complex(fl)
    c, w = W.genz_params(fam, d, d)
    return q.Integrand.genz(fam, c, w), O.genz(fam, c, w)


@pytest.mark.parametrize("tr", [("none",), ("baker",), ("korobov", 3), ("korobov", 1, 3), ("korobov", 8)])
@pytest.mark.parametrize("m,spb", [(1, 1), (2, 1), (2, 2), (3, 1)])
@pytest.mark.parametrize("fam,d", [(1, 5), (1, 16), (2, 5), (2, 16), (3, 5), (3, 16), (4, 5), (4, 16),
                                   ("sector", 5), ("feynman", 5)])
def test_batch_of_small_blocks(fam, d, m, spb, tr):
    import torch

    import paper_1811_11720_gb300 as q
    n = 257
    z = [v for v in range(3, 3 + 7 * d, 7)]
    D = q.make_shifts(d + m, m, d)
    f, fo = _integrand(q, fam, d)
    r = q.rule(n, z, torch.from_numpy(D.astype(np.int64)).cuda(), tr)
    b = q.Batch([(f.device_struct("cuda"), r, 0, n)] * 2)
    cfg = q.qmc_batch_config(spb, 16)
    ws = torch.empty(b.workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    out = torch.zeros(2, 4 * m, dtype=torch.float64, device="cuda")
    b.sums(ws, out, cfg=cfg)
    got = out.cpu().numpy()
    assert np.array_equal(got[0], got[1])
    o = O.shift_sums(fo, tr, n, z, D)
    for s, want in [(got[0, :2 * m], o["re"])] + ([(got[0, 2 * m:], o["im"])] if f.is_complex else []):
        assert np.all(np.abs(s.reshape(m, 2).sum(1) - want.sum(1)) <= 1e-12 * o["abs"])
