"""The block's shift table at its largest: many shifts and dimensions, and small blocks, for every
kind of family, single and batched, against the oracle."""
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


@pytest.mark.parametrize("fam,d,m", [(4, 16, 256), (1, 16, 300), ("sector", 8, 256), ("sector", 16, 128),
                                     ("sector", 5, 2), ("feynman", 6, 64), ("feynman", 6, 256), ("feynman", 8, 256),
                                     ("feynman", 3, 2)])
@pytest.mark.parametrize("tr", [("korobov", 3), ("baker",), ("korobov", 8)])
def test_sums_and_batches(fam, d, m, tr):
    import torch

    import paper_1811_11720_gb300 as q
    dev = torch.device("cuda:0")
    n = 1021
    z = np.arange(1, d + 1) * 76 % n
    D = q.make_shifts(d + m, m, d)
    f, fo = _integrand(q, fam, d)
    fd = f.device_struct(dev)
    r = q.rule(n, z, torch.from_numpy(D.astype(np.int64)).to(dev), tr)
    ws = torch.empty(q.sums_workspace_bytes(r, f.is_complex, 0, n), dtype=torch.uint8, device=dev)
    out = torch.zeros(4 * m, dtype=torch.float64, device=dev)
    q.sums(fd, r, 0, n, ws, out)
    s = out.cpu().numpy()
    o = O.shift_sums(fo, tr, n, z, D)
    for got, want in [(s[:2 * m], o["re"])] + ([(s[2 * m:], o["im"])] if f.is_complex else []):
        assert np.all(np.abs(got.reshape(m, 2).sum(1) - want.sum(1)) <= 1e-12 * o["abs"])
    if m > 256:
        return
    b = q.Batch([(fd, r, 0, n)] * 3)
    for cfg in [None] + ([q.qmc_batch_config(1, 16)] if fam in ("sector", "feynman") else []):
        bw = torch.empty(b.workspace_bytes(cfg), dtype=torch.uint8, device=dev)
        bs = torch.zeros(3, 4 * m, dtype=torch.float64, device=dev)
        b.sums(bw, bs, cfg=cfg)
        got = bs.cpu().numpy()
        assert np.array_equal(got[0], got[2])
        if cfg is None:
            assert np.array_equal(got[1], s)
        else:   # one stream a block: 2 to 256 threads
            assert np.all(np.abs((got[1] - s)[:2 * m].reshape(m, 2).sum(1)) <= 1e-12 * o["abs"])
