"""The block's search for its integral over the batch's tile sums: counts at the edges of its
rounds, uneven integrals, small and large blocks."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("count", [1, 2, 31, 32, 33, 255, 256, 257, 1025, 5000])
@pytest.mark.parametrize("m,spb", [(32, None), (32, 1), (1, 1), (3, 1)])
def test_every_integral_is_found(count, m, spb):
    import torch

    import paper_1811_11720_gb300 as q
    d = 2
    sizes = [3, 17, 101, 257]
    c, w = W.genz_params(4, d, 1)
    f = q.Integrand.genz(4, c, w).device_struct("cuda")
    D = q.make_shifts(m, m, d)
    Dd = torch.from_numpy(D.astype(np.int64)).cuda()
    rules = [q.rule(n, [1, 2], Dd, ("baker",)) for n in sizes]
    pick = np.random.default_rng(count).integers(0, len(sizes), count)
    b = q.Batch([(f, rules[k], 0, sizes[k]) for k in pick])
    cfg = None if spb is None else q.qmc_batch_config(spb, 8)
    ws = torch.empty(b.workspace_bytes(cfg), dtype=torch.uint8, device="cuda")
    out = torch.zeros(count, 4 * m, dtype=torch.float64, device="cuda")
    b.sums(ws, out, cfg=cfg)
    got = out.cpu().numpy()[:, :2 * m].reshape(count, m, 2).sum(2)
    for k, n in enumerate(sizes):
        o = O.shift_sums(O.genz(4, c, w), ("baker",), n, [1, 2], D)
        assert np.all(np.abs(got[pick == k] - o["re"].sum(1)) <= 1e-12 * o["abs"])
