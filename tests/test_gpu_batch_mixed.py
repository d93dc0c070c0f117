"""Batches of several transform kinds: their launches overlap, and every integral's sums, results and
counters are those of a call of its own, run after run, on any stream and from a captured graph."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

KINDS = [("none",), ("baker",), ("korobov", 3), ("korobov", 1, 3), ("korobov", 8), ("sidi", 2)]


def _batch(q, torch, fam, sizes, m):
    import workloads as W
    entries, want = [], []
    for i, n in enumerate(sizes):
        d = 3 + i % 3
        if fam == "sector":
            f = q.Integrand.polynomial(W.sector_like(i, d, 40, 60)).device_struct("cuda")
        else:
            f = q.Integrand.genz(fam, *W.genz_params(fam, d, i)).device_struct("cuda")
        D = torch.from_numpy(q.make_shifts(i, m, d).astype(np.int64)).cuda()
        r = q.rule(n, [v * 2 + 1 for v in range(d)], D, KINDS[(5 * i) % len(KINDS)])
        ws = torch.empty(q.sums_workspace_bytes(r, False, 0, n), dtype=torch.uint8, device="cuda")
        s = torch.zeros(2 * m, dtype=torch.float64, device="cuda")
        q.sums(f, r, 0, n, ws, s)
        want.append(s)
        entries.append((f, r, 0, n))
    return q.Batch(entries), torch.stack(want)


@pytest.mark.parametrize("fam,sizes,m", [(4, [257, 1021, 101, 64, 4691, 31, 257], 32), (1, [1021] * 24, 8),
                                         ("sector", [101, 1021, 257, 31, 64, 101], 16), (3, [200003, 101, 101, 50021], 32)])
def test_overlapping_launches(fam, sizes, m):
    import torch

    import paper_1811_11720_gb300 as q
    b, want = _batch(q, torch, fam, sizes, m)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    with torch.cuda.stream(stream):
        ws = torch.empty(b.workspace_bytes(), dtype=torch.uint8, device="cuda")
        sums = torch.zeros(len(sizes), 4 * m, dtype=torch.float64, device="cuda")
        res = torch.zeros(len(sizes), 4, dtype=torch.float64, device="cuda")
        cnt = torch.zeros(len(sizes), 2, dtype=torch.int64, device="cuda")
        plan = b.plan(ws, stream=stream)
        for _ in range(100):
            sums.zero_()
            plan.run(sums, res, cnt, stream=stream)
            assert torch.equal(sums[:, :2 * m], want)
        first = res.clone()
        g = torch.cuda.CUDAGraph()
        with torch.cuda.graph(g, stream=stream):
            plan.run(sums, res, cnt, stream=torch.cuda.current_stream())
        for _ in range(50):
            sums.zero_()
            res.zero_()
            g.replay()
            assert torch.equal(sums[:, :2 * m], want) and torch.equal(res, first)
        assert int(cnt.abs().sum()) == 0
