"""Host threads with streams and workspaces of their own, at sizes that need different amounts of the
same kernel's dynamic shared memory: every call is accepted and returns its own sums."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def _run(workers, calls):
    errors = []
    start = threading.Barrier(len(workers))

    def loop(fn):
        try:
            start.wait()
            for _ in range(calls):
                fn()
        except Exception as e:   # noqa: BLE001 - reported below
            errors.append(e)

    threads = [threading.Thread(target=loop, args=(w,)) for w in workers]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors[0]


@pytest.mark.parametrize("fam,shapes", [(4, [(256, 16), (64, 8), (32, 9), (128, 16)]), ("sector", [(256, 16), (64, 5)])])
def test_sums_from_several_threads(fam, shapes):
    import torch

    import paper_1811_11720_gb300 as q
    import workloads as W
    n = 257
    workers, checks = [], []
    for m, d in shapes:
        if fam == "sector":
            f = q.Integrand.polynomial(W.sector_like(d, d, 20, 20)).device_struct("cuda")
        else:
            f = q.Integrand.genz(fam, *W.genz_params(fam, d, 1)).device_struct("cuda")
        D = torch.from_numpy(q.make_shifts(m, m, d).astype(np.int64)).cuda()
        r = q.rule(n, [v * 2 + 1 for v in range(d)], D, ("korobov", 3))
        ws = torch.empty(q.sums_workspace_bytes(r, False, 0, n), dtype=torch.uint8, device="cuda")
        out, want = (torch.zeros(2 * m, dtype=torch.float64, device="cuda") for _ in range(2))
        q.sums(f, r, 0, n, ws, want)
        torch.cuda.synchronize()
        stream = torch.cuda.Stream()
        workers.append(lambda f=f, r=r, ws=ws, out=out, s=stream: q.sums(f, r, 0, n, ws, out, stream=s))
        checks.append((out, want))
    _run(workers, 3000)
    torch.cuda.synchronize()
    for out, want in checks:
        assert torch.equal(out, want)


def test_histograms_from_several_threads():
    import torch

    import paper_1811_11720_gb300 as q
    import workloads as W
    n = 257
    workers, checks = [], []
    for d, bins in [(16, 1280), (4, 100), (8, 1000)]:
        f = q.Integrand.genz(4, *W.genz_params(4, d, 1)).device_struct("cuda")
        sh = torch.from_numpy(q.make_shifts(d, 1, d)[0].astype(np.int64)).cuda()
        z = np.array([v * 2 + 1 for v in range(d)], dtype=np.uint64)
        ws = torch.empty(q.histogram_workspace_bytes(n, d, bins), dtype=torch.uint8, device="cuda")
        out, want = (torch.zeros(d, bins, dtype=torch.float64, device="cuda") for _ in range(2))
        q.histogram(f, n, z, sh, bins, want, ws)
        torch.cuda.synchronize()
        stream = torch.cuda.Stream()
        workers.append(lambda a=(f, n, z, sh, bins, out, ws), s=stream: q.histogram(*a, stream=s))
        checks.append((out, want))
    _run(workers, 2000)
    torch.cuda.synchronize()
    for out, want in checks:
        assert torch.equal(out, want)
