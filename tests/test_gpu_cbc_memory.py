"""qmc_cbc_korobov's device memory is the call's own; the plans it keeps serve several threads and
lengths."""
import threading

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SIZES = [1021, 8311, 108863, 1072187]


def test_memory_is_freed_before_returning():
    import torch

    import paper_1811_11720_gb300 as q
    for n in SIZES[::-1]:   # cuFFT's and the context's own first-call allocations, the largest first
        q.cbc_korobov(n, 3)
    torch.cuda.synchronize()
    before = torch.cuda.mem_get_info()[0]
    for n in SIZES + SIZES[::-1]:
        q.cbc_korobov(n, 3)
        # what the call needs at n = 1,072,187 is 43 MB; an allocation granule or two may move
        assert before - torch.cuda.mem_get_info()[0] <= 4 << 20, n


def test_threads_and_lengths():
    import torch

    import paper_1811_11720_gb300 as q
    want = {n: q.cbc_korobov(n, 5) for n in SIZES[:3]}
    bad = []

    def loop(k):
        s = torch.cuda.Stream()
        for i in range(12):
            n = SIZES[(i + k) % 3]
            z, e2 = q.cbc_korobov(n, 5, stream=s)
            if not (np.array_equal(z, want[n][0]) and np.array_equal(e2, want[n][1])):
                bad.append((k, n))

    threads = [threading.Thread(target=loop, args=(k,)) for k in range(4)]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not bad
