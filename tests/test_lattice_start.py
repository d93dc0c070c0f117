"""The closed-form start of a lattice stream (lattice_state_at): the quotient from the host's
reciprocal word with one conditional correction, restated in exact integers, and on the GPU
through qmc_points at the ends of the accepted range of n and i."""
import random

import numpy as np
import pytest

SIZES = [2, 3, 7, 1021, (1 << 31) - 1, (1 << 32) - 5, (1 << 32) + 15, (1 << 61) - 1, (1 << 62) + 1, (1 << 63) - 25, (1 << 63) - 1]


def state_at(i, z, n):
    """(F, rem) as the kernel forms them, in 64-bit words."""
    M = (1 << 64) - 1
    fz, remz = divmod(z << 128, n)
    rq = (remz << 64) // n
    lo = (i * (fz & M)) & M
    add = (i * rq) >> 64
    r = -((lo + add) & M) * n & M
    if r >= n:
        r, add = r - n, add + 1
    f_lo = (lo + add) & M
    return (((((i * (fz & M)) >> 64) + i * (fz >> 64) + (f_lo < lo)) & M) << 64) | f_lo, r


@pytest.mark.parametrize("n", SIZES)
def test_closed_form_start_is_exact(n):
    rng = random.Random(n)
    for _ in range(200):
        z = rng.randrange(1, n)
        for i in (0, 1, n - 1, rng.randrange(n), (1 << 63) - 1 - rng.randrange(1000)):
            F, rem = divmod(((i * z) % n) << 128, n)
            assert state_at(i, z, n) == (F, rem)
    remz = (z << 128) % n   # what a step adds to the remainder
    assert -((z << 128) // n) * n % (1 << 64) == remz


@pytest.mark.gpu
@pytest.mark.parametrize("n", SIZES)
@pytest.mark.parametrize("d,m", [(1, 1), (3, 2), (7, 37)])
def test_points_at_the_ends_of_the_range(n, d, m):
    import torch

    import oracle as O
    import paper_1811_11720_gb300 as q
    rng = random.Random(n + d)
    z = []
    while len(z) < d:
        v = rng.randrange(1, n)
        if np.gcd(v, n) == 1:
            z.append(v)
    D = q.make_shifts(n % 1000, m, d)
    Dd = torch.from_numpy(D.astype(np.int64)).cuda()
    count = min(n, 5)
    for begin in {0, n - count}:
        out = torch.full((count + 1, m, d), -1.0, dtype=torch.float64, device="cuda")
        q.points(q.rule(n, z, Dd), begin, count, out)
        got = out.cpu().numpy()
        want = [[[O.point_py((i * z[j]) % n, n, int(D[k, j])) for j in range(d)] for k in range(m)]
                for i in range(begin, begin + count)]
        assert np.array_equal(got[:count], np.array(want))
        assert (got[count:] == -1.0).all()


@pytest.mark.gpu
@pytest.mark.parametrize("n,begin,count,d,m", [
    (7, 0, 7, 1, 1), (1021, 3, 1018, 2, 3), (1021, 0, 1021, 5, 300), (10007, 0, 10007, 16, 16),
    (108863, 1, 108862, 3, 1), ((1 << 32) - 5, (1 << 32) - 70005, 70000, 1, 2),
    ((1 << 32) + 15, (1 << 32) - 70000, 70015, 1, 2)])
def test_every_point_of_a_long_run(n, begin, count, d, m):
    """All steps of the stepped streams, at the ends of the lattice, against the C oracle."""
    import torch

    import oracle as O
    import paper_1811_11720_gb300 as q
    z = [1, 76, 306, 400, 17, 19, 23, 29, 31, 37, 41, 43, 47, 53, 59, 61][:d]
    z = [v % n for v in z]
    D = q.make_shifts(n % 997, m, d)
    D[0, 0] = 0                       # exact multiples of 1/n, and 0 itself
    out = torch.empty(count, m, d, dtype=torch.float64, device="cuda")
    q.points(q.rule(n, z, torch.from_numpy(D.astype(np.int64)).cuda()), begin, count, out)
    want = O.points(n, z, D, begin, count)
    assert np.array_equal(out.cpu().numpy().view(np.uint64), want.view(np.uint64))
