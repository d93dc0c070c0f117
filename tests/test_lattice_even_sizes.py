"""Lattices of even n that is no power of two: rem(i) = i z 2^128 mod n vanishes inside the lattice,
at multiples of n's odd part, where a stepped stream must take its carry.  The 192-bit step in
exact integers, and points and untransformed sums on the GPU across such indices."""
import random

import numpy as np
import pytest

SIZES = [12, 3072, 999998, 1000000, 3 << 30]
M = 1 << 64


def odd_part(n):
    while n % 2 == 0:
        n //= 2
    return n


@pytest.mark.parametrize("rows", [1, 8, 32, 256])
@pytest.mark.parametrize("n", SIZES + [(1 << 31), (1 << 32) - 5, (1 << 32) - 2, 2, 3])
def test_stepped_state_is_exact(n, rows):
    """F by steps of `rows`, the third word started at i w and stepped by rows w, equals the exact
    floor(2^128 (i z mod n) / n) along streams across the zeros of rem and at the lattice's end."""
    rng = random.Random(n)
    o = odd_part(n)
    for _ in range(20):
        z = rng.randrange(1, n)
        while np.gcd(z, n) != 1:
            z = rng.randrange(1, n)
        fz, remz = divmod(z << 128, n)
        rq = (remz << 64) // n
        w = rq + (rq * n % M != 0)
        assert w == -(-(remz << 64) // n)
        step, step_w = ((rows * z % n) << 128) // n, rows * w % M
        for zero in (o, o * rng.randrange(1, n // o + 1), n):
            i = max(0, zero - rows * rng.randrange(0, 12))
            F, third = ((i * z % n) << 128) // n, i * w % M
            while i < min(n, zero + 12 * rows):
                assert F == ((i * z % n) << 128) // n
                total = (F << 64) + third + (step << 64) + step_w
                F, third = (total >> 64) % (1 << 128), total % M
                i += rows


def _vector(n, d):
    rng = random.Random(n + d)
    z = [1]
    while len(z) < d:
        v = rng.randrange(1, n)
        if np.gcd(v, n) == 1:
            z.append(v)
    return z


def _shifts(q, n, m, d):
    D = q.make_shifts(n % 997, m, d)
    D[0] = 0
    D[m - 1] = 1 << 52
    return D


@pytest.mark.gpu
@pytest.mark.parametrize("d,m", [(1, 1), (8, 4), (8, 32), (3, 20)])
@pytest.mark.parametrize("n", SIZES)
def test_points(n, d, m):
    import torch

    import oracle as O
    import paper_1811_11720_gb300 as q
    z, D = _vector(n, d), _shifts(q, n, m, d)
    r = q.rule(n, z, torch.from_numpy(D.astype(np.int64)).cuda())
    o = odd_part(n)
    for begin in {0, o, n // 2, max(0, n // 2 - 1), max(0, n - o - 100)}:
        count = min(n - begin, 30000)
        out = torch.empty(count, m, d, dtype=torch.float64, device="cuda")
        q.points(r, begin, count, out)
        want = O.points(n, z, D, begin, count)
        assert np.array_equal(out.cpu().numpy().view(np.uint64), want.view(np.uint64))


@pytest.mark.gpu
@pytest.mark.parametrize("m", [2, 20, 32])
@pytest.mark.parametrize("n", [12, 3072, 999998, 1000000])
def test_untransformed_sums(n, m):
    """Corner peak under no transform: its value at x = 0 is far from that at x = 1, so one sample
    at the wrong end of the interval shows at 1 / n."""
    import torch

    import oracle as O
    import paper_1811_11720_gb300 as q
    d = 1
    z, D = _vector(n, d), _shifts(q, n, m, d)
    c, w = np.full(d, 3.0), np.full(d, 0.5)
    f = q.Integrand.genz(3, c, w).device_struct("cuda")
    r = q.rule(n, z, torch.from_numpy(D.astype(np.int64)).cuda(), ("none",))
    for begin, end in [(0, n), (n // 2, n), (0, n // 2 + 1)]:
        ws = torch.empty(q.sums_workspace_bytes(r, False, begin, end), dtype=torch.uint8, device="cuda")
        out = torch.zeros(2 * m, dtype=torch.float64, device="cuda")
        q.sums(f, r, begin, end, ws, out)
        s = out.cpu().numpy().reshape(m, 2).sum(1)
        o = O.shift_sums(O.genz(3, c, w), ("none",), n, z, D, i0=begin, i1=end)
        assert np.all(np.abs(s - o["re"].sum(1)) <= 1e-12 * o["abs"])
