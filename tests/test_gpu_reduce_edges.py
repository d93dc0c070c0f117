"""The fold of tile partials at the edges of its halving tree: 1 tile to several per thread, every
shift apart, against exact sums."""
from fractions import Fraction as Fr

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 3, 32])
@pytest.mark.parametrize("tiles", [1, 2, 3, 16, 31, 32, 33, 63, 64, 65, 127, 128, 129, 200, 255, 256, 257, 511, 513, 1000])
def test_fold_is_exact_to_two_words(tiles, m):
    import torch

    import paper_1811_11720_gb300 as q
    rng = np.random.default_rng(1000 * tiles + m)
    part = np.empty((2, tiles, m, 2))
    part[..., 0] = rng.standard_normal((2, tiles, m)) * 2.0 ** rng.integers(-30, 30, (2, tiles, m))
    part[..., 1] = part[..., 0] * 2.0 ** -53 * rng.uniform(-1, 1, (2, tiles, m))
    out = torch.zeros(4 * m, dtype=torch.float64, device="cuda")
    q.reduce_tiles(torch.from_numpy(part).cuda(), tiles, m, True, out)
    got = out.cpu().numpy().reshape(2, m, 2)
    for comp in range(2):
        for k in range(m):
            want = sum(Fr(float(v)) for v in part[comp, :, k].reshape(-1))
            size = np.abs(part[comp, :, k]).sum()
            err = abs(Fr(float(got[comp, k, 0])) + Fr(float(got[comp, k, 1])) - want)
            # each addition's own error is at most 2^-53 of the sizes, kept in the low word, whose
            # additions err by 2^-53 of what it holds
            assert err <= Fr(size) * (tiles + 16) ** 2 / 2 ** 106
            assert abs(got[comp, k, 1]) <= abs(got[comp, k, 0]) * 2.0 ** -52
