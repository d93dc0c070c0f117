"""The complex family with U in the denominator, with and without a constant term to keep it from
zero, and to other powers: sums against the oracle."""
import numpy as np
import pytest

import oracle as O
import workloads as W

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("fit", [False, True])
@pytest.mark.parametrize("const_u", [0.0, 0.5, 40.0])
@pytest.mark.parametrize("a,b", [(1.0, 2.5), (0.5, 1.5), (2.0, 3.0), (-0.5, 2.0), (-1.0, 2.0), (-2.0, 3.0)])
@pytest.mark.parametrize("d", [3, 5, 6])
def test_powers_of_u(d, a, b, const_u, fit):
    import torch

    import paper_1811_11720_gb300 as q
    rng = np.random.default_rng(d)
    e0, e2 = np.zeros((1, d), np.int32), W.all_monomials(d, 2)
    ef = np.vstack([W.all_monomials(d, k) for k in (1, 2, 3)])
    cf = rng.uniform(0, 1, len(ef))
    U = W.Polynomial(np.concatenate([[const_u], rng.uniform(0.1, 1, len(e2))]), np.vstack([e0, e2]).astype(np.int32))
    F = W.Polynomial(np.concatenate([[0.5 * cf.sum()], cf]), np.vstack([e0, ef]).astype(np.int32))
    fl = W.FeynmanLike(U, F, a, b, 0.1, d)
    n, m = 4691, 16
    z = [1, 76, 306, 400, 17, 19][:d]
    D = q.make_shifts(d, m, d)
    p = W.fit_params_example(d, 3) if fit else None
    out = q.integrate_device(q.Integrand.polynomial(fl), n, z, torch.from_numpy(D.astype(np.int64)).cuda(),
                             ("korobov", 1), None if p is None else torch.from_numpy(p).cuda())
    s = out[1].cpu().numpy()
    o = O.shift_sums(O.feynman_complex(fl), ("korobov", 1), n, z, D, fitp=p)
    for got, want in [(s[:2 * m], o["re"]), (s[2 * m:4 * m], o["im"])]:
        assert np.all(np.abs(got.reshape(m, 2).sum(1) - want.sum(1)) <= 1e-12 * o["abs"])
