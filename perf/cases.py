"""What this integrator's speed is judged on: twelve calls a user's program makes, from the
smallest adaptive integral to a full Genz lattice, through the package's public functions.

A case is a dict of plain values; ``kind`` says which call it is:
  sums       per-shift lattice sums and their mean and error, device-resident (q.sums, q.finalize)
  integrate  the host-buffer call (q.integrate): adaptive, or on one lattice with the
             variance-reduction fit
  batch      many sector integrals in one launch (q.Batch plan)
  serve      requests with error goals through the serving loop (q.Server)
  points     the shifted lattice points themselves (q.points)
  cbc        construction of a generating vector (q.cbc_korobov)

``exact`` evaluates the same definitions with plain torch in FP64: lattice points
frac(i z/n + D 2^-53), the periodizing transforms from their closed forms, the integrands
term by term, sums by torch.
"""
from __future__ import annotations

import itertools
import math
import os

import numpy as np
import torch

import paper_1811_11720_gb300 as q

GENZ = {"oscillatory": 1, "product_peak": 2, "corner_peak": 3, "gaussian": 4, "c0": 5,
        "discontinuous": 6}
# ||c||_1 of the Genz families (the paper's difficulty table)
DIFFICULTY = {1: 6.0, 2: 18.0, 3: 2.2, 4: 15.2, 5: 16.1, 6: 16.4}
SHIFT_SEED = 7919   # times the case's seed: the seed of the shift stream
DEV = "cuda:0"

_table = None


def _rows():
    """The shipped generating vectors: {n: (z_1, .., z_10)}, ascending in n."""
    global _table
    if _table is None:
        path = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(q.__file__))),
                            "tables", "cbc_korobov_a2_s10.txt")
        with open(path) as fh:
            rows = [[int(t) for t in line.split()] for line in fh
                    if line.strip() and not line.startswith("#")]
        _table = {r[0]: tuple(r[1:]) for r in sorted(rows)}
    return _table


def _next_n(want: float) -> int:
    return next(n for n in _rows() if n >= want)


# ---- the cases --------------------------------------------------------------------------
def _sums(family, d, transform, n, m, r0=0, r1=0, terms=0):
    return {"kind": "sums", "family": family, "d": d, "transform": transform, "r0": r0, "r1": r1,
            "n": _next_n(n), "m": m, "terms": terms}


def _integrate(family, d, n, m, epsrel=0.0, maxeval=0, fit=False, terms=0):
    return {"kind": "integrate", "family": family, "d": d, "transform": "korobov", "r0": 3, "r1": 3,
            "n": _next_n(n), "m": m, "epsrel": epsrel, "maxeval": maxeval, "fit": fit, "terms": terms}


def listed():
    return [
        # One adaptive integral at the library's default starting size (minn 8191, 32
        # shifts) with a modest goal: what an interactive user waits for.
        {"name": "integrate_small_d5", **_integrate("oscillatory", 5, 8191, 32, 1e-6, 20_000_000)},
        # The d = 4 product peak on n = 108,863 with 16 shifts: the latency of one small
        # device-resident integral.
        {"name": "peak_d4_n1e5", **_sums("product_peak", 4, "korobov", 108863, 16, 3, 3)},
        # The Genz benchmark's body: families x {baker, Korobov-1..4} x d = 6, 8, 10 at m = 32,
        # here its cheapest map at n ~ 1e6 and its most usual one at n ~ 1e7.
        {"name": "osc_d6_baker_n1e6", **_sums("oscillatory", 6, "baker", 1072187, 32)},
        {"name": "gaussian_d10_kor3_n1e7", **_sums("gaussian", 10, "korobov", 10560653, 32, 3, 3)},
        # An asymmetric Korobov map (for integrands singular at one end only) with a number of
        # shifts that is no power of two, as an accuracy run picks it.
        {"name": "corner_d8_kor1x3_m20", **_sums("corner_peak", 8, "korobov", 256687, 20, 1, 3)},
        # A contour-deformed Feynman-parameter integral: complex, d = 5, 32 shifts.
        {"name": "feynman_d5_n1e6", **_sums("feynman", 5, "korobov", 1072187, 32, 3, 3)},
        # A large sector integrand, 200 + 200 monomials in 8 variables.
        {"name": "sector_d8_n1e6", **_sums("sector", 8, "korobov", 1072187, 32, 3, 3, 200)},
        # The same kind of integrand through the host call with the variance-reduction fit: a
        # histogram pass over n = 108,863 points, the fit, then the fitted lattice.
        {"name": "sector_d5_fit", **_integrate("sector", 5, 108863, 32, fit=True, terms=100)},
        # An amplitude's worth of sector integrals in one launch: uneven dimensions, sizes and
        # lattices, the fit map on half of them.
        {"name": "batch_sector_256", "kind": "batch", "count": 256, "m": 32, "nmin": 10000,
         "nmax": 100000},
        # A serving burst: 128 small integrals with goals from 1e-6 to 1e-3 at once.
        {"name": "serve_small_128", "kind": "serve", "count": 128, "m": 32, "maxeval": 4000000},
        # The points of a lattice written out, for a user's own integrand.
        {"name": "points_d8_m4", "kind": "points", "d": 8, "m": 4, "n": 1072187, "count": 1072187},
        # A generating vector for a size in the middle of the table.
        {"name": "cbc_n1e5_s10", "kind": "cbc", "n": 108863, "s": 10},
    ]


def _log_uniform(rng, lo, hi):
    return math.exp(rng.uniform(math.log(lo), math.log(hi)))


def draw(rng):
    kind = rng.choice(["genz", "genz", "genz", "genz", "poly", "poly", "integrate", "fit", "batch",
                       "serve", "points", "cbc"])
    if kind == "genz":
        d = rng.randint(3, 10)
        tr, r0, r1 = rng.choice([("korobov", r, r) for r in (1, 2, 3, 3, 4)] +
                                [("baker", 0, 0)] * 2 + [("korobov", *rng.sample(range(1, 5), 2))] +
                                [("sidi", rng.randint(1, 3), 0)])
        m = rng.choice([8, 10, 16, 20, 32, 32, 32, 50, 64])
        slow = tr == "sidi" or r0 != r1
        n = _log_uniform(rng, 1e3, 1e6 if slow else 8e6)
        return _sums(rng.choice(sorted(GENZ)), d, tr, n, m, r0, r1)
    if kind == "poly":
        m = rng.choice([16, 32, 32, 64])
        r = rng.choice([1, 2, 3, 3])
        if rng.random() < 0.5:
            return _sums("feynman", rng.randint(3, 6), "korobov", _log_uniform(rng, 3e3, 4e5), m, r, r)
        return _sums("sector", rng.randint(3, 8), "korobov", _log_uniform(rng, 3e3, 9e5), m, r, r,
                     rng.randint(10, 400))
    if kind == "integrate":
        return _integrate(rng.choice(["oscillatory", "gaussian", "product_peak", "corner_peak"]),
                          rng.randint(3, 8), rng.choice([1021, 8191, 30000]), rng.choice([16, 32]),
                          10 ** rng.uniform(-7, -4), 20_000_000)
    if kind == "fit":
        return _integrate("sector", rng.randint(3, 8), _log_uniform(rng, 1e4, 4e5), 32, fit=True,
                          terms=rng.randint(10, 400))
    if kind == "batch":
        return {"kind": "batch", "count": rng.randint(40, 256), "m": 32, "nmin": 10000,
                "nmax": rng.randint(30000, 100000)}
    if kind == "serve":
        return {"kind": "serve", "count": rng.randint(8, 128), "m": 32, "maxeval": 4000000}
    if kind == "points":
        d, m = rng.randint(2, 10), rng.choice([1, 3, 8, 16])
        n = _next_n(_log_uniform(rng, 1e3, 4e7 / (m * d)))
        return {"kind": "points", "d": d, "m": m, "n": n, "count": n - rng.randint(0, n // 8)}
    return {"kind": "cbc", "n": _next_n(_log_uniform(rng, 1e3, 1e6)), "s": rng.randint(3, 10)}


# ---- inputs -----------------------------------------------------------------------------
def _monomials(d, degree):
    out = np.zeros((math.comb(d + degree - 1, degree), d), np.int32)
    for row, combo in zip(out, itertools.combinations_with_replacement(range(d), degree)):
        for v in combo:
            row[v] += 1
    return out


def _params(family, d, rng, terms_u=0, terms_f=0):
    """The integrand's arrays, drawn as the paper's workloads draw them."""
    if family in GENZ:
        a = np.maximum(rng.uniform(0, 1, d), 1e-12)
        return {"c": DIFFICULTY[GENZ[family]] * a / a.sum(), "w": rng.uniform(0, 1, d)}
    if family == "sector":
        # U: quadratic monomials, F: a constant and cubic ones, positive coefficients
        e2, e3 = _monomials(d, 2), _monomials(d, 3)
        cf = rng.uniform(0, 1, terms_f)
        cf[0] = 0.25 + 0.5 * cf[0]
        return {"ucoef": rng.uniform(0, 1, terms_u), "uexp": e2[rng.integers(0, len(e2), terms_u)],
                "fcoef": cf, "fexp": np.vstack([np.zeros((1, d), np.int32),
                                                e3[rng.integers(0, len(e3), terms_f - 1)]])}
    # Feynman-like: U all quadratic monomials, F = 1 - 0.95 sum x(1-x) + small cubic terms,
    # which changes sign inside the cube and is positive on its faces
    e2, e3 = _monomials(d, 2), _monomials(d, 3)
    eye = np.eye(d, dtype=np.int32)
    return {"ucoef": rng.uniform(-1, 2, len(e2)), "uexp": e2,
            "fcoef": np.concatenate([[1.0], np.full(d, -0.95), np.full(d, 0.95),
                                     5e-4 * rng.uniform(-1, 2, len(e3))]),
            "fexp": np.vstack([np.zeros((1, d), np.int32), eye, 2 * eye, e3])}


def _integrand(family, d, p):
    if family in GENZ:
        return q.Integrand.genz(GENZ[family], p["c"], p["w"])
    return q.Integrand(family, d, **p, pa=1.0, pb=2.5, lam=0.5 if family == "feynman" else 0.0)


def _transform(case):
    t = case["transform"]
    return (t, case["r0"], case["r1"]) if t == "korobov" else (t, case["r0"]) if t == "sidi" else (t,)


def _case_params(case, seed):
    return _params(case["family"], case["d"], np.random.default_rng(seed), case["terms"], case["terms"])


def _batch_items(case, seed):
    """(d, integrand arrays, n, shift seed, PolySingular parameters or None) per integral."""
    rng = np.random.default_rng(seed)
    for i in range(case["count"]):
        d = int(rng.integers(3, 9))
        p = _params("sector", d, rng, int(rng.integers(10, 401)), int(rng.integers(10, 401)))
        n = _next_n(math.exp(rng.uniform(math.log(case["nmin"]), math.log(case["nmax"]))))
        fit = None
        if i % 2:
            fit = np.stack([1.001 + rng.uniform(0.05, 1, d), -0.001 - rng.uniform(0.05, 1, d),
                            rng.uniform(0, 0.3, d), rng.uniform(0, 0.3, d),
                            rng.uniform(0.2, 0.6, d), rng.uniform(-0.1, 0.1, d)], axis=1)
        yield d, p, n, SHIFT_SEED * seed + 31 * i, fit


def _requests(case, seed):
    """(family, c, w, relative goal, shift seed): d = 4 product peaks and Gaussians in turn."""
    rng = np.random.default_rng(seed)
    for i in range(case["count"]):
        if i % 2 == 0:
            family, c, w = "product_peak", np.full(4, 5.0), rng.uniform(0, 1, 4)
        else:
            family, (c, w) = "gaussian", _params("gaussian", 4, rng).values()
        yield family, c, w, float(10 ** rng.uniform(-6, -3)), SHIFT_SEED * seed + i


def _device_shifts(seed, m, d):
    return torch.from_numpy(q.make_shifts(seed, m, d).astype(np.int64)).to(DEV)


def prepare(case, seed):
    kind = case["kind"]
    if kind == "cbc":
        # the size is the whole input; the weight varies a little with the seed so that
        # inputs differ, by less than what changes a choice
        return {"kind": kind, "n": case["n"], "s": case["s"], "gamma": _gamma(seed)}
    table = q.GenvecTable.load()
    if kind == "points":
        rule = q.rule(case["n"], table.z_for(case["n"])[:case["d"]],
                      _device_shifts(SHIFT_SEED * seed, case["m"], case["d"]))
        out = torch.empty(case["count"], case["m"], case["d"], dtype=torch.float64, device=DEV)
        return {"kind": kind, "rule": rule, "begin": (case["n"] - case["count"]) // 2, "out": out}
    if kind == "serve":
        server = q.Server(table, memory_budget=1 << 28, max_slots=256, m=case["m"],
                          transform=("korobov", 3), step_evaluations=1 << 25)
        reqs = [(q.Integrand.genz(GENZ[f], c, w), eps, s) for f, c, w, eps, s in _requests(case, seed)]
        return {"kind": kind, "server": server, "requests": reqs, "maxeval": case["maxeval"]}
    if kind == "batch":
        entries = []
        for d, p, n, s, fit in _batch_items(case, seed):
            fs = _integrand("sector", d, p).device_struct(DEV)
            fit_dev = None if fit is None else torch.from_numpy(fit).to(DEV)
            entries.append((fs, q.rule(n, table.z_for(n)[:d], _device_shifts(s, case["m"], d),
                                       ("korobov", 3), fit_dev), 0, n))
        batch = q.Batch(entries)
        ws = torch.empty(batch.workspace_bytes(), dtype=torch.uint8, device=DEV)
        return {"kind": kind, "plan": batch.plan(ws),
                "sums": torch.zeros(case["count"], 4 * case["m"], dtype=torch.float64, device=DEV),
                "results": torch.zeros(case["count"], 4, dtype=torch.float64, device=DEV)}
    f = _integrand(case["family"], case["d"], _case_params(case, seed))
    if kind == "integrate":
        opts = (q.options(epsrel=case["epsrel"], epsabs=0.0, maxeval=case["maxeval"])
                if case["epsrel"] else None)
        return {"kind": kind, "f": f, "table": table, "n": case["n"], "m": case["m"],
                "transform": _transform(case), "seed": SHIFT_SEED * seed, "opts": opts,
                "fit": q.fit_options() if case["fit"] else None}
    n, m = case["n"], case["m"]
    rule = q.rule(n, table.z_for(n)[:case["d"]], _device_shifts(SHIFT_SEED * seed, m, case["d"]),
                  _transform(case))
    parts = 2 if f.is_complex else 1
    return {"kind": kind, "f": f.device_struct(DEV), "rule": rule, "n": n, "m": m,
            "complex": f.is_complex,
            "ws": torch.empty(q.sums_workspace_bytes(rule, f.is_complex, 0, n), dtype=torch.uint8,
                              device=DEV),
            "sums": torch.empty(2 * parts * m, dtype=torch.float64, device=DEV),
            "counters": torch.zeros(2, dtype=torch.int64, device=DEV),
            "result": torch.empty(4, dtype=torch.float64, device=DEV),
            "Q": torch.empty(parts, m, dtype=torch.float64, device=DEV)}


# ---- one pass ---------------------------------------------------------------------------
def run(s):
    kind = s["kind"]
    if kind == "sums":
        q.sums(s["f"], s["rule"], 0, s["n"], s["ws"], s["sums"], s["counters"])
        q.finalize(s["sums"], s["m"], s["n"], s["complex"], s["result"], s["Q"])
        return {"result": s["result"], "Q": s["Q"]}
    if kind == "integrate":
        o = q.integrate(s["f"], s["table"], s["n"], s["m"], s["transform"], fit=s["fit"],
                        seed=s["seed"], opts=s["opts"])
        return {"result": np.array([o["value"], o["err"]]), "n": o["n"], "m": o["m"],
                "evaluations": o["evaluations"]}
    if kind == "batch":
        s["plan"].run(s["sums"], s["results"])
        return {"results": s["results"], "sums": s["sums"]}
    if kind == "serve":
        srv = s["server"]
        ids = [srv.submit(f, epsrel=eps, minn=1021, maxeval=s["maxeval"], seed=seed)
               for f, eps, seed in s["requests"]]
        waiting = set(ids)
        while waiting:
            srv.step()
            waiting.difference_update(srv.completed())
        done = [srv.status(i) for i in ids]
        return {"result": np.array([[o["value"], o["err"]] for o in done]),
                "n": np.array([o["n"] for o in done]),
                "evaluations": np.array([o["evaluations"] for o in done])}
    if kind == "points":
        return q.points(s["rule"], s["begin"], s["out"].shape[0], s["out"])
    z, e2 = q.cbc_korobov(s["n"], s["s"], gamma=s["gamma"])
    return {"z": z.astype(np.int64), "e2": e2}


# ---- what a pass cannot do without ------------------------------------------------------
def _flops_per_eval(family, d, transform, r0, r1, terms=0):
    """FP64 operations of one evaluation as the formulas are written."""
    per_dim = {"korobov": 3 * max(r0, r1) + r0 + r1 + 2, "baker": 3, "sidi": 4 * r0 + 20, "none": 0}
    fl = d * (2 + per_dim[transform])
    quad, cubic = math.comb(d + 2, 2), math.comb(d + 3, 3)
    if family == "sector":
        return fl + 2 * (min(quad, terms) + min(cubic, terms)) + 10
    if family == "feynman":
        # F, U, their gradients and the Hessian at x, the Taylor terms at z, det J, the power
        return fl + 2 * (2 * cubic + 3 * quad) + d * d * (d + 1) + 8 * d ** 3 // 3 + 60
    return fl + {"oscillatory": 2, "corner_peak": 2}.get(family, 4) * d + 12


def work(case):
    kind = case["kind"]
    if kind == "cbc":
        half = case["n"] // 2
        return {"bytes": 8 * half * case["s"], "flops": case["s"] * half * (5 * math.log2(half) + 10)}
    if kind == "points":
        out = 8 * case["count"] * case["m"] * case["d"]
        return {"bytes": out, "flops": 2 * out / 8}
    if kind == "serve":
        return {"bytes": case["count"] * (64 + 32 * case["m"]),
                "flops": case["count"] * 4000 * case["m"] * _flops_per_eval("gaussian", 4, "korobov", 3, 3)}
    if kind == "batch":
        mean_n = (case["nmax"] - case["nmin"]) / math.log(case["nmax"] / case["nmin"])
        return {"bytes": case["count"] * (400 * 28 + 44 * case["m"]),
                "flops": case["count"] * mean_n * case["m"] * _flops_per_eval("sector", 6, "korobov", 3, 3, 200)}
    d, m = case["d"], case["m"]
    evals = case["n"] * m + (108863 if case.get("fit") else 0)
    return {"bytes": 8 * m * (d + 1) + 16 * d + 56 * case["terms"] + 32,
            "flops": evals * _flops_per_eval(case["family"], d, case["transform"], case["r0"], case["r1"],
                                             case["terms"])}


# ---- the definitions in plain torch, FP64 -----------------------------------------------
def _gamma(seed):
    return 0.1 * (1.0 + 1e-9 * (seed % 1000))


def _splitmix_shifts(seed, m, d):
    """D_kj: outputs of the SplitMix64 stream, top 53 bits."""
    with np.errstate(over="ignore"):
        x = np.uint64(seed & (2 ** 64 - 1)) + np.arange(1, m * d + 1, dtype=np.uint64) * np.uint64(0x9E3779B97F4A7C15)
        x = (x ^ (x >> np.uint64(30))) * np.uint64(0xBF58476D1CE4E5B9)
        x = (x ^ (x >> np.uint64(27))) * np.uint64(0x94D049BB133111EB)
        x = x ^ (x >> np.uint64(31))
    return (x >> np.uint64(11)).reshape(m, d)


def _coordinate(n, z, D, begin, count):
    """frac(i z/n + D 2^-53) for begin <= i < begin + count (i z < 2^63 for the table's n)."""
    r = (torch.arange(begin, begin + count, device=DEV) * int(z)) % n
    u = r.double() / n + float(D) * 2.0 ** -53
    return u - torch.floor(u)


def _map(case, u):
    """(phi(u), phi'(u)) of the case's transform."""
    t, r0, r1 = case["transform"], case["r0"], case["r1"]
    if t == "none":
        return u, None
    if t == "baker":
        return 1 - (2 * u - 1).abs(), None
    if t == "sidi":
        c, s = torch.cos(math.pi * u), torch.sin(math.pi * u)
        if r0 == 1:
            return 0.5 * (1 - c), 0.5 * math.pi * s
        if r0 == 2:
            return u - s * c / math.pi, 2 * s * s
        return 0.25 * (2 + c) * (1 - c) ** 2, 0.75 * math.pi * s ** 3
    v = 1 - u

    def half(x, y, a, b):
        return x ** (a + 1) * sum(math.comb(a + k, k) * y ** k for k in range(b + 1))

    x = torch.where(u <= 0.5, half(u, v, r0, r1), 1 - half(v, u, r1, r0))
    return x, (r0 + r1 + 1) * math.comb(r0 + r1, r0) * u ** r0 * v ** r1


def _fit_map(x, a):
    """PolySingular p(x) and p'(x)."""
    a0, a1, a2, a3, a4, a5 = (float(v) for v in a)
    a2, a3 = abs(a2), abs(a3)
    a6 = 1 - a2 - a3 - a4 - a5
    p = a2 * x * (a0 - 1) / (a0 - x) + a3 * x * (a1 - 1) / (a1 - x) + x * (a4 + x * (a5 + x * a6))
    dp = (a2 * a0 * (a0 - 1) / (a0 - x) ** 2 + a3 * a1 * (a1 - 1) / (a1 - x) ** 2 + a4 +
          x * (2 * a5 + 3 * x * a6))
    return p, dp


def _poly(coef, exps, x):
    """sum c prod x^e, as nested sums over one variable after the other."""
    terms = {}
    for c, e in zip(coef, exps):
        key = tuple(int(v) for v in e)
        terms[key] = terms.get(key, 0.0) + float(c)

    def nested(t, k):
        if k == len(x):
            return t[()] if () in t else 0.0
        by = {}
        for e, c in t.items():
            by.setdefault(e[0], {})[e[1:]] = c
        out = 0.0
        for power in range(max(by), -1, -1):
            out = out * x[k] if not isinstance(out, float) or out else out
            if power in by:
                out = out + nested(by[power], k + 1)
        return out

    return nested(terms, 0)


def _derivative(coef, exps, k):
    keep = exps[:, k] > 0
    e = exps[keep].copy()
    c = coef[keep] * e[:, k]
    e[:, k] -= 1
    return c, e


def _feynman(p, x, lam=0.5, b=2.5):
    d = len(x)
    grads = [_derivative(p["fcoef"], p["fexp"], k) for k in range(d)]
    g = [_poly(*t, x) for t in grads]
    z = [torch.complex(x[k], -lam * x[k] * (1 - x[k]) * g[k]) for k in range(d)]
    A = [[None] * d for _ in range(d)]
    for k in range(d):
        for l in range(d):
            im = -lam * x[k] * (1 - x[k]) * _poly(*_derivative(*grads[k], l), x)
            if k == l:
                im = im - lam * (1 - 2 * x[k]) * g[k]
            A[k][l] = torch.complex(torch.full_like(x[k], float(k == l)), im)
    det = 1.0
    for c in range(d):   # the Hermitian part of a matrix similar to this one is the identity
        det = det * A[c][c]
        for r in range(c + 1, d):
            f = A[r][c] / A[c][c]
            for l in range(c + 1, d):
                A[r][l] = A[r][l] - f * A[c][l]
    return _poly(p["ucoef"], p["uexp"], z) * torch.exp(-b * torch.log(_poly(p["fcoef"], p["fexp"], z))) * det


def _integrand_value(family, p, x):
    if family == "feynman":
        return _feynman(p, x)
    if family == "sector":
        return _poly(p["ucoef"], p["uexp"], x) * _poly(p["fcoef"], p["fexp"], x) ** -2.5
    c, w, d = [float(v) for v in p["c"]], [float(v) for v in p["w"]], len(x)
    if family == "oscillatory":
        return torch.cos(2 * math.pi * w[0] + sum(c[j] * x[j] for j in range(d)))
    if family == "product_peak":
        return 1 / math.prod(c[j] ** -2 + (x[j] - w[j]) ** 2 for j in range(d))
    if family == "corner_peak":
        return (1 + sum(c[j] * x[j] for j in range(d))) ** -(d + 1)
    if family == "gaussian":
        return torch.exp(-sum((c[j] * (x[j] - w[j])) ** 2 for j in range(d)))
    if family == "c0":
        return torch.exp(-sum(c[j] * (x[j] - w[j]).abs() for j in range(d)))
    f = torch.exp(sum(c[j] * x[j] for j in range(d)))
    return torch.where((x[0] > w[0]) | (x[1] > w[1]), torch.zeros_like(f), f)


def _shift_means(case, p, n, D, fit=None):
    """Q_k for every shift: complex for the complex family."""
    z = _rows()[n]
    Q = []
    for Dk in D:
        x, weight = [], None
        for j in range(len(Dk)):
            xj, wj = _map(case, _coordinate(n, z[j], Dk[j], 0, n))
            if fit is not None:
                xj, dp = _fit_map(xj, fit[j])
                wj = dp if wj is None else wj * dp
            x.append(xj)
            weight = wj if weight is None else weight if wj is None else weight * wj
        g = _integrand_value(case["family"], p, x)
        Q.append((g if weight is None else g * weight).sum() / n)
    return torch.stack(Q).cpu().numpy()


def _mean_err(Q):
    m = len(Q)
    return np.array([Q.mean(), math.sqrt(((Q - Q.mean()) ** 2).sum() / (m * (m - 1)))])


def _adaptive(case, p, n, m, shift_seed, epsrel, maxeval):
    """[value, error], n, evaluations of the escalation: the error is taken to fall like 1/n."""
    sizes = list(_rows())
    evals = 0
    D = _splitmix_shifts(shift_seed, m, len(p["c"]))
    while True:
        res = _mean_err(_shift_means(case, p, n, D))
        evals += n * m
        goal = epsrel * abs(res[0])
        if res[1] <= goal or evals >= maxeval:
            return res, n, evals
        want = int(n * max(res[1] / max(goal, 1e-300), 1.0)) + 1
        n2 = next((v for v in sizes if v >= max(want, n + 1)), sizes[-1])
        if n2 * m > maxeval - evals:
            fits = [v for v in sizes if v > n and v * m <= maxeval - evals]
            if not fits:
                return res, n, evals
            n2 = fits[-1]
        n = n2


def exact(case, seed):
    kind = case["kind"]
    if kind == "cbc":
        # z is a choice among whole numbers; e^2 of the table's vector by its definition
        n, z, gamma = case["n"], _rows()[case["n"]], _gamma(seed)
        k = torch.arange(n, device=DEV)
        prod, e2 = torch.ones(n, dtype=torch.float64, device=DEV), []
        for j in range(case["s"]):
            x = ((k * z[j]) % n).double() / n
            prod = prod * (1 + gamma * 2 * math.pi ** 2 * (x * x - x + 1 / 6))
            e2.append((prod.sum() / n - 1).item())
        return {"z": None, "e2": np.array(e2)}
    if kind == "points":
        D = _splitmix_shifts(SHIFT_SEED * seed, case["m"], case["d"])
        z, begin = _rows()[case["n"]], (case["n"] - case["count"]) // 2
        return torch.stack([torch.stack([_coordinate(case["n"], z[j], D[k, j], begin, case["count"])
                                         for j in range(case["d"])], dim=1)
                            for k in range(case["m"])], dim=1)
    kor3 = {"transform": "korobov", "r0": 3, "r1": 3}
    if kind == "serve":
        got = [_adaptive({**kor3, "family": f}, {"c": c, "w": w}, _next_n(1021), case["m"], s, eps,
                         case["maxeval"]) for f, c, w, eps, s in _requests(case, seed)]
        return {"result": np.array([g[0] for g in got]), "n": np.array([g[1] for g in got]),
                "evaluations": np.array([g[2] for g in got])}
    if kind == "batch":
        results, sums = [], []
        for d, p, n, s, fit in _batch_items(case, seed):
            Q = _shift_means({**kor3, "family": "sector"}, p, n, _splitmix_shifts(s, case["m"], d), fit)
            results.append(np.concatenate([_mean_err(Q), [0.0, 0.0]]))
            pairs = np.zeros(4 * case["m"])
            pairs[:2 * case["m"]:2] = Q * n
            sums.append(pairs)
        return {"results": np.array(results), "sums": np.array(sums)}
    p = _case_params(case, seed)
    if kind == "integrate":
        if case["fit"]:
            return None   # the fitted map ends where the least-squares iteration stops
        res, n, evals = _adaptive(case, p, case["n"], case["m"], SHIFT_SEED * seed, case["epsrel"],
                                  case["maxeval"])
        return {"result": res, "n": n, "m": case["m"], "evaluations": evals}
    Q = _shift_means(case, p, case["n"], _splitmix_shifts(SHIFT_SEED * seed, case["m"], case["d"]))
    parts = [Q.real, Q.imag] if np.iscomplexobj(Q) else [Q]
    res = np.concatenate([_mean_err(c) for c in parts] + [np.zeros(2)] * (2 - len(parts)))
    return {"result": res, "Q": np.stack(parts)}
