"""Iterations whose preconditioned direction is not a descent direction take the
residual instead (Sec. IV.C reading).  Attempts that carry T psi and T p along
transform that direction in one attempt more, with nothing left unknown for the
conjugate directions after it.  Attractive couplings make P_V drop to its floor on
part of the grid, where such steps happen; the oracle takes the same ones."""
import functools

import numpy as np
import pytest

import oracle as O
from paper_2510_24543_gb300 import egpe as E
from paper_2510_24543_gb300 import inputs as I

from ._common import oracle_case

pytestmark = pytest.mark.gpu

# name: box, trap, (g11, g12, g22), gdd, c, pv_floor, noise of the start, iterations
CASES = {
    # one fallback, a conjugate direction right after it
    "single": ((10.0, 2.5, 4.75), (5.4, 0.36, 2.07), (-71.7, 195.5, 271.9), 161.5, 0.7, 1e-2, 0.01, 12),
    # several, each followed by conjugate directions
    "several": ((7.6, 2.2, 7.5), (0.5, 1.0, 0.85), (161.0, -70.0, 28.0), 2.0, 21.0, 1e-2, 0.3, 20),
    # a fallback direction whose first trial is rejected
    "rejected": ((9.4, 9.35, 3.9), (1.4, 0.73, 2.06), (-57.7, 90.6, 257.0), 151.9, 66.2, 1e-2, 0.01, 10),
}


@functools.lru_cache(maxsize=None)
def _case(name):
    """Workload, options, start, the oracle's run and how far a run drifts whose start
    is 1e-13 (some hundred roundings) off."""
    L, trap, (g11, g12, g22), gdd, c, floor, noise, iters = CASES[name]
    w = I.Workload(name, (16, 16, 16), L, trap, ((g11, g12), (g12, g22)), ((gdd, gdd), (gdd, gdd)), c, 3,
                   "kinetic+diagonal", 8)
    g, prm = oracle_case(w)
    psi = I.gaussian_start(w, noise=noise)
    opts = dict(precond="kinetic+diagonal", tol_res=0.0, max_iter=iters, pv_floor=floor)
    trace = []
    ref, rep = O.ncg_solve(g, prm, psi, O.SolveOpts(**opts), trace=trace)
    near = psi * (1.0 + 1e-13 * np.random.default_rng(5).standard_normal(psi.shape))
    off, _ = O.ncg_solve(g, prm, near, O.SolveOpts(**opts))
    tol = 10.0 * np.linalg.norm(off - ref) / np.linalg.norm(ref) + 1e-12
    return w, opts, psi, ref, rep, trace, tol


def _handle(w, n=1):
    return E.egpe_create([E.make_grid(w.n, w.L)] * n, [E.params_from_workload(w)] * n, E.EGPE_FP64)


def _opts(opts, **kw):
    o = E.egpe_default_solve_opts()
    o.precond, o.tol_res, o.max_iter, o.pv_floor = E.PRECOND[opts["precond"]], 0.0, opts["max_iter"], opts["pv_floor"]
    for k, v in kw.items():
        setattr(o, k, v)
    return o


def _near(x, ref, tol):
    return np.linalg.norm(x.cpu().numpy() - ref) < tol * np.linalg.norm(ref)


def _launches(trace):
    """Attempts the run takes: its trials, and one more per fallback direction."""
    first = {t["n"]: t for t in trace}
    return sum(1 + t["armijo"] + (1 if t["fallback"] else 0) for t in first.values())


@pytest.mark.parametrize("name", sorted(CASES))
def test_follows_the_oracle(name):
    import torch
    w, opts, psi, ref, rep, trace, tol = _case(name)
    falls = [t for t in trace if t["fallback"]]
    assert falls and (name != "rejected" or any(t["armijo"] for t in falls))
    for kw in (dict(poll_every=1), dict(use_graph=0), dict()):
        h = _handle(w)
        try:
            x = torch.from_numpy(psi).cuda()
            _, (r,), tr = E.egpe_ncg_solve(h, [x], _opts(opts, **kw), 1, trace_cap=200)
        finally:
            E.egpe_destroy(h)
        assert r["iters"] == opts["max_iter"] and _near(x, ref, tol)
        assert {t["n"] for t in tr if t["flags"] & 4} == {t["n"] for t in falls}
        if kw.get("poll_every") == 1:  # one launch more finds the iteration limit
            assert r["graph_launches"] == _launches(trace) + 1


@pytest.mark.parametrize("name", sorted(CASES))
def test_stepping_and_batch(name):
    import torch
    w, opts, psi, ref, _, trace, tol = _case(name)
    h = _handle(w)
    try:
        x = torch.empty(psi.shape, dtype=torch.complex128, device="cuda")
        E.egpe_solver_start(h, 0, 0, torch.from_numpy(psi).cuda(), _opts(opts, max_iter=1000))
        E.egpe_solver_step(h, 0, 0, _launches(trace))
        assert E.egpe_solver_read(h, 0, 0, x)["iters"] == opts["max_iter"]
        assert _near(x, ref, tol)
    finally:
        E.egpe_destroy(h)
    h = _handle(w, 2)
    try:
        xs = [torch.from_numpy(np.ascontiguousarray(p)).cuda() for p in (psi, psi)]
        _, reps, _ = E.egpe_ncg_solve(h, xs, _opts(opts), 2)
        assert all(r["iters"] == opts["max_iter"] for r in reps)
        assert all(_near(y, ref, tol) for y in xs)
    finally:
        E.egpe_destroy(h)
