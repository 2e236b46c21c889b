"""FP64 solver attempts with the kinetic preconditioners carry T psi and T p along
instead of transforming p and the trial state (T z = w - alpha z); every 8th
attempt transforms the trial state.  The iterates against the oracle's, over more
than one such period, alone, without graphs and in a batch (FP32 attempts transform
both: the same iterates to FP32 accuracy)."""
import numpy as np
import pytest

import oracle as O
from paper_2510_24543_gb300 import egpe as E
from paper_2510_24543_gb300 import inputs as I

from ._common import mixed_workload, oracle_case, rel

pytestmark = pytest.mark.gpu

ITERS = 20
# On E; 100 times as much on psi.  Two oracle runs from starts that differ by 1e-13
# or 1e-7 end closer to each other (the iteration contracts), so what remains is
# the rounding of the last iterations, eps |H| with |H| ~ 1e3 on these grids.
TOL = {"fp64": 1e-12, "fp32": 1e-6}


def _solve(w, psis, prec, mode, use_graph=1, batch=1):
    import torch
    dt = torch.complex64 if prec == "fp32" else torch.complex128
    n = len(psis)
    h = E.egpe_create([E.make_grid(w.n, w.L)] * n, [E.params_from_workload(w)] * n,
                      E.EGPE_FP32 if prec == "fp32" else E.EGPE_FP64)
    try:
        o = E.egpe_default_solve_opts()
        o.precond, o.tol_res, o.max_iter, o.use_graph, o.batch = E.PRECOND[mode], 0.0, ITERS, use_graph, batch
        xs = [torch.from_numpy(p).cuda().to(dt) for p in psis]
        _, reps, _ = E.egpe_ncg_solve(h, xs, o, n)
        return [x.cpu().numpy() for x in xs], reps
    finally:
        E.egpe_destroy(h)


@pytest.mark.parametrize("prec,n", [("fp64", (16, 32, 16)), ("fp64", (48, 16, 32)), ("fp32", (32, 16, 48))])
@pytest.mark.parametrize("mode", ["kinetic", "kinetic+diagonal"])
def test_follows_the_oracle(prec, n, mode):
    w = mixed_workload(n)
    g, prm = oracle_case(w)
    psi = I.gaussian_start(w)
    ref, rep = O.ncg_solve(g, prm, psi, O.SolveOpts(precond=mode, tol_res=0.0, max_iter=ITERS,
                                                    accept_rtol=1e-13 if prec == "fp64" else 1e-6))
    for kw in (dict(), dict(use_graph=0)):
        (x,), (r,) = _solve(w, [psi], prec, mode, **kw)
        assert prec == "fp32" or r["iters"] == ITERS
        assert rel(r["E"], rep["E"]) < TOL[prec]
        assert np.linalg.norm(x - ref) < 100 * TOL[prec] * np.linalg.norm(ref)
    xs, rs = _solve(w, [psi, np.ascontiguousarray(psi[::-1])], prec, mode)  # two instances, batched
    assert np.linalg.norm(xs[0] - ref) < 100 * TOL[prec] * np.linalg.norm(ref)
    assert rel(rs[0]["E"], rep["E"]) < TOL[prec] and np.isfinite(rs[1]["E"])
