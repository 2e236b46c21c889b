"""Handles take the memory of the carried kinetic terms when they are created, so solves
allocate none, and FP64 attempts without those terms take the same iterates."""
import numpy as np
import pytest

from paper_2510_24543_gb300 import egpe as E
from paper_2510_24543_gb300 import inputs as I

from ._common import mixed_workload, workload

pytestmark = pytest.mark.gpu


def _opts(mode, iters, **kw):
    o = E.egpe_default_solve_opts()
    o.precond, o.tol_res, o.max_iter = E.PRECOND[mode], 0.0, iters
    for k, v in kw.items():
        setattr(o, k, v)
    return o


@pytest.mark.parametrize("n_inst", [1, 3])
def test_solves_allocate_nothing(n_inst):
    import torch
    w = workload("c2")  # 64^3: the carried terms are 42 MB per instance
    psi = torch.from_numpy(I.gaussian_start(w)).cuda()
    for _ in range(2):  # the first round loads the kernels
        h = E.egpe_create([E.make_grid(w.n, w.L)] * n_inst, [E.params_from_workload(w)] * n_inst, E.EGPE_FP64)
        xs = [psi.clone() for _ in range(n_inst)]
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        E.egpe_ncg_solve(h, xs, _opts("kinetic+diagonal", 10), n_inst)
        after = torch.cuda.mem_get_info()[0]
        E.egpe_destroy(h)
        del xs
    # graphs and the batch's pointer tables, well below one instance's terms
    assert before - after < 10 * 16 * 64 ** 3 // 2


@pytest.mark.parametrize("mode", ["kinetic", "kinetic+diagonal"])
@pytest.mark.parametrize("n", [(16, 32, 16), (48, 16, 32)])
def test_without_carried_terms(mode, n):
    """14 transforms per iteration instead of 8 and a refresh, and the same iterates (the
    bound of the comparison with the oracle, tests/test_gpu_carried_kinetic.py)."""
    import torch
    w = mixed_workload(n)
    psi = I.gaussian_start(w)
    out = {}
    for off in (False, True):
        for kw in (dict(), dict(use_graph=0), dict(n_inst=2)):
            m = kw.pop("n_inst", 1)
            h = E.egpe_create([E.make_grid(w.n, w.L)] * m, [E.params_from_workload(w)] * m, E.EGPE_FP64)
            try:
                if off:  # of one instance: a batch decides for all
                    E.egpe_set_tuning(h, m - 1, 0, [dict(key="carried kinetic terms", choice=0)])
                xs = [torch.from_numpy(psi).cuda() for _ in range(m)]
                _, reps, _ = E.egpe_ncg_solve(h, xs, _opts(mode, 20, **kw), m)
            finally:
                E.egpe_destroy(h)
            assert (reps[0]["ffts"] >= 20 * 14) == off
            out[off, m, kw.get("use_graph", 1)] = xs[0].cpu().numpy()
    ref = out[True, 1, 1]
    assert all(np.linalg.norm(x - ref) < 1e-10 * np.linalg.norm(ref) for x in out.values())
