"""The state an FP32 solve returns has the energy of its own normalised copy: its norms are
those of fields rounded to 24 bits, 2^-24 per value without a preferred sign, which
average out over the grid (4e-10 at 32^3) whatever the step's coefficients are."""
import numpy as np
import pytest

from paper_2510_24543_gb300 import egpe as E
from paper_2510_24543_gb300 import inputs as I

from ._common import workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("name,n", [("c1", (32, 32, 32)), ("c1", (48, 32, 16)), ("c2", (64, 64, 64))])
@pytest.mark.parametrize("iters", [1, 10, 30])
def test_norms(name, n, iters):
    import torch
    w = workload(name, n=n)
    h = E.egpe_create([E.make_grid(w.n, w.L)], [E.params_from_workload(w)], E.EGPE_FP32)
    try:
        o = E.egpe_default_solve_opts()
        o.precond, o.tol_res, o.max_iter = E.PRECOND["kinetic+diagonal"], 0.0, iters
        x = torch.from_numpy(I.gaussian_start(w)).cuda().to(torch.complex64)
        E.egpe_ncg_solve(h, [x], o, 1)
    finally:
        E.egpe_destroy(h)
    dV = np.prod([2.0 * w.L[a] / w.n[a] for a in range(3)])
    norm2 = (dV * x.to(torch.complex128).abs().square().sum(dim=(1, 2, 3))).cpu().numpy()
    # the FP32 sums behind ||psi||^2 and <psi, p> (float-float) add their terms' rounding:
    # 2^-24 per term, averaged the same way
    assert np.all(np.abs(norm2 - 1.0) < 2e-8)
