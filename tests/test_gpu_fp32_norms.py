"""Norms of the states that FP32 iterations leave.  A trial point a psi + b p costs one
rounding per value, without a preferred sign; what is left is the rounding of the
coefficient a to 24 bits: 2 da on ||psi_i||^2, da uniform within 2^-25 for a below 1,
so 2^-24/sqrt(3) = 3.4e-8 in the mean square."""
import numpy as np
import pytest

from paper_2510_24543_gb300 import egpe as E
from paper_2510_24543_gb300 import inputs as I

from ._common import workload

pytestmark = pytest.mark.gpu

BOUND = 1.4 * 2.0 ** -24 / 3 ** 0.5


def _norms(w, first=10, last=80):
    """||psi_i||^2 - 1 after the iterations `first` to `last`."""
    import torch
    h = E.egpe_create([E.make_grid(w.n, w.L)], [E.params_from_workload(w)], E.EGPE_FP32)
    try:
        x = torch.from_numpy(I.gaussian_start(w)).cuda().to(torch.complex64)
        dV = np.prod([2.0 * w.L[a] / w.n[a] for a in range(3)])
        o = E.egpe_default_solve_opts()
        o.precond, o.tol_res, o.max_iter = E.PRECOND["kinetic+diagonal"], 0.0, 1000
        E.egpe_solver_start(h, 0, 1, x, o)
        E.egpe_solver_step(h, 0, 1, first)
        out = []
        for _ in range(first, last):
            E.egpe_solver_step(h, 0, 1, 1)
            E.egpe_solver_read(h, 0, 1, x)
            out.append((dV * x.to(torch.complex128).abs().square().sum(dim=(1, 2, 3)) - 1.0).cpu().numpy())
        return np.array(out)
    finally:
        E.egpe_destroy(h)


def test_rounding_has_no_preferred_sign():
    v = np.concatenate([_norms(w) for w in (workload("c1"), workload("c2"), workload("c1", n=(48, 32, 16)),
                                            workload("c1", n=(16, 16, 16)))])
    assert np.sqrt(np.mean(v ** 2)) < BOUND
