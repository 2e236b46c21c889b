"""An LHY prefactor so small that its table entries leave the exponent range of the
fixed-point records is an LHY term of zero, not garbage."""
import numpy as np
import pytest

from paper_2510_24543_gb300 import egpe as E
from paper_2510_24543_gb300 import inputs as I

from ._common import mixed_workload

pytestmark = pytest.mark.gpu


def _evaluate(w, kappa):
    import torch
    p = E.make_params(w.g, w.gdd, kappa, w.eta_s, w.lhy_nodes, w.trap)
    h = E.egpe_create([E.make_grid(w.n, w.L)], [p], E.EGPE_FP64)
    try:
        psi = torch.from_numpy(I.random_state(w.n, w.L, 7)).cuda()
        d = torch.from_numpy(I.raw_direction(w.n, w.L, 8)).cuda()
        g = torch.empty_like(psi)
        e, mu = E.egpe_energy_grad(h, 0, psi, g)
        return np.array([e, *mu]), g.cpu().numpy(), np.array(E.egpe_line_coeffs(h, 0, psi, d))
    finally:
        E.egpe_destroy(h)


@pytest.mark.parametrize("kappa", [1e-270, 1e-285, 1e-295, 1e-305, 5e-324, -1e-300])
def test_tiny_prefactor(kappa):
    w = mixed_workload((16, 16, 16))
    for a, b in zip(_evaluate(w, kappa), _evaluate(w, 0.0)):
        assert np.array_equal(a, b)
