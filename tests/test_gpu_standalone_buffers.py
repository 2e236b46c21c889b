"""Standalone evaluations work on the caller's buffers directly where they are
element-aligned and through copies where they are not: the same bits either way, and
with the output in place of the input."""
import numpy as np
import pytest

from paper_2510_24543_gb300 import egpe as E
from paper_2510_24543_gb300 import inputs as I

from ._common import mixed_workload

pytestmark = pytest.mark.gpu


def _at(x, offset):
    """A copy of tensor x (viewed as reals) `offset` reals into a fresh buffer, and its address."""
    import torch
    r = torch.view_as_real(x).reshape(-1)
    buf = torch.zeros(r.numel() + 4, dtype=r.dtype, device="cuda")
    buf[offset:offset + r.numel()] = r
    return buf, buf.data_ptr() + offset * r.element_size()


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
@pytest.mark.parametrize("n", [(16, 32, 16), (48, 16, 32)])
@pytest.mark.parametrize("offset", [0, 1])
def test_same_results(prec, n, offset):
    import torch
    w = mixed_workload(n)
    dt = torch.complex128 if prec == "fp64" else torch.complex64
    psi = torch.from_numpy(I.random_state(w.n, w.L, 7)).cuda().to(dt)
    res = torch.from_numpy(I.raw_direction(w.n, w.L, 8)).cuda().to(dt)
    h = E.egpe_create([E.make_grid(w.n, w.L)], [E.params_from_workload(w)],
                      E.EGPE_FP64 if prec == "fp64" else E.EGPE_FP32)
    try:
        grad, z = torch.empty_like(psi), torch.empty_like(psi)
        ref = E.egpe_energy_grad(h, 0, psi, grad)
        dref = E.egpe_param_grad(h, 0, psi)
        m = torch.view_as_real(psi).numel()
        bp, pp = _at(psi, offset)
        bg, pg = _at(torch.zeros_like(psi), offset)
        assert E.egpe_energy_grad(h, 0, pp, pg) == ref
        assert torch.equal(bg[offset:offset + m], torch.view_as_real(grad).reshape(-1))
        assert E.egpe_param_grad(h, 0, pp) == dref
        assert torch.equal(bp[offset:offset + m], torch.view_as_real(psi).reshape(-1))
        for mode in range(5):
            for r in (None, res):
                E.egpe_precondition(h, 0, mode, psi, r, z)
                br, pr = _at(res, offset)
                E.egpe_precondition(h, 0, mode, pp, pr if r is not None else None, pg)
                assert torch.equal(bg[offset:offset + m], torch.view_as_real(z).reshape(-1))
        assert E.egpe_line_coeffs(h, 0, pp, pr) == E.egpe_line_coeffs(h, 0, psi, res)
        # outputs in place of the inputs
        E.egpe_precondition(h, 0, 3, psi, res, z)
        E.egpe_precondition(h, 0, 3, pp, pr, pr)
        assert torch.equal(br[offset:offset + m], torch.view_as_real(z).reshape(-1))
        assert E.egpe_energy_grad(h, 0, pp, pp) == ref
        assert torch.equal(bp[offset:offset + m], torch.view_as_real(grad).reshape(-1))
        assert np.isfinite(ref[0])
    finally:
        E.egpe_destroy(h)
