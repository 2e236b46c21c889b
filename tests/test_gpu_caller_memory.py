"""Standalone evaluations take buffers from any memory the runtime can copy: pinned host
memory gives the bits that device memory gives."""
import pytest

from paper_2510_24543_gb300 import egpe as E
from paper_2510_24543_gb300 import inputs as I

from ._common import mixed_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["fp64", "fp32"])
def test_pinned_host_buffers(prec):
    import torch
    w = mixed_workload((16, 32, 16))
    dt = torch.complex128 if prec == "fp64" else torch.complex64
    psi = torch.from_numpy(I.random_state(w.n, w.L, 7)).to(dt)
    pin, out = psi.pin_memory(), torch.empty_like(psi).pin_memory()
    dev, grad = psi.cuda(), torch.empty_like(psi, device="cuda")
    h = E.egpe_create([E.make_grid(w.n, w.L)], [E.params_from_workload(w)],
                      E.EGPE_FP64 if prec == "fp64" else E.EGPE_FP32)
    try:
        ref = E.egpe_energy_grad(h, 0, dev, grad)
        assert E.egpe_energy_grad(h, 0, pin.data_ptr(), out.data_ptr()) == ref
        torch.cuda.synchronize()
        assert torch.equal(out, grad.cpu())
        assert E.egpe_param_grad(h, 0, pin.data_ptr()) == E.egpe_param_grad(h, 0, dev)
        E.egpe_precondition(h, 0, 3, dev, None, grad)
        E.egpe_precondition(h, 0, 3, pin.data_ptr(), None, out.data_ptr())
        torch.cuda.synchronize()
        assert torch.equal(out, grad.cpu())
    finally:
        E.egpe_destroy(h)
