"""Algorithmic bytes that egpe_profile_attempt reports for the preconditioner's first
pass: H psi, psi and r, the two workspace fields, the B field of P_V, and in FP64
attempts that carry T psi along the two fields of P_V^{-1} r."""
import pytest

from paper_2510_24543_gb300 import egpe as E
from paper_2510_24543_gb300 import inputs as I

from ._common import mixed_workload

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,mode,fields", [("fp64", "kinetic", 8), ("fp64", "kinetic+diagonal", 11),
                                              ("fp32", "kinetic+diagonal", 9)])
def test_precond_first_pass(prec, mode, fields):
    import torch
    w = mixed_workload((16, 16, 16))
    f32 = prec == "fp32"
    h = E.egpe_create([E.make_grid(w.n, w.L)], [E.params_from_workload(w)], E.EGPE_FP32 if f32 else E.EGPE_FP64)
    try:
        psi = torch.from_numpy(I.gaussian_start(w)).cuda().to(torch.complex64 if f32 else torch.complex128)
        rows = E.egpe_profile_attempt(h, 0, int(f32), psi, E.PRECOND[mode], reps=1)
    finally:
        E.egpe_destroy(h)
    name, _, by = rows[0]
    assert name.startswith("x-fwd precond")
    assert by == fields * 16 ** 3 * (8 if f32 else 16)
