"""FP64 transforms run in 64-bit fixed point under one scale per line: every
length on every axis against numpy, fields far from unit magnitude, lines of very
different magnitude, zero fields and non-finite values."""
import numpy as np
import pytest

from paper_2510_24543_gb300 import egpe as E
from paper_2510_24543_gb300 import inputs as I

pytestmark = pytest.mark.gpu

# every supported length on the row axis (x) and on both strided axes
GRIDS = [(16, 32, 48), (32, 48, 64), (48, 64, 80), (64, 80, 96), (80, 96, 128), (96, 128, 16), (128, 256, 16),
         (256, 16, 32)]
# numpy's FP64 transform is itself a few 1e-16 off, the fixed-point one about 1.5e-16
TOL = 1e-15


def _fft(n, x, inverse):
    import torch
    w = I.PRESETS["c1"]
    h = E.egpe_create([E.make_grid(n, w.L)], [E.params_from_workload(w)], E.EGPE_FP64)
    try:
        t = torch.from_numpy(np.ascontiguousarray(x)).cuda()
        o = torch.empty_like(t)
        E.egpe_fft(h, 0, t, o, 1, inverse)
        return o.cpu().numpy()[0]
    finally:
        E.egpe_destroy(h)


def _field(n, seed):
    rng = np.random.default_rng(seed)
    s = (1, n[2], n[1], n[0])
    return rng.standard_normal(s) + 1j * rng.standard_normal(s)


def _err(got, x, inverse):
    ref = np.fft.ifftn(x[0], norm="forward") if inverse else np.fft.fftn(x[0])
    return np.linalg.norm(got - ref) / np.linalg.norm(ref)


@pytest.mark.parametrize("n", GRIDS)
@pytest.mark.parametrize("inverse", [False, True])
def test_random_field(n, inverse):
    x = _field(n, 1)
    assert _err(_fft(n, x, inverse), x, inverse) < TOL


@pytest.mark.parametrize("n", [(32, 16, 48), (80, 16, 16)])
@pytest.mark.parametrize("power", [-900, 900])
def test_scaled_field(n, power):
    """A power-of-two factor far from 1 changes nothing but the exponents."""
    x = _field(n, 2)
    a, b = _fft(n, x, False), _fft(n, np.ldexp(x.real, power) + 1j * np.ldexp(x.imag, power), False)
    assert np.array_equal(np.ldexp(a.real, power), b.real) and np.array_equal(np.ldexp(a.imag, power), b.imag)


@pytest.mark.parametrize("n", [(64, 32, 16), (96, 48, 16)])
def test_lines_of_different_magnitude(n):
    """A Gaussian envelope down to e^-300 along every axis, and one dominant point."""
    x = _field(n, 3)
    r = [np.linspace(-17.0, 17.0, k) ** 2 for k in n]
    x = x * np.exp(-r[2][:, None, None] - r[1][None, :, None] - r[0][None, None, :])
    x[0, 3, 5, 7] = 1e3
    assert _err(_fft(n, x, False), x, False) < TOL


@pytest.mark.parametrize("n", [(16, 16, 16), (48, 16, 32)])
def test_zero_and_nonfinite(n):
    x = np.zeros((1, n[2], n[1], n[0]), dtype=np.complex128)
    assert not np.any(_fft(n, x, False))
    for bad in (np.nan, np.inf):
        y = _field(n, 4)
        y[0, 1, 2, 3] = bad
        assert np.all(np.isnan(_fft(n, y, False)))


@pytest.mark.parametrize("n", [(16, 32, 48), (80, 16, 16)])
@pytest.mark.parametrize("tiny", [-1e-300, -0.0, -5e-324])
def test_lines_below_the_range(n, tiny):
    """Negative values below 2^-960 are zeros: alone, and in lines beside ordinary ones."""
    x = np.full((1, n[2], n[1], n[0]), tiny + 1j * tiny)
    assert not np.any(_fft(n, x, False))
    x[0, 4, 3] = _field(n, 5)[0, 4, 3]
    assert _err(_fft(n, x, False), x, False) < TOL
