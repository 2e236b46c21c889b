"""FP64 transforms of values next to the end of the exponent range: the exponents shift,
the bits stay, and what leaves the range is infinite."""
import numpy as np
import pytest

from .test_gpu_fixed_point_fft import _fft, _field

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [(32, 16, 48), (80, 16, 16), (16, 96, 128)])
@pytest.mark.parametrize("inverse", [False, True])
@pytest.mark.parametrize("power", [1009, 1012])  # outputs below 2^1023, lines on both sides of 2^1013
def test_large_values(n, inverse, power):
    x = _field(n, 2)
    a = _fft(n, x, inverse)
    b = _fft(n, np.ldexp(x.real, power) + 1j * np.ldexp(x.imag, power), inverse)
    assert np.array_equal(np.ldexp(a.real, power), b.real) and np.array_equal(np.ldexp(a.imag, power), b.imag)
    assert np.all(np.isfinite(b))


@pytest.mark.parametrize("n", [(32, 16, 16), (48, 16, 16)])
def test_overflow_is_infinite(n):
    """One point 2^1020 along x: the line's values all have that size; its sum over a constant
    line does not fit."""
    x = np.zeros((1, n[2], n[1], n[0]), dtype=np.complex128)
    x[0, 2, 3, 5] = 2.0 ** 1020
    assert np.allclose(np.abs(_fft(n, x, False)) / 2.0 ** 1020, 1.0, rtol=1e-14, atol=0.0)
    x[0, :, :, :] = 2.0 ** 1022
    y = _fft(n, x, False)
    assert not np.isfinite(y[0, 0, 0])
