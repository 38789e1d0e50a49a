"""Double fields of subnormal values, which FP64 arithmetic transforms without loss.

Values v 2^k are multiples of u = 2^-1074.  Sums of subnormal numbers are exact and a
product is off by u / 2 at most, so an element meets an error of at most about u for
each rotation on its way.  There are no more than 10 rotations an axis with both
products of a component rounded, so as independent errors they come to less than
sqrt(60) u < 8 u an input element, against rms values 2^k / sqrt(3) of the field: a
relative error below 16 u / 2^k.  The inverse transform divides by N0 N1 N2 at its end
and rounds once more, which its smaller results, of rms 2^k / sqrt(3 N0 N1 N2) here,
meet with u / 2."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import gpu_c2r, gpu_r2c, rel_l2

pytestmark = pytest.mark.gpu

# one-warp, paired, 24-element and two-warp z-lines; columns of one and of several stages
SHAPES = [(8, 16, 32), (32, 12, 1024), (3, 48, 384), (16, 8, 2048), (24, 512, 24)]
UNIT = -1074
UP = 1000  # exact: from multiples of 2^-1074 to multiples of 2^-74


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("k", [-1043, -1050, -1060])
def test_subnormal_field_r2c(shape, k):
    f = np.ldexp(synth.uniform_field(shape, 5), k)
    assert np.abs(f).max() < 2.0 ** -1042
    F = oracle.rfft3(np.ldexp(f, UP))
    X = gpu_r2c(f, "f64")
    X = np.ldexp(X.real, UP) + 1j * np.ldexp(X.imag, UP)
    assert rel_l2(X, F) <= 16 * 2.0 ** (UNIT - k)


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("k", [-1043, -1050])
def test_subnormal_spectrum_c2r(shape, k):
    n = float(np.prod(shape))
    F = oracle.rfft3(synth.uniform_field(shape, 6)) / np.sqrt(n)
    F = np.ldexp(F.real, k) + 1j * np.ldexp(F.imag, k)
    f = oracle.irfft3(np.ldexp(F.real, UP) + 1j * np.ldexp(F.imag, UP), shape)
    y = np.ldexp(gpu_c2r(F, shape, "f64"), UP)
    assert rel_l2(y, f) <= 16 * np.sqrt(n) * 2.0 ** (UNIT - k)


def test_smallest_constant_field_sums_exactly():
    """The DC entry of a constant 2^-1074 field is its number of points, every other entry zero."""
    for shape in [(16, 8, 32), (8, 4, 1024), (3, 6, 2048)]:
        X = gpu_r2c(np.full(shape, 2.0 ** UNIT), "f64")
        assert X[0, 0, 0] == np.ldexp(float(np.prod(shape)), UNIT)
        X[0, 0, 0] = 0
        assert not X.any()
