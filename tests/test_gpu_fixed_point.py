"""Double-precision transforms run in block fixed point, each line scaled by a
power of two of its own; lines outside the conversions' range take the FP64
path.  Here: fields over the whole exponent range, lines of very different
size in one field, zero lines, and non-finite values.  FP64 bound 1e-13, as in
the parity sweep."""
import numpy as np
import pytest

import oracle
import synth
from gpu_util import TOL, gpu_c2r, gpu_r2c, rel_l2

pytestmark = pytest.mark.gpu

# paired, one-warp, two-warp and 24-element z-lines; columns of one and of several stages
SHAPES = [(8, 16, 32), (32, 12, 1024), (3, 48, 384), (256, 8, 2048), (24, 512, 24)]


@pytest.mark.parametrize("shape", SHAPES, ids=lambda s: "x".join(map(str, s)))
@pytest.mark.parametrize("k", [-1000, -930, -895, -700, 0, 700, 880, 950])
def test_any_scale(shape, k):
    f = synth.uniform_field(shape, 5)
    F = oracle.rfft3(f)
    assert rel_l2(np.ldexp(1.0, -k) * gpu_r2c(f * np.ldexp(1.0, k), "f64"), F) <= TOL["f64"]
    assert rel_l2(np.ldexp(1.0, -k) * gpu_c2r(F * np.ldexp(1.0, k), shape, "f64"), f) <= TOL["f64"]


def test_lines_keep_their_own_scale():
    """Rows 2^60 apart: each row's own spectrum (the other axes have length 1)
    stays within the bound of that row."""
    for n2 in (24, 32, 96, 256, 768, 1536, 2048):
        f = synth.uniform_field((1, 1, n2), 6)
        for k in (-400, -60, 0, 60, 400):
            g = f * np.ldexp(1.0, k)
            assert rel_l2(gpu_r2c(g, "f64"), oracle.rfft3(g)) <= TOL["f64"]
    # columns: a field whose k2 = 3 part is 2^-60 of the rest keeps it (only one column set holds it)
    n = 32
    f = synth.uniform_field((n, n, n), 7)
    F = oracle.rfft3(f)
    F[:, :, 3] *= np.ldexp(1.0, -60)
    g = gpu_c2r(F, (n, n, n), "f64")
    assert rel_l2(g, oracle.irfft3(F, (n, n, n))) <= TOL["f64"]


def test_zero_lines_stay_zero():
    f = np.zeros((16, 24, 64))
    assert not gpu_r2c(f, "f64").any()
    assert not gpu_c2r(np.zeros((16, 24, 33), complex), f.shape, "f64").any()
    f[3, 5, 7] = 1.0
    assert rel_l2(gpu_r2c(f, "f64"), oracle.rfft3(f)) <= TOL["f64"]


@pytest.mark.parametrize("bad", [np.nan, np.inf, -np.inf])
def test_non_finite_values_stay_in_their_field(bad):
    import torch
    import paper_2202_12756_gb300 as fft3d
    shape = (16, 16, 64)
    f = np.stack([synth.uniform_field(shape, s) for s in (8, 9, 10)])
    f[1, 2, 3, 4] = bad
    x = torch.from_numpy(f).cuda()
    X = fft3d.rfft3(x)
    y = fft3d.irfft3(X, x.shape)
    X, y = X.cpu().numpy(), y.cpu().numpy()
    assert not np.isfinite(X[1]).any() and not np.isfinite(y[1]).any()
    for b in (0, 2):
        assert rel_l2(X[b], oracle.rfft3(f[b])) <= TOL["f64"]
        assert rel_l2(y[b], f[b]) <= TOL["f64"]
