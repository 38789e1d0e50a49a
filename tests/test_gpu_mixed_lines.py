"""Double lines and columns of every kind side by side in one launch: ordinary ones in fixed
point beside ones that take the FP64 path (infinities, values near both ends of the exponent
range) and ones of zeros.  Each is compared with its own transform in extended precision.

Bounds: one transform is off by 0.5 to 2.8e-16 of its line's norm, in fixed point and in
FP64 arithmetic, over lengths and kinds of data, so 5e-16 for a line and 1e-15 for two axes.
Single entries of a line are off by 1.8e-16 of its rms as independent errors in fixed point,
so 4 sigma stay below 2^-50 rms; the bound is twice that and the rounding of the entry."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROWS = 37  # odd: the last line of a pairing length has no partner
LENGTHS = [8, 32, 96, 384, 512, 1024, 1536, 2048]
COLUMNS = [8, 24, 48, 256, 512, 768, 1024, 2048]
LD = np.longdouble


def _l2(a, b):
    return float(np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel()))


def _rows(n2, rng):
    """[ROWS, n2] values, and for each row its kind and power of two."""
    f = rng.uniform(-1.0, 1.0, (ROWS, n2))
    f[3] = np.exp(-0.5 * ((np.arange(n2) - n2 / 2) / (n2 / 16)) ** 2)  # entries of its spectrum fall to zero
    f[5] = 0.0
    f[5, n2 // 3] = 1.0
    kinds, power = ["plain"] * ROWS, [0] * ROWS
    for i, r in enumerate(range(2, ROWS, 5)):
        kind, k = [("inf", 0), ("plain", 950), ("zero", 0), ("plain", -950)][i % 4]
        kinds[r], power[r] = kind, k
        if kind == "zero":
            f[r] = 0.0
    for r in (8, 10, 14):  # in range, far from their neighbours
        power[r] = {8: -600, 10: 0, 14: 700}[r]
    return f, kinds, power


def _alone(r, n2, kinds, power):
    """Whether row r shares its scale with no row of another size (lines of 1024 reals go in pairs)."""
    p = r ^ 1
    return n2 != 1024 or p >= ROWS or (kinds[p] == kinds[r] and power[p] == power[r])


def _check(got, want, n2, kinds, power):
    for r in range(ROWS):
        if not _alone(r, n2, kinds, power):
            continue
        if kinds[r] == "inf":
            assert not np.isfinite(got[r]).any(), r
        elif kinds[r] == "zero":
            assert not got[r].any(), r
        else:
            s = LD(2.0) ** -power[r]
            x = got[r].astype(want.dtype) * s
            assert _l2(x, want[r]) <= 5e-16, (r, kinds[r], power[r])
            rms = np.sqrt(np.mean(np.abs(want[r]) ** 2))
            assert (np.abs(x - want[r]) <= 2.0 ** -49 * rms + 2.0 ** -52 * np.abs(want[r])).all(), (r, power[r])


@pytest.mark.parametrize("inplace", [False, True], ids=["out", "in"])
@pytest.mark.parametrize("n2", LENGTHS)
def test_lines_of_every_kind_in_a_block(n2, inplace):
    import torch
    import paper_2202_12756_gb300 as fft3d
    plan = fft3d.Plan((1, 1, n2), torch.float64, batch=ROWS)
    f, kinds, power = _rows(n2, np.random.default_rng(n2))
    scale = np.ldexp(1.0, power)[:, None]

    F = np.fft.rfft(f.astype(LD), axis=1)
    g = f * scale
    g[[r for r in range(ROWS) if kinds[r] == "inf"], n2 // 2] = np.inf
    g = torch.from_numpy(g).reshape(plan.real_shape)
    if inplace:
        buf = plan.empty_padded()
        buf[..., :n2].copy_(g)
        X = plan.r2c_(buf)
    else:
        X = plan.r2c(g.cuda())
    _check(X.cpu().numpy().reshape(ROWS, -1), F, n2, kinds, power)

    # back from spectra of the rows' sizes, the ones of an infinity with one in an entry that counts
    G = F.astype(np.complex128)
    f = np.fft.irfft(G.astype(F.dtype), n2, axis=1)
    G = G * scale
    G[[r for r in range(ROWS) if kinds[r] == "inf"], n2 // 4] = np.inf
    G = torch.from_numpy(G).reshape(plan.half_shape)
    if inplace:
        buf = plan.empty_padded()
        buf.view(torch.complex128).copy_(G)
        y = plan.c2r_(buf)[..., :n2]
    else:
        y = plan.c2r(G.cuda())
    _check(y.cpu().numpy().reshape(ROWS, -1), f, n2, kinds, power)


@pytest.mark.parametrize("axis", [0, 1])
@pytest.mark.parametrize("n", COLUMNS)
def test_columns_of_every_kind_in_a_launch(n, axis):
    import torch
    import paper_2202_12756_gb300 as fft3d
    n2 = 64
    shape = (n, 1, n2) if axis == 0 else (1, n, n2)
    power = [0, 950, -950, 0]
    plan = fft3d.Plan(shape, torch.float64, batch=len(power))
    rng = np.random.default_rng(n + axis)
    scale = np.ldexp(1.0, power)[:, None, None, None]

    # tiles of the FP64 path beside fixed-point ones
    f = rng.uniform(-1.0, 1.0, plan.real_shape)
    F = np.fft.fft(np.fft.rfft(f.astype(LD), axis=3), axis=axis + 1)
    X = plan.r2c(torch.from_numpy(f * scale).cuda()).cpu().numpy()
    for b, k in enumerate(power):
        assert _l2(X[b].astype(F.dtype) * LD(2.0) ** -k, F[b]) <= 1e-15, (b, k)

    # columns of zeros, and in one field a tiny one, beside ordinary ones of a tile
    G = F.astype(np.complex128)
    G[..., 5] = 0.0
    G[..., 20:24] = 0.0
    G[3, ..., 7] *= np.ldexp(1.0, -960)
    want = np.fft.irfft(np.fft.ifft(G.astype(F.dtype), axis=axis + 1), n2, axis=3)
    y = plan.c2r(torch.from_numpy(G * scale).cuda()).cpu().numpy()
    for b, k in enumerate(power):
        assert _l2(y[b].astype(LD) * LD(2.0) ** -k, want[b]) <= 1e-15, (b, k)
