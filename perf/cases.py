"""The calls whose time matters, for a measuring program.

`listed()` names them, `draw(rng)` gives more of the same ranges, `prepare`
makes a case's inputs and plan on the GPU, `run` is one pass through the
package's public entry points, `work` the bytes and flops of that pass and
`exact` its outputs in 64 bits from torch.fft.

A case: `op` (what is called), `n0` x `n1` x `n2` (the grid), `batch` (fields
per call), `dtype` (real type) and `field` (what the data look like).

ops
  r2c      rfft3 of a dense field
  c2r      irfft3 of a half spectrum
  both     rfft3, then irfft3 of its result, out of place; both are returned
  inplace  Plan.r2c_ and Plan.c2r_ on one padded buffer (the solver's loop,
           and the layout of the largest grids, which have room for one copy)
  grad     a Gaussian filter in spectral space, rfft3 -> multiply -> irfft3,
           a squared-error loss and its backward pass (both adjoints)

fields
  uniform     iid uniform[-1, 1)
  turbulence  random phases with amplitudes |k|^(-11/6): the steep spectrum
              that pseudo-spectral flow solvers transform
"""
import math

import torch

import paper_2202_12756_gb300 as fft3d

_DTYPES = {"f32": torch.float32, "f64": torch.float64}

# lengths of axes 0 and 1, and of the halved axis 2
_COLUMNS = [8, 12, 16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024, 1536, 2048]
_LINES = [16, 24, 32, 48, 64, 96, 128, 192, 256, 384, 512, 768, 1024, 1536, 2048]


def _case(name, op, n0, n1, n2, dtype, field="uniform", batch=1):
    c = {"op": op, "n0": n0, "n1": n1, "n2": n2, "batch": batch, "dtype": dtype, "field": field}
    return {"name": name, **c} if name else c


def listed():
    return [
        # the smallest call: one transform of a coarse grid, where latency is all
        _case("r2c_32_f32", "r2c", 32, 32, 32, "f32"),
        # a laptop-sized grid in double precision, there and back
        _case("both_64_f64", "both", 64, 64, 64, "f64"),
        # a channel-like box, every axis of another length, back from a spectrum
        _case("c2r_96x48x384_f32", "c2r", 96, 48, 384, "f32", "turbulence"),
        _case("c2r_192x128x384_f64", "c2r", 192, 128, 384, "f64", "turbulence"),
        # three velocity components per call
        _case("both_3x256_f32", "both", 256, 256, 256, "f32", "turbulence", 3),
        # a training step through a spectral filter (forward and both adjoints)
        _case("grad_256_f32", "grad", 256, 256, 256, "f32"),
        # ordinary production grids
        _case("r2c_512_f32", "r2c", 512, 512, 512, "f32", "turbulence"),
        _case("inplace_512_f64", "inplace", 512, 512, 512, "f64"),
        # the headline grid in both precisions
        _case("inplace_1024_f32", "inplace", 1024, 1024, 1024, "f32"),
        _case("inplace_1024_f64", "inplace", 1024, 1024, 1024, "f64"),
        # the largest: 3 * 2^k lengths, and the longest columns
        _case("inplace_1536_f32", "inplace", 1536, 1536, 1536, "f32"),
        _case("inplace_2048x2048x1024_f32", "inplace", 2048, 2048, 1024, "f32"),
    ]


def draw(rng):
    op = rng.choice(["r2c", "c2r", "both", "inplace", "grad"])
    dtype = rng.choice(["f32", "f32", "f64"])
    batch = rng.choice([1, 1, 1, 2, 3, 5])
    # in 64 bits a pass costs about 20 times as much, and a training step holds several copies
    most = 2.0 ** ((31 if dtype == "f32" else 28) - (3 if op == "grad" else 0))
    while True:
        n0, n1, n2 = rng.choice(_COLUMNS), rng.choice(_COLUMNS), rng.choice(_LINES)
        if 2.0 ** 12 <= batch * n0 * n1 * n2 <= most:
            break
    small = batch * n0 * n1 * n2 <= 2 ** 28
    return _case(None, op, n0, n1, n2, dtype, rng.choice(["uniform", "turbulence"]) if small else "uniform", batch)


def _shape(case):
    s = (case["n0"], case["n1"], case["n2"])
    return (case["batch"],) + s if case["batch"] > 1 else s


def _wavenumbers_squared(case, dtype):
    n0, n1, n2 = case["n0"], case["n1"], case["n2"]
    k0 = torch.fft.fftfreq(n0, 1.0 / n0, device="cuda", dtype=dtype)
    k1 = torch.fft.fftfreq(n1, 1.0 / n1, device="cuda", dtype=dtype)
    k2 = torch.fft.rfftfreq(n2, 1.0 / n2, device="cuda", dtype=dtype)
    return k0[:, None, None] ** 2 + k1[:, None] ** 2 + k2 ** 2


def _uniform(case, seed):
    g = torch.Generator(device="cuda")
    g.manual_seed(seed)
    return torch.empty(_shape(case), dtype=_DTYPES[case["dtype"]], device="cuda").uniform_(-1.0, 1.0, generator=g)


def _turbulence_spectrum(case, seed):
    X = torch.fft.rfftn(_uniform(case, seed), dim=(-3, -2, -1))
    return X.mul_(_wavenumbers_squared(case, X.real.dtype).clamp_(min=1.0).pow_(-11.0 / 12.0))


def _field(case, seed):
    if case["field"] == "uniform":
        return _uniform(case, seed)
    return torch.fft.irfftn(_turbulence_spectrum(case, seed), s=_shape(case)[-3:], dim=(-3, -2, -1)).contiguous()


def _spectrum(case, seed):
    if case["field"] == "uniform":
        return torch.fft.rfftn(_uniform(case, seed), dim=(-3, -2, -1)).contiguous()
    return _turbulence_spectrum(case, seed).contiguous()


def _filter(case, dtype):
    n = min(case["n0"], case["n1"], case["n2"])
    return torch.exp_(_wavenumbers_squared(case, dtype).mul_(-16.0 / n ** 2))


def prepare(case, seed):
    op, dtype = case["op"], _DTYPES[case["dtype"]]
    state = {"op": op, "shape": _shape(case)}
    # the plan that a program keeps; rfft3 and irfft3 find it again by its sizes
    state["plan"] = plan = fft3d.get_plan((case["n0"], case["n1"], case["n2"]), dtype, "cuda", case["batch"])
    if op == "c2r":
        state["X"] = _spectrum(case, seed)
    elif op == "inplace":
        state["buf"] = plan.empty_padded()
        state["buf"][..., case["n2"]:] = 0
        state["buf"][..., :case["n2"]].copy_(_field(case, seed))
    else:
        state["x"] = _field(case, seed)
    if op == "grad":
        state["x"].requires_grad_(True)
        state["filter"] = _filter(case, dtype)
        state["target"] = _uniform(case, seed + 1)
    return state


def run(state):
    op, shape = state["op"], state["shape"]
    if op == "r2c":
        return fft3d.rfft3(state["x"])
    if op == "c2r":
        return fft3d.irfft3(state["X"], shape)
    if op == "both":
        X = fft3d.rfft3(state["x"])
        return X, fft3d.irfft3(X, shape)
    if op == "inplace":
        plan, buf = state["plan"], state["buf"]
        plan.r2c_(buf)
        plan.c2r_(buf)
        return buf[..., :shape[-1]]
    x = state["x"]
    x.grad = None
    y = fft3d.irfft3(fft3d.rfft3(x) * state["filter"], shape)
    loss = 0.5 * ((y - state["target"]) ** 2).sum()
    loss.backward()
    return y.detach(), x.grad


def work(case):
    n = case["n0"] * case["n1"] * case["n2"] * case["batch"]
    rows = case["n0"] * case["n1"] * case["batch"]
    size = 4 if case["dtype"] == "f32" else 8
    real, cplx = n * size, rows * (case["n2"] // 2 + 1) * 2 * size
    flops = 2.5 * n * math.log2(case["n0"] * case["n1"] * case["n2"])
    op = case["op"]
    if op in ("r2c", "c2r"):
        return {"bytes": real + cplx, "flops": flops}
    if op in ("both", "inplace"):
        return {"bytes": 2 * (real + cplx), "flops": 2 * flops}
    # forward and backward through both transforms (the saved spectrum is not read again: the
    # filter is linear), the filter twice, the loss and its gradient
    filt = cplx // 2 // case["batch"]
    return {"bytes": 4 * (real + cplx) + 2 * (2 * cplx + filt) + 4 * real, "flops": 4 * flops + 2 * cplx / size + 6 * n}


def exact(case, seed):
    op, shape, dims = case["op"], _shape(case), (-3, -2, -1)
    if op == "c2r":
        return torch.fft.irfftn(_spectrum(case, seed).to(torch.complex128), s=shape[-3:], dim=dims)
    if op == "inplace":
        return _field(case, seed).to(torch.float64)
    x = _field(case, seed).to(torch.float64)
    X = torch.fft.rfftn(x, dim=dims)
    if op == "r2c":
        return X
    if op == "both":
        return X, x
    filt = _filter(case, _DTYPES[case["dtype"]]).to(torch.float64)
    target = _uniform(case, seed + 1).to(torch.float64)
    y = torch.fft.irfftn(X * filt, s=shape[-3:], dim=dims)
    # the filter is real and even, so it is its own adjoint
    return y, torch.fft.irfftn(torch.fft.rfftn(y - target, dim=dims) * filt, s=shape[-3:], dim=dims)
