"""The transforms that this library is timed on, through its public entry points.

A case names a call (or the two calls of a round trip) as a program makes it: the
shape, the batch, the storage type, the direction, and whether the program goes
through ``fftn`` / ``ifftn`` on tensors, through a plan that it keeps, through
autograd, or through a ragged plan.  Shapes follow the configurations of the
bench and the tests: cubes of 32..1024 points, 1D 2^20 in a batch of 512, the 4096^2
plane, the batched 1D sweep, the 8 x 128^3 gradient step and the 256-shape ragged batch.
"""
import math

import numpy as np
import torch

from paper_2209_15040_gb300 import wsfft

_CODE = {"c32": wsfft.C32, "c16f": wsfft.C16F, "c16bf": wsfft.C16BF}
_TORCH = {"c16f": torch.float16, "c16bf": torch.bfloat16}
_RAGGED_AXES = (32, 64, 128, 256)


def _case(name, dims, batch=1, dtype="c32", steps="f", api="tensor"):
    return {"name": name, "kind": "transform", "dims": "x".join(str(d) for d in dims), "batch": batch,
            "dtype": dtype, "steps": steps, "api": api}


def listed():
    return [
        # one small cube at a time, plan and buffers kept: latency and launches
        _case("cube32_plan", (32, 32, 32), api="plan"),
        # a spectral solver's step on one mid-sized field that fits in L2
        _case("cube128_round_trip", (128, 128, 128), steps="fi"),
        # the same on a field of the size of L2
        _case("cube256_round_trip", (256, 256, 256), steps="fi"),
        # the benchmark's own step
        _case("cube512_round_trip", (512, 512, 512), steps="fi"),
        # the largest field: 8 GiB in, 8 GiB out
        _case("cube1024_forward", (1024, 1024, 1024)),
        # the benchmark's step in half-precision storage
        _case("cube512_fp16_round_trip", (512, 512, 512), dtype="c16f", steps="fi"),
        # bfloat16 storage, inverse only, overwriting its input: a solver that has no room for a second field
        _case("cube256_bf16_in_place", (256, 256, 256), batch=3, dtype="c16bf", steps="i", api="in_place"),
        # long signals, each longer than one block's pencil
        _case("line2e20_x512", (1 << 20,), batch=512),
        # a large image
        _case("plane4096_forward", (4096, 4096)),
        # the batched 1D sweep, with a batch that is no multiple of any tile
        _case("lines1024_x100003", (1024,), batch=100003),
        # a training step through the transform: loss = sum |W * FFT3(x)|^2, forward and gradient
        {"name": "gradient_8x128", "kind": "gradient", "dims": "128x128x128", "batch": 8},
        # 256 fields of uneven shapes in one launch
        {"name": "ragged_256", "kind": "ragged", "count": 256, "shape_seed": 4},
    ]


def _log2_between(rng, lo, hi):
    return 1 << rng.randint(lo, hi)


def draw(rng):
    known = [{k: v for k, v in c.items() if k != "name"} for c in listed()]
    while True:
        case = _drawn(rng)
        if case not in known:
            return case


def _drawn(rng):
    what = rng.random()
    if what < 0.10:
        n = _log2_between(rng, 5, 8)
        most = max(1, (1 << 26) // n ** 3)
        return {"kind": "gradient", "dims": "%dx%dx%d" % (n, n, n),
                "batch": int(round(2 ** rng.uniform(0, math.log2(min(most, 64)))))}
    if what < 0.22:
        return {"kind": "ragged", "count": int(round(2 ** rng.uniform(3, 8))), "shape_seed": rng.randint(5, 10000)}
    dtype = rng.choice(("c32", "c32", "c32", "c16f", "c16bf"))
    steps = rng.choice(("f", "f", "i", "fi"))
    shape = rng.random()
    if shape < 0.25:  # lines
        dims = (_log2_between(rng, 6, 22),)
    elif shape < 0.45:  # planes
        dims = (_log2_between(rng, 6, 12), _log2_between(rng, 6, 12))
    elif shape < 0.75:  # cubes
        dims = (_log2_between(rng, 5, 9),) * 3
    else:  # boxes
        dims = tuple(_log2_between(rng, 4, 9) for _ in range(3))
    n = math.prod(dims)
    total = 2 ** rng.uniform(max(17, math.log2(n)), 28)
    batch = max(1, int(total / n))
    if batch > 8:
        batch |= 1
    return {"kind": "transform", "dims": "x".join(str(d) for d in dims), "batch": batch, "dtype": dtype,
            "steps": steps, "api": "in_place" if steps != "fi" and dtype != "c32" and rng.random() < 0.3 else "tensor"}


def _dims(case):
    return tuple(int(d) for d in case["dims"].split("x"))


def _gen(seed):
    return torch.Generator(device="cuda").manual_seed(int(seed))


def _field(shape, dtype, seed):
    """N(0,1) real and imaginary parts (complex64), uniform[-1,1) in 16-bit storage."""
    g = _gen(seed)
    if dtype == "c32":
        return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda"))
    return (torch.rand(*shape, 2, generator=g, device="cuda", dtype=torch.float32) * 2 - 1).to(_TORCH[dtype])


def _ragged_shapes(case):
    rng = np.random.default_rng(case["shape_seed"])
    return [tuple(int(v) for v in s) for s in rng.choice(np.asarray(_RAGGED_AXES), size=(case["count"], 3))]


def _offsets(shapes):
    offs, at = [], 0
    for s in shapes:
        offs.append(at)
        at += math.prod(s)
    return offs, at


def prepare(case, seed):
    state = {"case": case}
    if case["kind"] == "gradient":
        shape = (case["batch"],) + _dims(case)
        state["x"] = _field(shape, "c32", seed).requires_grad_(True)
        state["w"] = torch.rand(*shape, generator=_gen(seed + 1_000_003), device="cuda")
        return state
    if case["kind"] == "ragged":
        shapes = _ragged_shapes(case)
        offs, total = _offsets(shapes)
        state["x"] = _field((total,), "c32", seed)
        state["y"] = torch.empty_like(state["x"])
        state["in"] = [state["x"].data_ptr() + 8 * o for o in offs]
        state["out"] = [state["y"].data_ptr() + 8 * o for o in offs]
        state["plan"] = wsfft.RaggedPlan(shapes)
        return state
    dims, batch = _dims(case), case["batch"]
    shape = ((batch,) if batch > 1 else ()) + dims
    state["x"] = _field(shape, case["dtype"], seed)
    state["rank"] = len(dims)
    if case["api"] != "tensor":
        direction = wsfft.INVERSE if case["steps"] == "i" else wsfft.FORWARD
        state["plan"] = wsfft.Plan(dims, _CODE[case["dtype"]], direction, batch)
        state["y"] = state["x"] if case["api"] == "in_place" else torch.empty_like(state["x"])
    return state


def run(state):
    case, x = state["case"], state["x"]
    if case["kind"] == "gradient":
        y = wsfft.fftn(x, rank=3)
        loss = (state["w"] * y).abs().pow(2).sum()
        (grad,) = torch.autograd.grad(loss, x)
        return {"loss": loss.detach(), "spectrum": y.detach(), "grad": grad}
    if case["kind"] == "ragged":
        state["plan"].execute(state["in"], state["out"])
        return state["y"]
    if case["api"] != "tensor":
        state["plan"].execute(x.data_ptr(), state["y"].data_ptr())
        return state["y"]
    rank = state["rank"]
    if case["steps"] == "f":
        return wsfft.fftn(x, rank=rank)
    if case["steps"] == "i":
        return wsfft.ifftn(x, rank=rank)
    spectrum = wsfft.fftn(x, rank=rank)
    return {"spectrum": spectrum, "field": wsfft.ifftn(spectrum, rank=rank)}


def _flops(dims, batch=1):
    n = math.prod(dims)
    return 5.0 * batch * n * math.log2(n)


def work(case):
    if case["kind"] == "gradient":
        dims, batch = _dims(case), case["batch"]
        n = batch * math.prod(dims)
        # forward: x and W read, spectrum written; backward: spectrum and W read, gradient written
        return {"bytes": float(n * (8 + 4 + 8 + 8 + 4 + 8)), "flops": 2 * _flops(dims, batch) + 10.0 * n}
    if case["kind"] == "ragged":
        shapes = _ragged_shapes(case)
        return {"bytes": 16.0 * sum(math.prod(s) for s in shapes), "flops": sum(_flops(s) for s in shapes)}
    dims, batch = _dims(case), case["batch"]
    elem = 8 if case["dtype"] == "c32" else 4
    calls = len(case["steps"])
    return {"bytes": 2.0 * elem * batch * math.prod(dims) * calls, "flops": calls * _flops(dims, batch)}


def _double(x):
    if x.is_complex():
        return x.to(torch.complex128)
    return torch.view_as_complex(x.to(torch.float64))


def exact(case, seed):
    if case["kind"] == "gradient":
        state = prepare(case, seed)
        x = state["x"].detach().to(torch.complex128).requires_grad_(True)
        y = torch.fft.fftn(x, dim=(-3, -2, -1))
        loss = (state["w"].double() * y).abs().pow(2).sum()
        (grad,) = torch.autograd.grad(loss, x)
        return {"loss": loss.detach(), "spectrum": y.detach(), "grad": grad}
    if case["kind"] == "ragged":
        shapes = _ragged_shapes(case)
        offs, total = _offsets(shapes)
        x = _field((total,), "c32", seed)
        out = torch.empty(total, dtype=torch.complex128, device="cuda")
        for s, o in zip(shapes, offs):
            n = math.prod(s)
            out[o:o + n] = torch.fft.fftn(x[o:o + n].to(torch.complex128).reshape(s)).reshape(-1)
        return out
    dims, batch = _dims(case), case["batch"]
    x = _field(((batch,) if batch > 1 else ()) + dims, case["dtype"], seed)
    axes = tuple(range(-len(dims), 0))
    norm = "backward" if case["dtype"] == "c32" else "ortho"  # the library's defaults for the two kinds of storage
    pairs = (lambda z: z) if case["dtype"] == "c32" else torch.view_as_real
    x = _double(x)
    if case["steps"] == "fi":
        spectrum = torch.fft.fftn(x, dim=axes, norm=norm)
        return {"spectrum": pairs(spectrum), "field": pairs(x)}
    if case["steps"] == "f":
        return pairs(torch.fft.fftn(x, dim=axes, norm=norm))
    return pairs(torch.fft.ifftn(x, dim=axes, norm=norm))
