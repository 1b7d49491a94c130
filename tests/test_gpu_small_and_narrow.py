"""Calls next to the limits of the tile kernels' rules, where the general kernels are the
faster ones: the schedule they run, told by launches or by the bytes of the
result (the two kernels round differently), and their error."""
import pytest
import torch

from paper_2209_15040_gb300 import wsfft as W
from tests._helpers import DT, TOL

pytestmark = pytest.mark.gpu


def _input(shape, dtype):
    x = torch.randn(*shape, 2, device="cuda", generator=torch.Generator("cuda").manual_seed(3))
    return torch.view_as_complex(x) if dtype == "c32" else x.to(torch.float16 if dtype == "c16f" else torch.bfloat16)


def _run(plan, x):
    out = torch.empty_like(x)
    plan.execute(x.data_ptr(), out.data_ptr())
    torch.cuda.synchronize()
    return out


def _same(a, b):
    a, b = (torch.view_as_real(t) if t.is_complex() else t for t in (a, b))
    return torch.equal(a, b)


def _diff(a, b):
    a, b = (torch.view_as_real(t) if t.is_complex() else t.float() for t in (a, b))
    return float((a - b).norm() / b.norm())


# points, stride, elements, general shape, tiled?
AXES = [("c16f", 4096, 8, 1 << 23, (16, 0), False), ("c16bf", 4096, 256, 1 << 23, (16, 0), False),
        ("c16f", 4096, 16, 1 << 25, (16, 0), False), ("c16f", 4096, 4096, 1 << 25, (16, 0), False),
        ("c16f", 4096, 32, 1 << 25, (16, 0), True), ("c16bf", 4096, 1024, 1 << 25, (16, 0), True),
        ("c32", 1024, 8, 1 << 25, (16, 3008), False), ("c32", 1024, 8, 1 << 22, (16, 3008), True),
        ("c32", 1024, 16, 1 << 25, (16, 3008), True)]


@pytest.mark.parametrize("dtype, n, inner, elems, general, tiled", AXES)
def test_strided_axis(dtype, n, inner, elems, general, tiled):
    batch = elems // (n * inner)
    x = _input((elems,), dtype)
    plan = W.AxisPlan(n, inner, DT[dtype], W.FORWARD, batch, W.NORM_ORTHO)
    default = _run(plan, x)
    plan.set_pass_variant(0, *general)
    chosen = _run(plan, x)
    plan.close()
    assert _same(default, chosen) != tiled
    assert _diff(default, chosen) < TOL[dtype]


# a strided superstep right after rows of 2048 or 4096 points, 16-bit storage
@pytest.mark.parametrize("dims, batch, general, tiled", [((512, 2048), 4, (16, 3016), False),
                                                         ((512, 4096), 2, (16, 3016), False),
                                                         ((128, 2048), 20, (16, 0), False),
                                                         ((512, 2048), 6, (16, 3016), True),
                                                         ((512, 1024), 8, (16, 3016), True)])
def test_after_long_rows(dims, batch, general, tiled):
    x = _input((batch,) + dims, "c16f")
    plan = W.Plan(dims, W.C16F, W.FORWARD, batch)
    default = _run(plan, x)
    plan.set_pass_variant(1, *general)
    chosen = _run(plan, x)
    plan.close()
    assert _same(default, chosen) != tiled
    assert _diff(default, chosen) < TOL["c16f"]


@pytest.mark.parametrize("dims, batch, wide", [((2048, 512), 2, False), ((2048, 512), 3, True),
                                               ((4096, 512), 1, True), ((2048, 1024), 1, True)])
def test_digit_of_2048_points_beside_512(dims, batch, wide):
    x = _input((batch,) + dims, "c16f")
    plan = W.Plan(dims, W.C16F, W.FORWARD, batch)
    default = _run(plan, x)
    plan.set_engine(4)  # one launch per superstep for this shape
    chosen = _run(plan, x)
    plan.close()
    assert _same(default, chosen) != wide
    assert _diff(default, chosen) < TOL["c16f"]


# 2^17 elements and next to them: one launch per axis where that is the faster
@pytest.mark.parametrize("dtype, dims, batch, launches", [
    ("c32", (32, 64, 64), 1, 3), ("c32", (64, 64), 32, 2), ("c32", (64, 64), 33, 1), ("c32", (2, 64, 128), 8, 3),
    ("c32", (32, 32), 128, 1), ("c32", (32, 32, 32), 4, 2), ("c32", (32, 32), 127, 1),
    ("c16f", (32, 64, 64), 1, 3), ("c16bf", (8, 128, 64), 2, 3), ("c16f", (64, 64), 32, 1)])
def test_fused_from_2_17_elements(dtype, dims, batch, launches):
    x = _input((batch,) + dims, dtype)
    for direction in (W.FORWARD, W.INVERSE):
        plan = W.Plan(dims, DT[dtype], direction, batch, W.NORM_ORTHO)
        plan.profile(8)
        default = _run(plan, x)
        assert len(plan.launch_times()) == launches
        plan.profile(0)
        plan.set_engine(4)
        assert _diff(default, _run(plan, x)) < TOL[dtype]
        plan.close()
