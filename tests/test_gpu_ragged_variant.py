"""Choosing a ragged plan's queue variant and going back: the values of a new
plan bring back what a new plan runs, and the same results."""
import ctypes

import pytest
import torch

from paper_2209_15040_gb300 import build
from paper_2209_15040_gb300 import wsfft as W

pytestmark = pytest.mark.gpu

SHAPES = [(32, 64, 32), (64, 64, 64), (128, 32, 64)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build_library()
    W.lib()
    torch.cuda.init()


def _execute(plan, xs):
    ys = [torch.empty_like(x) for x in xs]
    plan.execute([x.data_ptr() for x in xs], [y.data_ptr() for y in ys])
    n = ctypes.c_int()
    assert W.lib().wsfft_plan_launch_times(plan.handle, None, 0, ctypes.byref(n)) == 0
    return ys, n.value


@pytest.mark.parametrize("dtype", ["c32", "c16f"])
def test_default_values_restore_a_new_plan(dtype):
    g = torch.Generator(device="cuda").manual_seed(51)
    xs = [torch.randn(*s, 2, generator=g, device="cuda") for s in SHAPES]
    xs = [torch.view_as_complex(x) if dtype == "c32" else x.half() for x in xs]
    plan = W.RaggedPlan(SHAPES, W.C32 if dtype == "c32" else W.C16F)
    assert W.lib().wsfft_plan_profile(plan.handle, 64) == 0
    new, launches = _execute(plan, xs)
    plan.set_variant(3, 2)
    assert _execute(plan, xs)[1] == 1
    plan.set_variant(0, 1)
    back, again = _execute(plan, xs)
    assert again == launches and (launches > 1) == (dtype == "c32")
    for y, z in zip(new, back):
        assert torch.equal(y, z)
    plan.close()
