"""GPU parity of the fused tile schedule (csrc/tile_fused.cuh): every shape
the plan builder's rule accepts at the edges of its range -- whole slabs with
full and partial tiles, split middle axes with the fewest and the most classes
-- in and out of place, both directions, every storage type, against the FP64
oracle; and the schedule a plan falls back to."""
import pytest
import torch

import oracle
from paper_2209_15040_gb300 import build
from paper_2209_15040_gb300 import wsfft as W
from tests._helpers import DT, TOL, seeded, to_device, to_host_c128

pytestmark = pytest.mark.gpu

SLABS = [(n1, n2) for n1 in (32, 64, 128, 256) for n2 in (32, 64, 128, 256) if n1 * n2 <= 1 << 13]
# n0, n1, n2: XB = log2 n0 in 5..8 with 1..4 bits of classes; rows of 16 .. n2 elements
SPLIT = [(128, 64, 256), (128, 128, 128), (256, 64, 256), (64, 128, 128), (32, 64, 256), (256, 128, 128),
         (64, 256, 128), (32, 128, 256), (128, 128, 256), (32, 256, 256), (64, 256, 256), (32, 512, 256),
         (32, 1024, 128), (128, 512, 64), (256, 256, 64), (256, 512, 32)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build_library()
    W.lib()
    torch.cuda.init()


def _launches(plan, x, out):
    plan.profile(8)
    plan.execute(x.data_ptr(), out.data_ptr())
    n = len(plan.launch_times())
    plan.profile(0)
    return n


def _check(dims, batch, dtype, direction, passes):
    xs, xc = seeded((batch,) + dims, 23, "uniform", dtype)
    x = to_device(xs, dtype)
    ref = oracle.fftn(xc, rank=len(dims), sign=direction, norm=oracle.NORM_ORTHO)
    plan = W.Plan(dims, DT[dtype], direction, batch, W.NORM_ORTHO)
    try:
        out = torch.empty_like(x)
        assert _launches(plan, x, out) == passes
        same = x.clone()
        plan.execute(same.data_ptr(), same.data_ptr())
        torch.cuda.synchronize()
        assert torch.equal(x, to_device(xs, dtype))  # the input is not written
        for got in (out, same):
            assert oracle.rel_l2(to_host_c128(got, dtype).reshape(ref.shape), ref) < TOL[dtype]
    finally:
        plan.close()


@pytest.mark.parametrize("dtype", ["c32", "c16f", "c16bf"])
@pytest.mark.parametrize("n1,n2", SLABS)
def test_whole_slabs(dtype, n1, n2):
    # below 2^17 elements one launch per axis, but for complex64 batches of
    # 32 x 32 slabs from 2^15 elements up (tiles of 2^11); then tiles of 2^13;
    # the last tile partial
    per, small = (1 << 13) // (n1 * n2), n1 * n2 == 1 << 10 and dtype == "c32"
    _check((n1, n2), 1, dtype, W.FORWARD, 2)
    _check((n1, n2), 5 * per + 1, dtype, W.INVERSE, 1 if small else 2)
    _check((n1, n2), 16 * per + 1, dtype, W.INVERSE, 1)
    _check((2, n1, n2), 2 * per + 1, dtype, W.FORWARD, 2 if small else 3)
    _check((2, n1, n2), 8 * per + 1, dtype, W.FORWARD, 2)


@pytest.mark.parametrize("dtype", ["c32", "c16f", "c16bf"])
@pytest.mark.parametrize("dims", SPLIT)
def test_split_middle_axis(dtype, dims):
    _check(dims, 1, dtype, W.FORWARD if dims[0] > 32 else W.INVERSE, 2)


def test_shapes_outside_the_rule_keep_their_passes():
    for dims, passes in [((16, 32), 2), ((32, 16), 2), ((64, 512), 2), ((256, 256, 256), 3), ((16, 128, 128), 3),
                         ((64, 512, 32), 3), ((512, 128, 128), 3)]:
        plan = W.Plan(dims)
        x = torch.zeros(dims, dtype=torch.complex64, device="cuda")
        assert _launches(plan, x, torch.empty_like(x)) == passes == plan.passes()[0]
        plan.close()


@pytest.mark.parametrize("norm", [W.NORM_PAPER, W.NORM_NONE, W.NORM_ORTHO, W.NORM_FORWARD])
def test_normalisations_match_the_unfused_schedule(norm):
    g = torch.Generator(device="cuda").manual_seed(29)
    for dims in ((32, 64, 64), (64, 128, 128)):
        for direction in (W.FORWARD, W.INVERSE):
            x = torch.view_as_complex(torch.randn(2, *dims, 2, generator=g, device="cuda"))
            plan = W.Plan(dims, W.C32, direction, 2, norm)
            fused, plain = torch.empty_like(x), torch.empty_like(x)
            assert _launches(plan, x, fused) == 2
            plan.set_pass_variant(0, 8 if dims[2] == 64 else 16, 0)  # any chosen shape: one launch per superstep
            assert _launches(plan, x, plain) == 3
            plan.set_pass_variant(0, 0, 0)
            assert _launches(plan, x, fused) == 2
            torch.cuda.synchronize()
            plan.close()
            assert ((fused - plain).norm() / plain.norm()).item() < TOL["c32"]


# a long strided axis beside a last axis of 512..4096 points: each row length,
# the digit taken from the middle axis, from the outer one, and (4096 x 4096) a
# tile of 2^14 elements
WIDE = [((2048, 512), 2), ((4096, 1024), 2), ((2048, 2048), 2), ((2048, 4096), 2), ((4096, 4096), 2),
        ((2, 4096, 512), 3), ((2048, 2, 1024), 3), ((4096, 4, 512), 3), ((1024, 512, 512), 3)]


@pytest.mark.parametrize("dtype", ["c32", "c16f", "c16bf"])
@pytest.mark.parametrize("dims,passes", WIDE)
def test_digit_of_a_long_axis(dtype, dims, passes):
    n = 1
    for v in dims:
        n *= v
    if n > 1 << 24 and dtype == "c16bf":
        pytest.skip("the largest shape in two storage types")
    batch = max(1, (1 << 21) // n)
    _check(dims, batch, dtype, W.FORWARD if len(dims) == 2 else W.INVERSE, passes)


def test_axes_outside_the_wide_rule():
    # the general kernels and the wide tiles agree on the shapes next to the
    # rule's limits, whichever of them runs
    for dtype, dims, batch in [("c32", (2048, 256), 2), ("c32", (2048, 512), 1), ("c16f", (2048, 512), 1),
                               ("c16f", (2048, 512), 2), ("c32", (1024, 256, 512), 1), ("c32", (1024, 4096), 1)]:
        xs, xc = seeded((batch,) + dims, 31, "uniform", dtype)
        x = to_device(xs, dtype)
        outs = []
        for chosen in (False, True):
            plan = W.Plan(dims, DT[dtype], W.FORWARD, batch, W.NORM_ORTHO)
            if chosen:  # any chosen shape: one launch per superstep
                e = 8 if dims[-1] == 512 else 16
                plan.set_pass_variant(0, e, 8 if e == 8 else 0)
            out = torch.empty_like(x)
            plan.execute(x.data_ptr(), out.data_ptr())
            torch.cuda.synchronize()
            plan.close()
            outs.append(to_host_c128(out, dtype))
        assert oracle.rel_l2(outs[0], outs[1]) < TOL[dtype]
