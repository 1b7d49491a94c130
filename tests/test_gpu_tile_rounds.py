"""Tile kernels beyond one tile per block: whole slabs over several rounds of the
persistent loop with a partial tile in the last one, digits of an outer axis in
a batch, and the four-step over more than one workspace chunk -- each against
the FP64 oracle."""
import numpy as np
import pytest
import torch

import oracle
from paper_2209_15040_gb300 import build, inputs
from paper_2209_15040_gb300 import wsfft as W
from tests._helpers import DT, TOL, seeded, to_device, to_host_c128

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build_library()
    W.lib()
    torch.cuda.init()


def _check(dims, batch, dtype, direction, launches):
    xs, xc = seeded((batch,) + dims, 61, "uniform", dtype)
    x = to_device(xs, dtype)
    ref = oracle.fftn(xc, rank=len(dims), sign=direction, norm=oracle.NORM_ORTHO)
    plan = W.Plan(dims, DT[dtype], direction, batch, W.NORM_ORTHO)
    out = torch.full_like(x, float("nan"))
    plan.profile(8)
    plan.execute(x.data_ptr(), out.data_ptr())
    assert len(plan.launch_times()) == launches
    plan.profile(0)
    assert torch.equal(x, to_device(xs, dtype))  # the input is not written
    plan.execute(x.data_ptr(), x.data_ptr())
    torch.cuda.synchronize()
    plan.close()
    # transform by transform: a tile that went wrong is not averaged away
    for got in (out, x):
        diff = to_host_c128(got, dtype).reshape(ref.shape) - ref
        axes = tuple(range(1, ref.ndim))
        errors = np.sqrt((np.abs(diff) ** 2).sum(axis=axes) / (np.abs(ref) ** 2).sum(axis=axes))
        assert errors.max() < TOL[dtype]


@pytest.mark.parametrize("dtype", ["c32", "c16f", "c16bf"])
@pytest.mark.parametrize("n1,n2", [(32, 32), (64, 64), (32, 256), (256, 32)])
def test_slabs_over_several_rounds(dtype, n1, n2):
    sms = torch.cuda.get_device_properties(0).multi_processor_count
    blocks = sms * (2 if dtype == "c32" else 3)
    tiles = 2 * blocks + 3  # the third round is for three blocks
    # one slab more: a partial tile in that round (slabs of a whole tile: a fourth one)
    _check((n1, n2), tiles * ((1 << 13) // (n1 * n2)) + 1, dtype, W.FORWARD, 1)


@pytest.mark.parametrize("dtype", ["c32", "c16f", "c16bf"])
@pytest.mark.parametrize("dims", [(2048, 2, 512), (4096, 2, 1024)])
def test_digit_of_the_outer_axis_in_a_batch(dtype, dims):
    _check(dims, 3, dtype, W.INVERSE, 3)


@pytest.mark.parametrize("dtype,n,per_chunk", [("c32", 1 << 20, 512), ("c16f", 1 << 18, 4096)])
def test_four_step_over_two_chunks(dtype, n, per_chunk):
    batch = per_chunk + 3
    g = torch.Generator(device="cuda").manual_seed(62)
    x = torch.randn(batch, n, 2, generator=g, device="cuda", dtype=torch.float32 if dtype == "c32" else torch.float16)
    if dtype == "c32":
        x = torch.view_as_complex(x)
    out = torch.full_like(x, float("nan"))
    plan = W.Plan((n,), DT[dtype], W.FORWARD, batch, W.NORM_ORTHO)
    plan.profile(8)
    plan.execute(x.data_ptr(), out.data_ptr())
    assert len(plan.launch_times()) == 4  # two supersteps for each chunk of 4 GiB
    plan.close()
    for i in (0, 1, per_chunk - 1, per_chunk, batch - 1):
        ref = oracle.fftn(to_host_c128(x[i], dtype), rank=1, norm=oracle.NORM_ORTHO)
        assert oracle.rel_l2(to_host_c128(out[i], dtype).reshape(ref.shape), ref) < TOL[dtype]
    assert bool(torch.isfinite(torch.view_as_real(out) if dtype == "c32" else out).all())
