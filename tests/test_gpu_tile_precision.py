"""The tile kernels (csrc/tile.cuh, tile_fused.cuh) are at least as accurate in
complex64 as the one-tile-per-block kernels: rel-L2 against a double-precision
transform of the same inputs, both schedules of a plan.  From 2^18 elements up
the figure repeats within 0.2% over seeds, and the radices' roundings leave the
tile kernels 5-10% below, so no margin is allowed."""
import pytest
import torch

from paper_2209_15040_gb300 import build
from paper_2209_15040_gb300 import wsfft as W

pytestmark = pytest.mark.gpu

PAIR = 3000  # tile code of the split-form pencil pairs


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build_library()
    W.lib()
    torch.cuda.init()


def _field(shape, seed):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda"))


def _error(y, ref):
    return ((y.to(torch.complex128) - ref).norm() / ref.norm()).item()


def _execute(plan, x):
    y = torch.empty_like(x)
    plan.execute(x.data_ptr(), y.data_ptr())
    return y


# whole slabs, a split middle axis, a digit of a long axis beside rows of 4096
# and of 1024 points; values per thread that select the general kernel of pass 0
@pytest.mark.parametrize("dims,batch,general", [
    ((32, 32, 32), 8, (8, 0)), ((64, 64), 64, (8, 0)), ((32, 256), 64, (16, 0)), ((256, 32), 64, (8, 0)),
    ((128, 128, 128), 1, (16, 0)), ((32, 256, 256), 1, (16, 0)), ((256, 64, 256), 1, (16, 0)),
    ((4096, 4096), 1, (16, 0)), ((2048, 1024), 1, (32, 8))])
def test_fused_schedules(dims, batch, general):
    x = _field((batch,) + dims, 41)
    ref = torch.fft.fftn(x.to(torch.complex128), dim=tuple(range(1, len(dims) + 1)))
    plan = W.Plan(dims, W.C32, W.FORWARD, batch, W.NORM_NONE)
    fused = _error(_execute(plan, x), ref)
    plan.set_pass_variant(0, *general)  # any chosen shape: one launch per superstep
    plain = _error(_execute(plan, x), ref)
    plan.close()
    assert fused <= plain


def test_strided_axis_of_1024_points():
    x = _field((4, 1024, 1024), 42)
    ref = torch.fft.fft(x.to(torch.complex128), dim=1)
    plan = W.AxisPlan(1024, 1024, W.C32, W.FORWARD, 4, W.NORM_NONE)
    tiles = _error(_execute(plan, x), ref)
    plan.set_pass_variant(0, 16, PAIR + 8)
    pairs = _error(_execute(plan, x), ref)
    plan.close()
    assert tiles <= pairs


def test_four_step_of_2_20_points():
    # from 2^23 elements up the four-step runs on the tile kernels as 1024 x
    # 1024, below on the general ones as 2048 x 512
    x = _field((8, 1 << 20), 43)
    ref = torch.fft.fft(x.to(torch.complex128), dim=1)
    tiled = _error(W.fftn(x, rank=1, norm="none"), ref)
    parts = torch.cat([W.fftn(x[i:i + 4], rank=1, norm="none") for i in (0, 4)])
    assert tiled <= _error(parts, ref)


def test_ragged_groups():
    shapes = [(32, 64, 64), (128, 128, 128), (64, 256, 128)]
    xs = [_field(s, 44 + i) for i, s in enumerate(shapes)]
    plan = W.RaggedPlan(shapes, W.C32, W.FORWARD)
    errors = []
    for queue in (False, True):
        if queue:
            plan.set_variant(0, 2)
        ys = [torch.empty_like(x) for x in xs]
        plan.execute([x.data_ptr() for x in xs], [y.data_ptr() for y in ys])
        errors.append([_error(y, torch.fft.fftn(x.to(torch.complex128))) for x, y in zip(xs, ys)])
    plan.close()
    for groups, queue in zip(*errors):
        assert groups <= queue
