"""GPU parity of the grouped launches of a ragged batch (complex64 out of place):
all 64 shapes of 32..256 points per axis, one instance of a shape and several,
against the FP64 oracle; in-place instances and a chosen queue variant keep the
queue; capture into a graph and replay on new data; two executes with other
pointers in a row."""
import itertools

import numpy as np
import pytest
import torch

import oracle
from paper_2209_15040_gb300 import build, inputs
from paper_2209_15040_gb300 import wsfft as W
from tests._helpers import TOL

pytestmark = pytest.mark.gpu

AXES = (32, 64, 128, 256)


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build_library()
    W.lib()
    torch.cuda.init()


def _launches(plan, ins, outs):
    lib = W.lib()
    assert lib.wsfft_plan_profile(plan.handle, 256) == 0
    plan.execute([t.data_ptr() for t in ins], [t.data_ptr() for t in outs])
    import ctypes
    n = ctypes.c_int()
    assert lib.wsfft_plan_launch_times(plan.handle, None, 0, ctypes.byref(n)) == 0
    assert lib.wsfft_plan_profile(plan.handle, 0) == 0
    return n.value


@pytest.mark.parametrize("n0", AXES)
@pytest.mark.parametrize("direction", [W.FORWARD, W.INVERSE])
def test_every_shape(n0, direction):
    shapes = [(n0, n1, n2) for n1, n2 in itertools.product(AXES, AXES)] + [(n0, 64, 64), (n0, 128, 32)]
    xs = [inputs.complex_input(s, 900 + i, "normal", "c32") for i, s in enumerate(shapes)]
    xd = [torch.from_numpy(x).cuda() for x in xs]
    outs = [torch.empty_like(x) for x in xd]
    plan = W.RaggedPlan(shapes, W.C32, direction)
    assert _launches(plan, xd, outs) > 1
    torch.cuda.synchronize()
    assert plan.sync_status() == W.SUCCESS
    plan.close()
    for x, d, y in zip(xs, xd, outs):
        assert np.array_equal(d.cpu().numpy(), x)
        ref = oracle.fftn(x.astype(np.complex128), rank=3, sign=direction, norm=oracle.NORM_PAPER)
        assert oracle.rel_l2(y.cpu().numpy(), ref) < TOL["c32"]


def test_in_place_and_variants_keep_the_queue():
    shapes = [(32, 64, 32), (64, 128, 128), (32, 256, 64)]
    xs = [inputs.complex_input(s, 950 + i, "normal", "c32") for i, s in enumerate(shapes)]
    refs = [oracle.fftn(x.astype(np.complex128)) for x in xs]
    for variant, in_place in ((False, True), (True, False)):
        xd = [torch.from_numpy(x).cuda() for x in xs]
        outs = [torch.empty_like(x) for x in xd]
        if in_place:
            outs[1] = xd[1]
        plan = W.RaggedPlan(shapes, W.C32, W.FORWARD)
        if variant:
            plan.set_variant(0, 2)
        assert _launches(plan, xd, outs) == 1
        torch.cuda.synchronize()
        assert plan.sync_status() == W.SUCCESS
        plan.close()
        for y, ref in zip(outs, refs):
            assert oracle.rel_l2(y.cpu().numpy(), ref) < TOL["c32"]


def test_capture_replay_and_new_pointers():
    shapes = [(64, 64, 64), (32, 128, 128), (128, 32, 64), (256, 256, 128)]
    g = torch.Generator(device="cuda").manual_seed(5)
    new = lambda: [torch.view_as_complex(torch.randn(*s, 2, generator=g, device="cuda")) for s in shapes]  # noqa: E731
    xa, xb = new(), new()
    ya, yb = [torch.empty_like(x) for x in xa], [torch.empty_like(x) for x in xa]
    want = [[W.fftn(x) for x in v] for v in (xa, xb)]
    plan = W.RaggedPlan(shapes, W.C32, W.FORWARD)
    plan.execute([x.data_ptr() for x in xa], [y.data_ptr() for y in ya])
    plan.execute([x.data_ptr() for x in xb], [y.data_ptr() for y in yb])
    torch.cuda.synchronize()
    for got, ref in ((ya, want[0]), (yb, want[1])):
        for y, r in zip(got, ref):
            assert ((y - r).norm() / r.norm()).item() < TOL["c32"]
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.execute([x.data_ptr() for x in xb], [y.data_ptr() for y in yb])
    for x, src in zip(xb, xa):
        x.copy_(src)
    graph.replay()
    torch.cuda.synchronize()
    for y, r in zip(yb, want[0]):
        assert ((y - r).norm() / r.norm()).item() < TOL["c32"]
    plan.close()


def test_back_to_back_executes_wait_for_each_other():
    """Launches of one trip overlap; the next trip, the next execute and plain
    work on the stream wait for all of them.  Forward and inverse in a chain
    with copies between, and ten rounds grow the error by at most ten roundings
    of each transform."""
    rng = np.random.default_rng(17)
    shapes = [tuple(int(v) for v in rng.choice(np.asarray(AXES), size=3)) for _ in range(24)] + [(256, 256, 128)]
    fwd, inv = W.RaggedPlan(shapes, W.C32, W.FORWARD), W.RaggedPlan(shapes, W.C32, W.INVERSE)
    g = torch.Generator(device="cuda").manual_seed(8)
    x = [torch.view_as_complex(torch.randn(*s, 2, generator=g, device="cuda")) for s in shapes]
    a, b, c = ([torch.empty_like(v) for v in x] for _ in range(3))
    for v, w in zip(a, x):
        v.copy_(w)
    for _ in range(10):
        fwd.execute([v.data_ptr() for v in a], [v.data_ptr() for v in b])
        for v, w in zip(c, b):
            v.copy_(w)
        inv.execute([v.data_ptr() for v in c], [v.data_ptr() for v in b])
        torch._foreach_copy_(a, b)
    torch.cuda.synchronize()
    assert fwd.sync_status() == W.SUCCESS and inv.sync_status() == W.SUCCESS
    fwd.close()
    inv.close()
    for v, w in zip(a, x):
        assert ((v - w).norm() / w.norm()).item() < 20 * TOL["c32"]
