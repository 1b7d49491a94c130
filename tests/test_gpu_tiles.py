"""GPU parity of the pipelined tile kernels (csrc/tile.cuh): every instantiated
shape at the smallest stride it takes, with fewer tiles than resident blocks,
one tile, and a last round that only some blocks take; both directions; in
place; and the plan builder's rule against the general kernels on strides on
both sides of its limits.  Tolerances are those of the parity tests."""
import numpy as np
import pytest
import torch

import oracle
from paper_2209_15040_gb300 import build
from paper_2209_15040_gb300 import wsfft as W
from tests._helpers import DT, TOL, seeded, to_device, to_host_c128

pytestmark = pytest.mark.gpu

PIPE = 4000
# (points, values per thread, log2 elements per tile)
HALF = [(32, 8, 13), (64, 8, 13), (128, 16, 13), (256, 16, 13), (256, 16, 14), (512, 32, 13), (512, 32, 14),
        (1024, 32, 14), (2048, 16, 14), (4096, 16, 14)]
SHAPES = [(d, *s) for d in ("c16f", "c16bf") for s in HALF] + [("c32", 1024, 32, 14), ("c32", 1024, 32, 13),
                                                                      ("c32", 2048, 16, 14)]


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build_library()
    W.lib()
    torch.cuda.init()


def _axis(x, dtype, n, inner, batch, direction, variant):
    plan = W.AxisPlan(n, inner, DT[dtype], direction, batch, norm=W.NORM_ORTHO)
    try:
        if variant:
            plan.set_pass_variant(0, *variant)
        out = torch.empty_like(x)
        plan.execute(x.data_ptr(), out.data_ptr())
        same = x.clone()
        plan.execute(same.data_ptr(), same.data_ptr())
        torch.cuda.synchronize()
    finally:
        plan.close()
    assert torch.equal(out, same)  # in place: the same bytes
    return out


@pytest.mark.parametrize("dtype,n,e,tb", SHAPES)
@pytest.mark.parametrize("tiles", ["one", "few", "rounds"])
def test_strided_tile_shapes(dtype, n, e, tb, tiles):
    w = (1 << tb) // n
    inner = w if tiles == "one" else 2 * w
    blocks = torch.cuda.get_device_properties(0).multi_processor_count * (1 if tb == 14 else 2 if dtype == "c32" else 3)
    batch = {"one": 1, "few": 5, "rounds": blocks // 2 + 3}[tiles]
    direction = W.INVERSE if tiles == "few" else W.FORWARD
    xs, xc = seeded((batch, n, inner), 11, "uniform", dtype)
    got = to_host_c128(_axis(to_device(xs, dtype), dtype, n, inner, batch, direction, (e, PIPE + tb)), dtype)
    ref = oracle.fftn(np.ascontiguousarray(np.moveaxis(xc, 1, 2)), rank=1, sign=direction, norm=oracle.NORM_ORTHO)
    assert oracle.rel_l2(np.moveaxis(got.reshape(batch, n, inner), 1, 2), ref) < TOL[dtype]


@pytest.mark.parametrize("dtype", ["c32", "c16f"])
@pytest.mark.parametrize("n,inner", [(n, i) for n in (32, 64, 128, 256, 512, 1024, 2048, 4096)
                                     for i in (8, 16, 32, 128, 256, 1 << 14, 1 << 17)])
def test_rule_matches_the_general_kernels(dtype, n, inner):
    # strides that fill whole tiles and strides that do not, enough elements
    # for the rule to choose the tile kernels where it may
    total = 1 << (25 if dtype == "c32" else 22)
    batch = max(1, total // (n * inner))
    general = (16 if n >= 128 and n != 512 else 8, 0)
    g = torch.Generator(device="cuda").manual_seed(n + inner)
    x = torch.randn(batch, n, inner, 2, generator=g, device="cuda")
    x = torch.view_as_complex(x) if dtype == "c32" else x.half()
    a = _axis(x, dtype, n, inner, batch, W.FORWARD, None)
    b = _axis(x, dtype, n, inner, batch, W.FORWARD, general)
    a, b = (torch.view_as_real(t).double() if dtype == "c32" else t.double() for t in (a, b))
    assert ((a - b).norm() / b.norm()).item() < TOL[dtype]


def _plan(x, dtype, dims, direction, batch, layout=W.LAYOUT_NATURAL):
    plan = W.Plan(dims, DT[dtype], direction, batch, W.NORM_ORTHO)
    try:
        plan.set_layout(layout)
        out = torch.empty_like(x)
        plan.execute(x.data_ptr(), out.data_ptr())
        same = x.clone()
        plan.execute(same.data_ptr(), same.data_ptr())
        torch.cuda.synchronize()
    finally:
        plan.close()
    assert torch.equal(out, same)
    return out


@pytest.mark.parametrize("dtype,lg", [("c32", g) for g in (16, 17, 18, 19, 20, 21)] +
                         [("c16f", g) for g in range(13, 22)] + [("c16bf", 18)])
def test_four_step_tiles(dtype, lg):
    # one transform more than fills the range the rule starts at, so the last
    # round of tiles is uneven
    n = 1 << lg
    batch = ((1 << (23 if dtype == "c32" else 22)) // n) + 1
    direction = W.INVERSE if lg % 2 else W.FORWARD
    xs, xc = seeded((batch, n), 13, "uniform", dtype)
    got = to_host_c128(_plan(to_device(xs, dtype), dtype, (n,), direction, batch), dtype).reshape(batch, n)
    ref = oracle.fftn(xc, rank=1, sign=direction, norm=oracle.NORM_ORTHO)
    assert oracle.rel_l2(got, ref) < TOL[dtype]


@pytest.mark.parametrize("dtype,dims", [("c32", (1024, 64)), ("c32", (64, 1024))] +
                         [("c16f", d) for d in ((128, 64), (64, 128), (256, 512), (512, 256), (1024, 64))])
def test_swapped_layout_tiles(dtype, dims):
    batch = (1 << (23 if dtype == "c32" else 22)) // (dims[0] * dims[1]) + 1
    xs, xc = seeded((batch,) + dims, 17, "uniform", dtype)
    got = to_host_c128(_plan(to_device(xs, dtype), dtype, dims, W.FORWARD, batch, W.LAYOUT_SWAPPED), dtype)
    ref = oracle.fftn(xc, rank=2, sign=W.FORWARD, norm=oracle.NORM_ORTHO)
    assert oracle.rel_l2(got.reshape((batch,) + dims[::-1]), np.swapaxes(ref, 1, 2)) < TOL[dtype]


@pytest.mark.parametrize("dtype", ["c32", "c16f", "c16bf"])
@pytest.mark.parametrize("n,e", [(32, 8), (64, 8), (128, 16)])
def test_contiguous_tiles(dtype, n, e):
    # one pencil, a partial tile, whole tiles, a partial tile after several rounds
    per = (1 << 13) // n
    for batch in (1, per - 1, 2 * per, 500 * per + 3):
        xs, xc = seeded((batch, n), 19, "uniform", dtype)
        x = to_device(xs, dtype)
        plan = W.Plan((n,), DT[dtype], W.INVERSE, batch, W.NORM_ORTHO)
        try:
            plan.set_pass_variant(0, e, PIPE + 13)
            guard = torch.zeros((batch + per) * n * x.element_size() // 4 * (1 if dtype == "c32" else 2),
                                dtype=torch.int32, device="cuda")
            plan.execute(x.data_ptr(), guard.data_ptr())
            plan.execute(x.data_ptr(), x.data_ptr())
            torch.cuda.synchronize()
        finally:
            plan.close()
        words = x.numel() * x.element_size() // 4
        raw = (torch.view_as_real(x) if dtype == "c32" else x).contiguous().view(-1).view(torch.int32)
        assert torch.equal(guard[:words], raw) and not guard[words:].any()  # nothing beyond the last pencil
        ref = oracle.fftn(xc, rank=1, sign=W.INVERSE, norm=oracle.NORM_ORTHO)
        assert oracle.rel_l2(to_host_c128(x, dtype).reshape(batch, n), ref) < TOL[dtype]
