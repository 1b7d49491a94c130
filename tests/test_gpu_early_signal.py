"""Fused launches that let the next launch in at their start: chains of dependent executes,
each reading what the one before it wrote, give the bytes of the same chain with
the stream waited for after each execute."""
import pytest
import torch

from paper_2209_15040_gb300 import wsfft as W
from tests._helpers import DT, seeded, to_device

pytestmark = pytest.mark.gpu


# tiles of 2^13 elements: 16 and a part (late signal in complex64), 32, 64, 65, one per
# block, more than one per block; split middle axes (two fused launches)
@pytest.mark.parametrize("dtype", ["c32", "c16f", "c16bf"])
@pytest.mark.parametrize("dims, batch", [((64, 64), 33), ((64, 64, 64), 1), ((8, 128, 64), 8), ((32, 32, 32), 2),
                                         ((8, 128, 64), 9), ((64, 128, 64), 2), ((64, 128, 128), 1), ((64, 64), 2000)])
def test_chained_executes(dtype, dims, batch):
    xs, _ = seeded((batch,) + dims, 41, "uniform", dtype)
    x = to_device(xs, dtype)
    f, i = (W.Plan(dims, DT[dtype], d, batch, W.NORM_ORTHO) for d in (W.FORWARD, W.INVERSE))
    outs = []
    for wait in (True, False):
        a, b, c = x.clone(), torch.full_like(x, float("nan")), torch.full_like(x, float("nan"))
        torch.cuda.synchronize()
        for step in range(12):
            f.execute(a.data_ptr(), b.data_ptr())
            if wait:
                torch.cuda.synchronize()
            i.execute(b.data_ptr(), c.data_ptr())
            if wait:
                torch.cuda.synchronize()
            a, c = c, a
        torch.cuda.synchronize()
        outs.append(a.clone())
    f.close()
    i.close()
    assert torch.equal(torch.view_as_real(outs[0]) if dtype == "c32" else outs[0],
                       torch.view_as_real(outs[1]) if dtype == "c32" else outs[1])
    assert not torch.isnan(outs[0].abs() if dtype == "c32" else outs[0]).any()
