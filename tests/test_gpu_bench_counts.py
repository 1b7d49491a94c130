"""The launch counts that bench.py turns into bytes and rates are those of the calls it times."""
import pytest
import torch

import bench
from paper_2209_15040_gb300 import wsfft

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims, forward, in_place", [((32, 32, 32), 2, 2), ((128, 128, 128), 2, 3),
                                                     ((256, 256, 256), 3, 3), ((1 << 16,), 2, 2)])
def test_launches_of_a_call(dims, forward, in_place):
    x = torch.randn(*dims, dtype=torch.complex64, device="cuda")
    y = torch.empty_like(x)
    plan = wsfft.Plan(dims)
    assert bench.launches_of(plan, lambda: plan.execute(x.data_ptr(), y.data_ptr())) == forward
    assert bench.launches_of(plan, lambda: plan.execute(y.data_ptr(), y.data_ptr())) == in_place
    plan.close()


def test_rates_of_the_other_sizes_stay_below_the_memory():
    """Bytes counted per launch over arrays beyond the L2 cannot exceed what HBM3e moves (7.9 TB/s)."""
    recs = bench.sizes_leg(wsfft, torch.device("cuda:0"), torch.cuda.current_stream(), 6800.0, steps=3, warmup=1)
    by = {tuple(r["dims"]): r for r in recs if r["dtype"] == "complex64"}
    assert (by[(128, 128, 128)]["launches_forward"], by[(128, 128, 128)]["launches_inverse_in_place"]) == (2, 3)
    assert (by[(32, 32, 32)]["launches_forward"], by[(32, 32, 32)]["launches_inverse_in_place"]) == (2, 2)
    assert all(r["gb_per_s"] < 7900 for r in recs if "min_bytes_roofline_frac" in r)
