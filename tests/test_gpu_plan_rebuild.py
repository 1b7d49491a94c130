"""A change of normalisation on a plan whose tables are made already builds the
schedule only: no table memory is touched."""
import time

import pytest
import torch

from paper_2209_15040_gb300 import wsfft as W

pytestmark = pytest.mark.gpu


def _least(call):
    times = []
    for _ in range(300):
        t = time.perf_counter()
        call()
        times.append(time.perf_counter() - t)
    return min(times)


@pytest.mark.parametrize("dims", [(2,), (64, 64)])
def test_set_norm_costs_no_more_than_a_query(dims):
    torch.zeros(1, device="cuda")
    plan = W.Plan(dims)
    try:
        # one call through ctypes each, the query with two results to make room for;
        # with 50 KB of remembered roots cleared at each rebuild the first took 1.5 times the second
        assert _least(lambda: plan.set_norm(W.NORM_NONE)) < 1.2 * _least(lambda: plan.passes())
    finally:
        plan.close()
