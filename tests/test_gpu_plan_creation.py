"""What a plan costs to create: the tables of the fused, wide and grouped
schedules add little to those of one launch per axis.  Each pair compares a
plan that has them with one of the same library that does not, the least of
nine (what else runs on the host only adds); before the tables shared their
roots, their memory and their copy the ratios were 2.9, 1.3, 2.5 and 2.0."""
import time

import numpy as np
import pytest
import torch

from paper_2209_15040_gb300 import build
from paper_2209_15040_gb300 import wsfft as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build_library()
    W.lib()
    torch.cuda.init()
    torch.zeros(1, device="cuda")


def _least(make):
    times = []
    for _ in range(9):
        torch.cuda.synchronize()
        t = time.perf_counter()
        plan = make()
        times.append(time.perf_counter() - t)
        plan.close()
    return min(times)


@pytest.mark.parametrize("dims,plain", [((4096, 4096), (4096, 256)), ((128, 128, 128), (256, 256, 256))])
def test_split_axes(dims, plain):
    W.Plan(plain).close()
    assert _least(lambda: W.Plan(dims)) < 1.15 * _least(lambda: W.Plan(plain))


@pytest.mark.parametrize("count", [64, 256])
def test_ragged_groups(count):
    rng = np.random.default_rng(4)
    shapes = [tuple(int(v) for v in s) for s in rng.choice(np.asarray((32, 64, 128, 256)), size=(count, 3))]
    W.RaggedPlan(shapes, W.C32).close()
    # 16-bit storage: the queue alone
    assert _least(lambda: W.RaggedPlan(shapes, W.C32)) < 1.75 * _least(lambda: W.RaggedPlan(shapes, W.C16F))
