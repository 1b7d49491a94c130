"""What wsfft_autotune remembers: records timed against other schedules are not
read, and a ragged plan's fastest queue stays beside the grouped launches."""
import ctypes
import json

import pytest
import torch

from paper_2209_15040_gb300 import build, inputs
from paper_2209_15040_gb300 import wsfft as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build_library()
    W.lib()
    torch.cuda.init()


@pytest.fixture
def cache(tmp_path, monkeypatch):
    path = tmp_path / "tune.jsonl"
    monkeypatch.setenv("WSFFT_TUNE_CACHE", str(path))
    return path


def _launches(plan, execute):
    assert W.lib().wsfft_plan_profile(plan.handle, 256) == 0
    execute()
    n = ctypes.c_int()
    assert W.lib().wsfft_plan_launch_times(plan.handle, None, 0, ctypes.byref(n)) == 0
    return n.value


def _ragged(shapes):
    xs = [torch.zeros(tuple(s), dtype=torch.complex64, device="cuda") for s in shapes]
    ys = [torch.empty_like(x) for x in xs]
    return [x.data_ptr() for x in xs], [y.data_ptr() for y in ys], xs + ys


def _tuned_key(plan, cache):
    plan.autotune()
    plan.close()
    return json.loads(cache.read_text().strip().splitlines()[-1])["key"]


def test_records_of_earlier_schedules_are_not_read(cache):
    # as a library without the generation in its keys wrote them
    shapes = [(64, 64, 64), (32, 128, 64)]
    records = [(_tuned_key(W.RaggedPlan(shapes), cache), 1, [[-1, 0, 0]]),
               (_tuned_key(W.Plan((64, 64, 64)), cache), 0, [[0, 8, 0]])]
    cache.write_text("".join(
        json.dumps({"key": key.replace("|s2|", "|"), "mode": mode, "variants": variants, "us": 1.0}) + "\n"
        for key, mode, variants in records))
    ins, outs, keep = _ragged(shapes)
    plan = W.RaggedPlan(shapes)
    assert _launches(plan, lambda: plan.execute(ins, outs)) > 1  # grouped, not the queue's one
    plan.close()
    cube = W.Plan((64, 64, 64))
    assert _launches(cube, lambda: cube.execute(ins[0], outs[0])) == 2  # fused, not one per axis
    cube.close()
    torch.cuda.synchronize()


def test_the_queue_is_tuned_beside_the_groups(cache):
    # the queue's default (shape selection 0, lag 1) is not the fastest of its
    # variants on every batch
    chosen = []
    for seed in (4, 5, 6, 7):
        _tuned_key(W.RaggedPlan(inputs.ragged_shapes(48, seed)), cache)
        entry = json.loads(cache.read_text().strip().splitlines()[-1])
        chosen.append((entry["variants"][0][1], entry["mode"], entry["variants"][0][2]))
    assert any(grouped == 1 and (sel, lag) != (0, 1) for sel, lag, grouped in chosen), chosen
