"""fftn / ifftn on plain tensors skip the autograd Function: what they return,
on which stream they run, and that every caller the Function refuses or serves
(gradients, forward-mode levels, vmap, tracing) still meets it."""
import pytest
import torch
from torch.autograd import forward_ad

from paper_2209_15040_gb300 import build
from paper_2209_15040_gb300 import wsfft as W

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module", autouse=True)
def _lib():
    build.build_library()
    W.lib()


def _x(seed=0, shape=(4, 8, 16, 32)):
    g = torch.Generator(device="cuda").manual_seed(seed)
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device="cuda"))


@pytest.mark.parametrize("f", [W.fftn, W.ifftn])
def test_same_bytes_with_and_without_a_gradient(f):
    x = _x()
    plain = f(x, rank=3)
    tracked = f(x.clone().requires_grad_(True), rank=3)
    assert tracked.grad_fn is not None and plain.grad_fn is None
    assert torch.equal(plain, tracked.detach())
    with torch.no_grad():
        assert torch.equal(plain, f(x.clone().requires_grad_(True), rank=3))
    with torch.inference_mode():
        assert torch.equal(plain, f(x, rank=3))


def test_runs_on_the_current_stream():
    x = _x(1, (64, 64, 64))
    side = torch.cuda.Stream()
    want = W.fftn(x)
    torch.cuda.synchronize()
    with torch.cuda.stream(side):
        torch.cuda._sleep(20_000_000)  # the input arrives late on the side stream
        late = x.clone()
        got = W.fftn(late)
    side.synchronize()
    assert torch.equal(got, want)


def test_transforms_without_a_rule_are_refused():
    x = _x(2)
    with pytest.raises(RuntimeError):
        torch.func.vmap(lambda t: W.fftn(t, rank=2))(x)
    with forward_ad.dual_level():
        with pytest.raises((RuntimeError, NotImplementedError)):
            W.fftn(forward_ad.make_dual(x, torch.ones_like(x)), rank=3)


def test_traced_call_transforms_its_own_input():
    x, z = _x(3), _x(4)
    traced = torch.jit.trace(lambda t: W.fftn(t, rank=3), (x,), check_trace=False)
    assert torch.equal(traced(z), W.fftn(z, rank=3))
