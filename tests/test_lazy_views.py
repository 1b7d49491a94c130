"""Lazy conjugate and negative views: the library reads a tensor's storage, which
holds neither, so every entry point that takes a tensor resolves them first."""
import numpy as np
import pytest
import torch

import oracle
from paper_2209_15040_gb300 import inputs
from paper_2209_15040_gb300 import wsfft as W
from paper_2209_15040_gb300.distributed import SlabFFT3
from tests._dist_local import NumpyLocal

VIEWS = [torch.conj, torch._neg_view, lambda t: torch._neg_view(torch.conj(t))]


@pytest.mark.parametrize("view", VIEWS)
def test_materialized_holds_the_values_in_storage(view):
    x = torch.from_numpy(inputs.complex_input((4, 8), 1, "normal", "c32"))
    assert W.materialized(x) is x
    lazy = view(x)
    assert lazy.is_contiguous() and lazy.data_ptr() == x.data_ptr()
    got = W.materialized(lazy)
    assert not got.is_conj() and not got.is_neg() and got.data_ptr() != x.data_ptr()
    assert torch.equal(got, lazy)


@pytest.mark.parametrize("view", VIEWS)
def test_distributed_steps(view):
    dims = (4, 8, 4)
    x = torch.from_numpy(inputs.complex_input(dims, 2, "normal", "c32").astype(np.complex128))
    f = SlabFFT3(dims, world=1, rank=0, local_forward=NumpyLocal(-1), local_inverse=NumpyLocal(+1))
    want = oracle.fftn(view(x).resolve_conj().resolve_neg().numpy())
    assert oracle.rel_l2(f.forward(view(x)).numpy(), want) < 1e-12
    y = torch.from_numpy(oracle.fftn(x.numpy()))
    back = oracle.fftn(view(y).resolve_conj().resolve_neg().numpy(), sign=+1, norm=oracle.NORM_PAPER)
    assert oracle.rel_l2(f.inverse(view(y)).numpy(), back) < 1e-12
    recv = view(f.forward_pack(x))
    assert oracle.rel_l2(f.forward_finish(recv).numpy(),
                         np.fft.fft(recv.resolve_conj().resolve_neg().numpy(), axis=0)) < 1e-12


@pytest.mark.gpu
@pytest.mark.parametrize("view", VIEWS)
@pytest.mark.parametrize("f,ref", [(W.fftn, torch.fft.fftn), (W.ifftn, torch.fft.ifftn)])
def test_transforms_of_views(view, f, ref):
    # 5e-6: the library's bar in complex64 against a double-precision transform
    x = torch.from_numpy(inputs.complex_input((2, 8, 16, 32), 3, "normal", "c32")).cuda()
    dims = (-3, -2, -1)
    for tracked in (False, True):
        leaf = x.clone().requires_grad_(tracked)
        y = f(view(leaf), rank=3)
        want = ref(view(x).to(torch.complex128), dim=dims)
        assert ((y.detach() - want).norm() / want.norm()).item() < 5e-6


@pytest.mark.gpu
@pytest.mark.parametrize("view", VIEWS)
def test_gradient_through_a_view_of_the_result(view):
    x = torch.from_numpy(inputs.complex_input((8, 16, 32), 4, "normal", "c32")).cuda()
    w = torch.from_numpy(inputs.complex_input((8, 16, 32), 5, "normal", "c32")).cuda()
    grads = []
    for dtype, f in ((torch.complex64, lambda t: W.fftn(t, norm="none")), (torch.complex128, torch.fft.fftn)):
        leaf = x.to(dtype, copy=True).requires_grad_(True)
        (w.to(dtype) * view(f(leaf))).real.sum().backward()
        grads.append(leaf.grad)
    assert ((grads[0] - grads[1]).norm() / grads[1].norm()).item() < 5e-6
