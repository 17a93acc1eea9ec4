"""The autograd wrapper's buffers: whole calls write every pixel and every gradient column (their
tensors start uninitialised), partial ones leave the other views' images and gradients zero."""

import numpy as np
import pytest
import torch

from _helpers import scene, to_device

pytestmark = pytest.mark.gpu


def _poison(*shapes):
    """Fill memory that the caching allocator will hand out again with NaN."""
    held = [torch.full(s, float("nan"), device="cuda") for s in shapes for _ in range(3)]
    torch.cuda.synchronize()
    del held


@pytest.mark.parametrize("view_scene,begin,count,extra", [
    (None, 0, 3, 0), (None, 1, 1, 0), (None, 0, 3, 5), ([0, 1, 1], 0, 3, 0), ([0, 1, 1], 0, 1, 0), ([1, 1, 1], 0, 3, 0)])
def test_autograd_buffers_are_written_or_zero(cuda_lib, view_scene, begin, count, extra):
    from paper_2601_09417_gb300.autograd import render
    W, H, V = 70, 51, 3
    P, cams, _ = scene(seed=8, n=900, V=V, W=W, H=H)
    n = P.shape[1]
    P = np.concatenate([P, P[:, :extra]], axis=1)       # columns beyond the plan's Gaussians
    offset = [0, n] if view_scene is None else [0, 400, n]
    params, cams_dev = to_device(P, cams)
    params.requires_grad_(True)
    plan = cuda_lib.Plan(offset, V, W, H, view_scene=view_scene, pair_capacity=1 << 20)
    _poison((V, 3, H, W), P.shape)
    img = render(params, plan, cams_dev, view_begin=begin, view_count=count)
    called = list(range(begin, begin + count))
    ref = torch.zeros((V, 3, H, W), device="cuda")
    plan.forward(params.detach(), cams_dev, ref, view_begin=begin, view_count=count)
    assert torch.equal(img.detach(), ref)
    assert all((img[v] != 0).any() == (v in called) for v in range(V))
    _poison((V, 3, H, W), P.shape)
    grad, = torch.autograd.grad(img, params, torch.ones_like(img))
    assert torch.isfinite(grad).all()
    seen = torch.zeros(P.shape[1], dtype=torch.bool, device="cuda")
    for v in called:
        s = 0 if view_scene is None else view_scene[v]
        seen[offset[s]:offset[s + 1]] = True
    assert not grad[:, ~seen].any() and grad[:, seen].any()
