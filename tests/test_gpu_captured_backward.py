"""A backward captured by itself on a plan that has run before: whoever cleared the splat-gradient
records the last time, every replay starts from cleared ones."""

import numpy as np
import pytest
import torch

from _helpers import rel_group_error, to_device
from vbm_inputs import orbit_cameras
from vbm_inputs.gaussians import random_gaussians

pytestmark = pytest.mark.gpu

W, H, V, G = 96, 72, 2, 32


def _scene(vbm, flags, seg):
    P = random_gaussians(3000, 12.0, 20.0, seed=3, scale_range=(0.3, 1.2),
                         opacity_logit_range=(-4.5, -2.5)).astype(np.float32)
    params, cams_dev = to_device(P, orbit_cameras((G, G, G), V, W, H))
    w = torch.from_numpy(np.random.default_rng(V).standard_normal((V, 3, H, W)).astype(np.float32)).cuda()
    plan = vbm.Plan([0, P.shape[1]], V, W, H, pair_capacity=1 << 22, segment_len=seg, flags=flags)
    return plan, params, cams_dev, w, torch.zeros((V, 3, H, W), device="cuda"), torch.zeros_like(params)


def _same(g, ref):
    """Equal up to the order of the float32 sums."""
    g, ref = g.cpu().numpy(), ref.cpu().numpy()
    for lo, hi in [(0, 3), (3, 6), (6, 10), (10, 11), (11, 14)]:
        nrm, elt = rel_group_error(g[lo:hi], ref[lo:hi])
        assert nrm < 1e-5 and elt < 1e-4, (lo, nrm, elt)


@pytest.mark.parametrize("flags,seg", [(0, 0), (0, -1), (1, 0), (2, 0)])
def test_captured_backward_after_a_warm_up(cuda_lib, flags, seg):
    vbm = cuda_lib
    plan, params, cams_dev, w, img, grad = _scene(vbm, flags, seg)
    for _ in range(2):
        plan.forward(params, cams_dev, img)
        plan.backward(params, cams_dev, w, grad)
    ref = grad.clone()
    plan.forward(params, cams_dev, img)        # has cleared the records for the next backward
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.backward(params, cams_dev, w, grad)
    for _ in range(3):
        grad.fill_(float("nan"))
        graph.replay()
        _same(grad, ref)
    plan.backward(params, cams_dev, w, grad)   # and one outside the graph
    _same(grad, ref)
    plan.forward(params, cams_dev, img)        # a replay between a forward and its backward
    graph.replay()
    plan.backward(params, cams_dev, w, grad)
    _same(grad, ref)


@pytest.mark.parametrize("flags", [0, 1])
def test_captured_forward_clears_for_its_own_capture_only(cuda_lib, flags):
    """A forward that was captured but not replayed has cleared nothing; forward and backward in one
    graph, and in two graphs, replay to the same gradients."""
    vbm = cuda_lib
    plan, params, cams_dev, w, img, grad = _scene(vbm, flags, 0)
    for _ in range(2):
        plan.forward(params, cams_dev, img)
        plan.backward(params, cams_dev, w, grad)
    ref = grad.clone()
    torch.cuda.synchronize()
    fwd, both, bwd, idle = (torch.cuda.CUDAGraph() for _ in range(4))
    with torch.cuda.graph(idle):
        plan.forward(params, cams_dev, img)
    plan.backward(params, cams_dev, w, grad)   # of the last forward that ran
    _same(grad, ref)
    with torch.cuda.graph(both):
        plan.forward(params, cams_dev, img)
        plan.backward(params, cams_dev, w, grad)
    with torch.cuda.graph(fwd):
        plan.forward(params, cams_dev, img)
    with torch.cuda.graph(bwd):
        plan.backward(params, cams_dev, w, grad)
    for graphs in ((both,), (both,), (fwd, bwd), (bwd,), (fwd, bwd), (both,)):
        grad.fill_(float("nan"))
        for g in graphs:
            g.replay()
        _same(grad, ref)
