"""Plans that leave their launch configuration to the library: list segments without
persistence, their default length on either side of the batch-size rule, lanes and pixels."""

import numpy as np
import pytest
import torch

from _helpers import rel_group_error, to_device
from vbm_inputs import orbit_cameras
from vbm_inputs.gaussians import random_gaussians

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H,V,recompute,length", [
    (96, 72, 2, False, 64), (101, 67, 1, True, 64),        # small batches: segments of 64
    (1024, 1023, 1, False, 64), (1024, 1024, 1, True, 256),   # either side of 2^20 pixels
    (512, 512, 4, False, 256),
    (1040, 1024, 1, False, 256), (1040, 1024, 1, True, 256)])   # more than 4096 tiles: claims by the warp
def test_default_plan_splits_lists(cuda_lib, W, H, V, recompute, length):
    """The forward is unchanged bit for bit and the gradients equal those of whole walks
    (segment_len -1, 32-lane groups) up to FP32 rounding, also when the splats crowd a small
    part of the image and the checkpoint pool runs out; every list longer than the default
    length asks for a slot per boundary (and one for its final state in recompute plans)."""
    vbm = cuda_lib
    G = 32
    box = (12.0, 20.0) if W < 200 else (15.6, 16.4)
    P = random_gaussians(4000, *box, seed=W + V, scale_range=(0.05, 0.4) if W > 200 else (0.3, 1.2),
                         opacity_logit_range=(-4.5, -2.5)).astype(np.float32)
    cams = orbit_cameras((G, G, G), V, W, H)
    params, cams_dev = to_device(P, cams)
    w = torch.from_numpy(np.random.default_rng(V).standard_normal((V, 3, H, W)).astype(np.float32)).cuda()
    out = []
    for seg, gl, ppt in ((0, 0, 0), (-1, 32, 2)):
        plan = vbm.Plan([0, P.shape[1]], V, W, H, pair_capacity=1 << 22, segment_len=seg, group_lanes=gl,
                        pixels_per_thread=ppt, flags=vbm.PLAN_RECOMPUTE if recompute else 0)
        img = torch.zeros((V, 3, H, W), device="cuda")
        grads = []
        for _ in range(2):      # a second call finds its queue and records cleared
            plan.forward(params, cams_dev, img)
            grad = torch.zeros_like(params)
            plan.backward(params, cams_dev, w, grad)
            grads.append(grad.cpu().numpy())
        b = plan.buffers()
        seg_count = vbm.device_tensor(b.seg_count, (4,), np.int32).cpu().numpy() if b.seg_count else None
        ranges = vbm.device_tensor(b.ranges, (V * -(-W // 16) * -(-H // 16), 2), np.int32).cpu().numpy()
        out.append((img.cpu().numpy(), grads, seg_count, ranges[:, 1] - ranges[:, 0], b.checkpoint_slots))
        ok, need = plan.check()
        assert ok, need
    (img, grads, seg_count, lengths, slots), (img1, grads1, none, _, _) = out
    assert none is None
    long = lengths[lengths > length]
    segments = -(-long // length)
    assert long.size and seg_count[2] == (segments - 1 + recompute).sum()
    if seg_count[2] <= slots:
        assert seg_count[1] == long.size and seg_count[0] == segments.sum()
    else:
        assert 0 < seg_count[1] < long.size
    assert np.array_equal(img, img1)
    for g, ref in zip(grads, grads1):
        for lo, hi in [(0, 3), (3, 6), (6, 10), (10, 11), (11, 14)]:
            nrm, elt = rel_group_error(g[lo:hi], ref[lo:hi])
            assert nrm < 1e-4 and elt < 1e-4, (lo, nrm, elt)


@pytest.mark.parametrize("flags,seg", [(0, 0), (0, -1), (2, 0)])
def test_captured_backward_replays_after_one_forward(cuda_lib, flags, seg):
    """A backward captured by itself gives the same gradient at every replay: its splat
    gradients and its work queue are cleared each time."""
    vbm = cuda_lib
    W, H, V, G = 96, 72, 2, 32
    P = random_gaussians(3000, 12.0, 20.0, seed=3, scale_range=(0.3, 1.2),
                         opacity_logit_range=(-4.5, -2.5)).astype(np.float32)
    params, cams_dev = to_device(P, orbit_cameras((G, G, G), V, W, H))
    w = torch.from_numpy(np.random.default_rng(V).standard_normal((V, 3, H, W)).astype(np.float32)).cuda()
    plan = vbm.Plan([0, P.shape[1]], V, W, H, pair_capacity=1 << 22, segment_len=seg, flags=flags)
    img, grad = torch.zeros((V, 3, H, W), device="cuda"), torch.zeros_like(params)
    plan.forward(params, cams_dev, img)
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        plan.backward(params, cams_dev, w, grad)
    got = []
    for _ in range(3):
        grad.fill_(float("nan"))
        graph.replay()
        got.append(grad.cpu().numpy())
    ref = torch.zeros_like(params)
    plan.forward(params, cams_dev, img)
    plan.backward(params, cams_dev, w, ref)
    for g in got:
        for lo, hi in [(0, 3), (3, 6), (6, 10), (10, 11), (11, 14)]:
            nrm, elt = rel_group_error(g[lo:hi], ref.cpu().numpy()[lo:hi])
            assert nrm < 1e-5 and elt < 1e-4, (lo, nrm, elt)
