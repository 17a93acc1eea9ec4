"""Segment length of plans that leave it to the library, on either side of its items rule."""

import numpy as np
import pytest
import torch

from _helpers import rel_group_error, to_device
from vbm_inputs import orbit_cameras
from vbm_inputs.gaussians import random_gaussians

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("flags", [0, 2])
@pytest.mark.parametrize("n,V,length", [(54135, 2, 64), (54136, 2, 256), (400000, 1, 256)])   # 8 x 101 x 67
def test_items_set_the_default_length(cuda_lib, n, V, length, flags):
    """Every list longer than the default length asks for a slot per boundary; gradients equal those
    of whole walks up to FP32 rounding."""
    vbm = cuda_lib
    W, H, G = 101, 67, 32
    P = random_gaussians(n, 4.0, 28.0, seed=n, scale_range=(0.02, 0.1),
                         opacity_logit_range=(-5.0, -4.0)).astype(np.float32)
    params, cams_dev = to_device(P, orbit_cameras((G, G, G), V, W, H))
    w = torch.from_numpy(np.random.default_rng(V).standard_normal((V, 3, H, W)).astype(np.float32)).cuda()
    grads = []
    for seg in (0, -1):
        plan = vbm.Plan([0, n], V, W, H, pair_capacity=1 << 23, segment_len=seg, flags=flags)
        img, grad = torch.zeros((V, 3, H, W), device="cuda"), torch.zeros_like(params)
        plan.forward(params, cams_dev, img)
        plan.backward(params, cams_dev, w, grad)
        grads.append(grad.cpu().numpy())
        b = plan.buffers()
        if seg == 0:
            seg_count = vbm.device_tensor(b.seg_count, (4,), np.int32).cpu().numpy()
            ranges = vbm.device_tensor(b.ranges, (V * -(-W // 16) * -(-H // 16), 2), np.int32).cpu().numpy()
            lengths = ranges[:, 1] - ranges[:, 0]
        ok, need = plan.check()
        assert ok, need
    long = lengths[lengths > length]
    assert long.size and seg_count[2] == (-(-long // length) - 1).sum()
    for lo, hi in [(0, 3), (3, 6), (6, 10), (10, 11), (11, 14)]:
        nrm, elt = rel_group_error(grads[0][lo:hi], grads[1][lo:hi])
        assert nrm < 1e-4 and elt < 1e-4, (lo, nrm, elt)


@pytest.mark.parametrize("tile,flags", [((16, 16), 0), ((16, 16), 3), ((8, 8), 2)])
@pytest.mark.parametrize("n,W,H,scales", [(3000, 512, 512, (0.3, 0.6)), (20000, 1000, 1000, (0.1, 0.3))])
def test_default_pool_holds_every_boundary(cuda_lib, n, W, H, scales, tile, flags):
    """Few splats on many pixels are wide, several pairs an item: the checkpoints of a default plan
    still hold every list's boundaries (a list without is walked by one warp)."""
    vbm = cuda_lib
    P = random_gaussians(n, 6.0, 26.0, seed=n, scale_range=scales, opacity_logit_range=(-3.0, -2.0))
    P = P.astype(np.float32)
    params, cams_dev = to_device(P, orbit_cameras((32, 32, 32), 1, W, H))
    plan = vbm.Plan([0, n], 1, W, H, tile_w=tile[0], tile_h=tile[1], pair_capacity=1 << 23, flags=flags)
    img = torch.empty((1, 3, H, W), device="cuda")
    plan.forward(params, cams_dev, img)
    b = plan.buffers()
    units, tiles, asked, _ = vbm.device_tensor(b.seg_count, (4,), np.int32).cpu().numpy()
    ok, need = plan.check()
    assert ok, need
    assert tiles > 0 and asked <= b.checkpoint_slots
