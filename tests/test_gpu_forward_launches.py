"""Launches of a forward call: a plan that leaves its configuration to the library takes no more of
them than one whose lists are never split, so that a viewer's frame of a few splats, which is bound by
its chain of launches, costs no more with them."""

import numpy as np
import pytest
import torch

from _helpers import to_device
from vbm_inputs import orbit_cameras
from vbm_inputs.gaussians import random_gaussians

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("W,H", [(320, 240), (1040, 1024)])      # up to 4096 tiles, and more
def test_default_plan_takes_no_more_launches(cuda_lib, W, H):
    vbm = cuda_lib
    P = random_gaussians(500, 12.0, 20.0, seed=1).astype(np.float32)
    params, cams_dev = to_device(P, orbit_cameras((32, 32, 32), 1, W, H))
    img = torch.empty((1, 3, H, W), device="cuda")
    launches = []
    for seg in (0, -1):
        plan = vbm.Plan([0, P.shape[1]], 1, W, H, pair_capacity=1 << 20, segment_len=seg)
        before = vbm.kernel_launches()
        plan.forward(params, cams_dev, img)
        launches.append(vbm.kernel_launches() - before)
    assert launches[0] <= launches[1], launches
