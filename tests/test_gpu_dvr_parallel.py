"""Rays with a zero direction component pass over empty blocks like any other."""

import numpy as np
import pytest
import torch

from vbm_inputs import TF_KNOTS_RGBA, TF_KNOTS_X
from vbm_inputs.cameras import camera_array

pytestmark = pytest.mark.gpu


def test_axis_parallel_rays_skip_blocks(cuda_lib):
    """One ray along a long empty volume (8192 blocks, 1.3 M samples): exactly along x it takes no
    longer than with a slight tilt.  Asked sample by sample it would take over a hundred times as long,
    so a factor of 5 tells the two apart whatever the clocks do."""
    vbm = cuda_lib
    dims, step = (65536, 16, 16), 0.05
    F = torch.zeros((16, 16, 65536), device="cuda")
    tf = vbm.make_tf(TF_KNOTS_X, TF_KNOTS_RGBA)
    out = torch.empty((1, 4, 1, 1), device="cuda")
    ms = []
    for tilt in (0.0, 1e-5):
        R = np.array([[0.0, 1, 0], [0, 0, 1], [1, 0, 0]])
        cam = dict(R=R, t=-R @ np.array([-10.0, 4.1, 4.3]), fx=1.0, fy=1.0, cx=0.5 - tilt, cy=0.5 - tilt, znear=0.2,
                   width=1, height=1)
        cams_dev = vbm.cameras_to_device(camera_array([cam]))
        times = []
        for _ in range(4):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            vbm.render_dvr(F, dims, tf, cams_dev, 1, 1, 1, step, out)
            end.record()
            torch.cuda.synchronize()
            times.append(start.elapsed_time(end))
        ms.append(min(times))
        assert not out.any()
    assert ms[0] < 5 * ms[1], ms
