"""Empty-space skipping passes over samples without opacity only: with a transfer function that rises
steeply from the faces of the marked blocks, and where positions round coarsely against the step (small
steps, far cameras), the images equal the full march's bit for bit."""

import ctypes

import numpy as np
import pytest
import torch

from vbm_inputs.cameras import camera_array, look_at

pytestmark = pytest.mark.gpu

STEEP = (np.array([0.0, 0.5, 0.5002, 1.0]),
         np.array([[0.2, 0.3, 0.4, 0.0], [0.9, 0.5, 0.1, 0.0], [0.4, 0.9, 0.1, 0.6], [1, 1, 1, 0.9]]))


@pytest.mark.parametrize("step", [0.5, 0.01, 0.002])
@pytest.mark.parametrize("distance", [40.0, 5000.0, 60000.0])
def test_skipping_passes_over_empty_samples_only(cuda_lib, distance, step):
    vbm = cuda_lib
    dims, W, H = (32, 24, 40), 64, 48
    nx, ny, nz = dims
    # no opacity up to one face of a block along every axis, rising behind it
    q = np.maximum(np.maximum(np.arange(nx)[None, None, :] - 8, np.arange(ny)[None, :, None] - 16),
                   np.arange(nz)[:, None, None] - 24)
    F = (0.49999 + 0.3 * np.clip(q, 0, 1)).astype(np.float32)
    middle = np.asarray(dims) / 2.0
    cams = []
    for direction in ((1, 0.01, 0.02), (0.8, 0.5, 0.33), (0.3, 0.9, 0.3), (-0.5, -0.6, -0.62), (0.2, -0.7, 0.7)):
        u = np.asarray(direction) / np.linalg.norm(direction)
        R, t = look_at(middle - distance * u, middle)
        f = W * distance / 50.0                       # 50 voxels across the image at the volume's centre
        cams.append(dict(R=R, t=t, fx=f, fy=f, cx=W / 2 + 0.123, cy=H / 2 - 0.377, znear=0.2, width=W, height=H))
    V = len(cams)
    cams_dev = vbm.cameras_to_device(camera_array(cams))
    Fd, tf = torch.from_numpy(F).cuda(), vbm.make_tf(*STEEP)
    skip, full = torch.full((V, 4, H, W), 7.0, device="cuda"), torch.full((V, 4, H, W), 9.0, device="cuda")
    vbm.render_dvr(Fd, dims, tf, cams_dev, V, W, H, step, skip)
    assert vbm.load().vbm_render_dvr(vbm._ptr(Fd), vbm._dims(dims), ctypes.byref(tf), vbm._ptr(cams_dev), V, W, H,
                                     ctypes.c_float(step), vbm._ptr(full), vbm._stream()) == 0
    assert full[:, 3].max().item() > 0.5
    assert torch.equal(skip, full)
