"""Infinite voxels in the target renderer: the interpolated scalar is clamped to [0, 1], so a voxel
of +inf shows the transfer function's value at 1 and one of -inf its value at 0, with the occupancy
marks and without them."""

import ctypes

import numpy as np
import pytest
import torch

from vbm_inputs import TF_KNOTS_RGBA, TF_KNOTS_X, blob_volume, orbit_cameras, tf_mode
from vbm_inputs.cameras import camera_array

pytestmark = pytest.mark.gpu

FALLING = (np.array([0.0, 0.5, 0.8, 1.0]),
           np.array([[0.9, 0.4, 0.2, 0.6], [0.5, 0.8, 0.1, 0.3], [0.1, 0.2, 0.9, 0.0], [1, 1, 1, 0.0]]))
TFS = {"table": (TF_KNOTS_X, TF_KNOTS_RGBA), "mode": tf_mode(2), "falling": FALLING}


def _images(vbm, F, dims, tf, cams, W, H, step):
    """The views with the occupancy marks and without."""
    V = len(cams)
    cams_dev, Fd = vbm.cameras_to_device(camera_array(cams)), torch.from_numpy(F).cuda()
    skip, full = torch.full((V, 4, H, W), 7.0, device="cuda"), torch.full((V, 4, H, W), 9.0, device="cuda")
    vbm.render_dvr(Fd, dims, tf, cams_dev, V, W, H, step, skip)
    assert vbm.load().vbm_render_dvr(vbm._ptr(Fd), vbm._dims(dims), ctypes.byref(tf), vbm._ptr(cams_dev), V, W, H,
                                     ctypes.c_float(step), vbm._ptr(full), vbm._stream()) == 0
    return skip, full


@pytest.mark.parametrize("tf_name", list(TFS))
@pytest.mark.parametrize("sign", [1, -1])
@pytest.mark.parametrize("dims", [(32, 32, 32), (20, 40, 24)])
def test_infinite_voxels_are_clamped(cuda_lib, dims, sign, tf_name):
    """The images of a volume with infinite voxels are those with +-1e30 in their place, which every
    weight above 1e-30 takes past the clamp as well.  Only a weight of exactly 0 tells them apart
    (inf * 0 is not a number, which reads as 0): a few samples in a million."""
    vbm = cuda_lib
    nx, ny, nz = dims
    F = np.ascontiguousarray(blob_volume(40, 8, seed=5)[:nz, :ny, :nx]) * 0.6 + 0.3
    box = (slice(nz // 2 - 6, nz // 2 + 6), slice(ny // 2 - 6, ny // 2 + 6), slice(nx // 2 - 6, nx // 2 + 6))
    W, H = 61, 45
    cams = orbit_cameras(dims, 3, W, H)
    tf = vbm.make_tf(*TFS[tf_name])
    got = {}
    for value in (np.inf, 1e30, 0.5):
        G = F.copy()
        G[box] = 0.5 if value == 0.5 else sign * value
        got[value] = _images(vbm, G.astype(np.float32), dims, tf, cams, W, H, 0.5)
    for k in range(2):
        assert (got[np.inf][k] != got[1e30][k]).float().mean().item() < 1e-3
        assert (got[0.5][k] != got[1e30][k]).float().mean().item() > 0.01      # the voxels are seen


def test_marks_keep_blocks_that_interpolate_to_nan(cuda_lib):
    """A block of nothing but +inf is not empty where the transfer function has opacity at 0: a ray
    through voxel centres weighs neighbours by 0 and reads inf * 0, which counts as 0."""
    vbm = cuda_lib
    dims, W, H = (33, 33, 33), 31, 31
    F = np.full((33, 33, 33), 0.9, dtype=np.float32)     # no opacity
    F[7:28, 7:28, 7:28] = np.inf
    cams = []
    for axis in range(3):
        f = np.zeros(3)
        f[axis] = 1.0
        r = np.roll(f, 1)
        R = np.stack([r, np.cross(f, r), f])
        pos = np.full(3, 16.5)
        pos[axis] = -20.0
        cams.append(dict(R=R, t=-R @ pos, fx=W / 1.0, fy=W / 1.0, cx=(W // 2) + 0.5, cy=(H // 2) + 0.5, znear=0.2,
                         width=W, height=H))
    skip, full = _images(vbm, F, dims, vbm.make_tf(*FALLING), cams, W, H, 0.5)
    assert full[:, 3].max().item() > 0.5
    assert torch.equal(skip, full)
