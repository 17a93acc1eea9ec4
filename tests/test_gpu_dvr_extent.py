"""The target renderer at extents beyond a launch grid's and a float's: images of any height, volumes
whose voxel indices along an axis pass 2^23."""

import numpy as np
import pytest
import torch

from vbm_inputs import TF_KNOTS_RGBA, TF_KNOTS_X, blob_volume
from vbm_inputs.cameras import camera_array

pytestmark = pytest.mark.gpu

R = np.array([[0.0, 1, 0], [0, 0, 1], [1, 0, 0]])      # looks along x; the image's rows run along z


def test_image_taller_than_65535_blocks(cuda_lib):
    """Rows of an image of 600,001 rows equal the same rays' in images of one row."""
    vbm = cuda_lib
    dims, W, H = (16, 16, 16), 3, 600001
    F = torch.from_numpy(blob_volume(16, 6, seed=2)).cuda()
    tf = vbm.make_tf(TF_KNOTS_X, TF_KNOTS_RGBA)

    def render(height, cy):
        cam = dict(R=R, t=-R @ np.array([-16.0, 8.0, 8.0]), fx=6.0, fy=1048576.0, cx=1.5, cy=cy, znear=0.2, width=W,
                   height=height)
        out = torch.full((1, 4, height, W), 7.0, device="cuda")
        vbm.render_dvr(F, dims, tf, vbm.cameras_to_device(camera_array([cam])), 1, W, height, 0.5, out)
        return out

    tall = render(H, 300000.5)
    assert tall[:, 3].max().item() > 0.01
    for row in (0, 1, 299999, 524279, 524280, 600000):
        assert torch.equal(tall[:, :, row], render(1, 300000.5 - row)[:, :, 0]), row


def test_axis_of_more_than_2_to_the_23_voxels(cuda_lib):
    """The voxels at the far end of a long volume are the ones sampled there."""
    vbm = cuda_lib
    n, W, H = (1 << 24) + 64, 5, 5
    F = torch.zeros((n, 2, 2), device="cuda")
    F[n - 64:] = 1.0
    tf = vbm.make_tf(TF_KNOTS_X, TF_KNOTS_RGBA)
    out = torch.empty((1, 4, H, W), device="cuda")
    cam = dict(R=R, t=-R @ np.array([-10.0, 1.0, n - 30.0]), fx=200.0, fy=200.0, cx=2.5, cy=2.5, znear=0.2, width=W,
               height=H)
    vbm.render_dvr(F, (2, 2, n), tf, vbm.cameras_to_device(camera_array([cam])), 1, W, H, 0.5, out)
    # a chord of 2 voxels (to 2e-4) of alpha 0.7 and colour 1; float32 rounding of the march is below 1e-5
    assert (out - (1.0 - 0.3 ** 2)).abs().max().item() < 1e-3
