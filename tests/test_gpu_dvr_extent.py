"""The target renderer at extents beyond a launch grid's: images of any height."""

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
