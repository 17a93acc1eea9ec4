"""Empty-space skipping of the target renderer: the images of a call with the occupancy marks
equal those of the full march, over transfer functions, volume shapes and cameras where the marks
or the steps across a block could go wrong."""

import ctypes

import numpy as np
import pytest
import torch

from vbm_inputs import TF_KNOTS_RGBA, TF_KNOTS_X, blob_volume, orbit_cameras, tf_mode
from vbm_inputs.cameras import camera_array

pytestmark = pytest.mark.gpu


def _inside_camera(dims, W, H, axis):
    """A camera at the volume's centre looking exactly along an axis (rays parallel to slabs)."""
    f = np.zeros(3)
    f[axis] = 1.0
    r = np.roll(f, 1)
    R = np.stack([r, np.cross(f, r), f])
    pos = np.asarray(dims) / 2.0
    return dict(R=R, t=-R @ pos, fx=W / 2.0, fy=W / 2.0, cx=(W // 2) + 0.5, cy=(H // 2) + 0.5, znear=0.2, width=W,
                height=H)


TFS = {
    "table": (TF_KNOTS_X, TF_KNOTS_RGBA),                    # no opacity up to the second knot
    "mode": tf_mode(2),                                      # opacity over one inner interval
    "from zero": (np.array([0.0, 1.0]), np.array([[0.2, 0.3, 0.4, 0.0], [0.9, 0.5, 0.1, 0.5]])),
    "everywhere": (np.array([0.0, 0.5, 1.0]), np.array([[0.2, 0.3, 0.4, 0.1], [0.9, 0.5, 0.1, 0.5], [1, 1, 1, 0.2]])),
    "nowhere": (np.array([0.1, 0.9]), np.array([[0.2, 0.3, 0.4, 0.0], [0.9, 0.5, 0.1, 0.0]])),
}


@pytest.mark.parametrize("dims,tf_name,step", [
    ((32, 32, 32), "table", 0.5), ((32, 32, 32), "mode", 0.5), ((32, 32, 32), "from zero", 0.3),
    ((32, 32, 32), "everywhere", 0.5), ((32, 32, 32), "nowhere", 0.5),
    ((9, 17, 8), "table", 0.5), ((10, 7, 33), "mode", 1.0), ((1, 40, 24), "table", 0.5), ((264, 12, 20), "from zero", 2.5),
    ((300, 5, 9), "table", 0.5)])
def test_dvr_skip_equals_full_march(cuda_lib, dims, tf_name, step):
    vbm = cuda_lib
    nx, ny, nz = dims
    G = max(max(dims), 32)
    F = np.ascontiguousarray(blob_volume(G, 8, seed=G)[G // 2 - nz // 2:][:nz, G // 2 - ny // 2:, :][:, :ny, :nx])
    F[F < 0.06] = 0.0                       # the noise floor: exact empty space
    F[nz // 2, ny // 2, nx // 3] = np.nan   # is the transfer function's value at 0
    W, H = 61, 45
    cams = orbit_cameras(dims, 3, W, H) + [_inside_camera(dims, W, H, a) for a in range(3)]
    V = len(cams)
    cams_dev = vbm.cameras_to_device(camera_array(cams))
    Fd, tf = torch.from_numpy(F).cuda(), vbm.make_tf(*TFS[tf_name])
    skip, full = torch.full((V, 4, H, W), 7.0, device="cuda"), torch.full((V, 4, H, W), 9.0, device="cuda")
    vbm.render_dvr(Fd, dims, tf, cams_dev, V, W, H, step, skip)
    assert vbm.load().vbm_render_dvr(vbm._ptr(Fd), vbm._dims(dims), ctypes.byref(tf), vbm._ptr(cams_dev), V, W, H,
                                     ctypes.c_float(step), vbm._ptr(full), vbm._stream()) == 0
    # a sample on a block's face may be taken for the block next to it: the face's values,
    # off by the rounding of the position (about 1e-5 voxels), bound its opacity by 1e-4
    off = (skip - full).abs()
    assert off.max().item() <= 1e-4 and (off > 0).float().mean().item() < 1e-3
    if tf_name == "nowhere":
        assert not full.any()
    elif min(dims) > 8:
        assert full[:, 3].max().item() > 0.01


def test_dvr_workspace_is_checked(cuda_lib):
    vbm = cuda_lib
    F = torch.zeros((16, 16, 16), device="cuda")
    tf = vbm.make_tf(TF_KNOTS_X, TF_KNOTS_RGBA)
    cams_dev = vbm.cameras_to_device(camera_array(orbit_cameras((16, 16, 16), 1, 8, 8)))
    out, ws, size = torch.empty((1, 4, 8, 8), device="cuda"), torch.empty(64, device="cuda"), ctypes.c_size_t()
    lib = vbm.load()
    assert lib.vbm_render_dvr_workspace_size(vbm._dims((16, 16, 16)), ctypes.byref(size)) == 0 and size.value == 16
    args = (vbm._ptr(F), vbm._dims((16, 16, 16)), ctypes.byref(tf), vbm._ptr(cams_dev), 1, 8, 8, ctypes.c_float(0.5),
            vbm._ptr(out), vbm._ptr(ws))
    assert lib.vbm_render_dvr_ws(*args, size.value - 1, vbm._stream()) == vbm.VBM_ERR_ARG
    assert lib.vbm_render_dvr_ws(*args, size.value, vbm._stream()) == 0
