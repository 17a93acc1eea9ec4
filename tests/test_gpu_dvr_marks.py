"""The occupancy marks and the rule that leaves them out of small calls: the tests of the target renderer
with the marks in every call, and what a small call gains without them."""

import ctypes

import pytest
import torch

from test_gpu_dvr_extent import test_axis_of_more_than_2_to_the_23_voxels as marked_long_axis  # noqa: F401
from test_gpu_dvr_infinite import test_infinite_voxels_are_clamped as marked_infinite  # noqa: F401
from test_gpu_dvr_infinite import test_marks_keep_blocks_that_interpolate_to_nan as marked_nan  # noqa: F401
from test_gpu_dvr_margin import test_skipping_passes_over_empty_samples_only as marked_margin  # noqa: F401
from test_gpu_dvr_parallel import test_axis_parallel_rays_skip_blocks as marked_parallel  # noqa: F401
from test_gpu_dvr_skip import test_dvr_skip_equals_full_march as marked_skip  # noqa: F401
from vbm_inputs import TF_KNOTS_RGBA, TF_KNOTS_X, blob_volume, orbit_cameras
from vbm_inputs.cameras import camera_array

pytestmark = pytest.mark.gpu


@pytest.fixture
def always_marked(cuda_lib, monkeypatch):
    monkeypatch.setattr(cuda_lib, "dvr_marks_pay", lambda *a: True)
    return cuda_lib


@pytest.mark.parametrize("dims,tf_name,step", [
    ((32, 32, 32), "table", 0.5), ((32, 32, 32), "mode", 0.5), ((32, 32, 32), "from zero", 0.3),
    ((32, 32, 32), "everywhere", 0.5), ((32, 32, 32), "nowhere", 0.5),
    ((9, 17, 8), "table", 0.5), ((10, 7, 33), "mode", 1.0), ((1, 40, 24), "table", 0.5), ((264, 12, 20), "from zero", 2.5),
    ((300, 5, 9), "table", 0.5)])
def test_marked_calls_skip(always_marked, dims, tf_name, step):
    marked_skip(always_marked, dims, tf_name, step)


@pytest.mark.parametrize("tf_name", ["table", "mode", "falling"])
@pytest.mark.parametrize("sign", [1, -1])
def test_marked_calls_clamp_infinite_voxels(always_marked, sign, tf_name):
    marked_infinite(always_marked, (32, 32, 32), sign, tf_name)


def test_marked_calls_keep_nan_blocks(always_marked):
    marked_nan(always_marked)


@pytest.mark.parametrize("step", [0.5, 0.01, 0.002])
@pytest.mark.parametrize("distance", [40.0, 5000.0, 60000.0])
def test_marked_calls_pass_over_empty_samples_only(always_marked, distance, step):
    marked_margin(always_marked, distance, step)


def test_marked_calls_of_parallel_rays(always_marked):
    marked_parallel(always_marked)


def test_marked_calls_of_long_axes(always_marked):
    marked_long_axis(always_marked)


def test_small_calls_do_without_marks(cuda_lib):
    """100^2 rays through 256^3 voxels: no slower through the binding than without scratch (with the
    marks 1.5 times as long, so a quarter tells the two apart)."""
    vbm = cuda_lib
    dims, W, H, step = (256, 256, 256), 100, 100, 1.0
    F = torch.from_numpy(blob_volume(64, 8, seed=1)).cuda().repeat_interleave(4, 0).repeat_interleave(4, 1)
    F = F.repeat_interleave(4, 2).contiguous()
    tf = vbm.make_tf(TF_KNOTS_X, TF_KNOTS_RGBA)
    cams_dev = vbm.cameras_to_device(camera_array(orbit_cameras(dims, 1, W, H)))
    out = [torch.empty((1, 4, H, W), device="cuda") for _ in range(2)]
    assert not vbm.dvr_marks_pay(dims, 1, W, H, step) and vbm.dvr_marks_pay(dims, 8, 512, 512, step)

    def bound():
        vbm.render_dvr(F, dims, tf, cams_dev, 1, W, H, step, out[0])

    def bare():
        assert vbm.load().vbm_render_dvr(vbm._ptr(F), vbm._dims(dims), ctypes.byref(tf), vbm._ptr(cams_dev), 1, W, H,
                                         ctypes.c_float(step), vbm._ptr(out[1]), vbm._stream()) == 0

    ms = []
    for call in (bound, bare):
        times = []
        for _ in range(8):
            start, end = torch.cuda.Event(enable_timing=True), torch.cuda.Event(enable_timing=True)
            start.record()
            for _ in range(8):
                call()
            end.record()
            torch.cuda.synchronize()
            times.append(start.elapsed_time(end))
        ms.append(min(times))
    assert torch.equal(out[0], out[1])
    assert ms[0] < 1.25 * ms[1], ms
