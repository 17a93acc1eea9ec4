"""vbm_build's first level in slabs of the least height: wide planes, of which the scratch holds 16, so
that a slab gives four plane pairs and overlaps the next by as many planes as it gives."""

import pytest
import torch

from vbm_inputs import TF_KNOTS_RGBA, TF_KNOTS_X

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wavelet", [0, 1])
def test_build_pyramid_in_least_slabs(cuda_lib, wavelet):
    """The same bits as tf_apply followed by dwt3d."""
    vbm = cuda_lib
    dims = nx, ny, nz = 1024, 1040, 24
    n, plane = nx * ny * nz, nx * ny
    # floats of scratch: four channels whole, or the largest of 1.2 volumes, 2^26 and 64 planes
    assert max(n + n // 5, 1 << 26) < 64 * plane < 4 * n
    F = torch.rand((nz, ny, nx), generator=torch.Generator(device="cuda").manual_seed(3), device="cuda") * 1.4 - 0.2
    tf = vbm.make_tf(TF_KNOTS_X, TF_KNOTS_RGBA)
    want = torch.empty((4, nz, ny, nx), device="cuda")
    vbm.tf_apply(F, tf, want)
    vbm.dwt3d(want, 4, dims, 2, wavelet, torch.empty(2 * n, device="cuda"))
    coef = torch.empty_like(want)
    vbm.build(F, dims, tf, vbm.bank_build(2, wavelet), vbm.make_select(100), capacity=n, coef=coef)
    assert torch.equal(coef, want)
