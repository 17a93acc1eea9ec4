"""Wavelet passes of volumes whose z extent needs more blocks than a grid's second axis holds."""

import numpy as np
import pytest
import torch

from oracle.dwt import dwt3d
from oracle.filters import filter_bank
from vbm_inputs import TF_KNOTS_RGBA, TF_KNOTS_X

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("dims,J,wavelet", [((2, 2, 1 << 20), 1, 0), ((4, 2, 1 << 20), 1, 1), ((4, 4, 1 << 20), 2, 0)])
def test_long_volumes_match_oracle(cuda_lib, dims, J, wavelet):
    """The same bound as the other shapes': the float32 chains of at most 27 taps against FP64."""
    vbm = cuda_lib
    nx, ny, nz = dims
    x = np.random.default_rng(nz).standard_normal((nz, ny, nx)).astype(np.float32)
    data = torch.from_numpy(x).cuda()
    vbm.dwt3d(data, 1, dims, J, wavelet, torch.empty(2 * x.size, device="cuda"))
    ref = dwt3d(x.astype(np.float64), J, filter_bank(wavelet))
    assert np.abs(data.cpu().numpy() - ref).max() < 2e-6 * max(1.0, np.abs(ref).max())
    # vbm_build's pyramid of the same extent
    F = torch.rand((nz, ny, nx), generator=torch.Generator(device="cuda").manual_seed(nx), device="cuda")
    tf = vbm.make_tf(TF_KNOTS_X, TF_KNOTS_RGBA)
    want = torch.empty((4, nz, ny, nx), device="cuda")
    vbm.tf_apply(F, tf, want)
    vbm.dwt3d(want, 4, dims, J, wavelet, torch.empty(2 * F.numel(), device="cuda"))
    coef = torch.empty_like(want)
    vbm.build(F, dims, tf, vbm.bank_build(J, wavelet), vbm.make_select(100), capacity=F.numel(), coef=coef)
    assert torch.equal(coef, want)
