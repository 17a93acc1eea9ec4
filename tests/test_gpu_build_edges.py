"""vbm_build at the sizes where its band-parallel selection and map can go wrong: bands of one
element, of odd and of ragged counts, shorter than a mask word, longer than a marking chunk; ties,
empty space and constant volumes; budgets of none, of a few and of everything."""

import numpy as np
import pytest
import torch

from _helpers import oracle_bank
from oracle.dwt import subband_slices, subbands
from oracle.mapping import map_coefficients, select_all
from vbm_inputs import TF_KNOTS_RGBA, TF_KNOTS_X, blob_volume

pytestmark = pytest.mark.gpu


def _volume(kind, dims, seed):
    nx, ny, nz = dims
    rng = np.random.default_rng(seed)
    if kind == "noise":
        return rng.uniform(0.0, 1.0, (nz, ny, nx)).astype(np.float32)
    if kind == "steps":        # few distinct values: magnitudes tie, most are zero
        F = np.zeros((nz, ny, nx), dtype=np.float32)
        F[nz // 4: nz // 2 + 1, ny // 4: ny // 2 + 1] = 0.5
        F[nz // 2:, :, nx // 2:] = 0.75
        return F
    if kind == "flat":
        return np.full((nz, ny, nx), 0.6, dtype=np.float32)
    G = max(dims)
    return np.ascontiguousarray(blob_volume(G, 6, seed)[:nz, :ny, :nx])


@pytest.mark.parametrize("dims,J,K_tot,kind,wavelet,min_per_band", [
    ((2, 2, 2), 1, 5, "noise", 0, 10),              # one element a band
    ((6, 10, 14), 1, 100, "noise", 0, 10),          # 105 elements a band: odd count
    ((32, 32, 32), 5, 3000, "blobs", 0, 10),        # down to one element at the last level
    ((34, 18, 22), 1, 400, "blobs", 0, 10),         # 1683 elements: no multiple of 4 or 32
    ((68, 44, 52), 2, 6000, "blobs", 0, 10),        # 19,448 elements: chunks of 8192 and a remainder
    ((96, 64, 80), 4, 30000, "blobs", 1, 10),
    ((64, 32, 48), 3, 4000, "steps", 1, 10),        # ties at the K-th value, zero medians
    ((32, 32, 32), 2, 500, "flat", 1, 10),          # nothing but the approximation band
    ((32, 32, 32), 2, 10 ** 9, "blobs", 0, 10),     # budget above every band's size
    ((32, 32, 32), 2, 1, "blobs", 0, 0),            # most bands get a budget of 0
])
def test_build_edges_match_oracle(cuda_lib, dims, J, K_tot, kind, wavelet, min_per_band):
    vbm = cuda_lib
    F = _volume(kind, dims, seed=sum(dims) + J)
    tf = vbm.make_tf(TF_KNOTS_X, TF_KNOTS_RGBA)
    coef = torch.zeros(4 * F.size, device="cuda")
    keep = torch.full((F.size,), 7, dtype=torch.uint8, device="cuda")
    sel = vbm.make_select(K_tot, min_per_band=min_per_band)
    P, n = vbm.build(torch.from_numpy(F).cuda(), dims, tf, vbm.bank_build(J, wavelet), sel, capacity=F.size + 3,
                     coef=coef, keep=keep)
    A = coef.cpu().numpy().reshape(4, *F.shape)
    masks, _, _, _ = select_all(A, J, K_tot, min_per_band=min_per_band, dtype=np.float32)
    got = keep.cpu().numpy().reshape(F.shape)
    for (j, o), m in zip(subbands(J), masks):
        assert np.array_equal(got[subband_slices(F.shape, j, o)], m.astype(np.uint8)), (j, o)
    assert n == sum(int(m.sum()) for m in masks)
    ref = map_coefficients(A.astype(np.float64), masks, J, oracle_bank(J, wavelet))
    P = P.cpu().numpy()
    assert not P[:, n:].any()
    assert np.allclose(P[:10, :n], ref[:10], atol=1e-5 * max(dims))
    if n:
        assert np.allclose(P[10, :n], ref[10], atol=2e-5 * np.abs(ref[10]).max())
    assert np.allclose(P[11:14, :n], ref[11:14], rtol=1e-5, atol=1e-9)


def test_build_workspace_need_not_be_aligned(cuda_lib):
    """The workspace size holds at any address: the scratch is aligned inside it."""
    import ctypes
    vbm = cuda_lib
    F = torch.from_numpy(blob_volume(32, 4, 2)).cuda()
    tf, bank, sel = vbm.make_tf(TF_KNOTS_X, TF_KNOTS_RGBA), vbm.bank_build(2), vbm.make_select(3000)
    want, n = vbm.build(F, (32, 32, 32), tf, bank, sel, capacity=6000)
    size = ctypes.c_size_t()
    lib = vbm.load()
    assert lib.vbm_build_workspace_size(vbm._dims((32, 32, 32)), 2, ctypes.byref(size)) == 0
    for shift in (8, 200):
        ws = torch.empty(size.value + shift, dtype=torch.uint8, device="cuda")[shift:]
        P, m = torch.zeros((14, 6000), device="cuda"), ctypes.c_int64()
        args = (vbm._ptr(F), vbm._dims((32, 32, 32)), ctypes.byref(tf), ctypes.byref(bank), ctypes.byref(sel),
                vbm._ptr(P), 6000, ctypes.byref(m), None, None, vbm._ptr(ws))
        assert lib.vbm_build(*args, size.value - 1, vbm._stream()) == vbm.VBM_ERR_ARG
        assert lib.vbm_build(*args, size.value, vbm._stream()) == 0
        assert m.value == n and torch.equal(P, want)


@pytest.mark.parametrize("dims,J,wavelet", [
    ((2, 2, 2), 1, 0), ((2, 2, 2), 1, 1),           # every tap wraps, several times round
    ((6, 10, 14), 1, 0), ((6, 10, 14), 1, 1),       # halves of odd length: no paired stores
    ((4, 64, 2), 1, 0), ((264, 12, 20), 2, 0),      # one position beyond a 256-wide tile, and then some
    ((36, 28, 140), 2, 1), ((32, 32, 32), 5, 0),    # regions down to 2^3
    ((1028, 4, 12), 2, 0), ((8, 520, 8), 3, 0)])
def test_dwt_edges_match_oracle(cuda_lib, dims, J, wavelet):
    """Ragged regions of the wavelet passes against the oracle, at an aligned and at an
    odd address (the same bits); vbm_build's pyramid, whose first level reads the volume
    through the transfer function, equals tf_apply followed by dwt3d."""
    from oracle.dwt import dwt3d
    from oracle.filters import filter_bank
    vbm = cuda_lib
    nx, ny, nz = dims
    n = nx * ny * nz
    x = np.random.default_rng(n).standard_normal((3, nz, ny, nx)).astype(np.float32)
    got = []
    for shift in (0, 1):
        buf, tmp = torch.zeros(3 * n + shift, device="cuda"), torch.zeros(2 * n + shift, device="cuda")
        buf[shift:] = torch.from_numpy(x).cuda().reshape(-1)
        vbm.dwt3d(buf[shift:], 3, dims, J, wavelet, tmp[shift:])
        got.append(buf[shift:].cpu().numpy().reshape(x.shape))
    assert np.array_equal(got[0], got[1])
    ref = np.stack([dwt3d(c.astype(np.float64), J, filter_bank(wavelet)) for c in x])
    assert np.abs(got[0] - ref).max() < 2e-6 * max(1.0, np.abs(ref).max())
    _check_build_pyramid(vbm, dims, J, wavelet)


@pytest.mark.parametrize("dims,J,wavelet", [((256, 256, 272), 2, 0), ((256, 256, 272), 1, 1), ((1024, 2064, 8), 1, 0)])
def test_build_pyramid_in_slabs(cuda_lib, dims, J, wavelet):
    """Volumes whose four channels do not fit the scratch whole go slab by slab: the same bits."""
    _check_build_pyramid(cuda_lib, dims, J, wavelet)


def _check_build_pyramid(vbm, dims, J, wavelet):
    nx, ny, nz = dims
    F = torch.rand((nz, ny, nx), generator=torch.Generator(device="cuda").manual_seed(nx), device="cuda") * 1.4 - 0.2
    tf = vbm.make_tf(TF_KNOTS_X, TF_KNOTS_RGBA)
    want = torch.empty((4, nz, ny, nx), device="cuda")
    vbm.tf_apply(F, tf, want)
    vbm.dwt3d(want, 4, dims, J, wavelet, torch.empty(2 * F.numel(), device="cuda"))
    coef = torch.empty_like(want)
    vbm.build(F, dims, tf, vbm.bank_build(J, wavelet), vbm.make_select(100), capacity=F.numel(), coef=coef)
    assert torch.equal(coef, want)
