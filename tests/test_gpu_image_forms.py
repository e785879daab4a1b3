"""GPU: the four-pixel and single-pixel forms of the image kernels (smallest
size, arrays not aligned to 16 bytes, pixel counts that are not a multiple of
4) against the FP64 oracle."""
import math

import numpy as np
import pytest
import torch

from oracle import core as oc
from paper_2206_15117_gb300 import synthetic as sy
from tests.gpu_cases import TOL_FP32, rel_err

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2206_15117_gb300 import aw
    return aw.aw_create(0)


def _at(a, off, dtype):
    """`a` on the device, `off` elements into its storage."""
    t = torch.empty(a.size + off, dtype=dtype, device="cuda")[off:].view(a.shape)
    return t.copy_(torch.as_tensor(a))


@pytest.mark.parametrize("off", [0, 1])
@pytest.mark.parametrize("npol,N", [(1, 16), (4, 32), (4, 1024), (1, 2048)])
def test_image_and_grid(ctx, npol, N, off):
    from paper_2206_15117_gb300 import aw
    ks = aw.aw_make_kernels(ctx, N=N, dl=math.radians(2.0) / N, OS=2, npol=npol, supports=[8], role=aw.AW_ROLE_DEGRID)
    c = oc.grid_correction_1d(7.0, N)
    corr = (c[:, None] * c[None, :])[None]
    G = sy.random_grid(npol, N, seed=N + npol)
    img = _at(np.full((npol, N, N), 7.0, np.float32), off, torch.float32)
    aw.aw_fft_to_image(ctx, ks, _at(G, off, torch.complex64), 321.0, img)
    ref, got = oc.fft_to_image(G.astype(np.complex128), 7.0, 321.0), img.cpu().numpy()
    assert rel_err(got * corr, ref * corr)[0] < TOL_FP32     # the correction amplifies rounding at the edge
    assert np.all(got[:, 0, :] == 0) and np.all(got[:, :, 0] == 0)
    model = np.random.default_rng(N).standard_normal((npol, N, N)).astype(np.float32) * corr.astype(np.float32)
    grid = _at(np.zeros((npol, N, N), np.complex64), off, torch.complex64)
    aw.aw_image_to_grid(ctx, ks, _at(model, off, torch.float32), grid)
    a = model.astype(np.float64)
    a[:, 1:, 1:] /= corr[:, 1:, 1:]
    a[:, 0, :] = a[:, :, 0] = 0
    ax = (1, 2)
    F = np.fft.fftshift(np.fft.fft2(np.fft.ifftshift(a, axes=ax), axes=ax), axes=ax)
    assert rel_err(grid.cpu().numpy(), F)[0] < TOL_FP32


@pytest.mark.parametrize("N,off", [(32, 0), (33, 0), (32, 1), (1024, 0)])
@pytest.mark.parametrize("nf", [1, 6])
def test_gamma(ctx, N, off, nf):
    from paper_2206_15117_gb300 import aw
    B = np.random.default_rng(N + nf).uniform(0.0, 1.0, (nf, N, N)).astype(np.float32)
    B[:, 0, :] = 0.0
    gam = _at(np.full((N, N), 7.0, np.float32), off, torch.float32)
    aw.mosaic_gamma(ctx, _at(B, off, torch.float32), 0.2, gam)
    ref, got = oc.mosaic_gamma(B.astype(np.float64), 0.2), gam.cpu().numpy()
    s = np.sqrt((B.astype(np.float64) ** 2).sum(0))
    far = np.abs(s / s.max() - 0.2) > 1e-5
    np.testing.assert_allclose(got[far], ref[far], rtol=1e-5, atol=0)
