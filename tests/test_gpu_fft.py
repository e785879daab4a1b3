"""GPU: the library's own two-pass transforms at every size they take (and the
sizes next to them) and every step count, both directions, against FP64.  FP32 rounding grows with
the square root of the number of steps: 4e-7 relative L2 holds log2(N^2) = 24
steps of half an ulp of the larger operand with room for three."""
import math

import numpy as np
import pytest
import torch

from oracle import core as oc
from paper_2206_15117_gb300 import synthetic as sy

pytestmark = pytest.mark.gpu
TOL = 4e-7


@pytest.fixture(scope="module")
def ctx():
    from paper_2206_15117_gb300 import aw
    return aw.aw_create(0)


def _err(a, b):
    return np.linalg.norm((a - b).ravel()) / np.linalg.norm(b.ravel())


@pytest.mark.parametrize("npol,N", [(4, 128), (1, 256), (4, 256), (1, 512), (4, 1024), (1, 2048), (1, 4096), (1, 8192)])
def test_transforms(ctx, npol, N):
    from paper_2206_15117_gb300 import aw
    ks = aw.aw_make_kernels(ctx, N=N, dl=math.radians(2.0) / N, OS=2, npol=npol, supports=[8], role=aw.AW_ROLE_DEGRID)
    c = oc.grid_correction_1d(7.0, N)
    corr = (c[:, None] * c[None, :])[None]
    corr[:, 0, :] = corr[:, :, 0] = 0
    G = sy.random_grid(npol, N, seed=N + npol).astype(np.complex64)
    grid = torch.as_tensor(G, device="cuda")
    img = torch.full((npol, N, N), 7.0, device="cuda")
    aw.aw_fft_to_image(ctx, ks, grid, 2.0, img)
    Z = np.fft.ifft2(G.astype(np.complex128), axes=(1, 2)) * (N * N)
    assert _err(grid.cpu().numpy(), Z) < TOL                     # left transformed
    sign = 1 - 2.0 * (np.add.outer(np.arange(N), np.arange(N)) & 1)
    ref = np.fft.fftshift(Z.real, axes=(1, 2)) * sign / 2.0
    ref[:, 0, :] = ref[:, :, 0] = 0
    got = img.cpu().numpy()
    assert _err(got * corr, ref) < TOL
    assert np.all(got[:, 0, :] == 0) and np.all(got[:, :, 0] == 0)
    model = (np.random.default_rng(N).standard_normal((npol, N, N)) * corr).astype(np.float32)
    aw.aw_image_to_grid(ctx, ks, torch.as_tensor(model, device="cuda"), grid)
    a = model.astype(np.float64)
    a[:, 1:, 1:] /= corr[:, 1:, 1:]
    F = np.fft.fft2(np.fft.ifftshift(a * sign, axes=(1, 2)), axes=(1, 2))
    assert _err(grid.cpu().numpy(), F) < TOL
