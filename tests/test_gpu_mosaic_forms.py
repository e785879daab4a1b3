"""GPU: the forms of the mosaic kernels: position maps by expansion and in FP64
(wide fields, far frames, sizes that do not fill a tile), and the four-pixel and
single-pixel combination (odd sizes, unaligned arrays), against the FP64 oracle."""
import math

import numpy as np
import pytest
import torch

from oracle import core as oc
from oracle import mosaic as om
from tests.test_gpu_mosaic import _compare, _image

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def ctx():
    from paper_2206_15117_gb300 import aw
    return aw.aw_create(0)


@pytest.mark.parametrize("interp", [0, 1])
@pytest.mark.parametrize("dl_s,Ns,dl_d,Nd,dra,ddec", [
    (2e-4, 97, 2e-4, 63, 0.004, -0.003),        # below one tile, an odd source
    (2e-4, 130, 1e-4, 385, 0.01, 0.006),        # several tiles, a remainder on each axis
    (4e-3, 150, 3e-3, 200, 0.1, -0.2),          # wide: the expansion gives way to FP64
    (6e-4, 64, 1.2e-2, 160, 0.3, 0.4),          # the destination reaches the horizon
    (2e-4, 64, 2e-4, 70, 1.5, 0.9)])            # nothing but fill
def test_reproject_forms(ctx, interp, dl_s, Ns, dl_d, Nd, dra, ddec):
    src = om.frame(0.7, -0.5, dl_s, Ns)
    dst = om.frame(0.7 + dra, -0.5 + ddec, dl_d, Nd, cx=Nd / 2 + 0.3)
    _compare(ctx, _image(Ns, 3, seed=Ns), src, dst, interp, fill=-2.0)


@pytest.mark.parametrize("N,off", [(32, 0), (33, 0), (32, 1)])
@pytest.mark.parametrize("nf,nplane", [(1, 1), (5, 6), (9, 4)])
def test_combine_forms(ctx, N, off, nf, nplane):
    from paper_2206_15117_gb300 import aw
    rng = np.random.default_rng(N + nf)

    def dev(a):   # `off` floats into its storage
        t = torch.empty(a.size + off, dtype=torch.float32, device="cuda")[off:].view(a.shape)
        return t.copy_(torch.as_tensor(a))
    imgs = rng.normal(size=(nf, nplane, N, N)).astype(np.float32)
    beams = rng.uniform(0, 1, size=(nf, N, N)).astype(np.float32)
    gam = oc.mosaic_gamma(beams.astype(np.float64), 0.1).astype(np.float32)
    out = dev(np.zeros((nplane, N, N), np.float32))
    aw.aw_mosaic_combine(ctx, dev(imgs), dev(beams), dev(gam), out)
    ref = om.combine(imgs, beams, gam)
    assert np.abs(out.cpu().numpy() - ref).max() < 1e-5 * np.abs(ref).max()


# an output that shares memory with the images: in place, and from one plane before
# them on (a plane's output over the plane that has been read already)
@pytest.mark.parametrize("before", [0, 1])
@pytest.mark.parametrize("nplane", [4, 9])
def test_combine_over_its_images(ctx, nplane, before):
    from paper_2206_15117_gb300 import aw
    N, nf = 256, 3
    rng = np.random.default_rng(nplane)
    imgs = rng.normal(size=(nf, nplane, N, N)).astype(np.float32)
    beams = rng.uniform(0, 1, size=(nf, N, N)).astype(np.float32)
    gam = oc.mosaic_gamma(beams.astype(np.float64), 0.1).astype(np.float32)
    buf = torch.zeros((before + nf * nplane, N, N), dtype=torch.float32, device="cuda")
    buf[before:] = torch.as_tensor(imgs.reshape(-1, N, N))
    out = buf[:nplane]
    aw.aw_mosaic_combine(ctx, buf[before:].view(nf, nplane, N, N), torch.as_tensor(beams, device="cuda"),
                         torch.as_tensor(gam, device="cuda"), out)
    ref = om.combine(imgs, beams, gam)
    assert np.abs(out.cpu().numpy() - ref).max() < 1e-5 * np.abs(ref).max()
