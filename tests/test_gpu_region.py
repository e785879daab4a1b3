"""GPU: the region gridding kernel at the edges of its forms (footprint blocks
of 8, 16 and 24 taps and their mixtures, supports padded to a multiple of 8,
runs and tasks longer than a staging round) against the FP64 oracle."""
import math

import numpy as np
import pytest

from paper_2206_15117_gb300 import synthetic as sy
from tests.gpu_cases import case_fullpol, rel_err
from tests.test_gpu_grid import Case, _check_degrid, _check_grid

pytestmark = pytest.mark.gpu

REGION = 3


@pytest.fixture(scope="module")
def ctx():
    from paper_2206_15117_gb300 import aw
    return aw.aw_create(0)


def _stokes_i(supports, n_t=60, radius=120.0, N=256):
    ob = sy.small_observation(n_ant=14, radius_m=radius, n_t=n_t, freq=(1.2e9, 1.35e9, 1.5e9), seed=sy.BASE_SEED + 410)
    return ob, dict(N=N, dl=math.radians(3.0) / N, OS=8, W=7.0, npol=1, nw=len(supports), w_max=ob.w_max,
                    supports=list(supports))


@pytest.mark.parametrize("supports", [(7, 8, 12), (15, 16, 18), (20, 24, 28), (32, 40, 48), (56, 64, 72), (9, 10, 17)])
@pytest.mark.parametrize("npol", [1, 4])
def test_region_supports(ctx, npol, supports):
    from paper_2206_15117_gb300 import aw
    ob, kw = case_fullpol(supports=supports, n_t=30, radius=100.0) if npol == 4 else _stokes_i(supports)
    flags = (np.random.default_rng(5).random(ob.nvis) < 0.05).astype(np.uint8)
    c = Case(ctx, ob, kw, tune=aw.aw_tune(32, 256, 2, 256, REGION), flags=flags)
    _check_grid(c)
    _check_grid(c, batched=True)
    _check_degrid(c)


# runs of equal offset longer than a round of 64 and tasks longer than 1024, a
# non-finite visibility among them
@pytest.mark.parametrize("npol", [1, 4])
def test_region_long_runs(ctx, npol):
    from paper_2206_15117_gb300 import aw
    sup = (16, 24, 40)
    ob, kw = case_fullpol(supports=sup, n_t=400, radius=20.0) if npol == 4 else _stokes_i(sup, n_t=700, radius=20.0)
    c = Case(ctx, ob, kw, tune=aw.aw_tune(32, 256, 2, 256, REGION))
    co, ok = c.co, c.co.valid == 1
    run = np.stack([co.bin[ok], co.y0[ok] // 41, co.x0[ok] // 41, co.fy[ok], co.fx[ok]])
    assert np.unique(run, axis=1, return_counts=True)[1].max() > 64
    c.vis[17, 0] = np.nan
    _check_grid(c)
    _check_degrid(c)


@pytest.mark.parametrize("storage,tol", [(1, 4e-3), (2, 5e-4)])
def test_region_padded_support_reduced_precision(ctx, storage, tol):
    from paper_2206_15117_gb300 import aw
    ob, kw = case_fullpol(supports=(12, 20, 40), n_t=30, radius=100.0)
    c = Case(ctx, ob, kw, storage=storage, tune=aw.aw_tune(32, 256, 2, 256, REGION))
    l2, mx = rel_err(c.gpu_grid(batched=True)[0], c.oracle_grid()[0])
    assert l2 < tol and mx < 4 * tol, (l2, mx)
    l2, _ = rel_err(c.gpu_degrid(), c.oracle_degrid())
    assert l2 < tol, l2


# supports of at most 8 (one warp an item from 65536 visibilities, a CTA an item
# below); the subtraction adds one FP32 rounding to the prediction
@pytest.mark.parametrize("n_t", [200, 300])
def test_degrid_small_supports(ctx, n_t):
    import torch
    from paper_2206_15117_gb300 import aw
    ob, kw = _stokes_i((7, 8), n_t=n_t)
    flags = (np.random.default_rng(6).random(ob.nvis) < 0.05).astype(np.uint8)
    c = Case(ctx, ob, kw, tune=aw.aw_tune(32, 256, 2, 256, 1), flags=flags)
    assert (int((c.co.valid == 1).sum()) >= 65536) == (n_t == 300)
    _check_degrid(c)
    vis, out = torch.as_tensor(c.vis, device="cuda"), torch.zeros_like(torch.as_tensor(c.vis, device="cuda"))
    aw.aw_degrid_subtract(ctx, c.plan, c.kd, torch.as_tensor(c.model, device="cuda"), vis, out)
    pred = c.gpu_degrid()
    eps = 2.0 ** -23 * (np.abs(c.vis).max() + np.abs(pred).max())
    assert np.abs(out.cpu().numpy() - (c.vis - pred)).max() <= 2 * eps


# full-pol sets with few visibilities a bin and tile take OFFSETS alone
def test_sparse_set_takes_offsets(ctx):
    from paper_2206_15117_gb300 import aw
    ob, kw = case_fullpol(supports=(24, 32, 40), n_t=1, radius=200.0)
    c = Case(ctx, ob, kw, tune=aw.aw_tune(32, 256, 2, 256, REGION))
    info = aw.aw_plan_query(c.plan)
    assert info.region_lists == 0 and info.grid_kernels == 1
    _check_grid(c)
    _check_grid(c, batched=True)
    _check_degrid(c)


# dense Stokes-I sets whose degridding tasks are too short for the region kernel keep no
# list of them: as many device buffers as a sparse set's plan
def test_short_degridding_tasks_are_not_kept(ctx):
    from paper_2206_15117_gb300 import aw

    def buffers(n_t, radius):
        ob, kw = _stokes_i((16, 24, 40), n_t=n_t, radius=radius)
        ks = aw.aw_make_kernels(ctx, **kw)
        vd, keep = aw.device_observation(ob)
        live = aw.aw_debug_alloc_stats()[0]
        plan = aw.aw_plan_create(ctx, vd, ks, aw.aw_tune(32, 256, 2, 256, REGION))
        assert aw.aw_plan_query(plan).region_lists > 0
        return aw.aw_debug_alloc_stats()[0] - live
    # 31850 visibilities a bin and tile, 96 a task; 19 a bin and tile
    assert buffers(700, 20.0) == buffers(2, 200.0)


# a region schedule found on one set is used on sets that have its planes of supports up to
# 40, as before the schedule took every plane; sets of fewer planes take OFFSETS
def test_cached_region_tune_on_fewer_planes(ctx):
    from paper_2206_15117_gb300 import aw
    own = aw.aw_create(0)
    ob, kw = case_fullpol(supports=(16, 24, 48), n_t=2000, radius=50.0)
    vd, keep = aw.device_observation(ob)
    t = aw.aw_autotune(own, vd, aw.aw_make_kernels(own, **kw))
    if t.grid_mode != REGION:
        pytest.skip("another schedule was the fastest: %d" % t.grid_mode)
    assert t.split_planes == 2
    for supports, lists in (((16, 24), 1), ((16,), 0)):
        few = dict(kw, nw=len(supports), supports=list(supports))
        assert aw.aw_plan_query(aw.aw_plan_create(own, vd, aw.aw_make_kernels(own, **few))).region_lists == lists
