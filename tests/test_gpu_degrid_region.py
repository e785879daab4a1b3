"""GPU: the Stokes-I region degridding kernel (dense sets of more than a quarter of a
million visibilities) against the FP64 oracle: footprint blocks of 8, 16 and 24
taps, padded supports, wide supports on the item kernel beside it, runs of equal
offset that one warp takes and that the four share, flagged visibilities, the
subtracting form, the table precisions; full-pol sets with bins on and off the
region kernel; and both through the bounds-checked build."""
import json
import os
import subprocess
import sys
import textwrap

import numpy as np
import pytest
import torch

from paper_2206_15117_gb300 import synthetic as sy
from tests.gpu_cases import case_fullpol, rel_err
from tests.test_gpu_grid import Case, _check_degrid, _check_grid
from tests.test_gpu_region import REGION, _stokes_i

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))


@pytest.fixture(scope="module")
def ctx():
    from paper_2206_15117_gb300 import aw
    return aw.aw_create(0)


def _dense(ctx, supports, storage=0, radius=100.0, flagged=0.05, n_t=1200):
    from paper_2206_15117_gb300 import aw
    ob, kw = _stokes_i(supports, n_t=n_t, radius=radius)
    flags = (np.random.default_rng(8).random(ob.nvis) < flagged).astype(np.uint8)
    c = Case(ctx, ob, kw, storage=storage, flags=flags, tune=aw.aw_tune(32, 256, 2, 256, REGION))
    assert aw.aw_debug_region_tasks(c.plan)[1] > 0
    return c


def _subtract(c, in_place):
    from paper_2206_15117_gb300 import aw
    vis = torch.as_tensor(c.vis, device="cuda")
    out = vis if in_place else torch.full_like(vis, 7)
    aw.aw_degrid_subtract(c.ctx, c.plan, c.kd, torch.as_tensor(c.model, device="cuda"), vis, out)
    return out.cpu().numpy()


@pytest.mark.parametrize("supports", [(7, 8, 12), (15, 16, 18), (20, 24, 28), (32, 40, 48), (24, 48, 56), (9, 40, 64)])
def test_supports(ctx, supports):
    from paper_2206_15117_gb300 import aw
    c = _dense(ctx, supports)
    region = [s not in (9, 56, 64) for s in supports]      # those have no region form
    assert aw.aw_plan_query(c.plan).grid_kernels == 1 + (not all(region))
    co, ok = c.co, c.co.valid == 1
    bins = np.unique(co.bin[ok])
    assert len(bins) == len(supports) and (co.valid == 0).sum() > 100
    run = np.unique(np.stack([co.bin[ok], co.y0[ok] // 33, co.x0[ok] // 33, co.fy[ok], co.fx[ok]]), axis=1,
                    return_counts=True)[1]
    assert run.max() > 16 and run.min() < 4
    _check_degrid(c)
    _check_grid(c)
    # one FP32 rounding beside the prediction's
    pred = c.gpu_degrid()
    eps = 2.0 ** -23 * (np.abs(c.vis).max() + np.abs(pred).max())
    for in_place in (False, True):
        assert np.abs(_subtract(c, in_place) - (c.vis - pred)).max() <= 2 * eps


@pytest.mark.parametrize("storage,tol", [(1, 4e-3), (2, 5e-4)])
def test_reduced_precision(ctx, storage, tol):
    c = _dense(ctx, (12, 24, 56), storage=storage)
    V = c.oracle_degrid()
    l2, _ = rel_err(c.gpu_degrid(), V)
    assert 1e-6 < l2 < tol, l2
    l2, _ = rel_err(_subtract(c, True), np.where((c.co.valid == 1)[:, None], c.vis - V, c.vis))
    assert l2 < tol, l2


# footprints up to the grid's edge (some beyond it) and the flags off
def test_grid_edges(ctx):
    c = _dense(ctx, (16, 20, 40), radius=420.0, flagged=0.0, n_t=2400)
    ok = c.co.valid == 1
    assert c.co.x0[ok].min() == 0 and c.co.x0[ok].max() == 256 - 16 and (~ok).sum() > 100
    _check_degrid(c)


# full polarisation with bins that have a region form and bins that have none: the region
# kernel and OFFSETS on the second stream at once, direct and in the captured graph
@pytest.mark.parametrize("supports", [(9, 16, 24), (10, 17, 32)])
def test_fullpol_on_two_streams(ctx, supports):
    from paper_2206_15117_gb300 import aw
    ob, kw = case_fullpol(supports=supports, n_t=100, radius=60.0)
    c = Case(ctx, ob, kw, tune=aw.aw_tune(32, 256, 2, 256, REGION))
    info = aw.aw_plan_query(c.plan)
    assert info.region_lists == 1 and info.grid_kernels == 2
    _check_grid(c)
    _check_grid(c, batched=True)
    _check_grid(c, batched=True)  # the cached graph again
    _check_degrid(c)


# which sets have region tasks: some support above 8 and one with a region form
@pytest.mark.parametrize("supports,npol,lists,kernels", [
    ((7, 8, 12), 1, 1, 1), ((56, 64, 72), 1, 0, 1), ((9, 10, 17), 1, 0, 1), ((32, 40, 48), 1, 1, 1),
    ((7, 8, 12), 4, 1, 1), ((56, 64, 72), 4, 1, 1), ((9, 10, 17), 4, 0, 1), ((6, 7, 8), 4, 0, 1), ((48, 49), 1, 1, 2)])
def test_region_lists(ctx, supports, npol, lists, kernels):
    from paper_2206_15117_gb300 import aw
    ob, kw = (case_fullpol(supports=supports, n_t=100, radius=60.0) if npol == 4
              else _stokes_i(supports, n_t=100, radius=60.0))
    vd, keep = aw.device_observation(ob)
    plan = aw.aw_plan_create(ctx, vd, aw.aw_make_kernels(ctx, **kw), aw.aw_tune(32, 256, 2, 256, REGION))
    info = aw.aw_plan_query(plan)
    assert (info.region_lists, info.grid_kernels) == (lists, kernels)
    tasks = aw.aw_debug_region_tasks(plan)
    assert (tasks[0] > 0) == (lists == 1) and tasks[1] == 0


CHECKED = textwrap.dedent('''
    import json, sys
    import numpy as np
    import torch
    sys.path.insert(0, %r)
    from paper_2206_15117_gb300 import aw
    from tests.gpu_cases import case_fullpol, rel_err
    from tests.test_gpu_grid import Case
    from tests.test_gpu_degrid_region import REGION, _dense, _subtract
    assert aw.load()._name.endswith("libaw_checked.so"), aw.load()._name
    aw.aw_debug_bounds_status(reset=True)
    ctx = aw.aw_create(0)
    worst = 0.0
    ob, kw = case_fullpol(supports=(9, 16, 24), n_t=100, radius=60.0)
    for c in [_dense(ctx, (7, 18, 24)), _dense(ctx, (32, 48, 56)),
              Case(ctx, ob, kw, tune=aw.aw_tune(32, 256, 2, 256, REGION))]:
        V, G = c.oracle_degrid(), c.oracle_grid()[0]
        worst = max(worst, *rel_err(c.gpu_degrid(), V), *rel_err(c.gpu_grid()[0], G), *rel_err(c.gpu_grid(True)[0], G))
        worst = max(worst, *rel_err(_subtract(c, True), np.where((c.co.valid == 1)[:, None], c.vis - V, c.vis)))
    print("REPORT " + json.dumps(dict(status=aw.aw_debug_bounds_status(), worst=worst)))
''') % ROOT


def test_bounds_checked_build():
    from paper_2206_15117_gb300 import build as awbuild
    env = dict(os.environ, AW_LIBAW=awbuild.build(bounds_check=True))
    r = subprocess.run([sys.executable, "-c", CHECKED], env=env, capture_output=True, text=True, timeout=900, cwd=ROOT)
    assert r.returncode == 0, r.stdout[-3000:] + r.stderr[-3000:]
    rep = json.loads([l for l in r.stdout.splitlines() if l.startswith("REPORT ")][-1][len("REPORT "):])
    assert rep["status"] == 0 and rep["worst"] < 1e-5, rep
