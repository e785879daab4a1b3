"""GPU: the plan's sorts at the edges of their tiles (8192 keys) and key widths
(32 and 64 bits): the grid order is numpy's stable sort of the same keys, far-out
and non-finite coordinates come last, and the degridding items are the groups'."""
import numpy as np
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("wide", [False, True])
@pytest.mark.parametrize("n", [1, 31, 8191, 8192, 8193, 40001])
def test_orders(n, wide):
    from paper_2206_15117_gb300 import aw
    ctx = aw.aw_create(0)
    # (bin, tile, position) needs 33 bits when wide, 20 otherwise
    N, nw, npa, nfb = (4096, 8, 8, 8) if wide else (256, 2, 3, 2)
    rng = np.random.default_rng(n + wide)
    uvw = rng.uniform(-1.0, 1.0, (500, 3)) * 55.0
    uvw[7], uvw[8], uvw[9] = (np.inf, 0.0, 1.0), (1.0, np.nan, np.nan), (1e300, 1.0, -np.inf)
    row, chan = rng.integers(0, 500, n).astype(np.int32), rng.integers(0, 5, n).astype(np.int16)
    pa, fb = rng.integers(0, npa, 500).astype(np.uint8), rng.integers(0, nfb, 5).astype(np.uint8)
    freq = np.linspace(1.2e9, 1.5e9, 5)
    kw = dict(N=N, dl=0.4 / 256, OS=4, npol=4, nw=nw, w_max=270.0, supports=[8] * nw, pa=[0.1 * i for i in range(npa)],
              fbin_freqs=[1.3e9] * nfb)
    if wide:
        kw["dl"] = 1.0 / 4096
    ks = aw.aw_make_kernels(ctx, **kw)
    dev = [torch.as_tensor(x, device="cuda") for x in (uvw, row, chan, freq, pa, fb)]
    plan = aw.aw_plan_create(ctx, aw.vis_desc(*dev), ks, aw.aw_tune(32, 256, 2, 256, aw.AW_GRID_REGION))
    out = {k: torch.empty(n, dtype=torch.int32, device="cuda") for k in ("x0", "y0", "fx", "fy", "bin")}
    valid, flip = (torch.empty(n, dtype=torch.uint8, device="cuda") for _ in range(2))
    perm = torch.empty(n, dtype=torch.int32, device="cuda")
    aw.aw_plan_coords(plan, **out, flip=flip, valid=valid)
    aw.aw_plan_order(plan, perm)
    c = {k: v.cpu().numpy().astype(np.int64) for k, v in out.items()}
    ok = valid.cpu().numpy() == 1
    bad = np.isin(row, (7, 8, 9))
    assert not ok[bad].any() and np.all(c["x0"][bad] == 0)
    np.testing.assert_array_equal(flip.cpu().numpy() == 1, (uvw[row, 2] < 0))
    nt = N // 32
    key = ((c["bin"] * nt + c["y0"] // 32) * nt + c["x0"] // 32) * 1024 + c["y0"] % 32 * 32 + c["x0"] % 32
    key[~ok] = 1 << 60
    np.testing.assert_array_equal(perm.cpu().numpy(), np.argsort(key, kind="stable"))
    grp = ((c["bin"] * 64 + c["y0"] // 256) * 64 + c["x0"] // 256) * 16 + c["fy"] * 4 + c["fx"]
    cnt = np.unique(grp[ok], return_counts=True)[1]
    info = aw.aw_plan_query(plan)
    assert info.nitems_degrid == int(((cnt + 31) // 32).sum()) and info.nvalid == int(ok.sum())


# a descriptor whose nchan does not count every channel in use (C callers may leave it
# 0) gives the plan of the full one: the frequencies come from the caller's array
@pytest.mark.parametrize("nchan", [-1, 0, 2])
def test_channels_beyond_nchan(nchan):
    from paper_2206_15117_gb300 import aw
    ctx = aw.aw_create(0)
    n = 5000
    rng = np.random.default_rng(3)
    dev = [torch.as_tensor(x, device="cuda") for x in
           (rng.uniform(-1.0, 1.0, (200, 3)) * 50.0, rng.integers(0, 200, n).astype(np.int32),
            rng.integers(0, 5, n).astype(np.int16), np.linspace(1.2e9, 1.5e9, 5))]
    ks = aw.aw_make_kernels(ctx, N=256, dl=0.4 / 256, OS=4, npol=1, nw=2, w_max=260.0, supports=[8, 12])
    got = []
    for k in (5, nchan):
        vd = aw.vis_desc(*dev)
        vd.nchan = k
        plan = aw.aw_plan_create(ctx, vd, ks, aw.aw_tune(32, 256, 2, 256, aw.AW_GRID_REGION))
        out = {c: torch.empty(n, dtype=torch.int32, device="cuda") for c in ("x0", "y0", "fx", "fy", "bin")}
        perm = torch.empty(n, dtype=torch.int32, device="cuda")
        aw.aw_plan_coords(plan, **out)
        aw.aw_plan_order(plan, perm)
        got.append([x.cpu().numpy() for x in (*out.values(), perm)])
        assert aw.aw_plan_query(plan).nvalid > 1000
    for a, b in zip(*got):
        np.testing.assert_array_equal(a, b)


# what a REGION plan keeps beyond an OFFSETS plan where no bin takes a region (no support
# with a region form; a sparse full-pol set): the OFFSETS items, no second order
@pytest.mark.parametrize("kw", [dict(N=512, npol=1, nw=2, w_max=260.0, supports=[9, 17]),
                                dict(N=512, npol=1, nw=1, supports=[7]),
                                dict(N=4096, npol=4, nw=1, supports=[16], pa=[0.0, 0.1, 0.2, 0.3],
                                     fbin_freqs=[1.2e9, 1.3e9, 1.4e9, 1.5e9])])
def test_memory_without_regions(kw):
    from paper_2206_15117_gb300 import aw
    ctx = aw.aw_create(0)
    n, nrow = 2000000, 100000
    rng = np.random.default_rng(4)
    half = 0.45 * kw["N"] / 0.4                     # 0.45 of the grid at the highest frequency
    uvw = rng.uniform(-1.0, 1.0, (nrow, 3)) * (half * 299792458.0 / 1.5e9, half * 299792458.0 / 1.5e9, 50.0)
    pa, fb = rng.integers(0, 4, nrow).astype(np.uint8), rng.integers(0, 4, 16).astype(np.uint8)
    dev = [torch.as_tensor(x, device="cuda") for x in
           (uvw, rng.integers(0, nrow, n).astype(np.int32), rng.integers(0, 16, n).astype(np.int16),
            np.linspace(1.2e9, 1.5e9, 16), pa, fb)]
    ks = aw.aw_make_kernels(ctx, **kw, dl=0.4 / kw["N"], OS=4)
    vd = aw.vis_desc(*dev)

    def kept(mode):
        aw.aw_plan_destroy(aw.aw_plan_create(ctx, vd, ks, aw.aw_tune(32, 256, 2, 1024, mode)))
        free = torch.cuda.mem_get_info()[0]
        plan = aw.aw_plan_create(ctx, vd, ks, aw.aw_tune(32, 256, 2, 1024, mode))
        info = aw.aw_plan_query(plan)
        assert info.region_lists == 0 and info.nvalid > n // 2
        return free - torch.cuda.mem_get_info()[0], info.nitems_degrid
    (offsets, items), (region, _) = kept(aw.AW_GRID_OFFSETS), kept(aw.AW_GRID_REGION)
    assert region <= offsets + 16 * items + (4 << 20), (region, offsets, items)   # (two allocations' rounding)
