"""What is timed: the calls a user of the framework makes, over the range of
sizes, schedules and table precisions they are made at.

Geometry: the 36-antenna earth-rotation array of the package's synthetic
observations, with the row and channel of every visibility drawn from the
seed.  Kernel tables are made here (a tapered w chirp times a Mueller matrix
that varies over the support, as the synthesised kernels do) and handed over
with aw_kernel_set_import, so that exact() knows their values.
"""
import math

import numpy as np
import torch

from paper_2206_15117_gb300 import aw
from paper_2206_15117_gb300 import synthetic as sy

DEV = "cuda:0"
STORAGE = {"fp32": aw.AW_STORAGE_FP32, "bf16": aw.AW_STORAGE_BF16, "fp16": aw.AW_STORAGE_FP16}
MODES = {"tiles": aw.AW_GRID_TILES, "offsets": aw.AW_GRID_OFFSETS, "hybrid": aw.AW_GRID_HYBRID,
         "region": aw.AW_GRID_REGION}
EXACT_TAPS = 2.0e10   # visibility-taps above which the 64-bit sum takes too long


def _obs(kind, name, **kw):
    """An observation: N^2 grid of field `deg` degrees, npol, w planes nw, supports
    8..64 (+ extra), oversampling os, npa x nfb beam bins, nvis visibilities from n_t
    time samples of 630 baselines and nchan channels, and the gridding schedule."""
    c = dict(name=name, kind=kind, N=2048, deg=3.0, npol=4, nw=32, extra=0, os=8, npa=1, nfb=1, nvis=1000003,
             n_t=2000, nchan=16, storage="fp32", tune="region", weights=False, flags=False)
    c.update(kw)
    return c


def listed():
    return [
        # one Stokes-I major cycle of a small narrow-field image (no w term, 7-cell kernel):
        # model -> grid -> residual visibilities -> grid -> residual image; launches count
        _obs("cycle", "cycle_i_512", N=512, deg=1.0, npol=1, nw=1, os=4, nvis=126000, n_t=200, nchan=1, tune="default"),
        # the paper's workload: wide-field full-polarisation AW gridding and the degridding
        # of the model, one spectral window of a long track
        _obs("grid", "grid_aw_4096", N=4096, extra=8, npa=4, nfb=2, nvis=12000011, nchan=72),
        _obs("degrid", "degrid_aw_4096", N=4096, extra=8, npa=4, nfb=2, nvis=12000011, nchan=72),
        # Stokes-I w-projection imaging of a whole track, and its prediction
        _obs("grid", "grid_w_2048", npol=1, nvis=20160000),
        _obs("degrid", "degrid_w_2048", npol=1, nvis=20160000),
        # one mosaic field with 16-bit tables: imaging weights and flags as measured data have them
        _obs("grid", "grid_aw_2048_bf16", npa=3, nfb=2, nvis=3000017, storage="bf16", weights=True, flags=True),
        # the subtraction of a major cycle on one short snapshot set
        _obs("residual", "residual_aw_2048_fp16", npa=2, nfb=2, nvis=700001, storage="fp16", n_t=300),
        # uv grid -> the four dirty Stokes images (the uv grid is kept: the call transforms a copy)
        dict(name="image_4096", kind="image", N=4096, deg=3.0, npol=4, to_grid=False),
        # the plan of a new data set: coordinates, sort, work items
        _obs("plan", "plan_aw_4096", N=4096, extra=8, npa=4, nfb=2, nvis=12000011, nchan=72),
        # a Hogbom minor cycle on the four dirty images
        dict(name="hogbom_2048", kind="hogbom", N=2048, npol=4, iters=500, patch=256),
        # seven fields onto the mosaic frame, the weights of Eq. 1 and the combination
        dict(name="mosaic_7x2048", kind="mosaic", fields=7, N=2048, Nm=4096, deg=3.0, npol=4, interp="cubic"),
        # gridding with the learned kernels evaluated inline (no tables)
        _obs("learned", "learned_aw_2048", npa=2, nfb=2, nvis=100003, n_t=993, degrid=False),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["grid", "grid", "degrid", "degrid", "residual", "cycle", "image", "plan", "hogbom", "mosaic",
                       "learned"])
    if kind == "image":
        return dict(kind=kind, N=2 ** rng.randint(8, 12), deg=rng.uniform(0.5, 4.0), npol=rng.choice([1, 4]),
                    to_grid=rng.random() < 0.5)
    if kind == "hogbom":
        N = 2 ** rng.randint(8, 11)
        return dict(kind=kind, N=N, npol=rng.choice([1, 4]), iters=_log(rng, 20, 500),
                    patch=rng.randint(N // 32, N // 8))
    if kind == "mosaic":
        N = 2 ** rng.randint(8, 11)
        return dict(kind=kind, fields=rng.randint(2, 7), N=N, Nm=rng.choice([N + 2 * rng.randint(50, 200), 2 * N]),
                    deg=rng.uniform(1.0, 3.0), npol=rng.choice([1, 4]), interp=rng.choice(["cubic", "bilinear"]))
    npol = rng.choice([1, 4])
    N = 2 ** rng.randint(9 if kind == "cycle" else 10, 12)
    c = _obs(kind, "", npol=npol, N=N, deg=rng.uniform(1.0, 3.0) * N / 4096.0 + 0.5, nw=rng.choice([1, 8, 16, 32]),
             extra=rng.choice([0, 0, 8, 4]), os=rng.choice([4, 8, 8]), nchan=rng.randint(1, 48),
             n_t=_log(rng, 100, 2000), storage=rng.choice(["fp32", "fp32", "bf16", "fp16"]),
             tune=rng.choice(["region", "region", "offsets", "hybrid", "tiles", "default"]),
             weights=rng.random() < 0.5, flags=rng.random() < 0.3)
    if npol == 4:
        c["npa"], c["nfb"] = rng.randint(1, 4), rng.randint(1, min(2, c["nchan"]))
    top = 630 * c["n_t"] * c["nchan"]
    hi = {"learned": 100000, "cycle": 2000000, "plan": 8000000}.get(kind, 5000000 if npol == 4 else 12000000)
    c["nvis"] = min(_log(rng, 20000, hi), top)
    if kind == "learned":
        c["degrid"] = rng.random() < 0.5
        c["nw"], c["extra"] = rng.choice([8, 16, 32]), 0
    del c["name"]
    return c


# ---------------------------------------------------------------- inputs
def _rng(case, seed, tag):
    return np.random.default_rng([seed, sum(ord(c) for c in tag), case["N"]])


def _gen(seed, tag):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed * 1000003 + sum(ord(c) * 31 ** i for i, c in enumerate(tag)) % 1000003)
    return g


def _randc(g, *shape):
    return torch.view_as_complex(torch.randn(*shape, 2, generator=g, device=DEV))


def _supports(case):
    if case["nw"] == 1:
        return [7 if case["npol"] == 1 else 8 + case["extra"]]
    return sy.w_supports(case["nw"], extra=case["extra"])


def _geometry(case, seed):
    """The observation's arrays on the device, w_max and the spec of its kernels."""
    r = _rng(case, seed, "array")
    bxyz = sy.baselines_xyz(sy.antenna_enu(36, 1500.0, r), math.radians(sy.LAT_DEG))
    ha = np.linspace(-4.0, 4.0, case["n_t"]) * (math.pi / 12.0) * r.uniform(0.9, 1.0)
    dec = math.radians(sy.DEC_DEG + r.uniform(-5.0, 5.0))
    uvw = sy.earth_rotation_uvw(bxyz, ha, dec)
    # the longest baseline stays inside the grid with its footprint
    dl = math.radians(case["deg"]) / case["N"]
    half = (case["N"] / 2 - max(_supports(case))) / (case["N"] * dl)
    freq = np.linspace(1.2e9, 1.5e9, case["nchan"])
    reach = np.abs(uvw[:, :2]).max() * freq[-1] / sy.C_LIGHT
    if reach > 0.98 * half:
        uvw = uvw * (0.98 * half / reach)
    nrow = uvw.shape[0]
    g = _gen(seed, "rows")
    # channels of uneven counts: channel c holds a window of one random row order
    share = np.array([1.0 + 0.6 * math.sin(1.7 * c) for c in range(case["nchan"])])
    cum = np.round(np.cumsum(share) / share.sum() * case["nvis"]).astype(np.int64)
    cnt = np.diff(np.concatenate([[0], cum]))
    over = np.maximum(cnt - nrow, 0).sum()
    cnt = np.minimum(cnt, nrow)
    for c in range(case["nchan"]):
        add = min(over, nrow - cnt[c])
        cnt[c] += add
        over -= add
    perm = torch.randperm(nrow, generator=g, device=DEV)
    rows = []
    for c, n in enumerate(cnt):
        w = (torch.arange(int(n), device=DEV) + (c * 104729) % nrow) % nrow
        rows.append(torch.sort(perm[w])[0])
    row = torch.cat(rows).to(torch.int32)
    chan = torch.repeat_interleave(torch.arange(case["nchan"], device=DEV),
                                   torch.as_tensor(cnt, device=DEV)).to(torch.int16)
    pa = np.repeat(sy.parallactic_angle(ha, math.radians(sy.LAT_DEG), dec), bxyz.shape[0])
    lo, hi = pa.min(), pa.max()
    pa_bin = np.clip((pa - lo) / max(hi - lo, 1e-9) * case["npa"], 0, case["npa"] - 1).astype(np.uint8)
    fb = (np.arange(case["nchan"]) * case["nfb"] // case["nchan"]).astype(np.uint8)
    flags = None
    if case["flags"]:
        flags = (torch.rand(row.numel(), generator=g, device=DEV) < 0.02).to(torch.uint8)
    o = dict(uvw=torch.as_tensor(uvw, device=DEV), row=row, chan=chan, freq=torch.as_tensor(freq, device=DEV),
             pa_bin=torch.as_tensor(pa_bin, device=DEV), fbin=torch.as_tensor(fb, device=DEV), flags=flags)
    w_max = float(np.abs(uvw[:, 2]).max() * freq[-1] / sy.C_LIGHT) * (1.0 + 1e-9)
    spec = dict(N=case["N"], dl=dl, OS=case["os"], W=7.0, npol=case["npol"], nw=case["nw"],
                w_max=w_max if case["nw"] > 1 else 0.0, supports=_supports(case),
                pa=list(lo + (np.arange(case["npa"]) + 0.5) * (hi - lo) / case["npa"]),
                fbin_freqs=[float(freq[fb == b].mean()) for b in range(case["nfb"])],
                storage=STORAGE[case["storage"]])
    return o, spec


def _table(case, seed, b, degrid):
    """Bin b's kernel, complex64 [os^2][S^2][npol][npol] (out, in)."""
    nbf = case["npa"] * case["nfb"]
    p = b // nbf
    S, OS, npol = _supports(case)[p], case["os"], case["npol"]
    r = np.random.default_rng([seed, b, 17 + degrid])
    rho = (S - 2) * OS // 2
    t = ((torch.arange(S, device=DEV) * OS - rho)[None, :] - torch.arange(OS, device=DEV)[:, None]) / OS
    x = t / (0.5 * S + 1.0)                                            # (-1, 1) over the support
    k = torch.polar(torch.exp(-4.0 * x * x), (1 - 2 * degrid) * (0.3 + 0.35 * p) * math.pi * x * x)
    k = (k / k.abs().sum(1).mean()).to(torch.complex64)                # [os][S]
    K = (k[:, None, :, None] * k[None, :, None, :]).reshape(OS * OS, S * S, 1, 1)
    if npol == 1:
        return K
    T = np.array([[1, 0, 0, 1], [1, 0, 0, -1], [0, 1, 1, 0], [0, -1j, 1j, 0]]) / 2.0
    M = np.linalg.inv(T) if degrid else T
    leak = lambda s: (s * (r.standard_normal((2, 4, 4)) * [[[1]], [[1j]]]).sum(0))
    m0, mx, my = (torch.as_tensor(m, dtype=torch.complex64, device=DEV)
                  for m in (M + leak(0.03), leak(0.2), leak(0.2)))
    xx = x.to(torch.float32)
    fy = xx[:, None, :, None].expand(OS, OS, S, S).reshape(OS * OS, S * S, 1, 1)
    fx = xx[None, :, None, :].expand(OS, OS, S, S).reshape(OS * OS, S * S, 1, 1)
    return K * (m0 + fx * mx + fy * my)


def _kernels(ctx, case, seed, spec, degrid):
    nb = case["nw"] * case["npa"] * case["nfb"]
    tab = torch.cat([_table(case, seed, b, degrid).reshape(-1) for b in range(nb)])
    role = aw.AW_ROLE_DEGRID if degrid else aw.AW_ROLE_GRID
    return aw.aw_kernel_set_import(ctx, tab, role=role, **spec)


def _tune(case):
    if case["tune"] == "default":
        return None
    sup = _supports(case)
    if case["tune"] == "region":       # planes of supports up to 40 cells, as autotuning chooses
        split = sum(1 for s in sup if s <= 40)
    else:
        split = max(case["nw"] // 4, 1)
    mode = case["tune"] if not (case["tune"] == "hybrid" and case["nw"] == 1) else "tiles"
    return aw.aw_tune(32, 256, 2, 1024, MODES[mode], min(split, case["nw"]))


def _visibilities(case, seed, n):
    g = _gen(seed, "vis")
    vis = _randc(g, n, case["npol"])
    w = torch.rand(n, case["npol"], generator=g, device=DEV) + 0.5 if case["weights"] else None
    return vis, w


def _sources(case, seed, tag):
    """Stokes planes of a few hundred point sources in the inner half of the image."""
    r, N = _rng(case, seed, tag), case["N"]
    img = np.zeros((case["npol"], N, N), np.float32)
    n = 300
    y, x = r.integers(N // 4, 3 * N // 4, n), r.integers(N // 4, 3 * N // 4, n)
    img[:, y, x] = (r.uniform(0.1, 1.0, n) * np.array([1, 0.1, -0.05, 0.01])[:case["npol"], None]).astype(np.float32)
    return torch.as_tensor(img, device=DEV)


def _beams(case, g):
    """Gaussian primary beams of the mosaic's fields and their phase centres."""
    dl, Nm = math.radians(case["deg"]) / case["N"], case["Nm"]
    cen = [(math.radians(e / math.cos(math.radians(sy.DEC_DEG))) * case["deg"] / 3.0,
            math.radians(sy.DEC_DEG + no * case["deg"] / 3.0)) for e, no in sy.mosaic_offsets()[:case["fields"]]]
    q = (torch.arange(Nm, device=DEV) - Nm // 2) * dl
    beams = torch.empty(len(cen), Nm, Nm, device=DEV)
    for f, (ra, de) in enumerate(cen):
        r2 = (q[None, :] - ra * math.cos(de)) ** 2 + (q[:, None] - (de - math.radians(sy.DEC_DEG))) ** 2
        beams[f] = torch.exp(-r2 / (2 * math.radians(0.5) ** 2))
    return dl, cen, beams


def _network(case, seed):
    """SIREN parameters [5, 128 x 4, 32] (the usual initialisation) and the feature scales."""
    r = np.random.default_rng([seed, 99])
    sizes, out = [5, 128, 128, 128, 128, 2 * case["npol"] ** 2], []
    for i in range(5):
        lim = 1.0 / 5 if i == 0 else math.sqrt(6.0 / sizes[i]) / 30.0
        out.append((r.uniform(-lim, lim, (sizes[i + 1], sizes[i])).astype(np.float32),
                    r.uniform(-lim, lim, sizes[i + 1]).astype(np.float32)))
    return out


def prepare(case, seed):
    s = dict(case=case, ctx=aw.aw_create(0))
    ctx, N, kind = s["ctx"], case["N"], case["kind"]
    if kind == "image":
        s["ks"] = aw.aw_make_kernels(ctx, N=N, dl=math.radians(case["deg"]) / N, OS=2, npol=1 if case["npol"] == 1 else 4,
                                     supports=[8])
        if case["to_grid"]:
            s["model"] = _sources(case, seed, "model")
        else:
            s["uv"] = _randc(_gen(seed, "uv"), case["npol"], N, N)
        s["grid"] = torch.empty(case["npol"], N, N, dtype=torch.complex64, device=DEV)
        s["image"] = torch.empty(case["npol"], N, N, device=DEV)
    elif kind == "hogbom":
        q = torch.arange(N, device=DEV) - N // 2
        r = torch.sqrt((q[:, None] ** 2 + q[None, :] ** 2).float())
        s["psf"] = (torch.cos(0.55 * r) * torch.exp(-0.05 * r) + 0.02 * torch.cos(0.11 * r)) / 1.02
        sky = torch.fft.rfft2(_sources(case, seed, "sky"))
        dirty = torch.fft.irfft2(sky * torch.fft.rfft2(torch.fft.ifftshift(s["psf"])), s=(N, N))
        s["dirty"] = dirty + 0.01 * torch.randn(case["npol"], N, N, generator=_gen(seed, "noise"), device=DEV)
        s["residual"], s["model"] = torch.empty_like(dirty), torch.empty_like(dirty)
    elif kind == "mosaic":
        g = _gen(seed, "fields")
        dl, cen, s["beams"] = _beams(case, g)
        Nm, nf, npol = case["Nm"], case["fields"], case["npol"]
        s["images"] = torch.randn(nf, npol, N, N, generator=g, device=DEV)
        s["frames"] = [aw.sky_frame(ra, de, dl, N) for ra, de in cen]
        s["mframe"] = aw.sky_frame(0.0, math.radians(sy.DEC_DEG), dl, Nm)
        s["on"] = torch.empty(nf, npol, Nm, Nm, device=DEV)
        s["gamma"] = torch.empty(Nm, Nm, device=DEV)
        s["out"] = torch.empty(npol, Nm, Nm, device=DEV)
    else:
        o, spec = _geometry(case, seed)
        n = o["row"].numel()
        vd = aw.vis_desc(o["uvw"], o["row"], o["chan"], o["freq"], o["pa_bin"], o["fbin"], o["flags"])
        tune = _tune(case)
        s.update(obs=o, vd=vd, tune=tune)
        if kind in ("degrid", "residual"):
            s["kd"] = _kernels(ctx, case, seed, spec, 1)
        elif kind == "learned":
            s["kg"] = _kernels(ctx, case, seed, spec, int(case["degrid"]))
        else:
            s["kg"] = _kernels(ctx, case, seed, spec, 0)
        if kind == "cycle":
            s["kd"] = _kernels(ctx, case, seed, spec, 1)
        if kind == "plan":
            i32 = lambda: torch.empty(n, dtype=torch.int32, device=DEV)
            s["coords"] = [i32() for _ in range(5)] + [torch.empty(n, dtype=torch.uint8, device=DEV) for _ in range(2)]
            s["order"] = i32()
            return s
        s["plan"] = aw.aw_plan_create(ctx, vd, s.get("kg") or s["kd"], tune)
        if kind in ("grid", "residual", "cycle") or (kind == "learned" and not case["degrid"]):
            s["vis"], s["weight"] = _visibilities(case, seed, n)
        if kind in ("degrid", "residual") or (kind == "learned" and case["degrid"]):
            s["model"] = _randc(_gen(seed, "model"), case["npol"], N, N)
        if kind == "cycle":
            s["model"] = _sources(case, seed, "model")
            s["mgrid"] = torch.empty(case["npol"], N, N, dtype=torch.complex64, device=DEV)
            s["image"] = torch.empty(case["npol"], N, N, device=DEV)
            s["wsum"] = float(n if s["weight"] is None else s["weight"].mean(1).double().sum())
        if kind in ("grid", "cycle") or (kind == "learned" and not case["degrid"]):
            s["grid"] = torch.empty(case["npol"], N, N, dtype=torch.complex64, device=DEV)
        if kind in ("degrid", "residual", "cycle") or (kind == "learned" and case["degrid"]):
            s["out"] = torch.empty(n, case["npol"], dtype=torch.complex64, device=DEV)
        if kind == "learned":
            s["sur"] = aw.aw_surrogate_create(ctx, npol=case["npol"], norm_supports=_supports(case),
                                              w_max=spec["w_max"], f_c=1.35e9, f_h=0.15e9, chi_c=0.0, chi_h=1.5,
                                              out_scale=0.02)
            aw.aw_surrogate_set_params(s["sur"], np.concatenate([np.concatenate([w.ravel(), b])
                                                                 for w, b in _network(case, seed)]))
    return s


# ---------------------------------------------------------------- one pass
def run(s):
    c, ctx, kind = s["case"], s["ctx"], s["case"]["kind"]
    if kind == "grid":
        s["grid"].zero_()
        aw.aw_grid_batched(ctx, s["plan"], s["kg"], s["vis"], s["weight"], s["grid"])
        return s["grid"]
    if kind == "degrid":
        aw.aw_degrid(ctx, s["plan"], s["kd"], s["model"], s["out"])
        return s["out"]
    if kind == "residual":
        aw.aw_degrid_subtract(ctx, s["plan"], s["kd"], s["model"], s["vis"], s["out"])
        return s["out"]
    if kind == "cycle":
        aw.aw_image_to_grid(ctx, s["kd"], s["model"], s["mgrid"])
        aw.aw_degrid_subtract(ctx, s["plan"], s["kd"], s["mgrid"], s["vis"], s["out"])
        s["grid"].zero_()
        aw.aw_grid_batched(ctx, s["plan"], s["kg"], s["out"], s["weight"], s["grid"])
        aw.aw_fft_to_image(ctx, s["kg"], s["grid"], s["wsum"], s["image"])
        return {"model_grid": s["mgrid"], "residual": s["out"], "image": s["image"]}
    if kind == "image":
        if c["to_grid"]:
            aw.aw_image_to_grid(ctx, s["ks"], s["model"], s["grid"])
            return s["grid"]
        s["grid"].copy_(s["uv"])
        aw.aw_fft_to_image(ctx, s["ks"], s["grid"], 1000.0, s["image"])
        return s["image"]
    if kind == "plan":
        plan = aw.aw_plan_create(ctx, s["vd"], s["kg"], s["tune"])
        aw.aw_plan_coords(plan, *s["coords"])
        aw.aw_plan_order(plan, s["order"])
        aw.aw_plan_destroy(plan)
        return {"coords": list(s["coords"]), "order": s["order"]}
    if kind == "hogbom":
        N = c["N"]
        s["residual"].copy_(s["dirty"])
        s["model"].zero_()
        it = aw.aw_hogbom(ctx, s["residual"], s["psf"], 0.1, 0.0, c["iters"], c["patch"],
                          (N // 4, N // 4, 3 * N // 4, 3 * N // 4), s["model"])
        return {"residual": s["residual"], "model": s["model"], "iterations": it}
    if kind == "mosaic":
        interp = aw.AW_INTERP_CUBIC if c["interp"] == "cubic" else aw.AW_INTERP_BILINEAR
        for f, fr in enumerate(s["frames"]):
            aw.aw_reproject(ctx, s["images"][f], fr, s["on"][f], s["mframe"], interp)
        aw.mosaic_gamma(ctx, s["beams"], 0.1, s["gamma"])
        aw.aw_mosaic_combine(ctx, s["on"], s["beams"], s["gamma"], s["out"])
        return {"fields": s["on"], "gamma": s["gamma"], "mosaic": s["out"]}
    if c["degrid"]:
        aw.aw_degrid_learned(ctx, s["plan"], s["sur"], s["kg"], s["model"], s["out"])
        return s["out"]
    s["grid"].zero_()
    aw.aw_grid_learned(ctx, s["plan"], s["sur"], s["kg"], s["vis"], s["weight"], s["grid"])
    return s["grid"]


# ---------------------------------------------------------------- what a pass cannot do without
# share of the visibilities in a w plane falls off with |w| as in the array's track
def _mean_taps(case):
    sup = np.array(_supports(case), float)
    if case["nw"] == 1:
        return float(sup[0] ** 2)
    x = (np.arange(case["nw"]) + 0.5) / case["nw"]
    p = np.exp(-x / 0.19)
    return float((p * sup ** 2).sum() / p.sum())


def work(case):
    N, kind = case["N"], case["kind"]
    if kind == "image":
        fft = 5.0 * case["npol"] * N * N * 2 * math.log2(N)
        return {"bytes": case["npol"] * N * N * (12 if case["to_grid"] else 28), "flops": fft}
    if kind == "hogbom":
        it = case["iters"]
        patch = (2 * case["patch"] + 1) ** 2
        return {"bytes": 16 * case["npol"] * N * N + it * patch * (4 + 8 * case["npol"]),
                "flops": 2.0 * it * patch * case["npol"]}
    if kind == "mosaic":
        out, taps = case["Nm"] ** 2, 16 if case["interp"] == "cubic" else 4
        nf, npol = case["fields"], case["npol"]
        return {"bytes": 4 * (nf * npol * N * N + nf * npol * out + nf * out + out + npol * out),
                "flops": nf * npol * min(out, N * N) * 2.0 * taps + 2.0 * nf * (npol + 1) * out}
    nv, npol = case["nvis"], case["npol"]
    rec = 16     # sorted coordinates of a visibility
    if kind == "plan":   # rows, channels and uvw in; coordinates, flip, valid and order out
        return {"bytes": nv * (4 + 2 + 22 + 4) + 24 * 630 * case["n_t"], "flops": 20.0 * nv}
    taps = nv * _mean_taps(case)
    tab = case["nw"] * case["npa"] * case["nfb"] * case["os"] ** 2 * npol ** 2 * (8 if case["storage"] == "fp32" else 4)
    tab *= sum(x * x for x in _supports(case)) / case["nw"]
    flops, grid, vis = 8.0 * npol ** 2 * taps, 8 * npol * N * N, nv * (8 * npol + rec)
    if kind == "learned":
        per = 2.0 * (5 * 128 + 3 * 128 * 128 + 128 * 2 * npol ** 2)
        return {"bytes": vis + grid, "flops": taps * per + flops}
    if kind == "residual":
        vis += nv * 8 * npol
    if kind == "grid" and case["weights"]:
        vis += nv * 4 * npol
    if kind == "cycle":
        return {"bytes": 2 * (vis + tab + grid) + nv * 8 * npol + 8 * npol * N * N,
                "flops": 2 * flops + 20.0 * npol * N * N * math.log2(N)}
    return {"bytes": vis + tab + grid, "flops": flops}


# ---------------------------------------------------------------- the same in 64 bits
def _coords(case, o, spec):
    f = (o["freq"] / 299792458.0)[o["chan"].long()]
    r = o["row"].long()
    u, v, w = (o["uvw"][r, i] * f for i in range(3))
    flip = w < 0
    u, v, w = (torch.where(flip, -t, t) for t in (u, v, w))
    N, OS = case["N"], case["os"]
    uscale, half = float(N) * spec["dl"] * float(OS), float(N // 2 * OS)
    X, Y = ((torch.floor(t * uscale + half + 0.5)).long() for t in (u, v))
    p = torch.zeros_like(r)
    if spec["nw"] > 1:
        p = torch.floor(w * (float(spec["nw"]) / spec["w_max"])).long().clamp(0, spec["nw"] - 1)
    sup = torch.tensor(spec["supports"], device=DEV)
    S = sup[p]
    rho = (S - 2) * OS // 2
    ax, ay = X - rho, Y - rho
    x0, y0 = torch.div(ax, OS, rounding_mode="floor"), torch.div(ay, OS, rounding_mode="floor")
    ok = (x0 >= 0) & (y0 >= 0) & (x0 + S <= N) & (y0 + S <= N)
    if o["flags"] is not None:
        ok &= o["flags"] == 0
    b = (p * case["npa"] + o["pa_bin"][r].long()) * case["nfb"] + o["fbin"][o["chan"].long()].long()
    return dict(x0=x0, y0=y0, off=(ay - y0 * OS) * OS + ax - x0 * OS, bin=b, S=S, ok=ok, flip=flip,
                u=u, v=v, w=w)


def _unflip(v, flip):
    """P conj(V) where flipped ([n][npol] complex)."""
    f = v.conj()
    if v.shape[1] == 4:
        f = f[:, [0, 2, 1, 3]]
    return torch.where(flip[:, None], f, v)


def _rounded(case, seed, b, degrid, scale):
    t = _table(case, seed, b, degrid)
    if case["storage"] == "fp32":
        return t.to(torch.complex128)
    dt = torch.bfloat16 if case["storage"] == "bf16" else torch.float16
    r = (torch.view_as_real(t) * scale).to(dt).double() / scale
    return torch.view_as_complex(r.contiguous())


def _runs(case, seed, co, degrid):
    """(visibilities of one kernel block, their footprint cells [n][S^2], the block
    [S^2][out][in]) for every block in use."""
    scale = 1.0
    if case["storage"] == "fp16":
        nb = case["nw"] * case["npa"] * case["nfb"]
        mx = max(float(torch.view_as_real(_table(case, seed, b, degrid)).abs().max()) for b in range(nb))
        scale = 2.0 ** math.floor(-math.log2(mx))
    nblk = case["os"] ** 2
    idx = torch.nonzero(co["ok"]).flatten()
    key = co["bin"][idx] * nblk + co["off"][idx]
    key, perm = torch.sort(key)
    idx = idx[perm]
    uniq, cnt = torch.unique_consecutive(key, return_counts=True)
    pos, last, tab = 0, -1, None
    for k, n in zip(uniq.tolist(), cnt.tolist()):
        b = k // nblk
        if b != last:
            tab, last = _rounded(case, seed, b, degrid, scale), b
        S = _supports(case)[b // (case["npa"] * case["nfb"])]
        j = torch.arange(S * S, device=DEV)
        toff = (j // S) * case["N"] + j % S
        step = max(1, (1 << 23) // (S * S))
        for a in range(pos, pos + n, step):
            i = idx[a:min(a + step, pos + n)]
            yield i, (co["y0"][i] * case["N"] + co["x0"][i])[:, None] + toff, tab[k % nblk]
        pos += n


def _grid64(case, seed, co, vis, weight):
    npol, N = case["npol"], case["N"]
    v = _unflip(vis.to(torch.complex128) * (1.0 if weight is None else weight.double()), co["flip"])
    G = torch.zeros(N * N, 2 * npol, dtype=torch.float64, device=DEV)
    for i, cells, K in _runs(case, seed, co, 0):
        add = v[i] @ K.permute(2, 0, 1).reshape(npol, -1)               # [n][S^2 npol]
        G.index_add_(0, cells.flatten(), torch.view_as_real(add.reshape(-1, npol)).reshape(-1, 2 * npol))
    return torch.view_as_complex(G.reshape(N * N, npol, 2)).t().reshape(npol, N, N)


def _degrid64(case, seed, co, model):
    npol = case["npol"]
    m = model.to(torch.complex128).reshape(npol, -1).t().contiguous()
    out = torch.zeros(co["ok"].numel(), npol, dtype=torch.complex128, device=DEV)
    for i, cells, K in _runs(case, seed, co, 1):
        out[i] = m[cells].reshape(i.numel(), -1) @ K.permute(0, 2, 1).reshape(-1, npol)
    return _unflip(out, co["flip"])


def _taper(N):
    """psi0(2 l / F) at the image pixels, psi0(0) = 1, bandwidth 7 pi / 2: the top
    eigenfunction of the kernel cos(c x t) on Gauss-Legendre nodes, carried to the pixels."""
    c = math.pi * 7.0 / 2.0
    t, w = np.polynomial.legendre.leggauss(96)
    lam, vec = np.linalg.eigh(np.sqrt(w)[:, None] * np.cos(c * np.outer(t, t)) * np.sqrt(w)[None, :])
    f = vec[:, np.argmax(np.abs(lam))] * np.sqrt(w)
    x = (np.arange(N) - N // 2) * 2.0 / N
    psi = np.cos(c * np.outer(np.concatenate([[0.0], x]), t)) @ f
    return torch.as_tensor(psi[1:] / psi[0], device=DEV)


def _image64(grid, wsum):
    N = grid.shape[-1]
    z = torch.fft.fftshift(torch.fft.ifft2(torch.fft.ifftshift(grid.to(torch.complex128), dim=(-2, -1))),
                           dim=(-2, -1)).real * float(N) * N
    t = _taper(N)
    img = z / (t[:, None] * t[None, :]) / wsum
    img[:, 0, :] = 0.0
    img[:, :, 0] = 0.0
    return img


def _grid_of64(image):
    N = image.shape[-1]
    t = _taper(N)
    a = image.double() / (t[:, None] * t[None, :])
    a[:, 0, :] = 0.0
    a[:, :, 0] = 0.0
    return torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(a, dim=(-2, -1))), dim=(-2, -1))


def _axes(ra, dec):
    return torch.tensor([[-math.sin(ra), math.cos(ra), 0.0],
                         [-math.sin(dec) * math.cos(ra), -math.sin(dec) * math.sin(ra), math.cos(dec)],
                         [math.cos(dec) * math.cos(ra), math.cos(dec) * math.sin(ra), math.sin(dec)]],
                        dtype=torch.float64)


def _mosaic64(case, seed):
    g = _gen(seed, "fields")
    dl, cen, beams = _beams(case, g)
    N, Nm, nf, npol = case["N"], case["Nm"], case["fields"], case["npol"]
    images = torch.randn(nf, npol, N, N, generator=g, device=DEV).double()
    q = (torch.arange(Nm, device=DEV, dtype=torch.float64) - Nm // 2) * dl
    l, m = q[None, :].expand(Nm, Nm), q[:, None].expand(Nm, Nm)
    n = torch.sqrt((1.0 - l * l - m * m).clamp(min=0.0))
    on = torch.zeros(nf, npol, Nm, Nm, dtype=torch.float64, device=DEV)
    taps = [-1, 0, 1, 2] if case["interp"] == "cubic" else [0, 1]

    def weight(d):
        d = d.abs()
        if case["interp"] != "cubic":
            return 1.0 - d
        return torch.where(d <= 1, 1.5 * d ** 3 - 2.5 * d ** 2 + 1, -0.5 * d ** 3 + 2.5 * d ** 2 - 4 * d + 2)
    for f, (ra, de) in enumerate(cen):
        R = _axes(ra, de) @ _axes(0.0, math.radians(sy.DEC_DEG)).t()
        ls, ms, ns = (R[i, 0].item() * l + R[i, 1].item() * m + R[i, 2].item() * n for i in range(3))
        x, y = ls / dl + N // 2, ms / dl + N // 2
        x0, y0 = torch.floor(x), torch.floor(y)
        ok = (ns > 0) & (x0 + taps[0] >= 0) & (x0 + taps[-1] < N) & (y0 + taps[0] >= 0) & (y0 + taps[-1] < N)
        for ty in taps:
            for tx in taps:
                at = ((y0 + ty).clamp(0, N - 1) * N + (x0 + tx).clamp(0, N - 1)).long()
                wt = torch.where(ok, weight(y - y0 - ty) * weight(x - x0 - tx), 0.0)
                on[f] += wt * images[f].reshape(npol, -1)[:, at.flatten()].reshape(npol, Nm, Nm)
    b = beams.double()
    s2 = (b * b).sum(0)
    pbp = torch.sqrt(s2) / torch.sqrt(s2).max()
    gamma = torch.where((pbp >= 0.1) & (s2 > 0), pbp / s2, 0.0)
    return {"fields": on, "gamma": gamma, "mosaic": gamma * (b[:, None] * on).sum(0)}


def _learned64(case, seed, o, spec):
    co = _coords(case, o, spec)
    N, npol = case["N"], case["npol"]
    net = []
    for i, (w, b) in enumerate(_network(case, seed)):
        w = w if i == 0 else w.astype(np.float16)
        net.append((torch.as_tensor(w.astype(np.float64), device=DEV), torch.as_tensor(b.astype(np.float64), device=DEV)))
    sup = torch.tensor(spec["supports"], device=DEV)
    pn = torch.floor(co["w"] * len(spec["supports"]) / spec["w_max"]).long().clamp(0, len(spec["supports"]) - 1)
    scale = (sup[pn] // 2 + 1).double()
    cx, cy = (t * (N * spec["dl"]) + N // 2 for t in (co["u"], co["v"]))
    nbf = case["nfb"]
    fr = torch.tensor(spec["fbin_freqs"], device=DEV, dtype=torch.float64)[co["bin"] % nbf]
    pa = torch.tensor(spec["pa"], device=DEV, dtype=torch.float64)[co["bin"] // nbf % case["npa"]]
    fix = torch.stack([2 * co["w"] / spec["w_max"] - 1, (fr - 1.35e9) / 0.15e9, pa / 1.5], 1)
    if case["degrid"]:
        m = _randc(_gen(seed, "model"), npol, N, N).to(torch.complex128).reshape(npol, -1).t().contiguous()
        out = torch.zeros(co["ok"].numel(), npol, dtype=torch.complex128, device=DEV)
    else:
        vis, wt = _visibilities(case, seed, co["ok"].numel())
        v = _unflip(vis.to(torch.complex128) * (1.0 if wt is None else wt.double()), co["flip"])
        G = torch.zeros(N * N, 2 * npol, dtype=torch.float64, device=DEV)
    for S in sorted(set(spec["supports"])):
        idx = torch.nonzero(co["ok"] & (co["S"] == S)).flatten()
        j = torch.arange(S * S, device=DEV)
        jy, jx = j // S, j % S
        step = max(1, (1 << 20) // (S * S))
        for a in range(0, idx.numel(), step):
            i = idx[a:a + step]
            n = i.numel()
            du = (co["x0"][i, None] + jx - cx[i, None]) / scale[i, None]
            dv = (co["y0"][i, None] + jy - cy[i, None]) / scale[i, None]
            h = torch.cat([du.reshape(-1, 1), dv.reshape(-1, 1),
                           fix[i].repeat_interleave(S * S, 0)], 1)
            for k, (w, b) in enumerate(net):
                h = h @ w.t() + b
                if k < 4:
                    h = torch.sin(30.0 * h)
            K = torch.view_as_complex(h.reshape(n * S * S, npol, npol, 2)) * 0.02
            cells = ((co["y0"][i] * N + co["x0"][i])[:, None] + jy * N + jx).flatten()
            if case["degrid"]:
                p = (K @ m[cells][:, :, None]).reshape(n, S * S, npol)
                out[i] = p.sum(1)
            else:
                p = (K @ v[i].repeat_interleave(S * S, 0)[:, :, None])[:, :, 0]
                G.index_add_(0, cells, torch.view_as_real(p).reshape(-1, 2 * npol))
    if case["degrid"]:
        return _unflip(out, co["flip"])
    return torch.view_as_complex(G.reshape(N * N, npol, 2)).t().reshape(npol, N, N)


def exact(case, seed):
    kind, N = case["kind"], case["N"]
    if kind == "image":
        if case["to_grid"]:
            return _grid_of64(_sources(case, seed, "model"))
        return _image64(_randc(_gen(seed, "uv"), case["npol"], N, N), 1000.0)
    if kind == "mosaic":
        return _mosaic64(case, seed)
    if kind in ("plan", "hogbom"):   # whole numbers; a minor cycle's choices follow its 32-bit rounding
        return None
    if case["nvis"] * _mean_taps(case) > (EXACT_TAPS if kind != "learned" else 1.2e8):
        return None
    o, spec = _geometry(case, seed)
    if kind == "learned":
        return _learned64(case, seed, o, spec)
    co = _coords(case, o, spec)
    n = co["ok"].numel()
    if kind == "grid":
        return _grid64(case, seed, co, *_visibilities(case, seed, n))
    if kind == "degrid":
        return _degrid64(case, seed, co, _randc(_gen(seed, "model"), case["npol"], N, N))
    vis, weight = _visibilities(case, seed, n)
    if kind == "residual":
        return vis.to(torch.complex128) - _degrid64(case, seed, co, _randc(_gen(seed, "model"), case["npol"], N, N))
    mg = _grid_of64(_sources(case, seed, "model"))
    res = vis.to(torch.complex128) - _degrid64(case, seed, co, mg)
    img = _image64(_grid64(case, seed, co, res, weight),
                   float(n if weight is None else weight.mean(1).double().sum()))
    return {"model_grid": mg, "residual": res, "image": img}
