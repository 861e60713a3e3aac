"""Timed cases of the framework: what its users have it do, through its public entry points.

Every case names a `kind` of work and its sizes; `prepare` makes inputs on the GPU from a seed,
`run` makes one pass, `work` counts the bytes and flops a pass cannot do without, and `exact`
recomputes the outputs in float64 with plain torch from the method's definitions (Merry,
"Approximating W projection as a separable kernel", MNRAS 2015; the conventions of include/sepw.h).

Kinds:
  step        a gridding + prediction round on new coordinates: plan, grid, degrid a model grid
  batched     many grids (W-stacking layers x channels) planned and gridded in one call
  wstack      hybrid W stacking, both directions: plan, slice grids, image, model grids, prediction
  gradient    forward and backward of the weighted chi^2 of a model image, plan kept (autograd)
  correction  gridding and prediction with the stored correction F_w - F~_w, plan kept
  facet       one facet: shift in, plan, grid, image; predict the facet's model and shift out
  noalloc     one block of a real-time pipeline through the allocation-free gridder
  tables      set-up of a new geometry: the tap table and the stored-correction table
"""
import math

import numpy as np
import torch

import paper_1511_07152_gb300.sepw as sepw
from paper_1511_07152_gb300 import autograd

FORMS = {"tiled": sepw.FORM_TILED, "bf16": sepw.FORM_TC_BF16, "fp16": sepw.FORM_TC_FP16,
         "fp16x2": sepw.FORM_TC_FP16X2, "bf16x2": sepw.FORM_TC_BF16X2, "tf32": sepw.FORM_TC_TF32}
DEV = "cuda"
C128 = torch.complex128
C_LIGHT = 299792458.0
OMEGA_EARTH = 7.2921159e-5  # rad/s
FACET = (0.012, -0.007)     # facet centre, direction cosines


def _case(name, kind, n, N, S, OS, P, layout="tracks", form="tiled", weighted=True, **more):
    return {"name": name, "kind": kind, "n": n, "N": N, "S": S, "OS": OS, "P": P,
            "layout": layout, "form": form, "weighted": weighted, **more}


def listed():
    return [
        # a quick-look image of one short snapshot: the smallest call, bound by its launches
        _case("snapshot", "step", 20_000, 256, 8, 8, 32, layout="disk"),
        # the headline workload: a 64-antenna observation (2016 baselines x 1000 dumps x 16
        # channels) on a 4096^2 grid at support 16, default form
        _case("observation", "step", 32_256_000, 4096, 16, 16, 128),
        # a quarter of that observation in the hi + lo tensor-core form of FP32-class accuracy
        _case("observation_hi_lo", "step", 8_064_000, 4096, 16, 16, 128, form="bf16x2"),
        # the same in the one-part BF16 form: quick imaging at 16-bit accuracy
        _case("observation_bf16", "step", 8_064_000, 4096, 16, 16, 128, form="bf16"),
        # an odd-sized job away from the tuned sizes: support 10, oversampling that is no power
        # of two, a grid no tile divides, unit weights, some visibilities off the grid
        _case("ragged", "step", 333_337, 1000, 10, 7, 33, layout="disk", weighted=False),
        # 16 layers x 8 channels of 2048^2, counts spread over two decades (sparse tiles)
        _case("layers", "batched", 63_000_000, 2048, 12, 16, 32, layout="disk", grids=128),
        # a hybrid W-stacking cycle, 15 slices dense near w = 0
        _case("wstack", "wstack", 8_064_000, 4096, 8, 16, 32, slices=15),
        # model fitting: value and gradient of chi^2 for 2016 baselines x 1984 dumps
        _case("gradient", "gradient", 3_999_744, 2048, 8, 16, 64),
        # a major cycle with the stored correction on the separable kernel
        _case("correction", "correction", 3_999_744, 2048, 16, 16, 64, Sr=8, OSr=8),
        # one facet of a wide field
        _case("facet", "facet", 1_000_003, 1024, 8, 8, 32),
        # a real-time block of the largest size the fixed scratch takes
        _case("realtime", "noalloc", 524_288, 2048, 16, 16, 128),
        # tables of a new geometry, made once per observation
        _case("tables", "tables", 0, 1024, 12, 8, 32, Sr=8, OSr=8),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    kind = rng.choice(["step", "step", "step", "step", "batched", "wstack", "gradient",
                       "correction", "facet", "noalloc", "tables"])
    N = 2 * _log_int(rng, 100, 1200)
    OS = rng.choice([4, 7, 8, 8, 12, 16, 16])
    P = _log_int(rng, 8, 128)
    layout = rng.choice(["tracks", "tracks", "disk"])
    weighted = rng.random() < 0.75
    S = rng.choice([6, 8, 10, 12, 14, 16, 16])
    n = _log_int(rng, 3_000, 8_000_000)
    form, more = "tiled", {}
    if kind == "step":
        form = rng.choice(["tiled", "tiled", "tiled", "bf16", "fp16", "bf16x2", "fp16x2", "tf32"])
        if form == "tiled" and rng.random() < 0.15:
            S, n = rng.choice([4, 20, 24]), _log_int(rng, 3_000, 2_000_000)
    elif kind == "batched":
        layout = "disk"
        form = rng.choice(["tiled", "tiled", "bf16x2"])
        N = 2 * _log_int(rng, 100, 800)
        more = {"grids": rng.randint(2, 48)}
    elif kind == "wstack":
        layout, S, n = "tracks", rng.choice([6, 8]), _log_int(rng, 30_000, 4_000_000)
        form = rng.choice(["tiled", "tiled", "fp16x2"])
        more = {"slices": 2 * rng.randint(1, 8) + 1}
    elif kind == "gradient":
        layout, S = "tracks", rng.choice([6, 8])
    elif kind == "correction":
        S, OS, P = rng.choice([8, 12, 16]), 8, min(P, 48)
        N = 2 * _log_int(rng, 100, 512)
        n = _log_int(rng, 3_000, 2_000_000)
        more = {"Sr": S - rng.choice([0, 2, 4]), "OSr": rng.choice([4, 8])}
    elif kind == "facet":
        layout, S, OS = "tracks", rng.choice([6, 8]), rng.choice([8, 16])
    elif kind == "noalloc":
        n = _log_int(rng, 3_000, 524_288)
    elif kind == "tables":
        N, S, OS, P = 2 * _log_int(rng, 100, 400), rng.choice([6, 8, 12]), 8, min(P, 32)
        n, more = 0, {"Sr": S - rng.choice([0, 2, 4]), "OSr": rng.choice([2, 4, 8])}
    c = _case("", kind, n, N, S, OS, P, layout=layout, form=form, weighted=weighted, **more)
    del c["name"]
    return c


# ---- inputs -----------------------------------------------------------------


def _fov(c):
    return math.radians(1.0)


def _gen(seed):
    g = torch.Generator(device=DEV)
    g.manual_seed(seed)
    return g


def _tracks(c, g):
    """Earth-rotation tracks of 64 antennas uniform in a disk, [dump][baseline][channel]; the
    disk scales with the grid, so that the longest baseline fills a third of it (8 km at 4096
    cells); 8000 s at declination -30 deg seen from latitude -30.7 deg, 1.0-1.4 GHz."""
    n, nant = c["n"], 64
    nchan = 16 if n >= 16 * 2016 * 8 else 1
    nb = nant * (nant - 1) // 2
    ndumps = -(-n // (nb * nchan))
    f64 = dict(dtype=torch.float64, device=DEV)
    r = 4000.0 * c["N"] / 4096 * torch.sqrt(torch.rand(nant, generator=g, **f64))
    phi = 2.0 * math.pi * torch.rand(nant, generator=g, **f64)
    east, north = r * torch.cos(phi), r * torch.sin(phi)
    lat, dec = math.radians(-30.7), math.radians(-30.0)
    X, Y, Z = -math.sin(lat) * north, east, math.cos(lat) * north
    i, j = torch.triu_indices(nant, nant, 1, device=DEV)
    dX, dY, dZ = X[j] - X[i], Y[j] - Y[i], Z[j] - Z[i]
    H = OMEGA_EARTH * (8000.0 / ndumps) * (torch.arange(ndumps, **f64) - 0.5 * (ndumps - 1))
    sH, cH = torch.sin(H)[:, None], torch.cos(H)[:, None]
    um = sH * dX + cH * dY
    vm = -math.sin(dec) * cH * dX + math.sin(dec) * sH * dY + math.cos(dec) * dZ
    wm = math.cos(dec) * cH * dX - math.cos(dec) * sH * dY + math.sin(dec) * dZ
    lam = torch.linspace(1.0e9, 1.4e9, nchan, **f64) / C_LIGHT
    return [(x[:, :, None] * lam).reshape(-1)[:n].contiguous() for x in (um, vm, wm)]


def _disk(c, g, reach, w_top):
    """(u, v) uniform in a disk of `reach` cells, w uniform in [-w_top, w_top]."""
    n, du = c["n"], 1.0 / _fov(c)
    f64 = dict(dtype=torch.float64, device=DEV, generator=g)
    r = reach * du * torch.sqrt(torch.rand(n, **f64))
    phi = 2.0 * math.pi * torch.rand(n, **f64)
    w = w_top * (2.0 * torch.rand(n, **f64) - 1.0)
    return [r * torch.cos(phi), r * torch.sin(phi), w]


def _inputs(c, seed):
    """Everything a user has before the call, from the seed alone."""
    g = _gen(seed)
    n, N = c["n"], c["N"]
    d = {}
    if c["kind"] == "tables":
        # a geometry: the largest |w| of an observation to come
        d["w_max"] = 4000.0 + 500.0 * float(torch.rand(1, generator=g, device=DEV))
        return d
    if c["layout"] == "tracks":
        d["u"], d["v"], d["w"] = _tracks(c, g)
        d["w_max"] = float(d["w"].abs().max())
    elif c["kind"] == "batched":
        d["u"], d["v"], d["w"] = _disk(c, g, 0.45 * N, 1000.0)
        d["w_max"] = 1000.0
    else:
        # reaches past the last footprint, and a little past the last plane: a few are dropped
        d["u"], d["v"], d["w"] = _disk(c, g, N / 2 - c["S"] / 2 + 1.5, 2000.0)
        d["w_max"] = 1990.0
    if c["kind"] == "facet":
        # |w| stays; the facet's shift moves u, v by up to w l0
        d["u"] *= 0.8
        d["v"] *= 0.8
    d["vis"] = torch.randn(n, dtype=torch.complex64, device=DEV, generator=g)
    d["weight"] = (0.5 + 0.5 * torch.rand(n, dtype=torch.float32, device=DEV, generator=g)
                   if c["weighted"] else None)
    if c["kind"] in ("step", "correction", "facet"):
        # a model's grid (the degridder's input)
        d["model"] = torch.randn((N, N), dtype=torch.complex64, device=DEV, generator=g)
    if c["kind"] in ("gradient", "wstack"):
        # point sources and noise in the unpadded half of the field
        x = torch.zeros((N, N), dtype=torch.float32, device=DEV)
        q, h = N // 4, N // 2
        x[q:q + h, q:q + h] = 1e-4 * torch.randn((h, h), dtype=torch.float32, device=DEV,
                                                 generator=g)
        at = q + torch.randint(0, h, (2, 500), device=DEV, generator=g)
        flux = torch.exp(math.log(1e-3) * torch.rand(500, device=DEV, generator=g))
        x.index_put_((at[0], at[1]), flux, accumulate=True)
        d["image"] = x
    if c["kind"] == "batched":
        # counts per grid log-uniform over a factor of 200, in the total asked for
        rng = np.random.default_rng(seed)
        share = np.exp(rng.uniform(math.log(1e4), math.log(2e6), c["grids"]))
        cut = np.floor(np.cumsum(share) / share.sum() * n).astype(np.int64)
        d["offsets"] = np.concatenate([[0], cut[:-1], [n]]).astype(np.int64)
    if c["kind"] == "wstack":
        K = (c["slices"] - 1) // 2
        top = 0.93 * d["w_max"]
        pos = [top * (k / K) ** 1.5 for k in range(1, K + 1)]
        d["centres"] = [-x for x in reversed(pos)] + [0.0] + pos
        gaps = np.diff([0.0] + pos + [d["w_max"] + 0.07 * d["w_max"]])
        d["w_max"] = 0.51 * float(gaps.max())
    return d


def _params(c, d):
    return sepw.make_params(c["N"], _fov(c), c["S"], c["OS"], c["P"], d["w_max"],
                            form=FORMS[c["form"]])


def prepare(case, seed):
    c = case
    s = {"c": c, **_inputs(c, seed)}
    N, n = c["N"], c["n"]
    s["params"] = _params(c, s)
    ctx = s["ctx"] = sepw.sepw_create(s["params"])
    kind = c["kind"]
    c64 = dict(dtype=torch.complex64, device=DEV)
    if kind == "facet":
        sepw.sepw_set_facet(ctx, *FACET)
    if kind == "tables":
        s["taps"] = torch.empty((c["P"], c["OS"], c["S"]), **c64)
        s["table"] = torch.empty((c["P"], c["OSr"], c["OSr"], c["Sr"], c["Sr"]), **c64)
        return s
    s["taps"] = sepw.sepw_make_taps(ctx)
    s["dropped"] = torch.zeros(1, dtype=torch.int64, device=DEV)
    if kind == "gradient":
        sepw.sepw_plan(ctx, s["u"], s["v"], s["w"])
        return s
    if kind == "correction":
        s["table"] = sepw.sepw_make_residual(ctx, c["Sr"], c["OSr"])
        sepw.sepw_plan(ctx, s["u"], s["v"], s["w"])
    ng = {"batched": c.get("grids", 1), "wstack": c.get("slices", 1)}.get(kind, 1)
    s["grid"] = torch.empty((ng, N, N) if ng > 1 else (N, N), **c64)
    if kind != "batched" and kind != "noalloc":
        s["out"] = torch.empty(n, **c64)
    if kind == "wstack":
        s["dirty"] = torch.empty((N, N), **c64)
        s["image"] = s["image"].to(torch.complex64)
    if kind == "facet":
        s["fu"], s["fv"] = torch.empty_like(s["u"]), torch.empty_like(s["v"])
        s["fvis"] = torch.empty_like(s["vis"])
    return s


def run(state):
    s = state
    c, kind = s["c"], s["c"]["kind"]
    ctx = s["ctx"]
    if kind == "step":
        s["grid"].zero_()
        sepw.sepw_grid(ctx, s["taps"], s["u"], s["v"], s["w"], s["vis"], s["weight"], s["grid"],
                       n_dropped=s["dropped"])
        sepw.sepw_degrid_planned(ctx, s["taps"], s["model"], s["weight"], s["out"])
        return {"grid": s["grid"], "vis": s["out"], "dropped": s["dropped"]}
    if kind == "batched":
        s["grid"].zero_()
        sepw.sepw_grid_batched(ctx, s["taps"], s["offsets"], s["u"], s["v"], s["w"], s["vis"],
                               s["weight"], s["grid"], n_dropped=s["dropped"])
        return {"grid": s["grid"], "dropped": s["dropped"]}
    if kind == "wstack":
        sepw.sepw_wstack_plan(ctx, s["centres"], s["u"], s["v"], s["w"])
        s["grid"].zero_()
        sepw.sepw_grid_planned(ctx, s["taps"], s["vis"], s["weight"], s["grid"])
        sepw.sepw_wstack_image(ctx, s["grid"], s["dirty"])
        sepw.sepw_wstack_model_grids(ctx, s["image"], s["grid"])
        sepw.sepw_degrid_planned(ctx, s["taps"], s["grid"], None, s["out"])
        return {"dirty": s["dirty"], "vis": s["out"]}
    if kind == "gradient":
        x = s["image"].detach().requires_grad_(True)
        pred = autograd.predict(x, ctx, s["taps"])
        loss = autograd.chi2(pred, s["vis"], s["weight"])
        loss.backward()
        return {"vis": pred.detach(), "chi2": loss.detach(), "grad": x.grad}
    if kind == "correction":
        s["grid"].zero_()
        sepw.sepw_grid_planned(ctx, s["taps"], s["vis"], s["weight"], s["grid"])
        sepw.sepw_grid_residual_planned(ctx, s["table"], s["vis"], s["weight"], s["grid"])
        sepw.sepw_degrid_planned(ctx, s["taps"], s["model"], s["weight"], s["out"])
        sepw.sepw_degrid_residual_planned(ctx, s["table"], s["model"], s["weight"], s["out"])
        return {"grid": s["grid"], "vis": s["out"]}
    if kind == "facet":
        sepw.sepw_facet_shift(ctx, sepw.FACET_IN, s["u"], s["v"], s["w"], s["vis"], s["fu"],
                              s["fv"], s["fvis"])
        s["grid"].zero_()
        sepw.sepw_grid(ctx, s["taps"], s["fu"], s["fv"], s["w"], s["fvis"], s["weight"],
                       s["grid"], n_dropped=s["dropped"])
        sepw.sepw_image(ctx, sepw.GRID_TO_IMAGE, s["grid"])
        sepw.sepw_degrid_planned(ctx, s["taps"], s["model"], None, s["out"])
        sepw.sepw_facet_shift(ctx, sepw.FACET_OUT, s["u"], s["v"], s["w"], s["out"],
                              vis_out=s["out"])
        return {"dirty": s["grid"], "vis": s["out"], "dropped": s["dropped"]}
    if kind == "noalloc":
        s["grid"].zero_()
        status = sepw.sepw_grid_noalloc(s["params"], s["taps"], s["u"], s["v"], s["w"], s["vis"],
                                        s["weight"], s["grid"], n_dropped=s["dropped"])
        return {"grid": s["grid"], "dropped": s["dropped"], "status": status}
    sepw.sepw_make_taps(ctx, s["taps"])
    sepw.sepw_make_residual(ctx, c["Sr"], c["OSr"], s["table"])
    return {"taps": s["taps"], "table": s["table"]}


def work(case):
    """Each input read once, each output written once; 8 S^2 + 8 S flops per visibility and
    direction (S^2 complex multiply-adds and S partial products), 5 N^2 log2 N^2 per FFT."""
    c = case
    n, N, S, kind = c["n"], c["N"], c["S"], c["kind"]
    P, OS = c["P"], c["OS"]
    px = N * N
    taps = 8 * P * OS * S
    wt = 4 if c["weighted"] else 0
    each = 8.0 * S * S + 8.0 * S
    fft = 5.0 * px * 2 * math.log2(N)
    if kind == "step":
        return {"bytes": n * (24 + 8 + wt + 8) + 16 * px + taps, "flops": 2 * n * each}
    if kind == "batched":
        return {"bytes": n * (24 + 8 + wt) + 8 * px * c["grids"] + taps, "flops": n * each}
    if kind == "wstack":
        L = c["slices"]
        return {"bytes": n * (24 + 8 + wt + 8) + 16 * px + taps,
                "flops": 2 * n * each + 2 * L * fft}
    if kind == "gradient":
        return {"bytes": n * (24 + 8 + wt + 8) + 8 * px + taps, "flops": 2 * n * each + 2 * fft}
    if kind == "correction":
        cells = c["Sr"] ** 2
        return {"bytes": n * (24 + 8 + wt + 8) + 16 * px + taps + 8 * P * c["OSr"] ** 2 * cells,
                "flops": 2 * n * (each + 8 * cells)}
    if kind == "facet":
        return {"bytes": n * (24 + 8 + wt + 8) + 16 * px + 2 * taps, "flops": 2 * n * each + fft}
    if kind == "noalloc":
        return {"bytes": n * (24 + 8 + wt) + 8 * px + taps, "flops": n * each}
    rows = c["OSr"] * c["Sr"]
    # taps: a DFT of N samples per tap.  Correction: by planes, the rows' DFT of the N x N
    # pixels, then the columns' (the pixel screens are symmetric about the centre)
    return {"bytes": taps + 8 * P * rows * rows,
            "flops": 8.0 * P * (OS * S * N + rows * px / 4 + rows * rows * N / 2)}


# ---- float64 reference --------------------------------------------------------


def _taper64(c):
    """Transform of the Kaiser-Bessel window (beta = 2.34 S), normalised to 1 at nu = 0."""
    N, S = c["N"], c["S"]
    beta = 2.34 * S
    nu = (torch.arange(N, dtype=torch.float64, device=DEV) - N // 2) / N
    z2 = beta * beta - (math.pi * S * nu) ** 2  # positive for beta > pi S / 2
    z = torch.sqrt(z2)
    return (beta / z) * torch.exp(z - beta) * torch.expm1(-2.0 * z) / math.expm1(-2.0 * beta)


def _pixels(c):
    N = c["N"]
    return (torch.arange(N, dtype=torch.float64, device=DEV) - N // 2) / N * _fov(c)


def _planes(c, w_max):
    P = c["P"]
    return torch.arange(P, dtype=torch.float64, device=DEV) * (w_max / max(P - 1, 1))


def _cis(turns):
    ph = 2.0 * math.pi * (turns - torch.round(turns))
    return torch.complex(torch.cos(ph), torch.sin(ph))


def _dft(c, d):
    """exp(-2 pi i d nu_a), [len(d)][N], for offsets d in units of 1 / OS cells (integers)."""
    N, OS = c["N"], c["OS"]
    a = torch.arange(N, dtype=torch.int64, device=DEV) - N // 2
    m = torch.remainder(d[:, None] * a[None, :], N * OS)
    return _cis(-m.double() / (N * OS))


def _tap_offsets(c):
    S, OS = c["S"], c["OS"]
    o = torch.arange(OS, device=DEV)[:, None]
    j = torch.arange(S, device=DEV)[None, :]
    return ((j - S // 2 + 1) * OS - o).reshape(-1)


def _taps64(c, w_max, a2=-0.5, a4=-5.0 / 24.0):
    l, t = _pixels(c), _taper64(c).to(C128)
    w = _planes(c, w_max)
    screen = t[None, :] * _cis(w[:, None] * (a2 * l ** 2 + a4 * l ** 4)[None, :])
    return (screen @ _dft(c, _tap_offsets(c)).T / c["N"]).reshape(c["P"], c["OS"], c["S"])


def _residual64(c, w_max):
    """F_w - F~_w on the kept cells and offsets, [P][OSr][OSr][Sr][Sr]."""
    N, S, OS, Sr, OSr = c["N"], c["S"], c["OS"], c["Sr"], c["OSr"]
    step, k0 = OS // OSr, (S - Sr) // 2
    cc = torch.arange(OSr, device=DEV)[:, None]
    t = torch.arange(Sr, device=DEV)[None, :]
    E = _dft(c, ((k0 + t - S // 2 + 1) * OS - cc * step).reshape(-1))  # [OSr Sr][N]
    l, tp = _pixels(c), _taper64(c)
    r2 = l[None, :] ** 2 + l[:, None] ** 2
    nm1 = -r2 / (1.0 + torch.sqrt(1.0 - r2))
    taper2 = (tp[:, None] * tp[None, :]).to(C128)
    taps = _taps64(c, w_max)[:, ::step, k0:k0 + Sr].reshape(c["P"], -1)
    out = torch.empty((c["P"], OSr, OSr, Sr, Sr), dtype=C128, device=DEV)
    for p, w in enumerate(_planes(c, w_max)):
        K = (E @ (taper2 * _cis(w * nm1)) @ E.T) / (N * N)
        K -= taps[p][:, None] * taps[p][None, :]
        out[p] = K.reshape(OSr, Sr, OSr, Sr).permute(0, 2, 1, 3)
    return out


def _locate64(c, u, v, w, w_max):
    """Footprint origins, oversample indices, planes, conj and keep, as include/sepw.h says."""
    N, S, OS, P = c["N"], c["S"], c["OS"], c["P"]

    def axis(x):
        t = torch.floor((x * _fov(c) + float(N // 2)) * float(OS) + 0.5).long()
        cell = torch.div(t, OS, rounding_mode="floor")
        return cell - S // 2 + 1, t - cell * OS

    x0, ou = axis(u)
    y0, ov = axis(v)
    plane = torch.floor(w.abs() * ((P - 1) / w_max) + 0.5).long()
    keep = (x0 >= 0) & (x0 + S <= N) & (y0 >= 0) & (y0 + S <= N) & (plane <= P - 1)
    return x0, y0, ou, ov, plane, w < 0, keep


def _passes(c, u, v, w, w_max, tu, tv, res=None, base=None, vis=None, weight=None, grid=None,
            model=None, step=1 << 20):
    """Grids vis into `grid` (flat, complex128, += at base + cell) and degrids `model` (flat)."""
    N, S, OS = c["N"], c["S"], c["OS"]
    n = u.numel()
    out = torch.zeros(n, dtype=C128, device=DEV) if model is not None else None
    dropped = 0
    for a in range(0, n, step):
        sl = slice(a, min(n, a + step))
        x0, y0, ou, ov, pl, neg, keep = _locate64(c, u[sl], v[sl], w[sl], w_max)
        ids = torch.nonzero(keep).reshape(-1)
        dropped += keep.numel() - ids.numel()
        x0, y0, ou, ov, pl, neg = (t[ids] for t in (x0, y0, ou, ov, pl, neg))
        U, V = tu[pl, ou].T, tv[pl, ov].T  # [S][n]
        U = torch.where(neg, U.conj(), U).contiguous()
        V = torch.where(neg, V.conj(), V).contiguous()
        at = y0 * N + x0
        if base is not None:
            at += base[sl][ids]
        ids = ids + a
        wt = weight[ids].double() if weight is not None else 1.0
        if grid is not None:
            x = vis[ids].to(C128) * wt
            flat = torch.view_as_real(grid)
        R = None
        if res is not None:
            Sr, OSr = c["Sr"], c["OSr"]
            k0, q = (S - Sr) // 2, OS // OSr
            entry = (pl * OSr + torch.div(ov, q, rounding_mode="floor")) * OSr + \
                torch.div(ou, q, rounding_mode="floor")
            R = res.reshape(-1, Sr * Sr)
        acc = torch.zeros(ids.numel(), dtype=C128, device=DEV)
        for k in range(S):
            for j in range(S):
                kern = V[k] * U[j]
                if R is not None and k0 <= k < k0 + Sr and k0 <= j < k0 + Sr:
                    r = R[entry, (k - k0) * Sr + j - k0]
                    kern = kern + torch.where(neg, r.conj(), r)
                idx = at + (k * N + j)
                if grid is not None:
                    flat.index_add_(0, idx, torch.view_as_real(x * kern))
                if model is not None:
                    acc += kern.conj() * model[idx]
        if model is not None:
            out[ids] = acc * wt
    return out, torch.tensor([dropped], dtype=torch.int64, device=DEV)


def _correction64(c, l0=0.0, m0=0.0):
    """n, and n / (c1 c1) over the pixels [m][l]."""
    l, t = _pixels(c), _taper64(c)
    n = torch.sqrt(1.0 - ((l + l0)[None, :] ** 2 + (l + m0)[:, None] ** 2))
    return n, n / (t[None, :] * t[:, None])


def _to_image(g):
    return torch.fft.fftshift(torch.fft.ifft2(torch.fft.ifftshift(g), norm="forward"))


def _to_grid(x):
    return torch.fft.fftshift(torch.fft.fft2(torch.fft.ifftshift(x)))


def exact(case, seed):
    c = case
    d = _inputs(c, seed)
    N, kind = c["N"], c["kind"]
    w_max = d["w_max"]
    if kind == "tables":
        return {"taps": _taps64(c, w_max), "table": _residual64(c, w_max)}
    zeros = lambda k=1: torch.zeros(k * N * N, dtype=C128, device=DEV)  # noqa: E731
    if kind == "facet":
        l0, m0 = FACET
        n0 = math.sqrt(1.0 - l0 * l0 - m0 * m0)
        tu = _taps64(c, w_max, -0.5 * (1.0 / n0 + l0 * l0 / n0 ** 3), 0.0)
        tv = _taps64(c, w_max, -0.5 * (1.0 / n0 + m0 * m0 / n0 ** 3), 0.0)
        u, v, w = d["u"], d["v"], d["w"]
        turn = _cis(u * l0 + v * m0 + w * (n0 - 1.0))
        g = zeros()
        out, drop = _passes(c, u - (w * l0) / n0, v - (w * m0) / n0, w, w_max, tu, tv,
                            vis=d["vis"].to(C128) * turn, weight=d["weight"], grid=g)
        out, _ = _passes(c, u - (w * l0) / n0, v - (w * m0) / n0, w, w_max, tu, tv,
                         model=d["model"].to(C128).reshape(-1))
        return {"dirty": _to_image(g.reshape(N, N)) * _correction64(c, l0, m0)[1],
                "vis": out * turn.conj(), "dropped": drop}
    t = _taps64(c, w_max)
    if kind in ("step", "correction"):
        g = zeros()
        res = _residual64(c, w_max) if kind == "correction" else None
        out, drop = _passes(c, d["u"], d["v"], d["w"], w_max, t, t, res=res, vis=d["vis"],
                            weight=d["weight"], grid=g, model=d["model"].to(C128).reshape(-1))
        r = {"grid": g.reshape(N, N), "vis": out}
        return r if kind == "correction" else {**r, "dropped": drop}
    if kind == "noalloc":
        g = zeros()
        _, drop = _passes(c, d["u"], d["v"], d["w"], w_max, t, t, vis=d["vis"],
                          weight=d["weight"], grid=g)
        return {"grid": g.reshape(N, N), "dropped": drop, "status": None}
    if kind == "batched":
        g = zeros(c["grids"])
        counts = torch.from_numpy(np.diff(d["offsets"])).to(DEV)
        base = torch.repeat_interleave(torch.arange(c["grids"], device=DEV) * (N * N), counts)
        _, drop = _passes(c, d["u"], d["v"], d["w"], w_max, t, t, base=base, vis=d["vis"],
                          weight=d["weight"], grid=g)
        return {"grid": g.reshape(-1, N, N), "dropped": drop}
    if kind == "wstack":
        cen = torch.tensor(d["centres"], dtype=torch.float64, device=DEV)
        mid = 0.5 * (cen[1:] + cen[:-1])
        sl = torch.bucketize(d["w"], mid)
        wr = d["w"] - cen[sl]
        g = zeros(c["slices"])
        _passes(c, d["u"], d["v"], wr, w_max, t, t, base=sl * (N * N), vis=d["vis"],
                weight=d["weight"], grid=g)
        n, corr = _correction64(c)
        g = g.reshape(-1, N, N)
        dirty = torch.zeros((N, N), dtype=C128, device=DEV)
        for k in range(c["slices"]):
            ph = _cis(cen[k] * (n - 1.0))
            dirty += ph * _to_image(g[k])
            g[k] = _to_grid(d["image"].double() * ph.conj() * corr / (n * n))  # / (n c1 c1)
        out, _ = _passes(c, d["u"], d["v"], wr, w_max, t, t, base=sl * (N * N),
                         model=g.reshape(-1))
        return {"dirty": dirty * corr, "vis": out}
    # gradient
    n, corr = _correction64(c)
    fwd = corr / (n * n)  # 1 / (n c1 c1)
    m = _to_grid(d["image"].double() * fwd).reshape(-1)
    pred, _ = _passes(c, d["u"], d["v"], d["w"], w_max, t, t, model=m)
    r = pred - d["vis"].to(C128)
    wt = d["weight"].double() if d["weight"] is not None else torch.ones(c["n"], device=DEV)
    g = zeros()
    _passes(c, d["u"], d["v"], d["w"], w_max, t, t, vis=2.0 * wt * r, grid=g)
    return {"vis": pred, "chi2": (wt * (r.real ** 2 + r.imag ** 2)).sum(),
            "grad": (_to_image(g.reshape(N, N)) * fwd).real}
