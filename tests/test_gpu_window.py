"""The register-window gridder of the tiled form and the plan passes below it,
at the sizes where they can go wrong, against the FP64 oracle (FP32 bar: the
suite's relative L2 of 1e-5)."""
import math

import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_07152_gb300 import build
    build.build()
    import paper_1511_07152_gb300.sepw as S
    return torch, S


def rel_l2(a, b):
    a = np.asarray(a, np.complex128).ravel()
    b = np.asarray(b, np.complex128).ravel()
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


def _dev(torch, wl):
    return {k: torch.from_numpy(getattr(wl, k)).cuda() for k in ("u", "v", "w", "vis", "weight")}


def _run(env, wl, tile=0, form=None, schedule=None, vis=None):
    torch, S = env
    ctx = S.sepw_create(S.make_params(**wl.params(), tile=tile,
                                      form=S.FORM_TILED if form is None else form))
    if schedule:
        S.sepw_set_schedule(ctx, *schedule)
    taps = S.sepw_make_taps(ctx)
    d = _dev(torch, wl)
    N = wl.grid_size
    grid = torch.zeros((N, N), dtype=torch.complex64, device="cuda")
    S.sepw_grid(ctx, taps, d["u"], d["v"], d["w"], d["vis"] if vis is None else vis, d["weight"],
                grid)
    out = torch.empty(wl.nvis, dtype=torch.complex64, device="cuda")
    S.sepw_degrid_planned(ctx, taps, grid, d["weight"], out)
    return grid.cpu().numpy(), out.cpu().numpy()


def _check(env, wl, **kw):
    p = O.params_from(wl.params())
    T, loc = O.taps(p), O.locate(p, wl.u, wl.v, wl.w)
    grid, out = _run(env, wl, **kw)
    assert rel_l2(grid, O.grid_separable(p, loc, wl.vis, wl.weight, T)) <= TOL
    assert rel_l2(out, O.degrid_separable(p, loc, grid.astype(np.complex128), wl.weight, T)) <= TOL


@pytest.mark.parametrize("support", range(2, 33, 2))
@pytest.mark.parametrize("radius", [None, 9.0])
def test_every_support(env, support, radius):
    """Each support's rows and columns per lane, spread over the grid (moves
    between columns of blocks, windows over the grid's edge) and packed (steps
    down a column, several units per tile)."""
    _check(env, synth.random_case(300 + support, 3000, 98, support, 8, 5, radius_cells=radius,
                                  edge_fraction=0.2 if radius is None else 0.0))


@pytest.mark.parametrize("tile", [8, 10, 18, 30, 32, 34, 52])
def test_tile_sizes(env, tile):
    """Tiles that blocks of 4 x 4 origins do and do not divide, and those
    above 32 (the column gridder)."""
    _check(env, synth.random_case(340, 5000, 160, 10, 7, 9, edge_fraction=0.1), tile=tile)


@pytest.mark.parametrize("nvis", [1, 31, 32, 33, 2047, 2048, 2049])
@pytest.mark.parametrize("schedule", [None, (64, 1), (2048, 1), (2048, 16)])
def test_unit_edges(env, nvis, schedule):
    """Units and items at their edges, all visibilities in one or two tiles."""
    _check(env, synth.random_case(341, nvis, 96, 12, 8, 5, radius_cells=3.0), schedule=schedule)


@pytest.mark.parametrize("N,support,tile,form", [
    (2048, 8, 8, "tiled"),    # 65,025 tiles, one block each: a thread per tile
    (2400, 12, 12, "tiled"),  # 39,601 tiles of 9 blocks: 64 tiles per block of threads
    (1500, 6, 8, "tiled"),    # 34,969 tiles of 4 blocks
    (1088, 4, 32, "tiled"),   # 1,156 tiles of 64 blocks: two loads per lane
    (2048, 8, 8, "tc"),
])
def test_many_tiles(env, N, support, tile, form):
    torch, S = env
    _check(env, synth.random_case(342, 20000, N, support, 4, 3, w_max=50.0, edge_fraction=0.05),
           tile=tile, form=S.FORM_TILED if form == "tiled" else S.FORM_TC_BF16X2)


@pytest.mark.parametrize("support", [6, 10, 16, 20])
def test_non_finite_values_stay_in_their_footprints(env, support):
    """NaN, infinite and huge visibilities touch exactly their S x S cells, and
    a tap that is not finite only the cells it multiplies."""
    torch, S = env
    wl = synth.random_case(343, 400, 128, support, 4, 3)
    p = O.params_from(wl.params())
    T, loc = O.taps(p), O.locate(p, wl.u, wl.v, wl.w)
    bad = np.flatnonzero(loc["keep"])[[3, 50, 120]]
    vis = wl.vis.copy()
    vis[bad] = [complex(np.nan, 1), complex(1, np.inf), complex(3e38, 3e38)]
    grid, _ = _run(env, wl, vis=torch.from_numpy(vis).cuda())
    hit = np.zeros((p.N, p.N), bool)
    for i in bad[:2]:
        y, x = loc["cv"][i] - p.S // 2 + 1, loc["cu"][i] - p.S // 2 + 1
        hit[y:y + p.S, x:x + p.S] = True
    y, x = loc["cv"][bad[2]] - p.S // 2 + 1, loc["cu"][bad[2]] - p.S // 2 + 1
    huge = np.zeros_like(hit)
    huge[y:y + p.S, x:x + p.S] = True
    fine = np.isfinite(grid)
    assert not np.any(fine & hit & ~huge)  # the footprints of NaN and infinity
    assert np.all(fine[~hit & ~huge])      # nothing else
    keep = loc["keep"].copy()
    keep[bad] = False
    want = O.grid_separable(p, dict(loc, keep=keep), wl.vis, wl.weight, T)
    rest = ~hit & ~huge
    assert rel_l2(grid[rest], want[rest]) <= TOL
    # the same for prediction: a cell that is not finite reaches the footprints
    # that hold it, and no others
    model = np.random.default_rng(9).standard_normal((p.N, p.N, 2)).astype(np.float32)
    model = model.view(np.complex64)[:, :, 0]
    y0, x0 = loc["cv"][bad[0]] + 1, loc["cu"][bad[0]] - 1
    model[y0, x0] = complex(np.inf, 0)
    ctx = S.sepw_create(S.make_params(**wl.params(), form=S.FORM_TILED))
    t0 = S.sepw_make_taps(ctx)
    dd = _dev(torch, wl)
    out = torch.empty(wl.nvis, dtype=torch.complex64, device="cuda")
    S.sepw_degrid(ctx, t0, dd["u"], dd["v"], dd["w"], torch.from_numpy(model).cuda(),
                  dd["weight"], out)
    got = out.cpu().numpy()
    fy, fx = loc["cv"] - p.S // 2 + 1, loc["cu"] - p.S // 2 + 1
    holds = loc["keep"] & (fy <= y0) & (y0 < fy + p.S) & (fx <= x0) & (x0 < fx + p.S)
    assert holds.any() and np.array_equal(~np.isfinite(got), holds)
    clean = np.where(np.isfinite(model), model, 0)
    pw = O.degrid_separable(p, loc, clean.astype(np.complex128), wl.weight, T)
    assert rel_l2(got[~holds], pw[~holds]) <= TOL
    # a NaN tap: the same cells as the plain form, which reads no padded rows
    ctxs = [S.sepw_create(S.make_params(**wl.params(), form=f))
            for f in (S.FORM_PLAIN, S.FORM_TILED)]
    taps = S.sepw_make_taps(ctxs[0])
    taps[1, 2, p.S // 2] = complex(np.nan, 0.0)
    d = _dev(torch, wl)
    got = []
    for ctx in ctxs:
        g = torch.zeros((p.N, p.N), dtype=torch.complex64, device="cuda")
        S.sepw_grid(ctx, taps, d["u"], d["v"], d["w"], d["vis"], d["weight"], g)
        got.append(g.cpu().numpy())
    assert np.array_equal(np.isfinite(got[0]), np.isfinite(got[1]))
    ok = np.isfinite(got[0])
    assert 0 < (~ok).sum() < ok.size
    assert rel_l2(got[1][ok], got[0][ok]) <= TOL


@pytest.mark.parametrize("support,nvis", [(16, 4095), (16, 4097), (12, 4097)])
def test_correction_after_an_unsorted_plan(env, support, nvis):
    """The sort that the correction passes add to a plan made without it (dense
    enough or not), and the separable kernels on that plan before and after;
    S = 16 on both sides of the window gridder's density."""
    torch, S = env
    wl = synth.random_case(345, nvis, 128, support, 4, 3)
    p = O.params_from(wl.params())
    T, loc = O.taps(p), O.locate(p, wl.u, wl.v, wl.w)
    ctx = S.sepw_create(S.make_params(**wl.params(), form=S.FORM_TILED))
    taps = S.sepw_make_taps(ctx)
    d = _dev(torch, wl)
    rng = np.random.default_rng(7)
    R = (rng.standard_normal((p.P, 2, 2, 8, 8)) + 1j * rng.standard_normal((p.P, 2, 2, 8, 8)))
    table = torch.from_numpy(R.astype(np.complex64)).cuda()
    S.sepw_plan(ctx, d["u"], d["v"], d["w"])
    grid = torch.zeros((p.N, p.N), dtype=torch.complex64, device="cuda")
    out = torch.zeros(nvis, dtype=torch.complex64, device="cuda")
    S.sepw_grid_residual_planned(ctx, table, d["vis"], d["weight"], grid)
    want = O.grid_residual(p, loc, wl.vis, wl.weight, R.astype(np.complex64))
    assert rel_l2(grid.cpu().numpy(), want) <= TOL
    model = grid.clone()
    S.sepw_degrid_residual_planned(ctx, table, model, d["weight"], out)
    host = model.cpu().numpy()
    assert rel_l2(out.cpu().numpy(), O.degrid_residual(p, loc, host, wl.weight,
                                                       R.astype(np.complex64))) <= TOL
    grid.zero_()
    S.sepw_grid_planned(ctx, taps, d["vis"], d["weight"], grid)
    assert rel_l2(grid.cpu().numpy(), O.grid_separable(p, loc, wl.vis, wl.weight, T)) <= TOL
    S.sepw_degrid_planned(ctx, taps, model, d["weight"], out)
    assert rel_l2(out.cpu().numpy(), O.degrid_separable(p, loc, host, wl.weight, T)) <= TOL


def test_facet_tables(env):
    """Separate u and v tables (the v taps come from the second one)."""
    torch, S = env
    wl = synth.random_case(344, 6000, 128, 10, 8, 9, w_max=400.0, radius_cells=40.0,
                           fov=math.radians(2.0))
    ctx = S.sepw_create(S.make_params(**wl.params(), form=S.FORM_TILED))
    S.sepw_set_facet(ctx, 0.012, -0.007)
    taps = S.sepw_make_taps(ctx)
    p = O.params_from(wl.params())
    loc = O.locate(p, wl.u, wl.v, wl.w)
    Tu, Tv = O.taps_facet(p, 0.012, -0.007)
    d = _dev(torch, wl)
    grid = torch.zeros((p.N, p.N), dtype=torch.complex64, device="cuda")
    S.sepw_grid(ctx, taps, d["u"], d["v"], d["w"], d["vis"], d["weight"], grid)
    want = O.grid_separable(p, loc, wl.vis, wl.weight, Tu, Tv=Tv)
    assert rel_l2(grid.cpu().numpy(), want) <= TOL
