"""The window kernels' tap tables: allocated by the first plan that takes them,
and left alone where they are large for the call, against the FP64 oracle."""
import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5  # FP32 bar, relative L2


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


def test_a_context_without_a_plan_holds_none(env):
    """S = 12 with 524,288 tap rows: tables of 201 MB, the caller's taps 50 MB."""
    torch, S = env
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    ctx = S.sepw_create(S.make_params(64, 0.03, 12, 16, 32768, 500.0, form=S.FORM_TILED))
    assert free - torch.cuda.mem_get_info()[0] < 150e6
    ctx.close()


@pytest.mark.parametrize("support,planes", [(4, 5300), (12, 2750), (20, 1900)])
@pytest.mark.parametrize("nvis", [2_000, 20_000])
def test_large_tables(env, support, planes, nvis):
    """16.0 to 17.5 MB of tables, below and above 2048 bytes a visibility."""
    torch, S = env
    wl = synth.random_case(support, nvis, grid_size=128, support=support, oversample=16,
                           n_wplanes=planes)
    ctx = S.sepw_create(S.make_params(**wl.params(), form=S.FORM_TILED))
    taps = S.sepw_make_taps(ctx)
    d = _dev(torch, wl)
    grid = torch.zeros((128, 128), dtype=torch.complex64, device="cuda")
    out = torch.empty(nvis, dtype=torch.complex64, device="cuda")
    S.sepw_grid(ctx, taps, d["u"], d["v"], d["w"], d["vis"], d["weight"], grid)
    S.sepw_degrid_planned(ctx, taps, grid, d["weight"], out)
    p = O.params_from(wl.params())
    loc, T = O.locate(p, wl.u, wl.v, wl.w), taps.cpu().numpy().astype(np.complex128)
    g = grid.cpu().numpy()
    assert rel_l2(g, O.grid_separable(p, loc, wl.vis, wl.weight, T)) <= TOL
    assert rel_l2(out.cpu().numpy(),
                  O.degrid_separable(p, loc, g.astype(np.complex128), wl.weight, T)) <= TOL


def test_first_sparse_plan_inside_a_capture(env):
    """A context that has only made dense S = 16 plans has no tables yet: a sparse
    plan captured then does without."""
    torch, S = env
    wl = synth.random_case(7, 20_000, grid_size=200, support=16, oversample=8, n_wplanes=5)
    ctx = S.sepw_create(S.make_params(**wl.params(), form=S.FORM_TILED))
    taps = S.sepw_make_taps(ctx)
    d = _dev(torch, wl)
    grid = torch.zeros((200, 200), dtype=torch.complex64, device="cuda")
    S.sepw_grid(ctx, taps, d["u"], d["v"], d["w"], d["vis"], d["weight"], grid)
    n = 3_000  # below a visibility per four cells
    few = {k: x[:n] for k, x in d.items()}
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        grid.zero_()
        S.sepw_grid(ctx, taps, few["u"], few["v"], few["w"], few["vis"], few["weight"], grid)
    p = O.params_from(wl.params())
    loc = O.locate(p, wl.u[:n], wl.v[:n], wl.w[:n])
    want = O.grid_separable(p, loc, wl.vis[:n], wl.weight[:n], O.taps(p))
    for _ in range(2):
        graph.replay()
        assert rel_l2(grid.cpu().numpy(), want) <= TOL
    grid.zero_()
    S.sepw_grid(ctx, taps, few["u"], few["v"], few["w"], few["vis"], few["weight"], grid)
    assert rel_l2(grid.cpu().numpy(), want) <= TOL
