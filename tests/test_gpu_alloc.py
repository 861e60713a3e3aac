"""A plan whose k-th workspace allocation fails returns SEPW_ENOMEM and leaves a
context that plans again, also for sizes it had room for before the failure."""
import numpy as np
import pytest

import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_07152_gb300 import build
    build.build()
    import paper_1511_07152_gb300.sepw as S
    return torch, S


def _centres(kind):
    # more slices (or grids) than the plan before, so that their arrays grow, too
    n = {"wstack": 5, "batched": 5, "plain": 1}[kind]
    return [100.0 * (k - (n - 1) / 2) for k in range(n)]


def _plan(S, ctx, kind, d, n, wide):
    u, v, w = (d[k][:n] for k in ("u", "v", "w"))
    if kind == "wstack":
        c = _centres(kind)
        S.sepw_wstack_plan(ctx, c if wide else c[1:3], u, v, w)
    elif kind == "batched":
        g = 5 if wide else 2
        S.sepw_plan_batched(ctx, [n * k // g for k in range(g + 1)], u, v, w)
    else:
        S.sepw_plan(ctx, u, v, w)


def _grid(torch, S, ctx, taps, d, n, ng):
    N = ctx.params.grid_size
    g = torch.zeros((ng, N, N), dtype=torch.complex64, device="cuda")
    S.sepw_grid_planned(ctx, taps, d["vis"][:n], d["weight"][:n], g if ng > 1 else g[0])
    return g.cpu().numpy()


@pytest.mark.parametrize("form,S_,kind", [
    ("FORM_TILED", 8, "plain"), ("FORM_TILED", 12, "plain"), ("FORM_TILED", 12, "batched"),
    ("FORM_TC_BF16", 8, "plain"), ("FORM_TILED", 8, "wstack")])
def test_planning_after_a_failed_allocation(env, form, S_, kind):
    torch, S = env
    wl = synth.random_case(3, 9000, grid_size=160, support=S_, oversample=8, n_wplanes=4)
    d = {k: torch.from_numpy(getattr(wl, k)).cuda() for k in ("u", "v", "w", "vis", "weight")}
    params = S.make_params(**wl.params(), form=getattr(S, form))
    ng = {"plain": 1, "batched": 2, "wstack": 2}[kind]
    ctx = S.sepw_create(params)
    taps = S.sepw_make_taps(ctx)
    _plan(S, ctx, kind, d, 700, False)
    want = _grid(torch, S, ctx, taps, d, 700, ng)
    failed = 0
    for k in range(1, 40):
        for start in (0, 900):  # the failure in the first plan, or in a later larger one
            ctx = S.sepw_create(params)
            if start:
                _plan(S, ctx, kind, d, start, False)
            S.sepw_test_fail_alloc(ctx, k)
            try:
                _plan(S, ctx, kind, d, 9000, True)
            except S.SepwError as e:
                assert e.status == S.ENOMEM
                failed += 1
                if start:  # the plan before is gone
                    with pytest.raises(S.SepwError):
                        _grid(torch, S, ctx, taps, d, start, ng)
            S.sepw_test_fail_alloc(ctx, 0)
            _plan(S, ctx, kind, d, 700, False)
            got = _grid(torch, S, ctx, taps, d, 700, ng)
            assert np.linalg.norm(got - want) <= 1e-5 * np.linalg.norm(want)
    assert failed >= 12
