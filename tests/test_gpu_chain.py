"""Back-to-back calls on small plans, whose kernels overlap (programmatic
dependent launches): every call has to see the tap table, the grid and the
visibilities as the calls before it left them, with nothing in between.
Against the FP64 oracle (FP32 bar: the suite's relative L2 of 1e-5)."""
import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu

TOL = 1e-5


def rel_l2(a, b):
    a = np.asarray(a, np.complex128).ravel()
    b = np.asarray(b, np.complex128).ravel()
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("S,nvis", [(8, 20_000), (10, 20_000), (12, 5_003), (16, 20_000),
                                    (16, 1_000), (20, 9_001)])
def test_alternating_tables_and_grids(S, nvis):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_07152_gb300 import build
    build.build()
    import paper_1511_07152_gb300.sepw as sepw
    wl = synth.random_case(S, nvis, grid_size=256, support=S, oversample=8, n_wplanes=8)
    ctx = sepw.sepw_create(sepw.make_params(**wl.params(), form=sepw.FORM_TILED))
    u, v, w, vis, weight = (torch.from_numpy(getattr(wl, k)).cuda()
                            for k in ("u", "v", "w", "vis", "weight"))
    first = sepw.sepw_make_taps(ctx)
    # another table: planes reversed, another scale and phase
    tables = [first, (first.flip(0) * (0.5 - 0.25j)).contiguous()]
    sepw.sepw_plan(ctx, u, v, w)
    N = wl.grid_size
    rounds = 6
    grids = torch.zeros((rounds, N, N), dtype=torch.complex64, device="cuda")
    outs = torch.empty((rounds, nvis), dtype=torch.complex64, device="cuda")
    torch.cuda.synchronize()
    for k in range(rounds):  # predictions of one round are the next one's visibilities
        sepw.sepw_grid_planned(ctx, tables[k % 2], vis if k == 0 else outs[k - 1], weight,
                               grids[k])
        sepw.sepw_degrid_planned(ctx, tables[(k + 1) % 2], grids[k], weight, outs[k])
    torch.cuda.synchronize()
    p = O.params_from(wl.params())
    loc = O.locate(p, wl.u, wl.v, wl.w)
    T = [t.cpu().numpy().astype(np.complex128) for t in tables]
    g, o = grids.cpu().numpy(), outs.cpu().numpy()
    x = wl.vis
    for k in range(rounds):
        assert rel_l2(g[k], O.grid_separable(p, loc, x, wl.weight, T[k % 2])) <= TOL, k
        want = O.degrid_separable(p, loc, g[k].astype(np.complex128), wl.weight, T[(k + 1) % 2])
        assert rel_l2(o[k], want) <= TOL, k
        x = o[k]
