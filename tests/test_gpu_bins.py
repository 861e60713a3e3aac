"""The bins of a plan below the tile, on both sides of each line of the rule that
chooses them (few or many tiles, few or many visibilities, tile edges with and
without room for conj bins), against the FP64 oracle."""
import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu

# the suite's bars (relative L2): FP32-class forms 1e-5, 11-bit operands 1.5e-3,
# BF16 operands 1e-2
TOL = {"FORM_TILED": 1e-5, "FORM_TC_BF16X2": 1e-5, "FORM_TC_TF32": 1.5e-3,
       "FORM_TC_FP16": 1.5e-3, "FORM_TC_BF16": 1e-2}


def rel_l2(a, b):
    a = np.asarray(a, np.complex128).ravel()
    b = np.asarray(b, np.complex128).ravel()
    return float(np.linalg.norm(a - b) / np.linalg.norm(b))


@pytest.mark.parametrize("form,S,tile,N,nvis", [
    # 16-bit forms: one bin by few visibilities, edge 4 (T = 16 with conj bins,
    # 26, 24, 18 and 20 without room for them), edge 8, one bin by many tiles
    ("FORM_TC_BF16", 16, 0, 128, 32768), ("FORM_TC_BF16", 16, 0, 128, 32769),
    ("FORM_TC_FP16", 6, 0, 160, 40000), ("FORM_TC_BF16X2", 8, 0, 200, 40000),
    ("FORM_TC_FP16", 14, 0, 130, 40000), ("FORM_TC_BF16X2", 12, 8, 1100, 1300000),
    ("FORM_TC_BF16", 16, 8, 1060, 40000),
    # sorted plans: edge 4 with (T = 16) and without (32) conj bins, T > 32, edge 8
    ("FORM_TC_TF32", 16, 0, 128, 40000), ("FORM_TC_TF32", 6, 0, 160, 3000),
    ("FORM_TILED", 8, 0, 256, 40000), ("FORM_TILED", 16, 16, 128, 20000),
    ("FORM_TILED", 8, 40, 200, 20000), ("FORM_TILED", 16, 8, 1200, 400000),
    ("FORM_TILED", 8, 0, 1100, 30000)])
def test_step_against_the_oracle(form, S, tile, N, nvis):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_07152_gb300 import build
    build.build()
    import paper_1511_07152_gb300.sepw as sepw
    wl = synth.random_case(S + N, nvis, grid_size=N, support=S, oversample=8, n_wplanes=4,
                           edge_fraction=0.02)
    ctx = sepw.sepw_create(sepw.make_params(**wl.params(), tile=tile, form=getattr(sepw, form)))
    taps = sepw.sepw_make_taps(ctx)
    u, v, w, vis, weight = (torch.from_numpy(getattr(wl, k)).cuda()
                            for k in ("u", "v", "w", "vis", "weight"))
    rng = np.random.default_rng(N)
    X = (rng.standard_normal((N, N)) + 1j * rng.standard_normal((N, N))).astype(np.complex64)
    grid = torch.zeros((N, N), dtype=torch.complex64, device="cuda")
    out = torch.empty(nvis, dtype=torch.complex64, device="cuda")
    dropped = torch.zeros(1, dtype=torch.int64, device="cuda")
    sepw.sepw_grid(ctx, taps, u, v, w, vis, weight, grid, n_dropped=dropped)
    sepw.sepw_degrid_planned(ctx, taps, torch.from_numpy(X).cuda(), weight, out)
    assert sepw.sepw_device_status(ctx) == sepw.OK
    p = O.params_from(wl.params())
    T, loc = O.taps(p), O.locate(p, wl.u, wl.v, wl.w)
    assert int(dropped) == int(np.count_nonzero(~np.asarray(loc["keep"], bool)))
    assert rel_l2(grid.cpu().numpy(),
                  O.grid_separable(p, loc, wl.vis, wl.weight, T)) <= TOL[form]
    assert rel_l2(out.cpu().numpy(),
                  O.degrid_separable(p, loc, X.astype(np.complex128), wl.weight, T)) <= TOL[form]
