"""The window gridder's sums are no less exact than those of one atomic per
visibility and cell, at the supports where few visibilities meet in a cell."""
import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu


def _fma(a, b, c):
    # exact: the product of two FP32 numbers fits float64
    return (a.astype(np.float64) * b.astype(np.float64) + c.astype(np.float64)).astype(np.float32)


def _grid_one_by_one(p, loc, x, T):
    """FP32 grid with every visibility's W V F1 F1 (rounded as the kernels do)
    added to the cells on its own."""
    S = p.S
    grid = np.zeros((p.N, p.N, 2), np.float32)
    for i in np.flatnonzero(loc["keep"]):
        u = T[loc["plane"][i], loc["ou"][i]]
        v = T[loc["plane"][i], loc["ov"][i]]
        if loc["conj"][i]:
            u, v = u.conj(), v.conj()
        wx, wy = np.float32(x[i].real), np.float32(x[i].imag)
        pr = _fma(wx, u.real, -(wy * u.imag))
        pi = _fma(wx, u.imag, wy * u.real)
        vr, vi = v.real[:, None], v.imag[:, None]
        y, z = loc["cv"][i] - S // 2 + 1, loc["cu"][i] - S // 2 + 1
        cell = grid[y:y + S, z:z + S]
        cell[..., 0] += _fma(-vi, pi[None, :], vr * pr[None, :])
        cell[..., 1] += _fma(vi, pr[None, :], vr * pi[None, :])
    return grid[..., 0].astype(np.float64) + 1j * grid[..., 1]


@pytest.mark.parametrize("support", [2, 4, 6, 10])
def test_sums_are_as_exact_as_single_additions(support):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_07152_gb300 import build
    build.build()
    import paper_1511_07152_gb300.sepw as S
    wl = synth.random_case(support, 24_000, grid_size=112, support=support, oversample=8,
                           n_wplanes=4)
    ctx = S.sepw_create(S.make_params(**wl.params(), form=S.FORM_TILED))
    S.sepw_set_schedule(ctx, 2048, 8)  # units of 256: the most sums in registers
    taps = S.sepw_make_taps(ctx)
    u, v, w = (torch.from_numpy(getattr(wl, k)).cuda() for k in ("u", "v", "w"))
    vis = torch.from_numpy(wl.vis).cuda()
    grid = torch.zeros((112, 112), dtype=torch.complex64, device="cuda")
    S.sepw_grid(ctx, taps, u, v, w, vis, None, grid)
    p = O.params_from(wl.params())
    loc, T = O.locate(p, wl.u, wl.v, wl.w), taps.cpu().numpy()
    want = O.grid_separable(p, loc, wl.vis, np.ones(wl.nvis, np.float32),
                            T.astype(np.complex128))
    err = [np.linalg.norm(g - want) / np.linalg.norm(want)
           for g in (grid.cpu().numpy().astype(np.complex128),
                     _grid_one_by_one(p, loc, wl.vis, T))]
    assert err[0] <= err[1], err
