"""FP16 hi + lo gridding: the error is that of the FP32 sums, which depend on the
order of the visibilities within a tile.  The plan makes that order, so the input's
does not matter."""
import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

N_VIS, N, FOV, S_, OS, P, W_MAX = 30_000, 700, 0.02, 6, 8, 8, 500.0


def _visibilities(rng, side):
    """Uniform over a square of `side` cells, data that do not average out."""
    u, v = ((rng.random(N_VIS) - 0.5) * side / FOV for _ in range(2))
    w = 0.999 * W_MAX * rng.random(N_VIS)
    return u, v, w, (0.5 + rng.random(N_VIS)).astype(np.complex64)


@pytest.mark.parametrize("side", [104, 208])
def test_input_order_does_not_cost_accuracy(side):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_07152_gb300 import build
    build.build()
    import paper_1511_07152_gb300.sepw as S
    ctx = S.sepw_create(S.make_params(N, FOV, S_, OS, P, W_MAX, form=S.FORM_TC_FP16X2))
    taps = S.sepw_make_taps(ctx)
    p = O.Params(N, FOV, S_, OS, P, W_MAX)
    sq = [0.0, 0.0]
    for seed in range(6):
        a = _visibilities(np.random.default_rng(seed), side)
        loc = O.locate(p, *a[:3])
        assert loc["keep"].all()
        want = O.grid_separable(p, loc, a[3], np.ones(N_VIS, np.float32),
                                taps.cpu().numpy().astype(np.complex128))
        blocks = np.lexsort((loc["cu"] // 8, loc["cv"] // 8))  # 8 x 8 cells at a time
        for k, order in enumerate((blocks, np.arange(N_VIS))):
            grid = torch.zeros((N, N), dtype=torch.complex64, device="cuda")
            S.sepw_grid(ctx, taps, *(torch.from_numpy(x[order]).cuda() for x in a), None, grid)
            g = grid.cpu().numpy().astype(np.complex128)
            sq[k] += (np.linalg.norm(g - want) / np.linalg.norm(want)) ** 2 / 6
    by_blocks, as_drawn = np.sqrt(sq)
    # the same order of blocks either way; the order inside a block is free
    assert as_drawn <= 1.25 * by_blocks, (as_drawn, by_blocks)
