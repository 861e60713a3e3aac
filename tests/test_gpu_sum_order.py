"""Cells that many visibilities reach: the gridders' sums in two steps, within a
work unit and over the units, are as exact as units of the intended length make
them.  The data do not average out, as near the centre of the (u, v) plane."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

N_VIS, N, CELL, FOV, OS, P, W_MAX = 16_384, 256, 120, 0.02, 8, 4, 20.0


def fma(a, b, c):
    # the product of two FP32 numbers fits float64
    return (a.astype(np.float64) * b + c).astype(np.float32)


def emulate(x, tu, tv, unit):
    """FP32 grid cells [S][S] of visibilities x with tap rows tu, tv [n][S]: sums of
    `unit` of them at a time in the gridders' roundings, and then of those."""
    S = tu.shape[1]
    pr, pi, vr, vi = (np.asarray(a, np.float32).reshape(-1, unit, S) for a in (
        x.real[:, None] * tu.real, x.real[:, None] * tu.imag, tv.real, tv.imag))
    re = np.zeros((len(pr), S, S), np.float32)
    im = re.copy()
    for k in range(unit):
        a, b = vr[:, k, :, None], vi[:, k, :, None]
        p, q = pr[:, k, None, :], pi[:, k, None, :]
        if S <= 6:  # one rounded product
            re, im = re + fma(-b, q, a * p), im + fma(b, p, a * q)
        else:  # two FMAs
            re, im = fma(-b, q, fma(a, p, re)), fma(b, p, fma(a, q, im))
    re, im = (np.cumsum(a, axis=0, dtype=np.float32)[-1].astype(np.float64) for a in (re, im))
    return re + 1j * im


# schedule None: units of 32 would do for the size of the plan, but the tile holds
# all of it and gets the root of its number, 128; (2048, 1): whole items, cut to 256
# where the window gridder (S = 6, 10) keeps a cell's sum over all of a unit
@pytest.mark.parametrize("support, schedule, unit", [
    (6, None, 128), (8, None, 128), (10, None, 128), (16, None, 128),
    (6, (2048, 1), 256), (10, (2048, 1), 256)])
def test_units_of_dense_tiles(support, schedule, unit):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_07152_gb300 import build
    build.build()
    import paper_1511_07152_gb300.sepw as S
    ctx = S.sepw_create(S.make_params(N, FOV, support, OS, P, W_MAX, form=S.FORM_TILED))
    if schedule:
        S.sepw_set_schedule(ctx, *schedule)
    taps = S.sepw_make_taps(ctx)
    T = taps.cpu().numpy()

    def fine(t):
        return np.floor((t * FOV + N / 2) * OS + 0.5).astype(np.int64)

    y = CELL - support // 2 + 1
    got, emulated = [], []
    for seed in range(8):
        # all in one cell, at random offsets and planes
        rng = np.random.default_rng(seed)
        u, v = ((CELL - N // 2 + 0.9 * rng.random(N_VIS)) / FOV for _ in range(2))
        w = 0.999 * W_MAX * rng.random(N_VIS)
        x = (0.5 + rng.random(N_VIS)).astype(np.complex64)
        grid = torch.zeros((N, N), dtype=torch.complex64, device="cuda")
        S.sepw_grid(ctx, taps, *(torch.from_numpy(a).cuda() for a in (u, v, w, x)), None, grid)
        tu, tv, plane = fine(u), fine(v), np.floor(w * ((P - 1) / W_MAX) + 0.5).astype(np.int64)
        assert (tu // OS == CELL).all() and (tv // OS == CELL).all()
        rows, cols = T[plane, tv % OS], T[plane, tu % OS]
        want = np.einsum("n,ni,nj->ij", x.astype(np.complex128), rows.astype(np.complex128),
                         cols.astype(np.complex128))
        for out, g in ((got, grid.cpu().numpy()[y:y + support, y:y + support]),
                       (emulated, emulate(x, cols, rows, unit))):
            out.append(np.abs(g - want) / np.abs(want))
    rms = [float(np.sqrt(np.mean(np.square(e)))) for e in (got, emulated)]
    # 1.5: the order of the units' sums is free.  (Units of 32 at S = 6 are off twice
    # as far as 128, whole items at S = 10 nine times as far as 256.)
    assert rms[0] <= 1.5 * rms[1], rms
