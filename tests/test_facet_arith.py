"""The integer division by the facet centre's n0 (csrc/sepw_facet.cu), restated
in Python and checked against IEEE double, and the kernel's shift and phase bit
for bit / against extended precision on a GPU."""
import math
import struct

import numpy as np
import pytest


def _bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def _div(a, n0):
    """RN(a / n0) as the kernel computes it, or None where it falls back."""
    b = _bits(a)
    eb = (b >> 52) & 0x7FF
    nb = _bits(n0)
    ne = (nb >> 52) & 0x7FF
    mb = (nb & 0xFFFFFFFFFFFFF) | (1 << 52)
    recip = ((1 << 116) - 1) // mb
    assert recip < 1 << 64
    m = (b & 0xFFFFFFFFFFFFF) | (1 << 52)
    q = ((m << 11) * recip) >> 64
    e = eb - (ne - 1075) - 52
    if not q >> 63:
        q = (q << 1) & ((1 << 64) - 1)
        e -= 1
    low = q & 0x7FF
    if not q >> 63 or eb in (0, 0x7FF) or e < 1 or e > 2045 or 0x3FC <= low < 0x400:
        return None
    r = ((q >> 11) & 0xFFFFFFFFFFFFF) + (low >> 10)
    return struct.unpack("<d", struct.pack("<Q", (b & (1 << 63)) | ((e << 52) + r)))[0]


@pytest.mark.parametrize("n0", [1.0, 0.5, 1.0 - 2.0 ** -53, 0.9999037953722, 0.5 + 2.0 ** -53,
                                0.7071067811865476, 1.2e-8, 0.25 * (1 + 2.0 ** -52)])
def test_division_by_invariant_is_correctly_rounded(n0):
    rng = np.random.default_rng(int(n0 * 1e6) + 1)
    a = list(rng.uniform(-1e5, 1e5, 30000) * 10.0 ** rng.integers(-12, 12, 30000))
    for q in rng.uniform(0.5, 2.0, 5000):  # quotients next to half ways
        h = np.nextafter(q, 4.0)
        x = (q + (h - q) / 2) * n0
        a += [x, float(np.nextafter(x, 0)), float(np.nextafter(x, 4))]
        a += [q * n0, h * n0]
    a += [n0, -n0, 2 * n0, n0 * (1 - 2.0 ** -53), float(np.nextafter(n0, 2)),
          float(np.nextafter(n0, 0)), 5e-324, 1e-308, 1e308, 0.0, math.inf]
    done = 0
    for x in a:
        x = float(x)
        got = _div(x, n0)
        if got is None:
            continue
        done += 1
        assert _bits(got) == _bits(x / n0), (x, n0)
    assert done > 0.95 * len(a)


@pytest.mark.gpu
@pytest.mark.parametrize("l0,m0", [(0.0, 0.0), (0.012, -0.007), (0.6, 0.799999), (-0.5, 0.5),
                                   (1e-9, 0.3), (0.86602540378, 0.0)])
def test_shift_and_phase(l0, m0):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_07152_gb300 import build
    build.build()
    import paper_1511_07152_gb300.sepw as S
    rng = np.random.default_rng(17)
    n = 200_000
    u, v, w = (rng.uniform(-4e4, 4e4, n) * 10.0 ** rng.integers(-3, 3, n) for _ in range(3))
    special = [0.0, -0.0, 5e-324, -1e-310, 1e300, -1e308, math.inf, -math.inf, math.nan]
    for k, x in enumerate(special):
        w[k], u[20 + k], v[40 + k] = x, x, x
    vis = (rng.standard_normal(n) + 1j * rng.standard_normal(n)).astype(np.complex64)
    ctx = S.sepw_create(S.make_params(64, 0.02, 8, 8, 3, 100.0))
    S.sepw_set_facet(ctx, l0, m0)
    d = [torch.from_numpy(x).cuda() for x in (u, v, w)]
    uo, vo, out = torch.empty_like(d[0]), torch.empty_like(d[0]), torch.from_numpy(vis).cuda()
    S.sepw_facet_shift(ctx, S.FACET_IN, *d, out, uo, vo, out)
    n0 = math.sqrt(1.0 - l0 * l0 - m0 * m0)
    with np.errstate(all="ignore"):
        want_u, want_v = u - (w * l0) / n0, v - (w * m0) / n0
        L = np.longdouble
        ph = L(u) * L(l0) + L(v) * L(m0) + L(w) * L(n0 - 1.0)
    assert np.array_equal(uo.cpu().numpy(), want_u, equal_nan=True)
    assert np.array_equal(vo.cpu().numpy(), want_v, equal_nan=True)
    got = out.cpu().numpy()
    bad = ~(np.isfinite(u) & np.isfinite(v) & np.isfinite(w))
    assert np.all(np.isnan(got[bad])) and np.all(np.isfinite(got[~bad]))
    # extended precision still counts fractions of a turn below 2^40 turns
    ok = ~bad & (np.abs(u) < 1e9) & (np.abs(v) < 1e9) & (np.abs(w) < 1e9)
    turn = (ph[ok] - np.rint(ph[ok])).astype(np.float64)
    want = vis[ok] * np.exp(2j * np.pi * turn)
    # float32 phase (2^-25 turns) and rotation
    eps = 0.0 if np.finfo(L).nmant >= 63 else 2.0 ** -20
    assert np.max(np.abs(got[ok] - want) / np.abs(vis[ok])) <= 2 ** -25 * 2 * np.pi + 4e-7 + eps
    # back out: the opposite rotation
    S.sepw_facet_shift(ctx, S.FACET_OUT, *d, out, vis_out=out)
    assert np.max(np.abs(out.cpu().numpy()[ok] - vis[ok]) / np.abs(vis[ok])) <= 2e-6
