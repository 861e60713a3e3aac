"""The 32-bit fixed-point path of locate (csrc/sepw_internal.cuh), restated in
Python and checked against the IEEE double definition of the header."""
import math
import struct

import numpy as np
import pytest

M32 = 0xFFFFFFFF


def _bits(x):
    return struct.unpack("<Q", struct.pack("<d", x))[0]


def _fixed(b, ex):
    hi, lo, s = (b >> 32) & 0xFFFFF | 0x100000, b & M32, 20 - ex
    assert s >= 0
    if s >= 32:
        lo, hi, s = hi, 0, s - 32
    frac = hi if s >= 32 else ((hi << 32 | lo) >> s) & M32  # __funnelshift_rc clamps at 32
    return (hi >> s if s < 32 else 0), frac


def _bounds(N, os_log2):
    half_span, e = (N << os_log2) // 2, 0
    while e < 21 and (1 << (e + 1)) <= half_span:
        e += 1
    return e, ((N << os_log2) >> 21) + 3


def _axis(y, N, os_log2):
    """t = floor((y + N/2) OS + 1/2), or None where the kernel takes FP64."""
    elim, near = _bounds(N, os_log2)
    b = _bits(y)
    ey = ((b >> 52) & 0x7FF) - 1023 + os_log2
    if ey >= elim:
        return None
    whole, frac = _fixed(b, ey)
    if ((frac - 0x80000000 + near) & M32) <= 2 * near:
        return None
    n = whole + (frac >> 31)
    return ((N >> 1) << os_log2) + (-n if b >> 63 else n)


def _plane(x, P):
    """The plane of x = fl(|w| r), or None for a drop."""
    b = _bits(x)
    ex = ((b >> 52) & 0x7FF) - 1023
    whole, frac = _fixed(b, min(ex, 20))
    q = whole + (frac >> 31) + (b == 0x3FDFFFFFFFFFFFFF)
    return q if ex <= 20 and q <= P - 1 else None


@pytest.mark.parametrize("N,OS", [(16, 1), (96, 16), (256, 8), (1000, 4), (4096, 16), (8192, 256),
                                  (65536, 256), (65536, 1)])
def test_axis_equals_ieee(N, OS):
    lg, H = OS.bit_length() - 1, N // 2
    rng = np.random.default_rng(N + OS)
    ys = list(rng.uniform(-H - 5, H + 5, 20000))
    ys += list(rng.uniform(-1, 1, 3000) * 10.0 ** rng.integers(-30, 3, 3000))
    for k in rng.integers(-H * OS, H * OS, 3000):  # next to half-integers of y OS
        up = dn = (float(k) - 0.5) / OS
        ys.append(up)
        for _ in range(3):
            up, dn = float(np.nextafter(up, np.inf)), float(np.nextafter(dn, -np.inf))
            ys += [up, dn]
        for d in (1, 3, 10, 100):
            ys += [(float(k) - 0.5) / OS + s * d * 2.0 ** -32 / OS for s in (-1, 1)]
    ys += [0.0, -0.0, 5e-324, -5e-324, 1e-310, float(H), -float(H), 0.5 / OS, -0.5 / OS,
           math.inf, -math.inf, math.nan, 1e300]
    done = 0
    for y in ys:
        t = _axis(float(y), N, lg)
        if t is None:
            continue
        done += 1
        assert t == math.floor((y + float(H)) * OS + 0.5), (y, N, OS)
    # the path covers |y| OS < 2^elim of the N OS / 2 on the grid
    assert done > 15000 * min(1.0, 2.0 ** _bounds(N, lg)[0] / (N * OS / 2))


@pytest.mark.parametrize("P", [1, 2, 33, 128, 32768])
def test_plane_equals_ieee(P):
    rng = np.random.default_rng(P)
    xs = list(rng.uniform(0, P + 1, 20000)) + list(10.0 ** rng.uniform(-320, 300, 3000))
    for k in rng.integers(0, P + 1, 2000):
        h = float(k) + 0.5
        xs += [h, float(np.nextafter(h, 0)), float(np.nextafter(h, 1e9)), float(k)]
    xs += [0.0, 0.5 - 2.0 ** -54, 0.5, 2.0 ** 20, 2.0 ** 21 - 0.5, 2.0 ** 21, 2.0 ** 22, 1e18,
           math.inf, math.nan]
    for x in xs:
        x = float(x)
        want = None
        if math.isfinite(x):
            q = math.floor(x + 0.5)
            want = q if q <= P - 1 else None
        assert _plane(x, P) == want, x
