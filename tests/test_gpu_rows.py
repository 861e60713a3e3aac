"""The row transforms of the image step and of W stacking, for every size they
take and the ones beside it, against float64 FFTs (numpy)."""
import math

import numpy as np
import pytest

import oracle as O

pytestmark = pytest.mark.gpu

# FP32 transforms of 2^24 points: 1e-5, the bar of the image step, with the grid
# correction divided out where it amplifies rounding towards the edges
TOL = 1e-5
SIZES = [256, 510, 512, 1000, 1024, 2048, 4096]


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


def _terms(N, S_, fov):
    nu = (np.arange(N) - N // 2) / N
    c = O.kb_taper(nu, S_, 2.34 * S_)
    l = nu * fov
    n = np.sqrt(1.0 - l[None, :] ** 2 - l[:, None] ** 2)
    return n, n / np.outer(c, c)


def _to_image(g):
    return np.fft.fftshift(np.fft.ifft2(np.fft.ifftshift(g), norm="forward"))


def _to_grid(x):
    return np.fft.fftshift(np.fft.fft2(np.fft.ifftshift(x)))


def _random(rng, *shape):
    return (rng.standard_normal(shape) + 1j * rng.standard_normal(shape)).astype(np.complex64)


@pytest.mark.parametrize("N", SIZES)
def test_image_step(env, N):
    torch, S = env
    fov = math.radians(3.0)
    ctx = S.sepw_create(S.make_params(N, fov, 4, 3, 2, 100.0))
    n, corr = _terms(N, 4, fov)
    x = _random(np.random.default_rng(N), N, N)
    for direction, want, flat in (
            (S.GRID_TO_IMAGE, _to_image(x) * corr, corr),
            (S.IMAGE_TO_GRID_ADJOINT, _to_image(x) * corr / n ** 2, corr),
            (S.IMAGE_TO_GRID, _to_grid(x * corr / n ** 2), 1.0)):
        buf = torch.from_numpy(x).cuda()
        S.sepw_image(ctx, direction, buf)
        assert rel_l2(buf.cpu().numpy() / flat, want / flat) <= TOL, direction
    # a point in the grid: every frequency of one row and column pair
    p = np.zeros((N, N), np.complex64)
    p[N // 2 + 3, N // 2 - 5] = 1.0
    buf = torch.from_numpy(p).cuda()
    S.sepw_image(ctx, S.GRID_TO_IMAGE, buf)
    assert np.max(np.abs(buf.cpu().numpy() / corr - _to_image(p))) <= 1e-5


@pytest.mark.parametrize("N", [500, 512, 1024, 2048])
@pytest.mark.parametrize("layout", ["apart", "unaligned", "in_place"])
def test_wstack_directions(env, N, layout):
    """Slices to image and image to slices, with slice grids off 16-byte
    boundaries and with the image inside them (the general path)."""
    torch, S = env
    fov, L = math.radians(2.0), 3
    ctx = S.sepw_create(S.make_params(N, fov, 4, 4, 3, 500.0))
    centres = [-900.0, 10.0, 800.0]
    z = torch.zeros(1, dtype=torch.float64, device="cuda")
    S.sepw_wstack_plan(ctx, centres, z, z, z)
    n, corr = _terms(N, 4, fov)
    rng = np.random.default_rng(N)
    g = _random(rng, L, N, N)
    buf = torch.empty(L * N * N + 1, dtype=torch.complex64, device="cuda")
    grids = (buf[1:] if layout == "unaligned" else buf[:-1]).view(L, N, N)
    grids.copy_(torch.from_numpy(g))
    image = grids[0] if layout == "in_place" else torch.empty((N, N), dtype=torch.complex64,
                                                              device="cuda")
    S.sepw_wstack_image(ctx, grids, image)
    ph = [np.exp(2j * np.pi * w * (n - 1.0)) for w in centres]
    want = sum(ph[c] * _to_image(g[c]) for c in range(L))
    assert rel_l2(image.cpu().numpy() / corr, want) <= TOL
    x = _random(rng, N, N)
    image.copy_(torch.from_numpy(x))
    S.sepw_wstack_model_grids(ctx, image, grids)
    want = np.stack([_to_grid(x * np.conj(ph[c]) * corr / n ** 2) for c in range(L)])
    assert rel_l2(grids.cpu().numpy(), want) <= TOL


@pytest.mark.parametrize("warm,direction", [
    (None, "GRID_TO_IMAGE"), ("IMAGE_TO_GRID", "GRID_TO_IMAGE"),
    ("IMAGE_TO_GRID", "IMAGE_TO_GRID_ADJOINT"), ("GRID_TO_IMAGE", "IMAGE_TO_GRID")])
def test_first_call_in_a_direction_can_be_captured(env, warm, direction):
    """One call in any direction (towards the image: none) is all that a capture
    in another one needs."""
    torch, S = env
    N = 512
    ctx = S.sepw_create(S.make_params(N, math.radians(3.0), 4, 3, 2, 100.0))
    if warm:
        S.sepw_image(ctx, getattr(S, warm), torch.zeros((N, N), dtype=torch.complex64,
                                                        device="cuda"))
    d = getattr(S, direction)
    buf = torch.zeros((N, N), dtype=torch.complex64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        S.sepw_image(ctx, d, buf)
    x = torch.from_numpy(_random(np.random.default_rng(4), N, N)).cuda()
    buf.copy_(x)
    graph.replay()
    want = x.clone()
    S.sepw_image(ctx, d, want)
    assert torch.equal(torch.view_as_real(buf), torch.view_as_real(want))


def test_first_wstack_image_can_be_captured(env):
    torch, S = env
    N = 512
    ctx = S.sepw_create(S.make_params(N, math.radians(3.0), 4, 3, 2, 100.0))
    u = torch.zeros(4, dtype=torch.float64, device="cuda")
    S.sepw_wstack_plan(ctx, [-50.0, 50.0], u, u, u)
    g = torch.zeros((2, N, N), dtype=torch.complex64, device="cuda")
    image = torch.zeros((N, N), dtype=torch.complex64, device="cuda")
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        S.sepw_wstack_image(ctx, g, image)
    x = torch.from_numpy(_random(np.random.default_rng(5), 2, N, N)).cuda()
    g.copy_(x)
    graph.replay()
    got = image.clone()
    S.sepw_wstack_image(ctx, x, image)
    assert torch.equal(torch.view_as_real(got), torch.view_as_real(image))
