"""A call that the runtime refuses reports it and leaves nothing behind: later
calls on other streams work.  Refused here: planned calls into a capture that a
synchronisation has ended as invalid (an error of the host API alone)."""
import ctypes

import numpy as np
import pytest

import oracle as O
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("call", ["plan", "grid", "degrid"])
def test_refused_launch_leaves_no_error(call):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_07152_gb300 import build
    build.build()
    import paper_1511_07152_gb300.sepw as sepw
    wl = synth.random_case(3, 5_000, grid_size=128, support=8, oversample=8, n_wplanes=4)
    ctx = sepw.sepw_create(sepw.make_params(**wl.params(), form=sepw.FORM_TILED))
    u, v, w, vis, weight = (torch.from_numpy(getattr(wl, k)).cuda()
                            for k in ("u", "v", "w", "vis", "weight"))
    taps = sepw.sepw_make_taps(ctx)
    grid = torch.zeros((wl.grid_size, wl.grid_size), dtype=torch.complex64, device="cuda")
    out = torch.empty_like(vis)
    sepw.sepw_plan(ctx, u, v, w)
    torch.cuda.synchronize()

    rt = ctypes.CDLL("libcudart.so.13")
    stream = torch.cuda.Stream()
    s = ctypes.c_void_p(stream.cuda_stream)
    assert rt.cudaStreamBeginCapture(s, 2) == 0  # relaxed
    assert rt.cudaStreamSynchronize(s) != 0      # not in a capture, which is invalid from here on
    with pytest.raises(sepw.SepwError):
        if call == "plan":
            sepw.sepw_plan(ctx, u, v, w, stream=stream)
        elif call == "grid":
            sepw.sepw_grid_planned(ctx, taps, vis, weight, grid, stream=stream)
        else:
            sepw.sepw_degrid_planned(ctx, taps, grid, weight, out, stream=stream)
    graph = ctypes.c_void_p()
    assert rt.cudaStreamEndCapture(s, ctypes.byref(graph)) != 0 and not graph.value
    rt.cudaGetLastError()

    got = sepw.sepw_locate(ctx, u, v, w)
    want = O.locate(O.params_from(wl.params()), wl.u, wl.v, wl.w)
    keep = got["keep"].cpu().numpy().astype(bool)
    assert np.array_equal(keep, want["keep"])
    assert np.array_equal(got["cu"].cpu().numpy()[keep], want["cu"][keep])
