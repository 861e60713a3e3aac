"""Contexts of several host threads: kernels that they share (one function, one
set of attributes per device) are launched by all of them at once."""
import threading

import pytest

import synth

pytestmark = pytest.mark.gpu


def test_plans_of_different_sort_sizes_at_once(  # 8 KB and 32 KB of bins for the sort
):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1511_07152_gb300 import build
    build.build()
    import paper_1511_07152_gb300.sepw as S
    errors = []

    def work(tile, support):
        try:
            wl = synth.random_case(tile, 2000, grid_size=200, support=support, oversample=4,
                                   n_wplanes=3)
            s = torch.cuda.Stream()
            with torch.cuda.stream(s):
                ctx = S.sepw_create(S.make_params(**wl.params(), tile=tile, form=S.FORM_TILED))
                u, v, w = (torch.from_numpy(getattr(wl, k)).cuda() for k in ("u", "v", "w"))
                for _ in range(1500):
                    S.sepw_plan(ctx, u, v, w)
                s.synchronize()
        except Exception as e:  # the first error ends the thread
            errors.append(e)

    threads = [threading.Thread(target=work, args=a) for a in ((16, 8), (56, 8)) * 2]
    for t in threads:
        t.start()
    for t in threads:
        t.join()
    assert not errors, errors
