"""The autotuner on a render of few tiles, where several candidates come to the same launches."""
import pytest
import torch

import synthetic
from _helpers import to_device

SHAPES = [((16, 16), 4), ((16, 16), 2), ((16, 8), 4), ((16, 8), 2), ((8, 8), 2), ((32, 8), 2), ((16, 16), 1)]


@pytest.mark.gpu
def test_equal_launches_are_timed_once():
    """60 tiles of 16x16 (120 of 16x8) take one pixel per thread forward, whatever is asked for;
    the plain backward too, the persistent one two for four: 9 of the 14 first candidates differ.
    Among equal ones the larger request is the name kept."""
    from paper_2501_08174_gb300 import Rasterizer
    sc = synthetic.small_scene(802, 1500, 96, 80, degree=1, n_views=2)
    r = Rasterizer(0)
    g, cams = to_device(sc["gaussians"], r.device), sc["cameras"]
    P = 2 * 96 * 80
    score = torch.zeros(1500, device=r.device)
    d = dict(rgb=torch.ones(P, 3, device=r.device), alpha=torch.ones(P, device=r.device))
    all_14 = 0  # kernels of the 14 candidates, three passes each
    for tile, ppt in SHAPES:
        for persistent in (False, True):
            r.set_options(tile=tile, pixels_per_thread=ppt, persistent=persistent)
            before = r.kernel_launches()
            _, st = r.render(g, cams, score=score)
            r.render_backward(st, g, d)
            st.release()
            all_14 += 3 * (r.kernel_launches() - before)
    r.set_options()
    before = r.kernel_launches()
    res = r.autotune(g, cams)
    used = r.kernel_launches() - before
    assert res["n_tried"] >= 14
    if res["persistent"]:  # further candidates: the two-pass split, the batches of its backward
        assert used < 1.5 * all_14 and (res["tile"] != (16, 8) or res["pixels_per_thread"] == 4)
    else:
        assert used < 0.8 * all_14
        assert res["pixels_per_thread"] == (4 if res["tile"] in ((16, 16), (16, 8)) else 2) and res["batch"] == 32
    r.close()
