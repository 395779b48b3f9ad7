"""The image-free pass at every launch shape, on views of enough tiles to take the shape as given,
eager and captured: scores are bit for bit those of one pixel per thread."""
import numpy as np
import pytest
import torch

import synthetic
from _helpers import to_device

SHAPES = [((16, 16), 2, 32), ((16, 16), 4, 32), ((16, 16), 4, 16), ((16, 16), 2, 64), ((16, 16), 4, 64),
          ((16, 8), 4, 32), ((8, 8), 2, 32), ((32, 8), 2, 32)]


@pytest.mark.gpu
@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("axes", [2, 3])
def test_sweep_shapes_at_full_grids(axes, persistent):
    from paper_2501_08174_gb300 import Rasterizer
    rng = np.random.default_rng(axes)
    g = synthetic.object_scene(rng, 20_000, 1)
    if axes == 3:
        g["scale"] = synthetic.log_uniform(rng, (20_000, 3), 0.01, 0.1)
    cams = [synthetic.make_camera((0.2, -3.0, 0.3), 1136, 1136), synthetic.make_camera((2.0, 2.0, 0.9), 801, 1133)]
    want = None
    for tile, ppt, batch in [((16, 16), 1, 32)] + SHAPES:  # 5,041 + 3,621 tiles of 16x16
        r = Rasterizer(0, tile=tile, persistent=persistent, pixels_per_thread=ppt, batch=batch)
        gd = to_device(g, r.device)
        sweep = r.accumulate_contribution if axes == 2 else r.accumulate_contribution_3d
        scores = [sweep(gd, cams)]
        if axes == 2:
            graph = r.contribution_graph(gd, cams)
            scores.append(graph.launch().clone())
            r.sync()
            graph.close()
        r.close()
        want = scores[0] if want is None else want
        assert float(want.max()) > 0.5
        for s in scores:
            assert torch.equal(s, want), (tile, ppt, batch)
