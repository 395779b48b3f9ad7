"""Renders of more than 2^24 tiles: the tile sort's keys have 25 bits (four digits of 7)."""
import numpy as np
import pytest
import torch

import synthetic
from _helpers import to_device


@pytest.mark.gpu
@pytest.mark.parametrize("persistent", [False, True])
def test_sweep_over_more_than_2_24_tiles(persistent):
    """16 views of 8193x8192 have 16,793,600 tiles of 8x8; no result depends on the tile."""
    from paper_2501_08174_gb300 import Rasterizer
    rng = np.random.default_rng(5)
    n = 300
    g = synthetic._pack(synthetic.uniform_ball(rng, n, 1.0), synthetic.random_quats(rng, n),
                        synthetic.log_uniform(rng, (n, 2), 0.01, 0.05), rng.uniform(0.1, 0.9, size=n),
                        rng.normal(0.0, 0.3, size=(n, 1, 3)), 0)
    cams = [synthetic.make_camera(p, 8193, 8192) for p in synthetic.hemisphere_positions(rng, 16, 3.0)]
    scores = []
    for tile in ((8, 8), (16, 16)):
        r = Rasterizer(0, tile=tile, persistent=persistent)
        scores.append(r.accumulate_contribution(to_device(g, r.device), cams))
        r.sync()
        tiles = r.stats()["n_tiles"]
        r.close()
        if tile == (8, 8):
            assert tiles > 2 ** 24
    assert torch.equal(scores[0], scores[1]) and float(scores[0].min()) > 0.05
