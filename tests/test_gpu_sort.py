"""The radix sorts of the binning at the edges of their tiles: a front-to-back image depends on
the depth order of every record and on the tile order of every pair, so an item that is lost,
doubled or misplaced shows in it."""
import numpy as np
import pytest
import torch

import oracle
import synthetic
from _helpers import FWD_TOL, OUT_KEYS, to_device

TILE = 384 * 18  # items of one sort tile


def scene(n: int):
    rng = np.random.default_rng(n)
    g = synthetic._pack(synthetic.uniform_ball(rng, n, 1.0), synthetic.random_quats(rng, n),
                        synthetic.log_uniform(rng, (n, 2), 0.01, 0.1), rng.uniform(0.1, 0.9, size=n),
                        rng.normal(0.0, 0.3, size=(n, 1, 3)), 0)
    return g, synthetic.make_camera((0.3, -3.0, 0.4), 37, 21)


@pytest.mark.gpu
@pytest.mark.parametrize("persistent", [False, True])  # one pass, and two passes of binning
@pytest.mark.parametrize("n", [1, 2, 31, TILE - 1, TILE, TILE + 1, 2 * TILE + 33])
def test_records_around_a_sort_tile(n, persistent):
    from paper_2501_08174_gb300 import Rasterizer
    g, cam = scene(n)
    rast = Rasterizer(0, persistent=persistent)
    out, _ = rast.render(to_device(g, rast.device), [cam], keep_state=False)
    ref = oracle.render(g, cam)
    ok = ~ref["fragile"]
    assert ok.mean() > 0.5
    for k in OUT_KEYS:
        err = np.abs(out[k].double().cpu().numpy() - ref[k])[ok].max()
        assert err <= FWD_TOL, (n, k, err)
    rast.close()


@pytest.mark.gpu
def test_many_sort_tiles_in_one_look_back():
    """Hundreds of sort tiles in flight: the one-pass and the two-pass lists are built by sorts of
    different sizes and render the same bits."""
    from paper_2501_08174_gb300 import Rasterizer
    sc = synthetic.config4(seed=9, n=150_000, n_views=5, resolutions=((157, 93), (333, 251)))
    outs = []
    for front in (0.0, 0.1, 0.37):
        rast = Rasterizer(0, persistent=True, pixels_per_thread=4, front_fraction=front)
        g = to_device(sc["gaussians"], rast.device)
        score = torch.zeros(150_000, device=rast.device)
        out, _ = rast.render(g, sc["cameras"], score=score, keep_state=False)
        outs.append(dict(out, score=score))
        rast.close()
    for o in outs[1:]:
        for k in outs[0]:
            assert torch.equal(outs[0][k], o[k]), k
