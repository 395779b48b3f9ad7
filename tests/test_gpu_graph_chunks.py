"""The captured sweep over chunks of unequal size: its last chunk has fewer views than the others,
so that its sorts may use smaller tiles, and more of them, than those of the full chunks.  One
workspace serves all; the score is bit for bit the eager one's."""
import numpy as np
import pytest
import torch

import synthetic
from _helpers import to_device


def compare(g: dict, cams: list, **opts):
    from paper_2501_08174_gb300 import Rasterizer
    r = Rasterizer(0, **opts)
    gd = to_device(g, r.device)
    eager = r.accumulate_contribution(gd, cams)
    graph = r.contribution_graph(gd, cams)
    for _ in range(2):  # the second launch finds the workspace as the first left it
        got = graph.launch()
        r.sync()
        assert torch.equal(got, eager)
    assert float(eager.max()) > 0.1
    graph.close()
    r.close()


def ball(n: int):
    rng = np.random.default_rng(n)
    return synthetic._pack(synthetic.uniform_ball(rng, n, 1.0), synthetic.random_quats(rng, n),
                           synthetic.log_uniform(rng, (n, 2), 0.01, 0.05), rng.uniform(0.1, 0.9, size=n),
                           rng.normal(0.0, 0.3, size=(n, 1, 3)), 0)


def views(count: int, w: int, h: int):
    rng = np.random.default_rng(count)
    return [synthetic.make_camera(p, w, h) for p in synthetic.hemisphere_positions(rng, count, 3.0)]


@pytest.mark.gpu
@pytest.mark.parametrize("persistent", [False, True])
@pytest.mark.parametrize("n,count", [(20_000, 20), (20_000, 27), (50_000, 20), (15_000, 31)])
def test_records_of_a_short_last_chunk(n, count, persistent):
    compare(ball(n), views(count, 61, 47), persistent=persistent)


@pytest.mark.gpu
def test_tiles_of_a_short_last_chunk():
    """480,000 tiles in the first chunk, 210,000 in the second: the queue order's scratch."""
    compare(ball(2_000), views(23, 1600, 1200), tile=(8, 8), persistent=True)
