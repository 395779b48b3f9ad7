"""Every launch shape on a view of enough tiles to be taken as given (renders of few tiles use
fewer pixels per thread than the options ask for), and the sizes around those rules: images and
scores are bit for bit those of one pixel per thread, gradients agree to the rounding of their
sums (1e-5 of each group's largest entry, as for the two binning modes)."""
import numpy as np
import pytest
import torch

import synthetic
from _helpers import KEYS, to_device

SHAPES = [((16, 16), 2, 32), ((16, 16), 4, 32), ((16, 16), 4, 16), ((16, 16), 2, 64), ((16, 16), 4, 64),
          ((16, 8), 2, 32), ((16, 8), 4, 32), ((16, 8), 4, 64), ((8, 8), 2, 32), ((32, 8), 2, 32)]


def scene(w, h, n):
    rng = np.random.default_rng(n)
    return synthetic.object_scene(rng, n, 1), synthetic.make_camera((0.2, -3.0, 0.3), w, h)


def run(g, cam, planes, **opts):
    from paper_2501_08174_gb300 import Rasterizer
    r = Rasterizer(0, **opts)
    gd = to_device(g, r.device)
    score = torch.zeros(g["opacity"].shape[0], device=r.device)
    out, st = r.render(gd, [cam], score=score, depth2=True)
    P = cam["width"] * cam["height"]
    gen = torch.Generator(device="cpu").manual_seed(3)
    d = {k: torch.randn(P, 3, generator=gen) if k in ("rgb", "normal") else torch.randn(P, generator=gen)
         for k in planes}
    grads = r.render_backward(st, gd, {k: v.to(r.device) for k, v in d.items()})
    st.release()
    torch.cuda.synchronize()
    r.close()
    return dict(out, score=score), grads


def same(a, b):
    for k in a[0]:
        assert torch.equal(a[0][k], b[0][k]), k
    for k in KEYS:
        x, y = a[1][k].double(), b[1][k].double()
        assert (x - y).abs().max() <= 1e-5 * y.abs().max(), k


@pytest.mark.gpu
@pytest.mark.parametrize("planes", [("rgb", "alpha"), ("rgb", "alpha", "depth", "normal", "depth2")])
@pytest.mark.parametrize("persistent", [False, True])
def test_shapes_at_full_grids(planes, persistent):
    g, cam = scene(1136, 1136, 20_000)  # 5,041 tiles of 16x16
    base = run(g, cam, planes, tile=(16, 16), persistent=persistent, pixels_per_thread=1)
    for tile, ppt, batch in SHAPES:
        same(run(g, cam, planes, tile=tile, persistent=persistent, pixels_per_thread=ppt, batch=batch), base)


@pytest.mark.gpu
@pytest.mark.parametrize("tiles", [(1, 1), (19, 16), (61, 5), (32, 19), (29, 21), (64, 76), (65, 75)])
def test_shapes_around_the_rules(tiles):
    """304 / 305, 608 / 609 and 4,864 / 4,875 tiles, and a single one, ragged at the edges."""
    g, cam = scene(16 * tiles[0] - 3, 16 * tiles[1] - 5, 4_000)
    base = run(g, cam, ("rgb", "alpha"), pixels_per_thread=1)
    for persistent in (False, True):
        for ppt, batch in ((2, 32), (4, 32), (4, 64)):
            same(run(g, cam, ("rgb", "alpha"), persistent=persistent, pixels_per_thread=ppt, batch=batch), base)
