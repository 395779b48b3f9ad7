"""The depth sort at the edges of both of its tile sizes and at the switch between them
(csrc/sort_layout.h): surfels of distinct depths, so that the image and each surfel's score are the
same bits in whatever order the surfels are given.  A record lost, doubled or misplaced at an edge
of a tile shows: every surfel blends (opacities of 0.01 to 0.03), and every record is visible."""
import numpy as np
import pytest
import torch

from _helpers import to_device

SMALL, LARGE, SWITCH = 384 * 4, 384 * 18, 152 * 384 * 4
W, H = 157, 93


def scene(n: int) -> tuple:
    rng = np.random.default_rng(n)
    z = np.float32(2.0) + np.arange(n, dtype=np.float32) * np.float32(2.0 ** -21)  # distinct float32 depths
    x, y = rng.uniform(-0.9, 0.9, n) * z * 0.57, rng.uniform(-0.9, 0.9, n) * z * 0.57 * H / W
    size = 0.05 * min(1.0, (2000.0 / n) ** 0.5) + 0.005
    g = dict(xyz=np.stack([x, y, z], 1), quat=np.tile([1.0, 0.0, 0.0, 0.0], (n, 1)),
             scale=rng.uniform(0.5, 1.0, (n, 2)) * size, opacity=rng.uniform(0.01, 0.03, n),
             sh=rng.normal(0.0, 0.3, (n, 1, 3)))
    f = (W / 2.0) / np.tan(np.radians(30.0))
    cam = dict(viewmat=np.eye(4), fx=f, fy=f, cx=W / 2.0, cy=H / 2.0, width=W, height=H, near=0.2)
    return {k: np.asarray(v, np.float32) for k, v in g.items()}, cam


@pytest.mark.gpu
@pytest.mark.parametrize("n", [SMALL - 1, SMALL, SMALL + 1, 2 * SMALL + 33, SWITCH - 1, SWITCH, SWITCH + 1,
                               34 * LARGE - 1, 34 * LARGE, 34 * LARGE + 1])
def test_any_input_order_gives_the_same_image(n):
    from paper_2501_08174_gb300 import Rasterizer
    g, cam = scene(n)
    r = Rasterizer(0)
    rng = np.random.default_rng(n + 1)
    base = None
    for perm in (np.arange(n), np.arange(n)[::-1], rng.permutation(n)):
        gd = to_device({k: np.ascontiguousarray(v[perm]) for k, v in g.items()}, r.device)
        score = torch.zeros(n, device=r.device)
        out, _ = r.render(gd, [cam], score=score, keep_state=False)
        back = torch.empty_like(score)
        back[torch.tensor(perm.copy(), device=r.device)] = score
        out = dict(out, score=back)
        if base is None:
            base = out
            assert float(back.min()) > 0.0 and float(out["alpha"].max()) < 0.9999  # all blend
        for k in base:
            assert torch.equal(base[k], out[k]), (n, k)
    r.close()
