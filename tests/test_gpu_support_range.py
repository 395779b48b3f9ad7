"""Scenes in other units of length.  Multiplying every length by a power of two (positions, scales,
camera translations, near planes; a power of two changes no float32 mantissa) leaves colour,
opacity, normals and scores as they are, bit for bit, and scales depth, Q and the gradients: the
support test that bins the surfels must not leave float32's range before the rest does."""
import numpy as np
import pytest
import torch

import synthetic
from _helpers import KEYS, to_device

W, H = 333, 251  # 336 tiles of 16x16: the backward takes two pixels per thread


def scene():
    rng = np.random.default_rng(77)
    g = synthetic.object_scene(rng, 400, 1)
    # large background surfels, as a room around an object has them
    g["scale"][:60] = synthetic.log_uniform(rng, (60, 2), 0.2, 1.0)
    g["xyz"][:60] *= 2.0
    return g, [synthetic.make_camera((0.2, -5.0, 0.4), W, H), synthetic.make_camera((4.0, 3.0, 1.0), W, H)]


def run(k: float, **opts):
    """Planes, score, sweep and gradients of the scene in units 1 / k, brought back to units of 1."""
    from paper_2501_08174_gb300 import Rasterizer
    g, cams = scene()
    g = {key: np.array(g[key], np.float32) for key in KEYS}
    g["xyz"] = g["xyz"] * np.float32(k)
    g["scale"] = g["scale"] * np.float32(k)
    scaled = []
    for c in cams:
        vm = np.array(c["viewmat"], np.float64)
        vm[:3, 3] *= k
        scaled.append(dict(c, viewmat=vm, near=c["near"] * k))
    r = Rasterizer(0, **opts)
    gd = to_device(g, r.device)
    score = torch.zeros(400, device=r.device)
    out, st = r.render(gd, scaled, score=score, depth2=True)
    P = 2 * W * H
    gen = torch.Generator().manual_seed(4)
    grads = {}
    for planes in (("rgb", "alpha"), ("rgb", "alpha", "normal", "depth", "depth2")):
        d = {p: torch.randn(P, 3, generator=gen) if p in ("rgb", "normal") else torch.randn(P, generator=gen)
             for p in planes}
        for p, f in (("depth", k), ("depth2", k * k)):
            if p in d:
                d[p] /= f
        for key, v in r.render_backward(st, gd, {p: v.to(r.device) for p, v in d.items()}).items():
            grads[(len(planes), key)] = v * k if key in ("xyz", "scale") else v
    st.release()
    sweep = r.accumulate_contribution(gd, scaled)
    r.close()
    out["depth"], out["depth2"] = out["depth"] / k, out["depth2"] / (k * k)
    return dict(out, score=score, sweep=sweep), grads


@pytest.mark.gpu
@pytest.mark.parametrize("opts", [dict(), dict(persistent=True, pixels_per_thread=4)])
def test_results_do_not_depend_on_the_unit_of_length(opts):
    base, base_g = run(1.0, **opts)
    assert float((base["alpha"] > 0.0).float().mean()) > 0.5  # the large surfels reach most pixels
    for exp in (-10, 10, 12, 16):
        out, grads = run(2.0 ** exp, **opts)
        for key in base:
            assert torch.equal(base[key], out[key]), (exp, key)
        for key, want in base_g.items():  # atomics: another order of the sums
            assert (grads[key] - want).abs().max() <= 1e-5 * want.abs().max(), (exp, key)


@pytest.mark.gpu
@pytest.mark.parametrize("opts", [dict(), dict(pixels_per_thread=1), dict(persistent=True, pixels_per_thread=4)])
def test_surfels_far_outside_the_image_have_no_gradient(opts):
    """Finite centres whose projection overflows: they reach no tile, and their gradients are 0."""
    from paper_2501_08174_gb300 import Rasterizer
    rng = np.random.default_rng(3)
    g = synthetic.object_scene(rng, 200, 1)
    g = {key: np.array(g[key], np.float32) for key in KEYS}
    g["xyz"][:, 2] += 3.0
    far = [(1e36, 0.0, 0.5), (3e38, 0.0, 5.0), (0.0, -1e37, 0.5)]
    g["xyz"][:3], g["quat"][:3], g["scale"][:3] = far, (1.0, 0.0, 0.0, 0.0), 0.05
    cam = dict(viewmat=np.eye(4), fx=300.0, fy=300.0, cx=80.0, cy=60.0, width=160, height=120, near=0.2)
    r = Rasterizer(0, **opts)
    gd = to_device(g, r.device)
    _, st = r.render(gd, [cam], depth2=True)
    gen = torch.Generator().manual_seed(4)
    P = 160 * 120
    for planes in (("rgb", "alpha"), ("rgb", "alpha", "normal", "depth", "depth2")):
        d = {p: torch.randn(P, 3, generator=gen) if p in ("rgb", "normal") else torch.randn(P, generator=gen)
             for p in planes}
        grads = r.render_backward(st, gd, {p: v.to(r.device) for p, v in d.items()})
        for key in KEYS:
            assert torch.isfinite(grads[key]).all(), key
            assert (grads[key][:3] == 0).all() and float(grads[key].abs().max()) > 0, key
    st.release()
    r.close()
