"""What a user of the rasterizer has it do, as timed cases over the public entry points.

A case is a dict of plain values.  ``kind`` names the call or the block of calls, ``scene`` the
distribution of the surfels, ``n`` their number, ``degree`` the spherical-harmonics degree,
``sizes`` the views ("640x480*4,800x800*2" is six views), ``tuned`` the launch options: the fastest
configuration the README states, or the defaults of ``Rasterizer``.

``listed()`` gives the fixed cases, ``draw(rng)`` one more of the same ranges, ``prepare`` the state a
program holds before the call (seeded inputs on the GPU), ``run`` one pass, ``work`` the bytes and
operations a pass cannot do without and ``exact`` the results in float64 from plain torch, where that
takes seconds.
"""
from __future__ import annotations

import math

import numpy as np
import torch

from paper_2501_08174_gb300 import PARAM_KEYS, Rasterizer, n_pixels, render

TUNED = dict(tile=(16, 16), persistent=True, pixels_per_thread=4, front_fraction=0.1, batch=32)
GAMMA = 0.5           # background-loss weight
LAMBDA_DSSIM = 0.2    # D-SSIM share of the photometric loss
ALPHA_DIST = 1000.0   # depth-distortion weight
BETA_NORMAL = 0.05    # normal-consistency weight
TAU = 0.01            # pruning threshold
A_MIN = 0.5           # normal consistency counts pixels above this opacity
ADAM_LR = dict(xyz=1.6e-7, quat=1e-6, scale=5e-6, opacity=5e-5, sh=2.5e-6)
RESOLUTIONS = ("640x480", "800x800", "1024x768", "1600x1200")


def _case(name, kind, scene, n, degree, sizes, tuned=True):
    c = dict(kind=kind, scene=scene, n=n, degree=degree, sizes=sizes, tuned=tuned)
    return dict(name=name, **c) if name else c


def listed() -> list:
    mixed = "640x480*4,800x800*4,1024x768*4,1600x1200*4"
    return [
        # the smallest call: a thumbnail of a few surfels with its background loss, default options
        _case("frame_128_2k", "frame", "ball", 2_000, 0, "128x128", tuned=False),
        # one frame of a trained model for a viewer: forward only, no state kept
        _case("frame_1600_500k", "frame", "object", 500_000, 3, "1600x1200"),
        # one view per optimiser step through torch autograd, default options, as the README shows it
        _case("autograd_800_100k", "autograd", "object", 100_000, 3, "800x800", tuned=False),
        # a few crops of odd sizes, every plane and every cotangent, default options
        _case("crops_odd_6k", "backward", "ball", 6_001, 1, "157x93*2,61x203,97x97,33x150", tuned=False),
        # the batched training step: 16 views of uneven resolution, losses, backward, keep-set
        _case("step_500k_16v", "step", "object", 500_000, 3, mixed),
        # render, the loss of Eq. 3 in full and backward over the largest batch of views
        _case("iteration_1m_64v", "iteration", "object", 1_000_000, 3, "1600x1200*64"),
        # the periodic pruning sweep over all training views, then the keep-set
        _case("sweep_300k_100v", "sweep", "shells", 300_000, 3, "800x800*100"),
        # the same record as one captured graph, launched again after the parameters moved
        _case("graph_300k_32v", "graph", "shells", 300_000, 3, "800x800*32"),
        # the pruning record of the 3DGS variant
        _case("sweep3d_500k_16v", "sweep3d", "object", 500_000, 3, mixed),
        # every loss of Eq. 3 with its adjoint on rendered planes
        _case("losses_8v", "losses", "planes", 0, 0, "1600x1200*4,1024x768*3,801x533"),
        # the evaluation of one held-out view: masked PSNR and SSIM
        _case("metrics_1037", "metrics", "planes", 0, 0, "1037x691"),
        # the optimiser update and the pruning of parameters and moments
        _case("update_1m", "update", "object", 1_000_000, 3, "8x8"),
    ]


def _log(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng) -> dict:
    kind = rng.choice(("frame", "autograd", "backward", "step", "iteration", "sweep", "graph", "sweep3d", "losses",
                       "metrics", "update"))
    tuned = rng.random() < 0.7
    if kind == "frame":
        w = _log(rng, 128, 1600)
        return _case(None, kind, "object", _log(rng, 2_000, 500_000), rng.randint(0, 3),
                     f"{w}x{max(1, int(w * rng.uniform(0.6, 1.0)))}", tuned)
    if kind == "autograd":
        w = _log(rng, 200, 1000)
        return _case(None, kind, "object", _log(rng, 5_000, 200_000), rng.randint(0, 3), f"{w}x{_log(rng, 200, 1000)}",
                     tuned)
    if kind == "backward":
        sizes = ",".join(f"{_log(rng, 31, 400)}x{_log(rng, 31, 400)}" for _ in range(rng.randint(1, 6)))
        return _case(None, kind, "ball", _log(rng, 500, 30_000), rng.randint(0, 3), sizes, tuned)
    if kind in ("step", "sweep3d"):
        sizes = ",".join(f"{rng.choice(RESOLUTIONS)}*{rng.randint(1, 4)}" for _ in range(rng.randint(1, 4)))
        return _case(None, kind, "object", _log(rng, 20_000, 500_000), 3, sizes)
    if kind == "iteration":
        sizes = f"{_log(rng, 401, 1600)}x{_log(rng, 301, 1200)}*{_log(rng, 4, 48)}"
        return _case(None, kind, "object", _log(rng, 50_000, 1_000_000), 3, sizes)
    if kind in ("sweep", "graph"):
        side = _log(rng, 200, 800)
        return _case(None, kind, "shells", _log(rng, 50_000, 300_000), rng.randint(0, 3),
                     f"{side}x{side}*{_log(rng, 4, 100 if kind == 'sweep' else 32)}", tuned)
    if kind in ("losses", "metrics"):
        sizes = ",".join(f"{_log(rng, 100, 1600)}x{_log(rng, 100, 1200)}" for _ in range(rng.randint(1, 6)))
        return _case(None, kind, "planes", 0, 0, sizes)
    return _case(None, kind, "object", _log(rng, 10_000, 1_000_000), rng.randint(0, 3), "8x8")


# ----------------------------------------------------------------------------- seeded inputs
def _views(sizes: str) -> list:
    out = []
    for part in sizes.split(","):
        wh, _, count = part.partition("*")
        w, h = wh.split("x")
        out += [(int(w), int(h))] * int(count or 1)
    return out


def _look_at(pos) -> np.ndarray:
    """World->camera matrix (x right, y down, z forward) of a camera at ``pos`` facing the origin."""
    f = -pos / np.linalg.norm(pos)
    up = np.array([0.0, 0.0, 1.0]) if abs(f[2]) < 0.999 else np.array([0.0, 1.0, 0.0])
    x = np.cross(f, up)
    x /= np.linalg.norm(x)
    vm = np.eye(4)
    vm[:3, :3] = np.stack([x, np.cross(f, x), f])
    vm[:3, 3] = -vm[:3, :3] @ pos
    return vm.astype(np.float32).astype(np.float64)


def _cameras(sizes: str, seed: int) -> list:
    """Pinhole cameras of 60 degrees on the upper hemisphere of radius 3."""
    rng = np.random.default_rng(seed)
    cams = []
    for w, h in _views(sizes):
        d = rng.normal(size=3)
        d /= np.linalg.norm(d)
        d[2] = abs(d[2])
        fx = float(np.float32((w / 2.0) / math.tan(math.radians(30.0))))
        cams.append(dict(viewmat=_look_at(3.0 * d), fx=fx, fy=fx, cx=w / 2.0, cy=h / 2.0, width=w, height=h,
                         near=float(np.float32(0.2))))
    return cams


def _gen(seed: int) -> torch.Generator:
    return torch.Generator(device="cuda").manual_seed(seed)


def _sphere(g, n):
    d = torch.randn(n, 3, generator=g, device="cuda")
    return d / d.norm(dim=1, keepdim=True)


def _uni(g, lo, hi, *shape):
    return lo + (hi - lo) * torch.rand(*shape, generator=g, device="cuda")


def _gaussians(case: dict, seed: int, axes: int = 2) -> dict:
    """Surfels (or, with three axes, 3D Gaussians): an object ball with a background shell, a ball
    alone, or closed opaque shells of tangent surfels that hide a cloud."""
    g, n, k = _gen(seed), case["n"], (case["degree"] + 1) ** 2
    quat = torch.randn(n, 4, generator=g, device="cuda")
    quat = quat / quat.norm(dim=1, keepdim=True)
    scale = torch.exp(_uni(g, math.log(0.01), math.log(0.1), n, axes))
    opacity = _uni(g, 0.1, 0.9, n)
    d, u = _sphere(g, n), torch.rand(n, 1, generator=g, device="cuda")
    if case["scene"] == "ball":
        xyz = d * u ** (1 / 3)
    elif case["scene"] == "object":
        inside = torch.arange(n, device="cuda")[:, None] < round(0.7 * n)
        xyz = d * torch.where(inside, 0.8 * u ** (1 / 3), (8.0 + 56.0 * u) ** (1 / 3))
    else:
        m = round(0.6 * n)
        shell = torch.arange(n, device="cuda")[:, None] < m
        layer = torch.arange(n, device="cuda")[:, None] % 3
        xyz = d * torch.where(shell, 1.0 - 0.03 * layer, 0.7 * u ** (1 / 3))
        # tangent surfels: the shortest rotation of +z onto the radial direction
        tangent = torch.stack([1.0 + d[:, 2], -d[:, 1], d[:, 0], torch.zeros_like(d[:, 0])], 1)
        quat = torch.where(shell & (d[:, 2:] > -0.999), tangent, quat)
        size = math.sqrt(180_000 / max(m, 1))  # fewer surfels are larger, so that the shells stay closed
        scale = torch.where(shell, _uni(g, 0.04 * size, 0.06 * size, n, axes), scale)
        opacity = torch.where(shell[:, 0], torch.full_like(opacity, 0.95), opacity)
    sh = 0.2 * torch.randn(n, k, 3, generator=g, device="cuda")
    perm = torch.randperm(n, generator=g, device="cuda")
    return {key: v[perm].contiguous() for key, v in
            dict(xyz=xyz, quat=quat, scale=scale, opacity=opacity, sh=sh).items()}


def _masks(cams, radius: float = 0.8) -> torch.Tensor:
    """The silhouette of a sphere about the origin in every view, concatenated."""
    out = []
    for c in cams:
        x = (torch.arange(c["width"], device="cuda", dtype=torch.float64) + 0.5 - c["cx"]) / c["fx"]
        y = (torch.arange(c["height"], device="cuda", dtype=torch.float64) + 0.5 - c["cy"]) / c["fy"]
        t = c["viewmat"][:3, 3]  # the sphere's centre in the camera frame
        dot = x[None, :] * t[0] + y[:, None] * t[1] + t[2]
        inside = dot * dot >= (x[None, :] ** 2 + y[:, None] ** 2 + 1.0) * float(t @ t - radius * radius)
        out.append((inside & (dot > 0)).to(torch.uint8).reshape(-1))
    return torch.cat(out)


def _planes(cams, seed: int) -> dict:
    """Planes as a render leaves them: an opaque relief on the silhouette, a thin haze beside it."""
    g, P = _gen(seed), n_pixels(cams)
    mask, depth = _masks(cams), []
    for c in cams:
        x = torch.arange(c["width"], device="cuda")[None, :] / c["width"]
        y = torch.arange(c["height"], device="cuda")[:, None] / c["height"]
        depth.append((2.6 + 0.15 * torch.sin(9.0 * x + 2.0 * y) + 0.1 * torch.cos(7.0 * y)).reshape(-1))
    z = torch.cat(depth) + 0.002 * torch.randn(P, generator=g, device="cuda")
    alpha = torch.where(mask > 0, _uni(g, 0.9, 0.9999, P), _uni(g, 0.0, 0.3, P))
    n = torch.randn(P, 3, generator=g, device="cuda") * 0.3 + torch.tensor([0.0, 0.0, -1.0], device="cuda")
    n = n / n.norm(dim=1, keepdim=True)
    spread = _uni(g, 0.0, 0.02, P)
    target = torch.rand(P, 3, generator=g, device="cuda")
    rgb = (target + 0.1 * torch.randn(P, 3, generator=g, device="cuda")).clamp(0.0, 1.0)
    return dict(rgb=rgb, target=target, mask=mask, alpha=alpha, depth=alpha * z,
                depth2=alpha * (z * z + spread * spread), normal=alpha[:, None] * n)


def _zeros(like: dict) -> dict:
    return {k: torch.zeros_like(v) for k, v in like.items()}


# ----------------------------------------------------------------------------- state and one pass
def prepare(case: dict, seed: int) -> dict:
    kind = case["kind"]
    rast = Rasterizer(0, **(TUNED if case["tuned"] else {}))
    cams = _cameras(case["sizes"], seed)
    P = n_pixels(cams)
    s = dict(kind=kind, rast=rast, cams=cams)
    if kind in ("losses", "metrics"):
        s["planes"] = _planes(cams, seed)
        if kind == "losses":
            s["d"] = _zeros({k: s["planes"][k] for k in ("rgb", "alpha", "depth", "depth2", "normal")})
        return s
    s["g"] = _gaussians(case, seed, 3 if kind == "sweep3d" else 2)
    if kind == "update":
        gen = _gen(seed + 1)
        s["grads"] = {k: 1e-4 * torch.randn(v.shape, generator=gen, device="cuda") for k, v in s["g"].items()}
        s["m"] = {k: 1e-4 * torch.randn(v.shape, generator=gen, device="cuda") for k, v in s["g"].items()}
        s["v"] = {k: 1e-8 * torch.rand(v.shape, generator=gen, device="cuda") for k, v in s["g"].items()}
        # three Gaussians in ten were never blended; the keep-set has the same size for every seed
        score = (torch.arange(case["n"], device="cuda") / case["n"] - 0.3).clamp_min(0.0) * 0.9
        s["score"] = score[torch.randperm(case["n"], generator=gen, device="cuda")].contiguous()
        s["t"] = 100
        return s
    if kind in ("sweep", "sweep3d"):
        s["score"] = torch.zeros(case["n"], device="cuda")
        return s
    if kind == "graph":
        s["graph"] = rast.contribution_graph(s["g"], cams)
        return s
    s["mask"] = _masks(cams)
    if kind == "frame":
        return s
    gen = _gen(seed + 1)
    if kind == "backward":
        s["d"] = dict(rgb=torch.randn(P, 3, generator=gen, device="cuda"), alpha=torch.randn(P, generator=gen, device="cuda"),
                      depth=torch.randn(P, generator=gen, device="cuda"),
                      normal=torch.randn(P, 3, generator=gen, device="cuda"),
                      depth2=torch.randn(P, generator=gen, device="cuda"))
        return s
    s["target"] = torch.rand(P, 3, generator=gen, device="cuda")
    if kind == "autograd":
        for v in s["g"].values():
            v.requires_grad_(True)
        return s
    s["score"] = torch.zeros(case["n"], device="cuda")
    s["grads"] = _zeros(s["g"])
    s["d"] = dict(rgb=torch.zeros(P, 3, device="cuda"), alpha=torch.zeros(P, device="cuda"))
    if kind == "iteration":
        s["d"].update(depth=torch.zeros(P, device="cuda"), depth2=torch.zeros(P, device="cuda"),
                      normal=torch.zeros(P, 3, device="cuda"))
    return s


def _eq3(r, out, target, mask, cams, d) -> dict:
    """The loss of Eq. 3, its adjoints added into ``d``."""
    l1 = r.masked_l1(out["rgb"], target, mask, cams, weight=1.0 - LAMBDA_DSSIM, d_rgb=d["rgb"])
    ssim, ssim_m = r.ssim(out["rgb"], target, mask, cams, weight=LAMBDA_DSSIM, d_rgb=d["rgb"])
    ld = r.depth_distortion(out["alpha"], out["depth"], out["depth2"], cams, weight=ALPHA_DIST, grads=d)
    ln = r.normal_consistency(out["alpha"], out["depth"], out["normal"], cams, weight=BETA_NORMAL, a_min=A_MIN, grads=d)
    lb = r.background_loss(out["alpha"], mask, cams, gamma=GAMMA, d_alpha=d["alpha"])
    return dict(l1=l1, ssim=ssim, ssim_masked=ssim_m, distortion=ld, normal=ln, background=lb)


def run(s: dict):
    kind, r, cams = s["kind"], s["rast"], s["cams"]
    if kind == "frame":
        out, _ = r.render(s["g"], cams, keep_state=False)
        return dict(out, background=r.background_loss(out["alpha"], s["mask"], cams, gamma=GAMMA))
    if kind == "autograd":
        rgb, alpha, depth, normal = render(r, s["g"], cams)
        loss = (rgb - s["target"]).abs().mean() + GAMMA * (alpha * (1 - s["mask"])).mean()
        grads = torch.autograd.grad(loss, [s["g"][k] for k in PARAM_KEYS])
        return dict(rgb=rgb.detach(), alpha=alpha.detach(), loss=loss.detach(), grads=list(grads))
    if kind == "backward":
        out, st = r.render(s["g"], cams, depth2=True)
        grads = r.render_backward(st, s["g"], s["d"])
        st.release()
        return dict(out=out, grads=[grads[k] for k in PARAM_KEYS])
    if kind in ("step", "iteration"):
        s["score"].zero_()
        for v in (*s["d"].values(), *s["grads"].values()):
            v.zero_()
        out, st = r.render(s["g"], cams, score=s["score"], depth2=kind == "iteration")
        if kind == "iteration":
            loss = _eq3(r, out, s["target"], s["mask"], cams, s["d"])
        else:
            loss = dict(l1=r.masked_l1(out["rgb"], s["target"], s["mask"], cams, d_rgb=s["d"]["rgb"]),
                        background=r.background_loss(out["alpha"], s["mask"], cams, gamma=GAMMA,
                                                     d_alpha=s["d"]["alpha"]))
        r.render_backward(st, s["g"], s["d"], grads=s["grads"])
        st.release()
        kept, _, _ = r.prune(s["g"], s["score"], TAU)
        # the keep-set's size, not its rows: their number is another for every scene
        return dict(out=out, loss=loss, grads=[s["grads"][k] for k in PARAM_KEYS], score=s["score"],
                    n_kept=kept["xyz"].shape[0])
    if kind == "sweep":
        s["score"].zero_()
        r.accumulate_contribution(s["g"], cams, s["score"])
        kept, _, _ = r.prune(s["g"], s["score"], TAU)
        return dict(score=s["score"], n_kept=kept["xyz"].shape[0])
    if kind == "sweep3d":
        s["score"].zero_()
        return dict(score=r.accumulate_contribution_3d(s["g"], cams, s["score"]))
    if kind == "graph":
        return dict(score=s["graph"].launch())
    if kind == "losses":
        p, d = s["planes"], s["d"]
        for v in d.values():
            v.zero_()
        return dict(loss=_eq3(r, p, p["target"], p["mask"], cams, d), d=d)
    if kind == "metrics":
        p = s["planes"]
        ssim, ssim_m = r.ssim(p["rgb"], p["target"], p["mask"], cams)
        return dict(psnr=r.masked_psnr(p["rgb"], p["target"], p["mask"], cams), ssim=ssim, ssim_masked=ssim_m)
    s["t"] += 1
    r.adam_step(s["g"], s["grads"], s["m"], s["v"], ADAM_LR, step=s["t"])
    kept = [r.prune(x, s["score"], TAU)[0] for x in (s["g"], s["m"], s["v"])]
    return dict(g=[s["g"][k] for k in PARAM_KEYS], m=[s["m"][k] for k in PARAM_KEYS], v=[s["v"][k] for k in PARAM_KEYS],
                kept=[[x[k] for k in PARAM_KEYS] for x in kept])


# ----------------------------------------------------------------------------- work of a pass
def _blends(case: dict) -> float:
    """An estimate of the (pixel, Gaussian) pairs a front-to-back walk has to evaluate: the mean number of
    supports over a pixel of the object, at most the number after which it is opaque."""
    total = 0.0
    for w, h in _views(case["sizes"]):
        f = (w / 2.0) / math.tan(math.radians(30.0))
        # mean of the two scales' product (log-uniform in [0.01, 0.1]), mean |cos| of the facing, 2.4 sigma of support
        area = math.pi * 2.4 ** 2 * (0.09 / math.log(10.0)) ** 2 * 0.5 * (f / 3.0) ** 2
        total += w * h * min(case["n"] * area / (w * h), 60.0)
    return total


def work(case: dict) -> dict:
    kind, n, views = case["kind"], case["n"], _views(case["sizes"])
    P = sum(w * h for w, h in views)
    floats = 10 + 3 * (case["degree"] + 1) ** 2
    par, E = 4 * n * floats, _blends(case) if n else 0.0
    image, q = 32 * P, 4 * P
    losses = {"step": 49 * P + 13 * P, "losses": 0, "iteration": 0}
    eq3 = P * (25 + 24 + 16 + 20 + 4 + 8 * 9)  # images and mask, planes, every adjoint read and written
    if kind == "frame":
        return dict(bytes=par + image + 5 * P, flops=35 * E)
    if kind in ("autograd", "backward"):
        return dict(bytes=3 * par + 2 * image + (0 if kind == "autograd" else 2 * q), flops=135 * E)
    if kind == "step":
        return dict(bytes=4 * par + 2 * image + losses[kind], flops=135 * E)
    if kind == "iteration":
        return dict(bytes=4 * par + 2 * (image + q) + eq3, flops=135 * E + 1000 * P)
    if kind in ("sweep", "sweep3d", "graph"):
        return dict(bytes=par + 4 * n + (2 * par if kind == "sweep" else 0), flops=35 * E)
    if kind == "losses":
        return dict(bytes=eq3, flops=1000 * P)
    if kind == "metrics":
        return dict(bytes=25 * P, flops=400 * P)
    return dict(bytes=7 * par + 3 * 2 * par, flops=15 * n * floats)


# ----------------------------------------------------------------------------- float64 results
def _sh64(d: torch.Tensor, degree: int) -> torch.Tensor:
    """Real spherical harmonics with the Condon-Shortley phase at unit directions, m = -l..l."""
    x, y, z = d.unbind(-1)
    pi = math.pi
    out = [torch.full_like(x, 0.5 / math.sqrt(pi))]
    if degree >= 1:
        a = math.sqrt(3 / (4 * pi))
        out += [-a * y, a * z, -a * x]
    if degree >= 2:
        a, b = math.sqrt(15 / (4 * pi)), math.sqrt(5 / (16 * pi))
        out += [a * x * y, -a * y * z, b * (2 * z * z - x * x - y * y), -a * x * z, a / 2 * (x * x - y * y)]
    if degree >= 3:
        a, b, c = math.sqrt(70 / pi) / 8, math.sqrt(105 / pi) / 2, math.sqrt(42 / pi) / 8
        e, f = math.sqrt(7 / pi) / 4, math.sqrt(105 / pi) / 4
        out += [-a * y * (3 * x * x - y * y), b * x * y * z, -c * y * (4 * z * z - x * x - y * y),
                e * z * (2 * z * z - 3 * x * x - 3 * y * y), -c * x * (4 * z * z - x * x - y * y),
                f * z * (x * x - y * y), -a * x * (x * x - 3 * y * y)]
    return torch.stack(out, -1)


def _project64(p: dict, c: dict, degree: int) -> dict:
    """Splat-to-pixel matrices, colours and normals of the surfels one view can blend, in depth order."""
    vm = torch.tensor(c["viewmat"], dtype=torch.float64, device="cuda")
    R, t = vm[:3, :3], vm[:3, 3]
    w, x, y, z = (p["quat"] / p["quat"].norm(dim=-1, keepdim=True)).unbind(-1)
    tu = torch.stack([1 - 2 * (y * y + z * z), 2 * (x * y + w * z), 2 * (x * z - w * y)], -1) @ R.T
    tv = torch.stack([2 * (x * y - w * z), 1 - 2 * (x * x + z * z), 2 * (y * z + w * x)], -1) @ R.T
    nr = torch.linalg.cross(tu, tv)
    U, V, X = p["scale"][:, :1] * tu, p["scale"][:, 1:] * tv, p["xyz"] @ R.T + t
    nr = torch.where(((nr * X).sum(-1, keepdim=True) > 0), -nr, nr)
    d = p["xyz"] + R.T @ t
    d = d / d.norm(dim=-1, keepdim=True)
    col = ((_sh64(d, degree)[:, :, None] * p["sh"]).sum(1) + 0.5).clamp_min(0.0)
    keep = (X[:, 2] - 3 * (U[:, 2].abs() + V[:, 2].abs()) > c["near"]) & (p["opacity"] >= 1 / 255)
    order = torch.sort(X[:, 2].detach().float(), stable=True).indices
    order = order[keep[order]]
    K = torch.tensor([[c["fx"], 0, c["cx"]], [0, c["fy"], c["cy"]], [0, 0, 1]], dtype=torch.float64, device="cuda")
    T = (K @ torch.stack([U, V, X], -1))[order]
    return dict(T=T, z=X[order, 2], o=p["opacity"][order], col=col[order], n=nr[order])


def _composite64(v: dict, px: torch.Tensor, py: torch.Tensor) -> dict:
    """Front-to-back compositing of the view's surfels at the pixel centres (px, py)."""
    T = v["T"]
    hu = px[:, None, None] * T[None, :, 2] - T[None, :, 0]
    hv = py[:, None, None] * T[None, :, 2] - T[None, :, 1]
    cr = torch.linalg.cross(hu, hv)
    den = torch.where(cr[..., 2] == 0, torch.full_like(cr[..., 2], 1e-300), cr[..., 2])
    u, w = cr[..., 0] / den, cr[..., 1] / den
    rho3 = u * u + w * w
    cx, cy = T[:, 0, 2] / T[:, 2, 2], T[:, 1, 2] / T[:, 2, 2]
    rho2 = 2 * ((px[:, None] - cx) ** 2 + (py[:, None] - cy) ** 2)
    surf = rho3 <= rho2
    rho = torch.where(surf, rho3, rho2)
    alpha = (v["o"] * torch.exp(-rho / 2)).clamp_max(0.99)
    alpha = torch.where((rho <= 9) & (alpha >= 1 / 255), alpha, torch.zeros_like(alpha))
    after = torch.cumprod(1 - alpha, 1)
    stop = torch.cummax(((after < 1e-4) & (alpha > 0)).to(torch.uint8), 1).values > 0
    alpha = torch.where(stop, torch.zeros_like(alpha), alpha)
    after = torch.cumprod(1 - alpha, 1)
    wt = alpha * torch.cat([torch.ones_like(after[:, :1]), after[:, :-1]], 1)
    z = torch.where(surf, u * T[:, 2, 0] + w * T[:, 2, 1] + T[:, 2, 2], v["z"].expand_as(u))
    return dict(rgb=wt @ v["col"], alpha=wt.sum(1), depth=(wt * z).sum(1), normal=wt @ v["n"], depth2=(wt * z * z).sum(1))


def _render64(case: dict, seed: int, d=None):
    """Planes of every view, and the parameter gradients of sum <d, planes> when ``d`` is given."""
    g = _gaussians(case, seed)
    p = {k: v.double().requires_grad_(d is not None) for k, v in g.items()}
    planes, grads, off = [], [torch.zeros_like(p[k]) for k in PARAM_KEYS], 0
    for c in _cameras(case["sizes"], seed):
        n_pix = c["width"] * c["height"]
        chunk = max(32, int(2e7 / case["n"]))
        for lo in range(0, n_pix, chunk):
            i = torch.arange(lo, min(lo + chunk, n_pix), device="cuda")
            with torch.set_grad_enabled(d is not None):
                out = _composite64(_project64(p, c, case["degree"]), (i % c["width"]).double() + 0.5,
                                   torch.div(i, c["width"], rounding_mode="floor").double() + 0.5)
                if d is not None:
                    loss = sum((out[k] * d[k][off + lo:off + lo + len(i)]).sum() for k in d)
                    for a, b in zip(grads, torch.autograd.grad(loss, [p[k] for k in PARAM_KEYS])):
                        a += b
            planes.append({k: v.detach() for k, v in out.items()})
        off += n_pix
    return {k: torch.cat([x[k] for x in planes]) for k in planes[0]}, grads


def _ssim_map64(x1, x2):
    """SSIM map of two [3,H,W] images under an 11x11 Gaussian window of sigma 1.5, zero outside."""
    t = torch.arange(-5, 6, dtype=torch.float64, device="cuda")
    w = torch.exp(-t * t / (2 * 1.5 * 1.5))
    w = w / w.sum()

    def blur(x):
        x = torch.nn.functional.pad(x, (5, 5, 5, 5))
        x = sum(w[i] * x[:, :, i:x.shape[2] - 10 + i] for i in range(11))
        return sum(w[i] * x[:, i:x.shape[1] - 10 + i] for i in range(11))

    m1, m2 = blur(x1), blur(x2)
    v1, v2, v12 = blur(x1 * x1) - m1 * m1, blur(x2 * x2) - m2 * m2, blur(x1 * x2) - m1 * m2
    return ((2 * m1 * m2 + 1e-4) * (2 * v12 + 9e-4)) / ((m1 * m1 + m2 * m2 + 1e-4) * (v1 + v2 + 9e-4))


def _normal64(c, A, D, Nr):
    """Sum over the counted pixels of A - N . Nr, divided by the pixels of the view ([H,W] planes)."""
    H, W = A.shape
    x = (torch.arange(W, device="cuda") + 0.5 - c["cx"]) / c["fx"]
    y = (torch.arange(H, device="cuda") + 0.5 - c["cy"]) / c["fy"]
    ok = A.detach() > np.float32(A_MIN)
    z = D / torch.where(ok, A, torch.ones_like(A))
    Pt = torch.stack([z * x[None, :], z * y[:, None], z], -1)
    dx, dy = Pt[1:-1, 2:] - Pt[1:-1, :-2], Pt[2:, 1:-1] - Pt[:-2, 1:-1]
    counted = ok[1:-1, 1:-1] & ok[1:-1, 2:] & ok[1:-1, :-2] & ok[2:, 1:-1] & ok[:-2, 1:-1]
    n = torch.linalg.cross(dx, dy)
    ln = n.detach().norm(dim=-1)
    counted = counted & (ln > 0)
    n = n[counted] / n[counted].norm(dim=-1, keepdim=True)
    n = torch.where((n * Pt[1:-1, 1:-1][counted]).sum(-1, keepdim=True) > 0, -n, n)
    return (A[1:-1, 1:-1][counted] - (n * Nr[1:-1, 1:-1][counted]).sum(-1)).sum() / (H * W)


def _losses64(case: dict, seed: int):
    cams = _cameras(case["sizes"], seed)
    pl, off = _planes(cams, seed), 0
    names = ("l1", "ssim", "ssim_masked", "distortion", "normal", "background")
    loss, d = {k: [] for k in names}, {k: [] for k in ("rgb", "alpha", "depth", "depth2", "normal")}
    for c in cams:
        H, W = c["height"], c["width"]
        one = {k: v[off:off + H * W].double().reshape(H, W, *v.shape[1:]) for k, v in pl.items()}
        off += H * W
        x = {k: one[k].clone().requires_grad_(True) for k in d}
        m = one["mask"][..., None]
        smap = _ssim_map64((one["target"] * m).permute(2, 0, 1), (x["rgb"] * m).permute(2, 0, 1))
        val = dict(l1=((one["target"] - x["rgb"]) * m).abs().mean(), ssim=smap.mean(),
                   ssim_masked=smap[:, one["mask"] > 0].mean(),
                   distortion=(2 * (x["alpha"] * x["depth2"] - x["depth"] ** 2)).mean(),
                   normal=_normal64(c, x["alpha"], x["depth"], x["normal"]),
                   background=(x["alpha"] * (1 - one["mask"])).mean())
        total = ((1 - LAMBDA_DSSIM) * val["l1"] + LAMBDA_DSSIM * (1 - val["ssim"]) + ALPHA_DIST * val["distortion"]
                 + BETA_NORMAL * val["normal"] + GAMMA * val["background"])
        for k, v in zip(d, torch.autograd.grad(total, list(x.values()))):
            d[k].append(v.reshape(H * W, *v.shape[2:]))
        for k in names:
            loss[k].append(val[k].detach())
    return dict(loss={k: torch.stack(v) for k, v in loss.items()}, d={k: torch.cat(v) for k, v in d.items()})


def _metrics64(case: dict, seed: int):
    cams = _cameras(case["sizes"], seed)
    pl, off = _planes(cams, seed), 0
    out = dict(psnr=[], ssim=[], ssim_masked=[])
    for c in cams:
        H, W = c["height"], c["width"]
        one = {k: pl[k][off:off + H * W].double().reshape(H, W, *pl[k].shape[1:]) for k in ("rgb", "target", "mask")}
        off += H * W
        m = one["mask"] > 0
        smap = _ssim_map64(*((one[k] * m[..., None]).permute(2, 0, 1) for k in ("target", "rgb")))
        out["psnr"].append(-10 * torch.log10(((one["target"] - one["rgb"])[m] ** 2).mean()))
        out["ssim"].append(smap.mean())
        out["ssim_masked"].append(smap[:, m].mean())
    return {k: torch.stack(v) for k, v in out.items()}


def _update64(case: dict, seed: int):
    s = prepare(case, seed)
    t = s["t"] + 1
    new = dict(g=[], m=[], v=[])
    for k in PARAM_KEYS:
        p, gr, m, v = (s[x][k].double() for x in ("g", "grads", "m", "v"))
        m, v = 0.9 * m + 0.1 * gr, 0.999 * v + 0.001 * gr * gr
        new["g"].append(p - ADAM_LR[k] * (m / (1 - 0.9 ** t)) / ((v / (1 - 0.999 ** t)).sqrt() + 1e-15))
        new["m"].append(m)
        new["v"].append(v)
    keep = s["score"] > TAU
    return dict(new, kept=[[x[keep] for x in new[k]] for k in ("g", "m", "v")])


def exact(case: dict, seed: int):
    kind = case["kind"]
    pairs = case["n"] * sum(w * h for w, h in _views(case["sizes"]))
    if kind == "frame" and pairs <= 2e9:
        out, _ = _render64(case, seed)
        mask, lb, off = _masks(_cameras(case["sizes"], seed)).double(), [], 0
        for w, h in _views(case["sizes"]):
            lb.append((out["alpha"][off:off + w * h] * (1 - mask[off:off + w * h])).mean())
            off += w * h
        del out["depth2"]
        return dict(out, background=torch.stack(lb))
    if kind == "backward" and pairs <= 5e8:
        out, grads = _render64(case, seed, prepare(case, seed)["d"])
        return dict(out=out, grads=grads)
    if kind == "losses":
        return _losses64(case, seed)
    if kind == "metrics":
        return _metrics64(case, seed)
    if kind == "update":
        return _update64(case, seed)
    return None  # a float64 render of these sizes takes minutes
