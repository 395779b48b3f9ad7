"""The pruning compaction at the edges of its blocks (256 Gaussians, 8 blocks per count block),
for every SH degree and for arrays that leave the vector copies unaligned."""
import numpy as np
import pytest
import torch

from _helpers import KEYS

TAU = 0.01


def arrays(n, degree, shift, dev):
    """Parameters whose scale, opacity and sh start `shift` floats into their buffer."""
    rng = np.random.default_rng(n + degree)
    shapes = dict(xyz=(n, 3), quat=(n, 4), scale=(n, 2), opacity=(n,), sh=(n, (degree + 1) ** 2, 3))
    out = {}
    for k, sh in shapes.items():
        off = shift if k in ("xyz", "opacity", "sh") else 0  # quat and scale must be aligned
        buf = torch.empty(int(np.prod(sh)) + off, device=dev)
        v = buf[off:].view(sh)
        v.copy_(torch.tensor(rng.normal(size=sh).astype(np.float32)))
        out[k] = v
    return out


@pytest.mark.gpu
@pytest.mark.parametrize("degree,shift", [(0, 0), (1, 1), (2, 0), (3, 0), (3, 1)])
@pytest.mark.parametrize("n", [1, 255, 256, 257, 2047, 2049, 70_001])
def test_prune_matches_a_boolean_index(n, degree, shift):
    from paper_2501_08174_gb300 import Rasterizer
    rast = Rasterizer(0)
    g = arrays(n, degree, shift, rast.device)
    rng = np.random.default_rng(n)
    score = rng.uniform(0.0, 0.03, size=n).astype(np.float32)
    score[rng.random(n) < 0.1] = np.float32(TAU)            # on the threshold: borderline, not kept
    score[rng.random(n) < 0.05] = np.nan                    # compares false: neither
    s = torch.tensor(score, device=rast.device)
    kept, border, n_border = rast.prune(g, s, TAU, borderline_cap=max(1, n // 20))
    keep = torch.tensor(score > np.float32(TAU), device=rast.device)
    for k in KEYS:
        assert torch.equal(kept[k], g[k][keep]), (k, n)
    want = np.nonzero(np.abs(score - np.float32(TAU)) <= np.float32(1e-6))[0]
    assert n_border == len(want)
    assert np.array_equal(border.cpu().numpy(), want[:max(1, n // 20)])
    rast.close()


@pytest.mark.gpu
@pytest.mark.parametrize("value", [0.0, 1.0])
def test_prune_none_and_all(value):
    from paper_2501_08174_gb300 import Rasterizer
    rast = Rasterizer(0)
    g = arrays(3000, 3, 0, rast.device)
    kept, _, n_border = rast.prune(g, torch.full((3000,), value, device=rast.device), 0.5)
    assert n_border == 0 and kept["xyz"].shape[0] == int(3000 * value)
    for k in KEYS:
        assert torch.equal(kept[k], g[k][:kept[k].shape[0]])
    rast.close()


@pytest.mark.gpu
@pytest.mark.parametrize("n", [524_288, 524_289, 1_300_003])
def test_prune_over_many_count_blocks(n):
    """More than 256 blocks of 2,048: the last block scans several totals per thread."""
    from paper_2501_08174_gb300 import Rasterizer
    rast = Rasterizer(0)
    g = arrays(n, 0, 0, rast.device)
    gen = torch.Generator(device=rast.device).manual_seed(n)
    s = torch.rand(n, generator=gen, device=rast.device)
    s[::1000] = 0.5
    kept, border, n_border = rast.prune(g, s, 0.5, borderline_cap=n)
    for k in KEYS:
        assert torch.equal(kept[k], g[k][s > 0.5]), k
    want = torch.nonzero((s - 0.5).abs() <= 1e-6).reshape(-1)
    assert n_border == len(want) and torch.equal(border, want)
    rast.close()
