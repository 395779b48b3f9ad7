"""A look-back that is given up is replaced by counting the earlier items.  The library is built once
more with a spin limit of 0, which gives up every one, and must render the same bits: small and
large sort tiles, the queue orders, and the scan of the open tiles of a two-pass render."""
import glob
import os
import subprocess
import sys

import pytest
import torch

from paper_2501_08174_gb300 import build

HERE = os.path.dirname(os.path.abspath(__file__))


def results() -> list:
    """Planes, scores and gradients of a few renders (the caller chooses the library)."""
    import synthetic
    from _helpers import to_device
    from paper_2501_08174_gb300 import Rasterizer
    out = []
    for n, tile, persistent in ((3_000, (16, 16), False), (60_000, (8, 8), True), (60_000, (16, 16), False)):
        sc = synthetic.config4(seed=9, n=n, n_views=5, resolutions=((157, 93), (333, 251)))
        sc["cameras"] = [dict(c, width=333, height=251) for c in sc["cameras"]]
        r = Rasterizer(0, tile=tile, persistent=persistent)
        g = to_device(sc["gaussians"], r.device)
        score = torch.zeros(n, device=r.device)
        planes, st = r.render(g, sc["cameras"], score=score)
        assert persistent is False or r.stats()["n_tiles"] > 4096  # more than one tile of the open scan
        st.release()
        out += [planes["rgb"], planes["alpha"], planes["depth"], planes["normal"], score,
                r.accumulate_contribution(g, sc["cameras"])]
        graph = r.contribution_graph(g, sc["cameras"])
        out.append(graph.launch().clone())
        r.sync()
        graph.close()
        r.close()
    return [t.cpu() for t in out]


@pytest.mark.gpu
def test_no_result_depends_on_a_wait(tmp_path):
    objs = [build._compile(s, [], False) for s in sorted(glob.glob(os.path.join(build.CSRC, "*.cu")))
            if not s.endswith("sort.cu")]
    sort, lib, got = str(tmp_path / "sort.o"), str(tmp_path / "libocgs_nowait.so"), str(tmp_path / "got.pt")
    subprocess.run([build.nvcc(), *build.ARCH, *build.NVCC_FLAGS, "-DOCGS_SPIN_LIMIT=0", "-c",
                    os.path.join(build.CSRC, "sort.cu"), "-o", sort], check=True)
    subprocess.run([build.nvcc(), *build.ARCH, "-shared", "-o", lib, sort, *objs], check=True)
    code = ("import sys, torch; from paper_2501_08174_gb300 import _lib; _lib.LIB_PATH = sys.argv[1]; "
            "import test_gpu_given_up_waits as t; torch.save(t.results(), sys.argv[2])")
    env = dict(os.environ, PYTHONPATH=os.pathsep.join([os.path.dirname(HERE), HERE]))
    subprocess.run([sys.executable, "-c", code, lib, got], check=True, env=env, timeout=300)
    want = results()
    have = torch.load(got)
    assert len(want) == len(have)
    for a, b in zip(want, have):
        assert torch.equal(a, b)
