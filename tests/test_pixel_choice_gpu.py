"""The library's own choice of pixels per thread: which kernel runs on both sides of
its lines (one pixel up to 608 16-pixel tiles forward and 456 backward, two beyond;
two with 8-pixel tiles and in persistent launches), by the names of the kernels the
profiler sees, and the adjoint there against the stated forms."""
import re

import pytest

torch = pytest.importorskip("torch")

from paper_2603_09277_gb300 import scenes
from paper_2603_09277_gb300.rasterize import Rasterizer, scene_to_device

pytestmark = pytest.mark.gpu


def _pass(r, p):
    r.preprocess(p)
    r.bin_sort()
    r.render_fwd()
    return {k: v.clone() for k, v in r.render_bwd(p, torch.ones_like(r.image), None).items()}


def _forms(r, p):
    """{fwd, bwd: pixels per thread of the kernel that ran}"""
    act = [torch.profiler.ProfilerActivity.CUDA]
    for _ in range(2):  # (the first profile of a process may come back empty)
        with torch.profiler.profile(activities=act) as prof:
            _pass(r, p)
            torch.cuda.synchronize()
    out = {}
    for e in prof.events():
        m = re.search(r"render_(fwd|bwd)_kernel<([^>]*)>", e.name.replace("(int)", ""))
        if m:
            out[m.group(1)] = int(m.group(2).split(",")[2])
    return out


def _scene(n):
    import numpy as np
    s = scenes.box_scene(n, 5, ls_mean=-3.0)
    s["log_scales"][::3] = [-1.2, -1.5, -6.0]  # discs over many tiles
    s["means"] = np.ascontiguousarray(s["means"])
    return scene_to_device(s)


@pytest.mark.parametrize("tiles,kw,fwd,bwd", [
    (1, {}, 1, 1), (456, {}, 1, 1), (457, {}, 1, 2), (608, {}, 1, 2), (609, {}, 2, 2),
    (100, {"tile": 8}, 2, 2), (100, {"persistent": 64}, 2, 2)])
def test_choice(tiles, kw, fwd, bwd):
    tile, pers = kw.get("tile", 16), kw.get("persistent", 0)
    p = _scene(300)
    cams = [scenes.camera(tile * tiles - 3, tile, 600.0)]
    make = lambda ppt: Rasterizer(cams, scenes.params(tile=tile), 300, persistent=pers,
                                  pixels_per_thread=ppt)
    r = make(0)
    ran = _forms(r, p)
    if not ran:
        pytest.skip("the profiler reports no kernels here")
    assert ran == {"fwd": fwd, "bwd": bwd}
    got = _pass(r, p)
    for ppt in (1, 2):
        want = _pass(make(ppt), p)
        for k, v in want.items():
            # sums of FP32 terms in another order
            assert float((got[k] - v).norm()) <= 1e-4 * float(v.norm()) + 1e-12, (k, ppt)
