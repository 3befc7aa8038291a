"""A grid barrier of the one-launch sort whose wait runs out (the bounds-checked
debug build, with the wait shortened to no read at all, so that every block gives
up at its first barrier): GS_ERR_TIMEOUT as the return value or, without a
synchronisation, in the status word; no pairs, empty ranges; nothing hangs, and the
next call with the usual wait is whole again.  Up to 32,768 rows the barriers are
the hardware's and do not wait that way."""
import os
import subprocess
import sys

import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

CHILD = r'''
import torch
from paper_2603_09277_gb300 import gs, scenes
from paper_2603_09277_gb300.rasterize import Rasterizer, scene_to_device

polls = gs._lib.gs_debug_sort_polls

def lists(n):
    scene, cams, _, prm = scenes.config1(n=n)
    r = Rasterizer(cams, prm, n)
    r.preprocess(scene_to_device(scene))
    P = r.bin_sort()
    assert P > 0
    return r, P, r.tile_ranges.clone(), r.sorted_vals[:P].clone()

def whole(r, P, ranges, vals, sync):
    r.tile_ranges.fill_(-1)
    r.bin_sort(sync=sync)
    assert int(r.status_dev) == gs.GS_OK and int(r.num_pairs_dev) == P
    assert torch.equal(r.tile_ranges, ranges) and torch.equal(r.sorted_vals[:P], vals)

case = lists(32769)
r = case[0]
for sync in (True, False):
    polls(0)
    r.tile_ranges.fill_(-1)
    try:
        r.bin_sort(sync=sync)
        assert not sync, "no error"
    except gs.GsError as e:
        assert sync and e.status == gs.GS_ERR_TIMEOUT, e
    torch.cuda.synchronize()
    assert int(r.status_dev) == gs.GS_ERR_TIMEOUT
    assert int(r.num_pairs_dev) == 0 and int(r.tile_ranges.abs().sum()) == 0
    r.render_fwd()
    assert float(r.image.abs().max()) == 0.0 and float(r.final_T.min()) == 1.0
    polls(-1)
    whole(*case, sync=sync)
case = lists(32768)
polls(0)
whole(*case, sync=True)
whole(*case, sync=False)
print("time-out reported")
'''


def test_a_barrier_that_runs_out_is_reported():
    from paper_2603_09277_gb300 import build
    env = dict(os.environ, GS_LIBRARY=build.build(debug=True))
    r = subprocess.run([sys.executable, "-c", CHILD], env=env, cwd=ROOT, capture_output=True,
                       text=True, timeout=900)
    assert r.returncode == 0, r.stdout[-2000:] + r.stderr[-4000:]
    assert "time-out reported" in r.stdout
