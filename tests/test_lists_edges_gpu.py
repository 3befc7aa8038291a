"""Per-tile lists of hand-made projections at the edges of the list kernels:
super-tiles of 31..4097 rows (warps, the 64-row writes and the 1024-row segments
with a remainder of one either way), ragged super-tiles at the view's edges,
several views, and views too wide for the packed descriptors.  The reference
walks every rect in (depth, row) order in numpy; lists, ranges and keys are
compared exactly."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _reference(depth, rects, views, N):
    """views: (TX, TY, first tile); returns the lists by tile."""
    T = sum(tx * ty for tx, ty, _ in views)
    lists = [[] for _ in range(T)]
    for row in np.lexsort((np.arange(len(depth)), depth)):
        x0, y0, x1, y1 = rects[row]
        TX, _, off = views[row // N]
        for y in range(y0, y1):
            for x in range(x0, x1):
                lists[off + y * TX + x].append(row)
    return lists


def _check(sizes, N, seed, big, visible=0.9):
    from paper_2603_09277_gb300 import scenes
    from paper_2603_09277_gb300.rasterize import Rasterizer
    rng = np.random.default_rng(seed)
    cams = [scenes.camera(w, h, w) for w, h in sizes]
    views, off = [], 0
    for w, h in sizes:
        tx, ty = -(-w // 16), -(-h // 16)
        views.append((tx, ty, off))
        off += tx * ty
    R = N * len(sizes)
    rects = np.zeros((R, 4), np.int32)
    for row in range(R):
        TX, TY, _ = views[row // N]
        if rng.random() < visible:
            x0, y0 = rng.integers(0, TX), rng.integers(0, TY)
            dx, dy = (1 + rng.integers(0, big) for _ in range(2))
            rects[row] = (x0, y0, min(TX, x0 + dx), min(TY, y0 + dy))
    area = (rects[:, 2] - rects[:, 0]) * (rects[:, 3] - rects[:, 1])
    # few distinct depths: ties go by row
    depth = rng.choice(np.float32([0.5, 1.0, 1.5, 2.25, 7.0, 100.0, 3e4]), R).astype(np.float32)
    r = Rasterizer(cams, scenes.params(), N, keep_debug=True)
    r.depth.copy_(torch.as_tensor(depth))
    r.tiles_touched.copy_(torch.as_tensor(area.astype(np.int32)))
    r.rect.copy_(torch.as_tensor(rects))
    p8 = rects[:, 0] | rects[:, 1] << 8 | rects[:, 2] << 16 | rects[:, 3] << 24
    r.rect8.copy_(torch.as_tensor(p8.astype(np.int64).astype(np.uint32).view(np.int32)))
    P = r.bin_sort(keys=True)
    want = _reference(depth, rects, views, N)
    flat = np.array([x for q in want for x in q], np.int64)
    assert P == flat.size
    ranges = r.tile_ranges.cpu().numpy()
    lens = np.array([len(q) for q in want])
    np.testing.assert_array_equal(ranges[:, 1] - ranges[:, 0], lens)
    starts = np.cumsum(lens) - lens
    np.testing.assert_array_equal(ranges[:, 0], np.where(lens > 0, starts, 0))
    np.testing.assert_array_equal(r.sorted_vals[:P].cpu().numpy(), flat)
    keys = (np.repeat(np.arange(len(want), dtype=np.int64), lens) << 32) | (
        depth.view(np.int32)[flat].astype(np.int64))
    np.testing.assert_array_equal(r.sorted_keys[:P].cpu().numpy(), keys)
    r.sorted_vals.zero_()
    r.bin_sort(sync=False)  # the form without keys and without a host count
    np.testing.assert_array_equal(r.sorted_vals[:P].cpu().numpy(), flat)


@pytest.mark.parametrize("N", [1, 31, 33, 63, 64, 65, 127, 1023, 1025, 4097])
def test_lists_of_one_super_tile(N):
    _check([(128, 128)], N, N, 8, visible=1.0)


@pytest.mark.parametrize("N,sizes,big", [(700, [(272, 150)], 3), (2500, [(272, 150)], 20),
                                         (900, [(1, 1), (200, 129), (16, 640)], 9)])
def test_lists_of_ragged_views(N, sizes, big):
    _check(sizes, N, N + big, big)


def test_lists_of_a_view_too_wide_for_packed_descriptors():
    _check([(16 * 8003 + 5, 40)], 3000, 5, 30)


@pytest.mark.parametrize("lo,hi", [(1.0, 1.0), (1.0, 1.00001), (0.9, 1.1), (0.25, 3e4)])
@pytest.mark.parametrize("N", [1, 1000, 4095, 4097, 152 * 4096, 152 * 4096 + 1, 1 << 21,
                               (1 << 21) + 1])
def test_depth_order_on_both_sides_of_the_one_launch_sort(N, lo, hi):
    """One tile, so that its list is the visible rows by (depth, row): up to 2^21
    rows the sort runs in one launch, above in separate passes; depth ranges of 0
    to 4 digits."""
    from paper_2603_09277_gb300 import scenes
    from paper_2603_09277_gb300.rasterize import Rasterizer
    g = torch.Generator(device="cuda").manual_seed(N)
    r = Rasterizer([scenes.camera(16, 16, 16)], scenes.params(), N, pair_capacity=N)
    u = torch.rand(N, generator=g, device="cuda", dtype=torch.float64)
    depth = (lo * (hi / lo) ** u).float()
    vis = torch.rand(N, generator=g, device="cuda") < 0.7
    r.depth.copy_(depth)
    r.tiles_touched.copy_(vis.int())
    r.rect8.copy_(torch.where(vis, 1 << 16 | 1 << 24, 0))
    rows = torch.nonzero(vis)[:, 0]
    want = rows[torch.argsort(depth[rows], stable=True)]
    for sync in (True, False):
        r.sorted_vals.fill_(-1)
        r.bin_sort(sync=sync)
        assert int(r.num_pairs_dev) == rows.numel() and int(r.status_dev) == 0
        assert torch.equal(r.sorted_vals[:rows.numel()].long(), want)
