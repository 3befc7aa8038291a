"""The blending kernels' per-warp blocks: 8x4, 8x8 and 8x16 pixels (1, 2 and 4
pixels per thread).  A list entry is left out of a warp's walk where no pixel
of its block can pass the alpha test; whatever the block shape, a pixel meets
the same entries, so the forward outputs agree bit for bit and the gradients to
the rounding of their sums.  Scenes of needles, discs of many tiles and points,
at image sizes that cut the tiles' blocks."""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def _scene(n, seed):
    from paper_2603_09277_gb300 import scenes
    s = scenes.box_scene(n, seed, ls_mean=-3.0)
    rng = np.random.default_rng(seed + 1)
    kind = rng.integers(0, 4, n)
    ls = s["log_scales"]
    ls[kind == 0] = [-1.0, -7.0, -7.0]   # needles
    ls[kind == 1] = [-1.2, -1.5, -6.0]   # discs over many tiles
    ls[kind == 2] = -7.0                 # points (the dilation alone)
    return s


@pytest.mark.parametrize("tile,ppts", [(16, (1, 2, 4)), (8, (1, 2))])
@pytest.mark.parametrize("w,h", [(1, 1), (9, 70), (56, 41), (250, 133)])
def test_block_shapes_agree(tile, ppts, w, h):
    from paper_2603_09277_gb300 import scenes
    from paper_2603_09277_gb300.rasterize import Rasterizer, scene_to_device, targets_to_device
    scene = _scene(600, w)
    cams = [scenes.camera(w, h, max(w, 32))]
    tgt = targets_to_device(scenes.noise_targets(cams, 3))
    p = scene_to_device(scene)
    out = []
    for ppt in ppts:
        r = Rasterizer(cams, scenes.params(tile=tile), 600, pixels_per_thread=ppt)
        r.step(p, tgt, scenes.GAMMA)
        out.append((r.image.clone(), r.final_T.clone(), r.last_idx.clone(), r.entropy.clone(),
                    {k: v.clone() for k, v in r.grads.items()}))
    assert float(out[0][0].abs().max()) > 0.0
    for o in out[1:]:
        for a, b in zip(out[0][:4], o[:4]):
            assert torch.equal(a, b)
        for k, a in out[0][4].items():
            # sums of up to w h FP32 terms in another order; the moments of needles
            # cancel to a few per cent of their terms
            tol = 1e-4 * float(a.norm()) + 1e-12
            assert float((a - o[4][k]).norm()) <= tol, k


def test_one_pixel_per_thread_is_chosen_for_few_tiles():
    """The library's own choice (0) gives the outputs of the stated ones, on
    both sides of its lines (456 and 608 tiles)."""
    from paper_2603_09277_gb300 import scenes
    from paper_2603_09277_gb300.rasterize import Rasterizer, scene_to_device
    p = scene_to_device(_scene(300, 5))
    for tx in (456, 457, 608, 609):
        cams = [scenes.camera(16 * tx - 3, 16, 600)]
        r = [Rasterizer(cams, scenes.params(), 300, pixels_per_thread=k) for k in (0, 2)]
        for x in r:
            x.preprocess(p)
            x.bin_sort()
            x.render_fwd()
        assert torch.equal(r[0].image, r[1].image) and torch.equal(r[0].last_idx, r[1].last_idx)
