"""The projection adjoint takes the rows the blending adjoint marked: a bitmap
over all views' rows, whose words straddle two views wherever the Gaussian
count is not a multiple of 32, read in chunks of Gaussians.  The gradients of a
batch of views are the mean of the single views' gradients (the loss is the
mean over the views), Gaussians that lie behind every pixel's last blended
entry get exact zeros, and the gradient buffers may start off 16-byte
boundaries."""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SIZES = [(50, 40), (96, 64), (33, 70)]
YAWS = [0.0, 9.0, -7.0]


def _grads(scene, cams, tgts, shift=0, attr="f32"):
    from paper_2603_09277_gb300 import gs, scenes
    from paper_2603_09277_gb300.rasterize import Rasterizer, scene_to_device, targets_to_device
    N = scene["means"].shape[0]
    r = Rasterizer(cams, scenes.params(), N, attr_dtype=attr)
    p = scene_to_device(scene)
    r.step(p, targets_to_device(tgts), scenes.GAMMA)
    if not shift:
        return r, {k: v.clone() for k, v in r.grads.items()}
    g = {}
    for k, v in r.grads.items():  # the same call into buffers off by `shift` floats
        o = 0 if k == "quats" else shift  # (16-byte aligned by contract)
        g[k] = torch.full((v.numel() + 8,), float("nan"), device="cuda")[o:o + v.numel()]
    gs.gs_render_bwd(r.proj_c, r.N, r.cams_c, r.prm_c, r.sorted_vals, r.tile_ranges, r.final_T,
                     r.last_idx, r.dL_dimage, r.dL_dentropy, p["means"], p["log_scales"],
                     p["quats"], p["opacity_logits"], p["sh"], r.grad2d, g["means"],
                     g["log_scales"], g["quats"], g["opacity_logits"], g["sh"])
    return r, {k: v.reshape(r.grads[k].shape) for k, v in g.items()}


@pytest.mark.parametrize("attr", ["f32", "bf16"])
@pytest.mark.parametrize("N", [1, 31, 33, 127, 2049, 5000])
def test_batch_is_the_mean_of_its_views(N, attr):
    from paper_2603_09277_gb300 import scenes
    scene = scenes.box_scene(N, N)
    cams = scenes.yaw_cameras(SIZES, YAWS)
    tgts = scenes.noise_targets(cams, 7)
    r, got = _grads(scene, cams, tgts, attr=attr)
    want = None
    for c, t in zip(cams, tgts):
        g = _grads(scene, [c], [t], attr=attr)[1]
        want = g if want is None else {k: want[k] + g[k] for k in g}
    for k in got:
        w = want[k] / len(cams)
        # the same terms, summed in another order over the pixels and the views
        assert float((got[k] - w).norm()) <= 1e-4 * float(w.norm()), k
    _, off = _grads(scene, cams, tgts, shift=1, attr=attr)
    for k in got:
        assert float((got[k] - off[k]).norm()) <= 1e-4 * float(got[k].norm()), k


def test_rows_behind_the_last_blended_entry_get_zeros():
    from paper_2603_09277_gb300 import scenes
    N = 4000
    scene = scenes.box_scene(N, 3, opacity_mean=3.0)
    hidden = torch.arange(N) % 3 == 0
    scene["means"][hidden.numpy(), 2] += 50.0  # visible, behind opaque ones
    scene["means"][hidden.numpy(), :2] *= 0.05
    cams = scenes.yaw_cameras(SIZES[:2], YAWS[:2])
    r, got = _grads(scene, cams, scenes.noise_targets(cams, 8))
    # a row is reached when it stands, in some tile's list, before the last
    # blended entry of one of the tile's pixels
    ranges, vals = r.tile_ranges.cpu(), r.sorted_vals.cpu()
    reached = torch.zeros(2 * N, dtype=torch.bool)
    tile = off = 0
    for c in cams:
        W, H = c["width"], c["height"]
        last = r.last_idx[off:off + W * H].reshape(H, W).cpu()
        off += W * H
        for y in range(0, H, 16):
            for x in range(0, W, 16):
                b = int(ranges[tile, 0])
                reached[vals[b:b + int(last[y:y + 16, x:x + 16].max())].long()] = True
                tile += 1
    reached = reached.reshape(2, N).any(0)
    seen = (r.tiles_touched.reshape(2, N) != 0).any(0).cpu()
    assert bool((seen & hidden & ~reached).any()) and bool(reached.any())
    for k, v in got.items():
        assert bool((v.reshape(N, -1).cpu()[~reached] == 0).all()), k
    # (a reached Gaussian may pass no pixel's alpha test; most do)
    g = got["opacity_logits"].cpu()
    assert bool((g[reached] != 0).any()) and bool(torch.isfinite(g).all())
