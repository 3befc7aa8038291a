"""One pixel per thread: a pixel's gradient that is not finite reaches the Gaussians
this pixel blends, no others (the pixel's warp sums one entry's parts over all of its
lanes).  Large discs that leave out a corner of the image, whose gradient is NaN."""
import pytest

torch = pytest.importorskip("torch")

from paper_2603_09277_gb300 import scenes
from paper_2603_09277_gb300.rasterize import Rasterizer

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("value", [float("nan"), float("inf")])
def test_a_pixel_that_blends_nothing_adds_nothing(value):
    n = 40
    g = torch.Generator(device="cuda").manual_seed(2)
    # (centres within 2 pixels of each other, standard deviations of about 3 pixels)
    means = torch.rand(n, 3, generator=g, device="cuda") * 0.1
    means[:, 0] -= 0.45
    means[:, 2] += 2.0
    p = {"means": means, "log_scales": -1.6 + 0.3 * torch.randn(n, 3, generator=g, device="cuda"),
         "quats": torch.randn(n, 4, generator=g, device="cuda"),
         "opacity_logits": torch.zeros(n, device="cuda"),
         "sh": torch.rand(n, 16, 3, generator=g, device="cuda")}
    r = Rasterizer([scenes.camera(32, 32, 32.0)], scenes.params(), n, pixels_per_thread=1)
    r.preprocess(p)
    r.bin_sort()
    r.render_fwd()
    last = r.last_idx.view(32, 32)
    empty = last == 0
    # a warp takes 8x4 pixels; some block holds both kinds, with more than 24 that blend
    per = (last > 0).view(8, 4, 4, 8).permute(0, 2, 1, 3).reshape(-1, 32).sum(1)
    assert bool(((per > 24) & (per < 32)).any())
    d = torch.ones(32, 32, 3, device="cuda")
    want = {k: v.clone() for k, v in r.render_bwd(p, d.view(-1, 3), None).items()}
    d[empty] = value
    got = r.render_bwd(p, d.view(-1, 3), None)
    for k, v in want.items():
        # (float atomics: the order of the sums differs)
        assert float((got[k] - v).norm()) <= 1e-4 * float(v.norm()), k
