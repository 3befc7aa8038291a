"""The projection adjoint over scenes whose ids follow space.  Every Gaussian that
a view's blending reached is taken, whatever CTA and word its id falls to: its opacity
gradient is the sum over the views of grad2d's sum of dd, times 1 - sigma, and the
others' is zero, at counts around the words (32), the runs of consecutive ids (128)
and the chunks of a CTA.  Tolerance: three FP32 terms and a product, below 1e-6 of
the terms' magnitudes (1 - sigma is at most 1 and rounds to 2^-24).  And the time does
not depend on the order: a view that touches one range of ids takes at most 1.3 times
what it takes with the same Gaussians at random ids (the same work; the events resolve
2 of some 40 us).  With a chunk of consecutive ids per CTA it was 1.8 times."""
import pytest

torch = pytest.importorskip("torch")

from paper_2603_09277_gb300 import gs, scenes
from paper_2603_09277_gb300.rasterize import Rasterizer

pytestmark = pytest.mark.gpu

KEYS = ("means", "log_scales", "quats", "opacity_logits", "sh")


def _scene(n, seen, scale):
    """The first `seen` Gaussians in front of the cameras, the others behind them."""
    g = torch.Generator(device="cuda").manual_seed(n)
    u = torch.rand(n, 3, generator=g, device="cuda")
    means = torch.stack([3.0 * u[:, 0] - 1.5, 2.0 * u[:, 1] - 1.0, 3.0 + u[:, 2]], 1)
    means[seen:, 2] *= -1.0
    return {"means": means, "log_scales": scale + 0.3 * torch.randn(n, 3, generator=g, device="cuda"),
            "quats": torch.randn(n, 4, generator=g, device="cuda"),
            "opacity_logits": torch.randn(n, generator=g, device="cuda"),
            "sh": 0.2 * torch.randn(n, 16, 3, generator=g, device="cuda")}


def _backward(r, p):
    r.preprocess(p)
    r.bin_sort()
    r.render_fwd()
    r.render_bwd(p, torch.ones_like(r.image), None)
    return {k: v.clone() for k, v in r.grads.items()}


@pytest.mark.parametrize("degree", [0, 2, 3])
@pytest.mark.parametrize("n", [31, 129, 4 * 128 + 1, 152 * 3 * 128 + 129, 152 * 5 * 128 * 2 + 1])
def test_every_reached_gaussian_is_taken(n, degree):
    seen = max(1, n // 16)
    p = _scene(n, seen, -4.0 if n > 1000 else -2.5)
    cams = scenes.yaw_cameras([(97, 75), (150, 90), (64, 64)], [0.0, 5.0, -5.0])
    r = Rasterizer(cams, scenes.params(sh_degree=degree), n)
    for order in (None, torch.randperm(n, device="cuda")):
        q = p if order is None else {k: p[k][order].contiguous() for k in KEYS}
        got = _backward(r, q)["opacity_logits"].double()
        dd = r.grad2d.view(3, n, 12)[:, :, 5].double()
        want = dd.sum(0) * (1.0 - torch.sigmoid(q["opacity_logits"].double()))
        assert int((want != 0).sum()) > (0 if n < 1000 else seen // 4)
        assert bool(((got - want).abs() <= 1e-6 * dd.abs().sum(0)).all())


def test_time_does_not_depend_on_the_order_of_ids():
    n = 1_000_000
    p = _scene(n, 70_000, -5.0)
    order = torch.randperm(n, generator=torch.Generator(device="cuda").manual_seed(1),
                           device="cuda")
    r = Rasterizer([scenes.camera(1237, 822, 1237.0)], scenes.params(sh_degree=3), n)
    times = []
    for q in (p, {k: p[k][order].contiguous() for k in KEYS}):
        ev = [torch.cuda.Event(enable_timing=True) for _ in range(2)]
        for e in ev:
            e.record()
        t = []
        for _ in range(12):
            gs.gs_stage_events(3, *ev)
            _backward(r, q)
            gs.gs_stage_events(3, None, None)
            torch.cuda.synchronize()
            t.append(ev[0].elapsed_time(ev[1]))
        times.append(sorted(t)[len(t) // 2])
    assert times[0] <= 1.3 * times[1], times
