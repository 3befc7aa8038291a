"""D-SSIM at the edges of its blocks (32x32 pixels, quarters of 16x16) and on
both sides of the line between one CTA per block and channel and one CTA per
block (1,216 blocks), against a plain FP64 PyTorch form of the same loss.
Tolerances as for the oracle: the loss 1e-5 relative, dL/dC 1e-4 relative in norm
and 1e-4 of its largest entry element by element (FP32 sums of 121 taps: below
121 * 2^-24 = 7e-6 of the terms, times the 1 / (variance + C2) of the quotient)."""
import pytest

torch = pytest.importorskip("torch")

from paper_2603_09277_gb300 import scenes

pytestmark = pytest.mark.gpu


def _ssim64(x, y):
    k = torch.exp(-torch.arange(-5, 6, dtype=torch.float64, device=x.device) ** 2 / (2 * 1.5 ** 2))
    k = k / k.sum()

    def blur(t):
        t = torch.nn.functional.conv2d(t, k.view(1, 1, 1, 11), padding=(0, 5))
        return torch.nn.functional.conv2d(t, k.view(1, 1, 11, 1), padding=(5, 0))

    x, y = (t.permute(2, 0, 1)[:, None] for t in (x, y))
    mx, my = blur(x), blur(y)
    sxx, syy, sxy = blur(x * x) - mx * mx, blur(y * y) - my * my, blur(x * y) - mx * my
    c1, c2 = 0.01 ** 2, 0.03 ** 2
    return ((2 * mx * my + c1) * (2 * sxy + c2)
            / ((mx * mx + my * my + c1) * (sxx + syy + c2))).mean()


@pytest.mark.parametrize("sizes", [
    [(1, 1)], [(15, 17)], [(16, 33)], [(32, 32)], [(33, 31), (48, 65), (17, 16)],
    [(1184, 1024)],    # 37 x 32 = 1,184 blocks: a CTA per channel
    [(1216, 1024)],    # 1,216: the last size of that form
    [(1217, 1024)],    # 1,248: a CTA for the three channels
    [(640, 1000), (641, 999)]])
def test_dssim_blocks(sizes):
    from paper_2603_09277_gb300 import gs
    g = torch.Generator(device="cuda").manual_seed(5)
    cams = gs.make_cameras([scenes.camera(w, h, float(w)) for w, h in sizes])
    P, lam, V = sum(w * h for w, h in sizes), 0.2, len(sizes)
    tgt = torch.rand(P, 3, generator=g, device="cuda")
    img = (tgt + 0.1 * torch.randn(P, 3, generator=g, device="cuda")).clamp_(0, 1)
    ent = torch.zeros(P, device="cuda")
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    dimg, dent = torch.zeros(P, 3, device="cuda"), torch.zeros(P, device="cuda")
    ws = torch.empty(gs.gs_loss_base_workspace_size(cams), dtype=torch.uint8, device="cuda")
    gs.gs_loss_base(img, tgt, ent, cams, lam, 0.0, loss, dimg, dent, ws)
    x = img.double().requires_grad_(True)
    y, ref, p = tgt.double(), 0.0, 0
    for w, h in sizes:
        a, b = x[p:p + w * h].view(h, w, 3), y[p:p + w * h].view(h, w, 3)
        ref = ref + ((1 - lam) * (a - b).abs().mean() + lam * (1 - _ssim64(a, b))) / V
        p += w * h
    ref.backward()
    assert float(loss) == pytest.approx(float(ref.detach()), rel=1e-5)
    d = (dimg.double() - x.grad).abs()
    assert float((dimg.double() - x.grad).norm() / x.grad.norm()) <= 1e-4
    assert float(d.max()) <= 1e-4 * float(x.grad.abs().max())
