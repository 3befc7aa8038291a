"""The D-SSIM gradient on smooth images close to their targets, where the window
sums cancel most (noise, as the other D-SSIM tests use, hides it): a ramp, a
sinusoid and a constant, across 32x32 blocks and with the last quarter's centre
outside the image.  lambda = 1 leaves the D-SSIM part alone.  Bounds: the error in
norm that an FP32 restatement of five correlations over 16x16 blocks about each
block's first pixel has on these images (the figures below, computed on the CPU),
times 1.25 for the other order and fused products of the kernel's sums."""
import math

import pytest

torch = pytest.importorskip("torch")

from paper_2603_09277_gb300 import scenes
from test_dssim_blocks_gpu import _ssim64

pytestmark = pytest.mark.gpu


def _image(kind, w, h):
    y, x = torch.meshgrid(torch.arange(h, dtype=torch.float64), torch.arange(w, dtype=torch.float64),
                          indexing="ij")
    if kind == "ramp":
        return x, (x / w + y / h) / 2
    if kind == "sin":
        return x, 0.5 + 0.4 * torch.sin(x / 9) * torch.cos(y / 13)
    return x, torch.full_like(x, 0.6)


@pytest.mark.parametrize("w,h,kind,eps,err", [
    (96, 96, "ramp", 1e-2, 3.25e-5), (96, 96, "ramp", 1e-3, 3.45e-4),
    (96, 96, "sin", 1e-2, 7.78e-5), (96, 96, "sin", 1e-3, 7.56e-4),
    (96, 96, "const", 1e-2, 2.79e-5), (96, 96, "const", 1e-3, 2.20e-4),
    (101, 69, "ramp", 1e-2, 4.12e-5), (101, 69, "ramp", 1e-3, 4.07e-4),
    (101, 69, "sin", 1e-2, 8.07e-5), (101, 69, "sin", 1e-3, 7.78e-4),
    (101, 69, "const", 1e-2, 3.38e-5), (101, 69, "const", 1e-3, 2.51e-4)])
def test_smooth_images(w, h, kind, eps, err):
    from paper_2603_09277_gb300 import gs
    x, t = _image(kind, w, h)
    img = (t * (1 - eps) + eps * 0.5 * torch.sin(x / 5)).clamp(0, 1)
    img, t = (v.float()[..., None].expand(h, w, 3).reshape(-1, 3).contiguous().cuda()
              for v in (img, t))
    cams = gs.make_cameras([scenes.camera(w, h, float(w))])
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    dimg, dent = torch.zeros(w * h, 3, device="cuda"), torch.zeros(w * h, device="cuda")
    ws = torch.empty(gs.gs_loss_base_workspace_size(cams), dtype=torch.uint8, device="cuda")
    gs.gs_loss_base(img, t, dent, cams, 1.0, 0.0, loss, dimg, dent.clone(), ws)
    x = img.double().requires_grad_(True)
    (1 - _ssim64(x.view(h, w, 3), t.double().view(h, w, 3))).backward()
    got = float((dimg.double() - x.grad).norm() / x.grad.norm())
    assert math.isfinite(got) and got <= 1.25 * err, got
