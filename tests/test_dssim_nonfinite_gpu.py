"""A NaN or an infinity in one pixel of the image or the target reaches the D-SSIM
gradient only where the definition takes it: within two window radii (10 pixels), not
over the whole 32x32 block whose constants that pixel would give."""
import pytest

torch = pytest.importorskip("torch")

from paper_2603_09277_gb300 import scenes

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("where", ["image", "target"])
@pytest.mark.parametrize("value", [float("nan"), float("inf")])
@pytest.mark.parametrize("y,x", [(48, 48), (32, 32), (80, 16)])
def test_stays_within_the_windows(where, value, y, x):
    from paper_2603_09277_gb300 import gs
    w = h = 96
    g = torch.Generator(device="cuda").manual_seed(3)
    img, tgt = (torch.rand(h, w, 3, generator=g, device="cuda") for _ in range(2))
    (img if where == "image" else tgt)[y, x, 1] = value
    cams = gs.make_cameras([scenes.camera(w, h, float(w))])
    loss = torch.zeros(1, dtype=torch.float64, device="cuda")
    dimg, dent = torch.zeros(h, w, 3, device="cuda"), torch.zeros(h, w, device="cuda")
    ws = torch.empty(gs.gs_loss_base_workspace_size(cams), dtype=torch.uint8, device="cuda")
    gs.gs_loss_base(img, tgt, dent, cams, 1.0, 0.0, loss, dimg, dent.clone(), ws)
    bad = ~torch.isfinite(dimg)
    assert bool(bad[y, x, 1]) and not bool(bad[..., 0].any() | bad[..., 2].any())
    bad[y - 10:y + 11, x - 10:x + 11] = False
    assert int(bad.sum()) == 0
