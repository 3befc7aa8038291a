"""Kernels issued to a stream without any wait between them (each placed while
the one before still runs) give what the same calls give with the device idle in
between: parameters written by a PyTorch kernel just before the call, every
output read by one just after it, on the default and on a side stream, eagerly
and captured.  The forward outputs are bit-identical (no float atomics there)."""
import pytest

torch = pytest.importorskip("torch")

from paper_2603_09277_gb300 import scenes
from paper_2603_09277_gb300.rasterize import Rasterizer, scene_to_device, targets_to_device

pytestmark = pytest.mark.gpu


def _pass(r, p, base, target, shift, wait):
    w = torch.cuda.synchronize if wait else (lambda: None)
    p["means"].copy_(base + shift)
    w()
    r.preprocess(p)
    w()
    r.bin_sort(sync=False)
    w()
    r.render_fwd()
    w()
    r.loss(target, scenes.GAMMA, lam=0.2)
    w()
    r.render_bwd(p)
    w()
    return [t.clone() for t in (r.image, r.final_T, r.entropy, r.last_idx, r.loss_dev,
                                r.dL_dimage, r.tile_ranges)], r.grads["means"].clone()


@pytest.mark.parametrize("side", [False, True])
def test_back_to_back_is_one_at_a_time(side):
    scene, cams, targets, prm = scenes.config1()
    r = Rasterizer(cams, prm, scene["means"].shape[0])
    p, target = scene_to_device(scene), targets_to_device(targets)
    base = p["means"].clone()
    r.preprocess(p)
    r.bin_sort()  # sizes the pair buffers
    r.loss(target, scenes.GAMMA, lam=0.2)
    shifts = [0.01 * k for k in range(8)]
    want = [_pass(r, p, base, target, s, True) for s in shifts]
    torch.cuda.synchronize()
    stream = torch.cuda.Stream() if side else torch.cuda.current_stream()
    with torch.cuda.stream(stream):
        got = [_pass(r, p, base, target, s, False) for s in shifts]
    torch.cuda.synchronize()
    graph = torch.cuda.CUDAGraph()
    with torch.cuda.graph(graph):
        out = _pass(r, p, base, target, shifts[-1], False)
    graph.replay()
    torch.cuda.synchronize()
    for a, b in zip(want + [want[-1]], got + [out]):
        for x, y in zip(a[0], b[0]):
            assert torch.equal(x, y)
        # (float atomics: the order of the sums differs)
        assert float((a[1] - b[1]).norm() / a[1].norm()) <= 1e-5
