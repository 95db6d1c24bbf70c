"""NCC of large images, whose query sums run in more blocks (one for every 8192 samples past
2.5 million, 2432 at most), against FP64 over the same render and query: the sums of the
render carry 2^-36 of their size and the query's FP64, so scores agree to 1e-9; the gray
values are formed in FP32 (2^-23 each, independent), 1e-7.  And a view scores the same bits
alone and with another query."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("w,h", [(900, 910), (1111, 777), (1920, 1080), (3840, 2160)])
@pytest.mark.parametrize("gray", [0, 1])
def test_scores(w, h, gray):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    g = sg.tiny_scene().gaussians
    cam = sg.Camera(w, h, 0.4 * w, 0.4 * w, 0.5 * w, 0.5 * h)
    pose = sg.pose_from_xyz_yaw(0.0, -14.0, 2.0, np.pi / 2)
    ctx = R.Context(R.reloc_default_config(ncc_gray=gray))
    ctx.load_map(g)
    rgb = torch.empty((1, 3, h, w), device="cuda:0")
    ctx.render([(0, g.n)], pose[None], cam, rgb=rgb)
    gen = torch.Generator(device="cuda:0").manual_seed(w)
    q = rgb[0] * 0.7 + 0.3 * torch.rand((3, h, w), generator=gen, device="cuda:0")
    score, _ = ctx.score([(0, g.n)], pose[None], cam, q)
    a, b = rgb[0].double(), q.double()
    if gray:
        a, b = a.mean(0), b.mean(0)
    a, b = a - a.mean(), b - b.mean()
    want = float((a * b).sum() / (a.square().sum().sqrt() * b.square().sum().sqrt()))
    assert abs(score[0] - want) <= (1e-7 if gray else 1e-9)
    other = torch.rand((3, h, w), generator=gen, device="cuda:0")
    qs = [(x, pose, 40.0, (1, 1, 1, 1.0, 1.0)) for x in (other, q)]
    _, alone = ctx.localize_batch(qs[1:], cam)
    _, both = ctx.localize_batch(qs, cam)
    assert alone[0][0] == both[1][0]
    ctx.close()
