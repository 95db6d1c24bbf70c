"""Network inputs of the learned proposal.  Box averages at every scale f (47 f x 176 f
images), from images on 16 bytes and off them, against the same sums in numpy: FP32,
row by row, column by column, (r + g) + b first, one rounding to BF16 at the end, so
the bits are equal.  And calls of more queries than one launch takes (64) against the
same queries alone: equal results."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture(scope="module")
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc
    return reloc


@pytest.mark.parametrize("f", [1, 2, 3, 4, 8, 12])
@pytest.mark.parametrize("shift", [0, 1, 4])
def test_input_bits(R, f, shift):
    h, w = 47 * f, 176 * f
    cam = sg.Camera(w, h, float(w), float(w), 0.5 * w, 0.5 * h)
    images = [sg.random_image(f + 40, 3, h, w).astype(np.float32), sg.random_image(f + 41, 3, h, w).astype(np.float32)]
    dev = []
    for k, img in enumerate(images):
        flat = torch.empty(3 * h * w + 8, device="cuda:0")
        t = flat[shift * (1 - k):][:3 * h * w].view(3, h, w)
        t.copy_(torch.tensor(img))
        dev.append(t)
    out = torch.zeros((47, 176, 2), dtype=torch.int16, device="cuda:0")
    ctx = R.Context()
    ctx.proposal_make_input(dev[0], dev[1], cam, out)
    got = out.cpu().numpy()
    for ch, img in enumerate(images):
        s = np.zeros((47, 176), np.float32)
        for y in range(f):
            for x in range(f):
                r, g, b = img[:, y::f, x::f]
                s += (r + g) + b
        want = torch.tensor(s / np.float32(3 * f * f)).to(torch.bfloat16).view(torch.int16).numpy()
        assert np.array_equal(got[..., ch], want), ch
    ctx.close()


def test_more_queries_than_a_launch(R):
    n, Q = 1500, 67
    r = sg.Rng(3)
    mean = np.stack([r.uniform(n, 4.0, 9.0), r.uniform(n, -3.0, 3.0), r.uniform(n, -1.0, 1.0)], 1).astype(np.float32)
    q = np.tile(np.float32([1, 0, 0, 0]), (n, 1))
    g = sg.Gaussians(mean, r.uniform(3 * n, 0.05, 0.3).reshape(n, 3).astype(np.float32), q,
                     r.uniform(n, 0.1, 0.8).astype(np.float32),
                     r.uniform(3 * n, -1.0, 1.0).reshape(n, 1, 3).astype(np.float32), 0)
    cam = sg.Camera(176, 47, 120.0, 120.0, 88.0, 23.5)
    ctx = R.Context(R.reloc_default_config(block_size=1000.0))
    ctx.load_map(g)
    ctx.proposal_init(seed=8)
    ctx.set_proposal(True, 4, -1.0)
    images = torch.tensor(np.stack([sg.random_image(60 + k, 3, 47, 176) for k in range(Q)]).astype(np.float32), device="cuda:0")
    qs = [(images[k], sg.pose_from_xyz_yaw(0.02 * k, 0.01 * k, 0.0, 0.0), 1e4, (4, 4, 4, 0.5, 2.0)) for k in range(Q)]
    res, sc = ctx.localize_batch(qs, cam)
    for k in (0, 1, 31, 63, 64, 65, 66):
        one, one_sc = ctx.localize_batch([qs[k]], cam)
        assert one[0].best_index == res[k].best_index and one[0].best_score == res[k].best_score
        assert np.array_equal(one_sc[0], sc[k], equal_nan=True) and (~np.isnan(sc[k])).sum() == 4
    ctx.close()
