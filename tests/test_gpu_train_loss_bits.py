"""The training loss's L1 sum carries FP64 from the first addition: against the exact sum
of the same FP32 differences.  All terms are positive, so the relative error is at most
2^-53 for each addition on the longest path (8 samples of a thread, 5 butterfly steps,
8 warps, the blocks' adds) and for the two roundings of the scale.  Samples of a wide
range, where a sum in pairs of FP32 would lose some seven bits to that."""
import math

import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("w,h", [(33, 31), (130, 67)])
def test_l1_sum_is_fp64(w, h):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    n = 300
    r = sg.Rng(8)
    mean = np.stack([r.uniform(n, 2.0, 6.0), r.uniform(n, -2.0, 2.0), r.uniform(n, -1.5, 1.5)], 1).astype(np.float32)
    g = sg.Gaussians(mean, np.full((n, 3), 0.2, np.float32), np.tile(np.float32([1, 0, 0, 0]), (n, 1)),
                     np.full(n, 0.5, np.float32), r.uniform(3 * n).reshape(n, 1, 3).astype(np.float32), 0)
    cam = sg.Camera(w, h, 0.8 * w, 0.8 * w, 0.5 * w, 0.5 * h)
    ctx = R.Context(R.reloc_default_config(block_size=1000.0))
    ctx.load_map(g)
    pose = sg.pose_from_xyz_yaw(0.0, 0.1, 0.0, 0.0)[None]
    rgb = torch.empty((1, 3, h, w), device="cuda:0")
    ctx.render([(0, n)], pose, cam, rgb=rgb)
    C = rgb.cpu().numpy()
    grad = torch.zeros((14, n), device="cuda:0")
    bound = (8 + 5 + 8 + math.ceil(C.size / 2048) + 2) * 2.0 ** -53
    for seed in range(16):
        t = np.exp(sg.Rng(seed).uniform(C.size, -4.0, 12.0)).reshape(C.shape).astype(np.float32)
        got = ctx.train_grad([(0, n)], pose, cam, torch.tensor(t, device="cuda:0"), grad, lambda_dssim=0.0, w_reproj=0.0)
        want = math.fsum(np.abs(C - t).astype(np.float64).ravel().tolist()) / C.size
        assert abs(got - want) <= bound * want, (seed, (got - want) / want, bound)
    ctx.close()
