"""Map training where every tile's list holds more than 1024 records (the backward
blend hands those out first) beside tiles with short and empty ones: gradients along
random directions against the oracle's derivatives, at the tolerance of the other
training tests (1e-3 of the absolute sum of the terms)."""
import numpy as np
import pytest

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("w,h,views", [(24, 20, 1), (24, 20, 3), (90, 20, 2)])
def test_gradients_of_long_lists(w, h, views):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    n = 2600
    r = sg.Rng(11)
    # a cluster in front of the image's left tiles; a wide image's right tiles see a few Gaussians
    mean = np.stack([r.uniform(n, 6.0, 9.0), r.uniform(n, -0.6, 0.6), r.uniform(n, -0.5, 0.5)], 1)
    mean[:, 1] += np.where(np.arange(n) % 100 == 0, -1.5, 0.0)
    q = r.normal(4 * n).reshape(n, 4)
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    g = sg.Gaussians(mean.astype(np.float32), r.uniform(3 * n, 0.1, 0.5).reshape(n, 3).astype(np.float32),
                     q.astype(np.float32), r.uniform(n, 0.01, 0.05).astype(np.float32),
                     r.uniform(3 * n, -1.0, 1.0).reshape(n, 1, 3).astype(np.float32), 0)
    cam = sg.Camera(w, h, 60.0, 60.0, 12.0, 10.0)
    ctx = R.Context(R.reloc_default_config(block_size=1000.0))
    ctx.load_map(g)
    g = g.subset(ctx.map_order())
    poses = np.stack([sg.pose_from_xyz_yaw(0.2 * k, 0.05 * k, 0.0, 0.0) for k in range(views)])
    tg = r.uniform(views * 3 * h * w).reshape(views, 3, h, w).astype(np.float32)
    grad = torch.zeros((14, n), device="cuda:0")
    ctx.train_grad([(0, n)], poses, cam, torch.tensor(tg, device="cuda:0"), grad, lambda_dssim=0.0, w_reproj=0.0)
    G = grad.cpu().numpy().astype(np.float64)
    ranges = torch.empty((views, ((h + 15) // 16) * ((w + 15) // 16), 2), dtype=torch.int32, device="cuda:0")
    ctx.export_debug(ranges=ranges)
    length = (ranges[..., 1] - ranges[..., 0]).cpu().numpy()
    assert (length >= 1024).sum() >= 4 * views and (w == 24 or (length < 1024).any())
    dirs = (r.u64(n * 14 * 6) % np.uint64(3)).astype(np.float64).reshape(n, 14, 6) - 1.0
    _, jv = oracle.photo_loss_jvp(g, poses, cam, tg.astype(np.float64), dirs)
    for k in range(6):
        terms = G.T * dirs[:, :, k]
        mine, mass = terms.sum(), np.abs(terms).sum()
        print(k, mine, jv[k], mass)
        assert abs(mine - jv[k]) <= 1e-3 * mass + 1e-12
    ctx.close()
