"""A training gradient does not depend on the order in which the blend's warps add
their sums: repeats of one call on long thin Gaussians that many tiles share.  The
scale and quaternion rows come from the conic's gradients alone, whose sums over the
warps are FP64: their order moves them by 2^-53 of the terms each, and so the FP32
value they are rounded to once in some 2^24 sums; with FP32 sums nearly every entry
differs between repeats.  Bound: one entry in 10^4."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("w,h,views", [(200, 120, 1), (330, 200, 3)])
def test_conic_rows_repeat(w, h, views):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    n = 1500
    r = sg.Rng(3)
    mean = np.stack([r.uniform(n, 4.0, 9.0), r.uniform(n, -2.0, 2.0), r.uniform(n, -1.5, 1.5)], 1)
    scale = np.stack([r.uniform(n, 0.5, 1.5), r.uniform(n, 0.002, 0.01), r.uniform(n, 0.002, 0.01)], 1)
    q = r.normal(4 * n).reshape(n, 4)
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    g = sg.Gaussians(mean.astype(np.float32), scale.astype(np.float32), q.astype(np.float32),
                     r.uniform(n, 0.05, 0.3).astype(np.float32),
                     r.uniform(3 * n, -1.0, 1.0).reshape(n, 1, 3).astype(np.float32), 0)
    cam = sg.Camera(w, h, 0.8 * w, 0.8 * w, 0.5 * w, 0.5 * h)
    ctx = R.Context(R.reloc_default_config(block_size=1000.0))
    ctx.load_map(g)
    poses = np.stack([sg.pose_from_xyz_yaw(0.2 * k, 0.05 * k, 0.0, 0.0) for k in range(views)])
    tg = torch.tensor(r.uniform(views * 3 * h * w).reshape(views, 3, h, w).astype(np.float32), device="cuda:0")
    runs = []
    for _ in range(6):
        grad = torch.zeros((14, n), device="cuda:0")
        ctx.train_grad([(0, n)], poses, cam, tg, grad)
        runs.append(grad.cpu().numpy())
    ctx.close()
    assert (runs[0][3:10] != 0).mean() > 0.5
    for k in range(1, 6):
        assert (runs[k][3:10] != runs[0][3:10]).mean() <= 1e-4
