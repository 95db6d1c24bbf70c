"""The workspace of a call does not grow with what the call before it saw: 40 views of
500,000 Gaussians after a view of none take about the memory that they take in a fresh
context (the binning's per-chunk counts are 83 MB at the largest chunks, 660 MB at the
smallest)."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_counts_after_an_empty_view():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    n, views = 500_000, 40
    r = sg.Rng(2)
    mean = np.stack([r.uniform(n, 4.0, 30.0), r.uniform(n, -3.0, 3.0), r.uniform(n, -1.0, 1.0)], 1)
    g = sg.Gaussians(mean.astype(np.float32), np.full((n, 3), 0.01, np.float32),
                     np.tile(np.float32([1, 0, 0, 0]), (n, 1)), np.full(n, 0.1, np.float32),
                     r.uniform(3 * n).reshape(n, 1, 3).astype(np.float32), 0)
    cam = sg.Camera(1408, 376, 552.0, 552.0, 704.0, 188.0)
    see = np.stack([sg.pose_from_xyz_yaw(0.01 * k, 0.0, 0.0, 0.0) for k in range(views)])
    away = sg.pose_from_xyz_yaw(0.0, 0.0, 0.0, np.pi)[None]
    rgb = torch.empty((views, 3, 376, 1408), device="cuda:0")
    used, image = [], []
    for first in (see[:1], away, see[:1], away):      # the first pair: the driver's own allocations
        ctx = R.Context(R.reloc_default_config(block_size=1000.0))
        ctx.load_map(g)
        torch.cuda.synchronize()
        free = torch.cuda.mem_get_info()[0]
        ctx.render([(0, n)], first, cam, rgb=rgb[:1])
        ctx.render([(0, n)], see, cam, rgb=rgb)
        torch.cuda.synchronize()
        used.append(free - torch.cuda.mem_get_info()[0])
        image.append(rgb.clone())
        ctx.close()
    assert used[3] <= used[2] + (128 << 20), used
    assert all(torch.equal(x, image[0]) for x in image)
