"""Tile lists of images whose grids sit at the emission's edges: up to 32 tile rows
(the rows' bits) and more (row tests), up to 128 tile columns and more, chunk lengths
that are no multiple of 32 or of 512, rectangles of one tile and of the whole image.
Every list must hold exactly the Gaussians whose exported rectangle covers the tile,
by (depth, index).  Whole numbers: equal."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("w,h", [(16, 16), (40, 512), (40, 528), (2048, 24), (2064, 40)])
@pytest.mark.parametrize("n,views", [(31, 1), (700, 1), (2600, 2)])
def test_lists(w, h, n, views):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    r = sg.Rng(n + w)
    mean = np.stack([r.uniform(n, 3.0, 9.0), r.uniform(n, -4.0, 4.0), r.uniform(n, -4.0, 4.0)], 1)
    q = np.tile(np.float32([1, 0, 0, 0]), (n, 1))
    scale = (10.0 ** r.uniform(3 * n, -3.0, 0.3)).reshape(n, 3)
    g = sg.Gaussians(mean.astype(np.float32), scale.astype(np.float32), q, np.full(n, 0.5, np.float32),
                     np.full((n, 1, 3), 0.5, np.float32), 0)
    cam = sg.Camera(w, h, 0.5 * max(w, h), 0.5 * max(w, h), 0.5 * w, 0.5 * h)
    ctx = R.Context(R.reloc_default_config(block_size=1000.0))
    ctx.load_map(g)
    poses = np.stack([sg.pose_from_xyz_yaw(0.3 * k, 0.1 * k, 0.0, 0.0) for k in range(views)])
    ctx.render([(0, n)], poses, cam, rgb=torch.empty((views, 3, h, w), device="cuda:0"))
    k = ctx.last_counts()
    ntx, nty = (w + 15) // 16, (h + 15) // 16
    rec = torch.empty((views, n, 12), device="cuda:0")
    rects = torch.empty((views, n, 4), dtype=torch.int32, device="cuda:0")
    lists = torch.empty((views, k.inst_stride), dtype=torch.int32, device="cuda:0")
    ranges = torch.empty((views, nty * ntx, 2), dtype=torch.int32, device="cuda:0")
    ctx.export_debug(records=rec, rects=rects, inst_gauss=lists, ranges=ranges)
    rec, rects, lists, ranges = (t.cpu().numpy() for t in (rec, rects, lists, ranges))
    total = 0
    for v in range(views):
        seen = np.nonzero(rects[v, :, 0] >= 0)[0]
        order = seen[np.argsort(rec[v, seen, 2], kind="stable")]
        x0, y0, x1, y1 = rects[v, order].T
        for t in range(nty * ntx):
            y, x = divmod(t, ntx)
            want = order[(x0 <= x) & (x <= x1) & (y0 <= y) & (y <= y1)]
            a, b = ranges[v, t]
            assert np.array_equal(lists[v, a:b], want), (v, t)
            total += len(want)
    assert total == k.n_instances and total > 0
    ctx.close()
