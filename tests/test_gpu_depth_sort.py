"""The depth order of a view against numpy's stable sort, through a 16 x 16 image
whose single tile lists every visible Gaussian: sizes at the edges of a warp's
round, of a block's share and of the cluster, one to forty views (the cluster
halves past 32), equal depths, culled Gaussians in between, and more Gaussians
than the cluster path takes (the launch chain per pass).  Whole numbers: equal."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,views", [(1, 1), (31, 1), (33, 3), (513, 1), (2048, 2), (2049, 1), (16385, 9), (40001, 33),
                                     (140_000, 1), (140_003, 12), (600_001, 2), ((1 << 20) + 77, 1)])
def test_depth_order(n, views):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    r = sg.Rng(n)
    # along the optical axis (+x), a third of them behind the camera, depths on a coarse lattice: many ties
    x = np.round(r.uniform(n, -20.0, 40.0) * 512) / 512
    mean = np.stack([x, np.zeros(n), np.zeros(n)], 1).astype(np.float32)
    q = np.tile(np.float32([1, 0, 0, 0]), (n, 1))
    g = sg.Gaussians(mean, np.full((n, 3), 0.01, np.float32), q, np.full(n, 0.5, np.float32),
                     np.full((n, 1, 3), 0.5, np.float32), 0)
    cam = sg.Camera(16, 16, 20.0, 20.0, 8.0, 8.0)
    ctx = R.Context(R.reloc_default_config(block_size=1000.0))
    ctx.load_map(g)
    poses = np.stack([sg.pose_from_xyz_yaw(0.37 * k, 0.0, 0.0, 0.0) for k in range(views)])
    ctx.render([(0, n)], poses, cam, rgb=torch.empty((views, 3, 16, 16), device="cuda:0"))
    k = ctx.last_counts()
    rec = torch.empty((views, n, 12), device="cuda:0")
    rects = torch.empty((views, n, 4), dtype=torch.int32, device="cuda:0")
    lists = torch.empty((views, k.inst_stride), dtype=torch.int32, device="cuda:0")
    count = ctx.export_debug(records=rec, rects=rects, inst_gauss=lists)
    for v in range(views):
        seen = np.nonzero(rects[v, :, 0].cpu().numpy() >= 0)[0]
        depth = rec[v, :, 2].cpu().numpy()[seen]
        want = seen[np.argsort(depth, kind="stable")]
        assert count[v] == len(seen)
        assert np.array_equal(lists[v, :len(seen)].cpu().numpy(), want)
    ctx.close()
