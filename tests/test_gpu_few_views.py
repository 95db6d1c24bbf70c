"""Images of few views (a pixel to a lane, half a 64-pixel block to a warp) against
the same views among four (whole blocks): every tile shape, image sizes that are no
multiple of a block, lists from empty to longer than 1024 records.  The pixel
arithmetic is the same, so the images are equal bit for bit."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("tile", [(16, 16), (8, 8), (32, 8), (16, 8), (8, 16), (32, 16)])
@pytest.mark.parametrize("w,h", [(1, 1), (9, 5), (16, 4), (67, 45), (130, 33)])
def test_few_views_equal_many(tile, w, h):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    n = 6000
    r = sg.Rng(7)
    mean = np.stack([r.uniform(n, 2.0, 9.0), r.uniform(n, -3.0, 3.0), r.uniform(n, -2.0, 2.0)], 1).astype(np.float32)
    q = r.normal(4 * n).reshape(n, 4).astype(np.float32)
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    g = sg.Gaussians(mean, r.uniform(3 * n, 0.02, 0.3).reshape(n, 3).astype(np.float32), q,
                     r.uniform(n, 0.02, 0.6).astype(np.float32), r.uniform(3 * n, -1.0, 1.0).reshape(n, 1, 3).astype(np.float32), 0)
    cam = sg.Camera(w, h, 0.7 * w, 0.7 * w, 0.5 * w, 0.5 * h)
    ctx = R.Context(R.reloc_default_config(block_size=1000.0, tile_w=tile[0], tile_h=tile[1]))
    ctx.load_map(g)
    poses = np.stack([sg.pose_from_xyz_yaw(x, y, 0.0, yaw) for x, y, yaw in
                      ((0.0, 0.0, 0.0), (1.0, 0.5, 0.4), (0.0, 0.0, 2.9), (-1.0, 0.2, -0.3))])

    def images(sel, export):
        out = dict(rgb=torch.empty((len(sel), 3, h, w), device="cuda:0"))
        if export:
            out.update(depth=torch.empty((len(sel), h, w), device="cuda:0"),
                       alpha=torch.empty((len(sel), h, w), device="cuda:0"))
        ctx.render([(0, n)], poses[sel], cam, **out)
        return {k: v.cpu().numpy() for k, v in out.items()}

    for export in (True, False):
        many = images([0, 1, 2, 3], export)
        assert many["rgb"][0].any()
        for sel in ([0], [2, 1], [3, 0, 1]):
            few = images(sel, export)
            for k in few:
                assert np.array_equal(few[k].view(np.int32), many[k][sel].view(np.int32)), (k, sel)
    ctx.close()
