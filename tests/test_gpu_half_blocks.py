"""Image launches take half blocks up to 8,512 64-pixel blocks (views times tiles) and whole
ones beyond; a view's image, depth and alpha are the same bits either way, on sizes whose
right and lower tiles are ragged, at every tile shape's number of blocks to a tile, with
lists of over 1024 records, and for the winners that a sweep exports."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def scene():
    n = 6000
    r = sg.Rng(21)
    mean = np.stack([r.uniform(n, 3.0, 12.0), r.uniform(n, -4.0, 4.0), r.uniform(n, -2.0, 2.0)], 1)
    mean[:2000] = np.stack([r.uniform(2000, 4.0, 5.0), r.uniform(2000, -0.2, 0.2), r.uniform(2000, -0.2, 0.2)], 1)
    q = r.normal(4 * n).reshape(n, 4)
    q /= np.linalg.norm(q, axis=1, keepdims=True)
    return sg.Gaussians(mean.astype(np.float32), np.exp(r.uniform(3 * n, -4.0, -1.0)).reshape(n, 3).astype(np.float32),
                        q.astype(np.float32), r.uniform(n, 0.02, 0.9).astype(np.float32),
                        r.uniform(3 * n).reshape(n, 1, 3).astype(np.float32), 0)


@pytest.mark.parametrize("tile", [(16, 16), (8, 8), (32, 8), (16, 8), (8, 16), (32, 16)])
@pytest.mark.parametrize("w,h,views", [(700, 301, 5), (1403, 371, 2), (90, 50, 200)])
def test_views_alone_and_together(tile, w, h, views):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    per = -(-w // tile[0]) * -(-h // tile[1]) * (tile[0] * tile[1] // 64)
    assert per <= 8512 < per * views
    g = scene()
    cam = sg.Camera(w, h, 0.6 * w, 0.6 * w, 0.5 * w, 0.5 * h)
    poses = np.stack([sg.pose_from_xyz_yaw(0.01 * k, 0.02 * k, 0.0, 0.001 * k) for k in range(views)])
    ctx = R.Context(R.reloc_default_config(block_size=1000.0, tile_w=tile[0], tile_h=tile[1]))
    ctx.load_map(g)
    runs = [(0, g.n)]
    all_ = [torch.empty((views, c, h, w), device="cuda:0") for c in (3, 1, 1)]
    ctx.render(runs, poses, cam, rgb=all_[0], depth=all_[1], alpha=all_[2])
    colour = torch.empty((views, 3, h, w), device="cuda:0")
    ctx.render(runs, poses, cam, rgb=colour)
    assert torch.equal(colour, all_[0])
    for k in (0, views - 1):
        one = [torch.empty((1, c, h, w), device="cuda:0") for c in (3, 1, 1)]
        ctx.render(runs, poses[k:k + 1], cam, rgb=one[0], depth=one[1], alpha=one[2])
        for a, b in zip(one, all_):
            assert torch.equal(a[0], b[k])
    ctx.close()


def test_exported_winners():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    g, w, h = scene(), 400, 200                       # 1,300 blocks a winner: eight in whole blocks, one in half
    cam = sg.Camera(w, h, 0.6 * w, 0.6 * w, 0.5 * w, 0.5 * h)
    ctx = R.Context(R.reloc_default_config(block_size=1000.0))
    ctx.load_map(g)
    img = torch.tensor(sg.random_image(9, 3, h, w).astype(np.float32), device="cuda:0")
    qs = [(img, sg.pose_from_xyz_yaw(0.1 * k, 0.0, 0.0, 0.0), 50.0, (2, 2, 2, 0.2, 1.0)) for k in range(8)]
    rgb = torch.empty((8, 3, h, w), device="cuda:0")
    depth = torch.empty((8, h, w), device="cuda:0")
    ctx.localize_batch(qs, cam, best_rgb=rgb, best_depth=depth)
    for k in (0, 7):
        one, d = torch.empty((1, 3, h, w), device="cuda:0"), torch.empty((1, h, w), device="cuda:0")
        ctx.localize_batch(qs[k:k + 1], cam, best_rgb=one, best_depth=d)
        assert torch.equal(one[0], rgb[k]) and torch.equal(d[0], depth[k])
    ctx.close()
