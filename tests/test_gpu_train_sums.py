"""The training loss's sums over pixels, against numpy's FP64 sums of the same FP32
images: sizes of less than a block, odd sizes and several blocks; targets within the
colour range and far outside it (single differences of 1e36: sums past FP32's range),
infinite and NaN ones.  The image is the renderer's own, so only the summation is
compared: the L1 sum is good to 2^-47 per block of samples and FP64 beyond, hence 1e-12
of the sum; the SSIM values are FP32 (11-tap windows, two passes: 40 roundings of
2^-24 amplified by the statistics' cancellation), compared through the oracle's map at
1e-4 of the sum."""
import numpy as np
import pytest

import oracle
import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def scene():
    n = 500
    r = sg.Rng(5)
    mean = np.stack([r.uniform(n, 2.0, 6.0), r.uniform(n, -2.0, 2.0), r.uniform(n, -1.5, 1.5)], 1).astype(np.float32)
    q = np.tile(np.float32([1, 0, 0, 0]), (n, 1))
    return sg.Gaussians(mean, r.uniform(3 * n, 0.05, 0.3).reshape(n, 3).astype(np.float32), q,
                        r.uniform(n, 0.1, 0.8).astype(np.float32),
                        r.uniform(3 * n, -1.0, 1.0).reshape(n, 1, 3).astype(np.float32), 0)


@pytest.mark.parametrize("w,h", [(1, 1), (7, 5), (33, 31), (130, 67)])
def test_loss_sums(w, h):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    g = scene()
    cam = sg.Camera(w, h, 0.8 * w, 0.8 * w, 0.5 * w, 0.5 * h)
    ctx = R.Context(R.reloc_default_config(block_size=1000.0))
    ctx.load_map(g)
    poses = np.stack([sg.pose_from_xyz_yaw(x, 0.1, 0.0, 0.0) for x in (0.0, 0.5)])
    rgb = torch.empty((2, 3, h, w), device="cuda:0")
    ctx.render([(0, g.n)], poses, cam, rgb=rgb)
    C = rgb.cpu().numpy()
    tg = sg.Rng(w * h).uniform(C.size).reshape(C.shape).astype(np.float32)
    grad = torch.zeros((14, g.n), device="cuda:0")

    def loss(target, lam):
        grad.zero_()
        return ctx.train_grad([(0, g.n)], poses, cam, torch.tensor(target, device="cuda:0"), grad, lambda_dssim=lam,
                              w_reproj=0.0)

    def l1(target):
        return float(np.abs((C - target).astype(np.float64)).mean())

    far = tg.copy()
    far.reshape(-1)[::3] = np.float32(1e36)
    for t in (tg, far):
        assert abs(loss(t, 0.0) - l1(t)) <= 1e-12 * l1(t)
    inf, nan = tg.copy(), tg.copy()
    inf.reshape(-1)[0] = np.inf
    nan.reshape(-1)[-1] = np.nan
    assert loss(inf, 0.0) == np.inf and np.isnan(loss(nan, 0.0)) and np.isnan(loss(nan, 0.2))
    dssim = float(np.mean([1.0 - oracle.ssim_map(C[v, ch].astype(np.float64), tg[v, ch].astype(np.float64))
                           for v in range(2) for ch in range(3)]))
    want = 0.8 * l1(tg) + 0.2 * dssim
    assert abs(loss(tg, 0.2) - want) <= 1e-4 * want
    ctx.close()
