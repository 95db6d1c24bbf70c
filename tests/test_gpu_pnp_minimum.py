"""Where the PnP solve with outliers stops, no step lowers the cost beyond the rounding of
the pairs' own costs.  With D = -g . step / 2 the decrease that the full step promises at
the returned pose (a lower bound of the true one: the quadratic touches the Huber cost from
above), a stop means that the measured change of the cost was not negative: the noise of
the measurement exceeded D.  A pair's cost changes by min(e, k) times its residual's
rounding (1.5 * 2^-53 of the pixel coordinate, image width at least) and by 2^-53 of itself
at each of the two poses; independent over the pairs, so their root sum of squares, taken
four times.  Judging by the summed cost adds the rounding of the whole sum: its ulp is some
twenty times sigma at the larger size."""
import numpy as np
import pytest

import oracle
import scenegen as sg
from pnp_cases import make_pairs, tiny_views
from test_gpu_pnp_halved import cost, gauss_newton, gradient

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n", [9000, 200_000])
def test_stops_at_the_minimum(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    s, Wq, Wr = tiny_views()
    cam, k, ctx = s.camera, 2.0, R.Context()
    for seed in range(8):
        depth, alpha, clean = make_pairs(s, Wq, Wr, step=1)
        pairs = clean[np.arange(n) % len(clean)]
        r = sg.Rng(100 + seed)
        pairs[:, 2:] += 0.3 * r.normal(2 * n).reshape(n, 2)
        out = r.uniform(n) < 0.15
        pairs[out, 2:] = np.stack([r.uniform(n, 0, cam.width), r.uniform(n, 0, cam.height)], 1)[out]
        dev = [torch.tensor(np.ascontiguousarray(x), device="cuda:0") for x in (depth, alpha, pairs)]
        res = ctx.refine_pnp(Wr, cam, *dev, max_iters=100)
        assert res.iters < 100 and res.n_used == n
        X, _ = oracle.pnp_backproject(Wr, cam, depth, alpha, pairs[:, :2].astype(np.float64))
        W, q = np.array(res.pose).reshape(4, 4), pairs[:, 2:].astype(np.float64)
        d, _, c = gauss_newton(W, X, q, cam)
        _, P, r, e = cost(W, X, q, cam)
        pixel = np.maximum(np.abs(r + q).max(1), cam.width)
        w = np.minimum(e, k)
        ci = np.where(e <= k, 0.5 * e * e, k * (e - 0.5 * k))
        sigma = np.sqrt(2 * ((w * 1.5 * 2.0 ** -53 * pixel) ** 2 + (2.0 ** -53 * ci) ** 2).sum())
        g = gradient(W, X, q, cam)
        assert -0.5 * g @ d <= 4 * sigma, (seed, -0.5 * g @ d, sigma, c)
    ctx.close()
