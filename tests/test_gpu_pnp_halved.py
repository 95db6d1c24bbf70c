"""PnP iterations whose full step does not lower the cost: the solve takes the first of
ten halved steps that does.  Starts whose first step the FP64 restatement here halves
h = 1 .. 10 times (the cost of step h is below the start's by 1e-9 of it, those of the
steps before are not below it by as much), noise-free pairs, one iteration.

Tolerance on the pose after it: the step solves a 6 x 6 system of condition number k in
FP64.  Its entries are sums of some hundred products (100 * 2^-53), and a pair's terms go
with 1 / z^2, z a difference of terms of the points' distance P: 4 P / z_min roundings
more.  So two solves differ by up to k (100 + 4 P / z_min) 2^-53 of the step, and of the
pose's entries (1 and the step's length)."""
import numpy as np
import pytest

import oracle
from pnp_cases import make_pairs, tiny_views

N = 60
# start offset (rho, phi) from the render pose, halvings
STARTS = [([-5.361689, 3.07533, -0.428737, -2.143932, 0.667062, -1.828619], 1),
          ([-5.32732, 3.064225, -0.208939, -2.078038, 0.705885, -1.794979], 2),
          ([-0.30685, -5.348945, -0.660063, -1.159226, 0.759543, 0.909114], 3),
          ([-0.463136, -5.323591, -0.702865, -1.138392, 0.760892, 0.883539], 4),
          ([-2.126507, -5.757379, 5.337788, -1.15926, 0.999138, 0.796218], 5),
          ([-6.419658, -2.204545, 1.273877, -0.381952, 0.938093, 0.189162], 6),
          ([-1.755586, -2.466927, -5.51102, -0.483352, 0.786304, 0.306842], 7),
          ([5.118471, 1.726951, -4.390029, 0.214336, -1.220838, 0.203729], 8),
          ([5.117628, 1.725354, -4.3892, 0.214224, -1.220308, 0.203108], 9),
          ([-1.965622, -0.957177, -5.925883, -0.235682, 0.756139, 0.213132], 10)]


def cost(W, X, q, cam, k=2.0):
    P = X @ W[:3, :3].T + W[:3, 3]
    front = P[:, 2] > 1e-6
    P, q = P[front], q[front]
    r = np.stack([cam.fx * P[:, 0] / P[:, 2] + cam.cx - q[:, 0], cam.fy * P[:, 1] / P[:, 2] + cam.cy - q[:, 1]], 1)
    e = np.hypot(r[:, 0], r[:, 1])
    return np.where(e <= k, 0.5 * e * e, k * (e - 0.5 * k)).sum(), P, r, e


def system(W, X, q, cam, k=2.0):
    """Normal equations (H, g) of the Huber cost at W."""
    _, P, r, e = cost(W, X, q, cam, k)
    x, y, z = P.T
    o = np.zeros_like(x)
    Jp = np.stack([np.stack([cam.fx / z, o, -cam.fx * x / z ** 2], 1), np.stack([o, cam.fy / z, -cam.fy * y / z ** 2], 1)], 1)
    M = np.stack([np.stack([o + 1, o, o, o, z, -y], 1), np.stack([o, o + 1, o, -z, o, x], 1),
                  np.stack([o, o, o + 1, y, -x, o], 1)], 1)
    J = Jp @ M
    w = np.where(e <= k, 1.0, k / np.maximum(e, 1e-300))
    return np.einsum("n,nra,nrb->ab", w, J, J), np.einsum("n,nra,nr->a", w, J, r)


def gradient(W, X, q, cam):
    return system(W, X, q, cam)[1]


def gauss_newton(W, X, q, cam, k=2.0):
    """(step, condition number of the system, cost at W)."""
    H, g = system(W, X, q, cam, k)
    H = H + 1e-9 * np.trace(H) / 6 * np.eye(6)
    return np.linalg.solve(H, -g), np.linalg.cond(H), cost(W, X, q, cam, k)[0]


def problem():
    s, Wq, Wr = tiny_views()
    depth, alpha, pairs = make_pairs(s, Wq, Wr, step=1, seed=5)
    pairs = pairs[np.linspace(0, len(pairs) - 1, N).astype(int)]
    X, use = oracle.pnp_backproject(Wr, s.camera, depth, alpha, pairs[:, :2].astype(np.float64))
    assert use.all()
    return s, Wr, depth, alpha, pairs, X, pairs[:, 2:].astype(np.float64)


def halvings(p, W):
    """(halvings of the step at W, whether each decision has a margin, step, condition number)."""
    s, Wr, depth, alpha, pairs, X, q = p
    d, k, c = gauss_newton(W, X, q, s.camera)
    clear = True
    for h in range(11):
        t = cost(oracle.pnp_apply(W, d, 0.5 ** h), X, q, s.camera)[0]
        clear = clear and abs(t - c) > 1e-9 * c
        if t < c:
            return h, clear, d, k
    return None, clear, d, k


def bound(p, W, h, d, k):
    X = p[5]
    far, near = 0.0, np.inf
    for V in (W, oracle.pnp_apply(W, d, 0.5 ** h)):
        P = X @ V[:3, :3].T + V[:3, 3]
        far, near = max(far, np.abs(P).max()), min(near, np.abs(P[:, 2]).min())
    return k * (100 + 4 * far / near) * 2.0 ** -53 * max(1.0, np.abs(0.5 ** h * d).max())


@pytest.mark.parametrize("offset,h", STARTS)
def test_starts_are_halved(offset, h):
    """The oracle's one iteration is the restatement's step, halved h times."""
    p = problem()
    s, Wr, depth, alpha, pairs = p[:5]
    W = oracle.pnp_apply(Wr, np.array(offset))
    got_h, clear, d, k = halvings(p, W)
    assert got_h == h and clear
    ref = oracle.refine_pnp(Wr, s.camera, depth, alpha, pairs, pose_init=W, max_iters=1)
    assert np.abs(ref["pose"] - oracle.pnp_apply(W, d, 0.5 ** h)).max() <= bound(p, W, h, d, k)


@pytest.mark.gpu
@pytest.mark.parametrize("offset,h", STARTS)
def test_halved_step(offset, h):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    p = problem()
    s, Wr, depth, alpha, pairs = p[:5]
    W = oracle.pnp_apply(Wr, np.array(offset))
    _, _, d, k = halvings(p, W)
    ref = oracle.refine_pnp(Wr, s.camera, depth, alpha, pairs, pose_init=W, max_iters=1)
    dev = [torch.tensor(np.ascontiguousarray(x), device="cuda:0") for x in (depth, alpha, pairs)]
    ctx = R.Context()
    res = ctx.refine_pnp(Wr, s.camera, *dev, pose_init=W, max_iters=1)
    ctx.close()
    assert res.iters == ref["iters"] == 1
    assert np.abs(np.array(res.pose).reshape(4, 4) - ref["pose"]).max() <= bound(p, W, h, d, k)
