"""The PnP solve ends by its step tolerance after each possible number of iterations: the
iteration count is the oracle's, the pose agrees as in the noise-free parity test
(1e-9 m, 1e-10 rad), and repeats are the same bit for bit (the exit is decided by every
warp of every block for itself, from the same values).  Tolerances lie at the geometric
mean of two consecutive steps' largest entries, so rounding does not decide."""
import numpy as np
import pytest

import oracle
from pnp_cases import make_pairs, pose_error, tiny_views

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def steps(Wr, cam, depth, alpha, pairs, W0, n):
    """Largest entry of each of the first n steps, from the oracle cut off after 0, 1, .. iterations."""
    poses = [oracle.refine_pnp(Wr, cam, depth, alpha, pairs, pose_init=W0, max_iters=k)["pose"] for k in range(n + 1)]
    out = []
    for a, b in zip(poses, poses[1:]):
        D = b[:3, :3] @ a[:3, :3].T
        phi = 0.5 * np.array([D[2, 1] - D[1, 2], D[0, 2] - D[2, 0], D[1, 0] - D[0, 1]])
        out.append(max(np.abs(b[:3, 3] - D @ a[:3, 3]).max(), np.abs(phi).max()))
    return out


@pytest.mark.parametrize("n", [40, 3000])
def test_exit_by_tolerance(n):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    s, Wq, Wr = tiny_views()
    depth, alpha, pairs = make_pairs(s, Wq, Wr, step=1, seed=5)
    pairs = pairs[np.linspace(0, len(pairs) - 1, n).astype(int)]
    W0 = oracle.pnp_apply(Wr, np.array([0.5, -0.4, 0.3, 0.05, -0.04, 0.1]))
    st = steps(Wr, s.camera, depth, alpha, pairs, W0, 4)
    assert all(b < 0.3 * a for a, b in zip(st, st[1:])), st
    dev = [torch.tensor(np.ascontiguousarray(x), device="cuda:0") for x in (depth, alpha, pairs)]
    ctx = R.Context()
    for k in range(len(st) - 1):
        tol = float(np.sqrt(st[k] * st[k + 1]))
        ref = oracle.refine_pnp(Wr, s.camera, depth, alpha, pairs, pose_init=W0, tol=tol)
        assert ref["iters"] == k + 2
        got = [ctx.refine_pnp(Wr, s.camera, *dev, pose_init=W0, tol=tol) for _ in range(5)]
        assert all(g.iters == ref["iters"] and list(g.pose) == list(got[0].pose) and g.cost == got[0].cost for g in got)
        dt, dr = pose_error(np.array(got[0].pose).reshape(4, 4), ref["pose"])
        assert dt < 1e-9 and dr < 1e-10, (k, dt, dr)
    ctx.close()
