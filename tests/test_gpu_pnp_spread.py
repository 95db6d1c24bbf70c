"""The PnP solve's spread over warps and blocks: fewer pairs than a warp, a
block's edge, more pairs than one pair per thread covers; a far start, whose
steps may have to be halved; solves cut off after a number of iterations.
Noise-free pairs: both sides converge quadratically to the same pose and differ
in the order of the sums only, so they agree as in the noise-free parity test
(1e-9 m, 1e-10 rad)."""
import numpy as np
import pytest

import oracle
from pnp_cases import make_pairs, pose_error, tiny_views

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,max_iters,far", [(31, 30, 0.0), (64, 30, 0.0), (65, 30, 0.0), (500, 0, 0.0), (500, 2, 0.0),
                                             (500, 30, 2.0), (9729, 30, 0.0), (20000, 30, 0.0)])
def test_spread_matches_oracle(n, max_iters, far):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    s, Wq, Wr = tiny_views()
    depth, alpha, pairs = make_pairs(s, Wq, Wr, step=1, seed=5)
    pairs = pairs[np.linspace(0, len(pairs) - 1, n).astype(int)]
    W0 = oracle.pnp_apply(Wr, far * np.array([0.5, -0.4, 0.3, 0.05, -0.04, 0.1]))
    opt = {"max_iters": max_iters}
    ref = oracle.refine_pnp(Wr, s.camera, depth, alpha, pairs, pose_init=W0, **opt)
    dev = [torch.tensor(np.ascontiguousarray(x), device="cuda:0") for x in (depth, alpha, pairs)]
    ctx = R.Context()
    res = ctx.refine_pnp(Wr, s.camera, *dev, pose_init=W0, **opt)
    dt, dr = pose_error(np.array(res.pose).reshape(4, 4), ref["pose"])
    assert res.n_used == ref["n_used"] == n
    assert dt < 1e-9 and dr < 1e-10, (dt, dr)
    assert abs(res.rms_px - ref["rms_px"]) <= 1e-6 * max(1.0, ref["rms_px"])
    ctx.close()
