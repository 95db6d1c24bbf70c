"""The depth sort's two routes (one cluster launch, or a launch chain per pass where the last
call's visible share lets expect many) give the same tile lists: the same views after calls
that saw nothing and after calls that saw everything.  The chain is told by its launches."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("n,views", [(262_145, 1), (270_000, 9), (400_001, 2)])
def test_routes_agree(n, views):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    r = sg.Rng(n)
    x = np.round(r.uniform(n, 2.0, 40.0) * 512) / 512                # ties
    mean = np.stack([x, r.uniform(n, -0.2, 0.2), r.uniform(n, -0.2, 0.2)], 1).astype(np.float32)
    q = np.tile(np.float32([1, 0, 0, 0]), (n, 1))
    g = sg.Gaussians(mean, np.full((n, 3), 0.01, np.float32), q, np.full(n, 0.05, np.float32),
                     r.uniform(3 * n).reshape(n, 1, 3).astype(np.float32), 0)
    cam = sg.Camera(40, 24, 30.0, 30.0, 20.0, 12.0)
    ctx = R.Context(R.reloc_default_config(block_size=1000.0))
    ctx.load_map(g)
    see = np.stack([sg.pose_from_xyz_yaw(0.01 * k, 0.0, 0.0, 0.0) for k in range(views)])
    away = sg.pose_from_xyz_yaw(0.0, 0.0, 0.0, np.pi)[None]
    rgb = torch.empty((views, 3, 24, 40), device="cuda:0")
    got = []
    for before in (away, see):
        ctx.render([(0, n)], before, cam, rgb=rgb[:len(before)])
        ctx.render([(0, n)], see, cam, rgb=rgb)
        k = ctx.last_counts()
        assert k.n_visible == n * views
        lists = torch.empty((views, k.inst_stride), dtype=torch.int32, device="cuda:0")
        count = ctx.export_debug(inst_gauss=lists)
        got.append((k.kernel_launches, rgb.cpu().numpy(), [lists[v, :count[v]].cpu().numpy() for v in range(views)]))
    assert got[1][0] == got[0][0] + 11                               # four passes of three launches for one
    assert np.array_equal(got[0][1], got[1][1])
    assert all(np.array_equal(a, b) for a, b in zip(got[0][2], got[1][2]))
    ctx.close()
