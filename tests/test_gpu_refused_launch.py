"""A batch that the runtime refuses to launch (more views in a sub-batch than a grid has
rows) reports it once: the next call on the context finds no error left."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("graph", [False, True])
def test_refusal_is_reported_once(graph):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    g = sg.tiny_scene(n=40).gaussians
    cam = sg.Camera(16, 16, 10.0, 10.0, 8.0, 8.0)
    pose = sg.pose_from_xyz_yaw(0.0, -14.0, 2.0, np.pi / 2)
    img = torch.rand((3, 16, 16), device="cuda:0")
    ctx = R.Context()
    ctx.load_map(g)
    ctx.set_batch_options(use_graph=graph)
    query = (img, pose, 40.0, (16, 16, 16, 0.1, 0.1))
    first, scores = ctx.localize_batch([query] * 2, cam)
    with pytest.raises(R.RelocError) as e:
        ctx.localize_batch([query] * 16, cam)                # 65,536 views
    assert e.value.status == R.ECUDA
    again, scores2 = ctx.localize_batch([query] * 2, cam)
    assert [r.best_index for r in again] == [r.best_index for r in first]
    assert all(np.array_equal(a, b) for a, b in zip(scores, scores2))
    ctx.close()
