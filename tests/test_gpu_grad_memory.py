"""Pose gradients keep the forward's render only where memory allows: when its allocation
fails, or the batch memory budget has no room for it, the call composites again and gives
the same result (scores bit for bit; gradients to the order of their FP32 atomic sums, a few
2^-24 of sums of many terms: 1e-4 of the norm, as the gradient tests allow)."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.fixture
def R():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc
    yield reloc
    reloc.reloc_inject_faults(reloc.FAULT_ALLOC, 0)


def setup(R, views, scale=1.0):
    g = sg.tiny_scene(n=3000).gaussians
    cam = sg.Camera(int(1408 * scale), int(376 * scale), 552.0 * scale, 552.0 * scale, 704.0 * scale, 188.0 * scale)
    poses = np.stack([sg.pose_from_xyz_yaw(0.1 * k, -14.0, 2.0, np.pi / 2) for k in range(views)])
    img = torch.tensor(sg.random_image(3, 3, cam.height, cam.width).astype(np.float32), device="cuda:0")
    return g, cam, poses, img


def same(a, b):
    assert np.array_equal(a[0], b[0])
    assert np.linalg.norm(a[1] - b[1]) <= 1e-4 * np.linalg.norm(b[1])


def test_falls_back_when_the_image_cannot_be_had(R):
    g, cam, poses, img = setup(R, 2)
    _, small, _, simg = setup(R, 2, 0.25)
    runs = [(0, g.n)]
    ref_ctx = R.Context()
    ref_ctx.load_map(g)
    ref = ref_ctx.score_grad(runs, poses, cam, img)
    ctx = R.Context()
    ctx.load_map(g)
    ctx.score(runs, poses, cam, img)                 # all but the gradients' buffers at full size
    ctx.score_grad(runs, poses, small, simg)         # those, and a small image
    R.reloc_inject_faults(R.FAULT_ALLOC, 1)
    got = ctx.score_grad(runs, poses, cam, img)      # only the image has to grow
    other = R.Context()
    other.load_map(g)                                # the fault was taken by the image
    same(got, ref)
    same(ctx.score_grad(runs, poses, cam, img), ref)
    for c in (ref_ctx, ctx, other):
        c.close()


def test_image_counts_towards_the_budget(R):
    g, cam, poses, img = setup(R, 16)                # an image of 102 MB
    runs = [(0, g.n)]
    used, out = [], []
    for budget in (16 << 30, 64 << 20, 16 << 30, 64 << 20):
        ctx = R.Context()
        ctx.load_map(g)
        ctx.set_batch_options(mem_budget=budget)
        torch.cuda.synchronize()
        before = torch.cuda.mem_get_info()[0]
        out.append(ctx.score_grad(runs, poses, cam, img))
        used.append(before - torch.cuda.mem_get_info()[0])
        ctx.close()
    assert used[2] - used[3] >= 90 << 20, used
    for o in out[1:]:
        same(o, out[0])
