"""A destroyed context gives back the device memory that its calls took: pose gradients and
map training (their image and gradient buffers are tens of megabytes here), refinement,
the proposal and a split GEMM.  After one round (the driver's own lazy allocations), the
free memory does not fall."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def use(R, what, g, cam, poses, img, targets, grad):
    ctx = R.Context(R.reloc_default_config(block_size=1000.0))
    ctx.load_map(g)
    runs = [(0, g.n)]
    if what == "grad":
        ctx.score_grad(runs, poses, cam, img)
    elif what == "train":
        ctx.train_grad(runs, poses, cam, targets, grad)
        ctx.train_step(runs, poses, cam, targets)
    elif what == "pnp":
        pairs = torch.rand((200_000, 4), device="cuda:0") * 90.0
        with pytest.raises(R.RelocError):            # no pair has a usable depth
            ctx.refine_pnp(poses[0], cam, torch.zeros_like(img[0]), torch.zeros_like(img[0]), pairs)
    else:
        ctx.proposal_init(1)
        x = torch.zeros((64, 47, 176, 2), dtype=torch.int16, device="cuda:0")
        ctx.proposal_train_step(x, torch.zeros(64, dtype=torch.int32, device="cuda:0"), 1e-3)
        a = torch.zeros((2048, 1024), dtype=torch.bfloat16, device="cuda:0")
        ctx.gemm_bf16(a, a, torch.empty((2048, 2048), device="cuda:0"), split_k=4)
    ctx.close()


@pytest.mark.parametrize("what", ["grad", "train", "pnp", "proposal"])
def test_destroyed_contexts_leave_nothing(what):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    g = sg.tiny_scene(n=3000).gaussians
    cam = sg.Camera(704, 188, 276.0, 276.0, 352.0, 94.0)
    poses = np.stack([sg.pose_from_xyz_yaw(0.2 * k, -14.0, 2.0, np.pi / 2) for k in range(8)])
    img = torch.rand((3, 188, 704), device="cuda:0")
    targets = torch.rand((8, 3, 188, 704), device="cuda:0")
    grad = torch.zeros((14, g.n), device="cuda:0")
    free = []
    for _ in range(4):
        use(R, what, g, cam, poses, img, targets, grad)
        torch.cuda.synchronize()
        torch.cuda.empty_cache()
        free.append(torch.cuda.mem_get_info()[0])
    assert min(free[1:]) >= free[0], free
