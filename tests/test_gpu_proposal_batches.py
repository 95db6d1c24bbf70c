"""A training batch's gradient against the mean of its 64-sample parts', each
from the same parameters: more output tiles, row blocks and K splits than one
part has (the operands read as they lie, the fused ReLU and col2im, the column
sums' partials).  The parts' signals are those of the batch times a power of two,
exactly, and so are their BF16 terms; only FP32 sums of up to K = 2 * 64 * 2112 *
(batch / 64) products are taken in another order, each off by at most
sqrt(K) 2^-24 of the products' root sum of squares for random signs.  Cancellation
makes a gradient smaller than that root sum, by a factor of about 30 at most
(sqrt(K) 2^-24 30 < 2e-3 of the tensor's norm)."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("batch", [64, 128, 256, 512])
def test_batch_gradient_is_the_mean_of_its_parts(batch):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    ctx = R.Context()
    ctx.proposal_init(9)
    gen = torch.Generator(device="cuda:0")
    gen.manual_seed(batch)
    x = torch.rand((batch, R.PROPOSAL_H, R.PROPOSAL_W, 2), generator=gen, device="cuda:0").to(torch.bfloat16)
    y = torch.randint(0, 64, (batch,), generator=gen, device="cuda:0", dtype=torch.int32)
    loss = ctx.proposal_train_step(x, y, 0.0, update=False)
    got = ctx.proposal_get(1).astype(np.float64)
    parts, losses = [], []
    for k in range(0, batch, 64):
        losses.append(ctx.proposal_train_step(x[k:k + 64].contiguous(), y[k:k + 64].contiguous(), 0.0, update=False))
        parts.append(ctx.proposal_get(1).astype(np.float64))
    want = np.mean(parts, axis=0)
    assert abs(loss - np.mean(losses)) < 1e-5 * abs(loss)
    at = 0
    cin, cout = (2, 32, 64, 64, 128), (32, 64, 64, 128, 128)
    sizes = [n for i, o in zip(cin, cout) for n in (o * 9 * i, o)] + [1024 * 1536, 1024, 64 * 1024, 64]
    for n in sizes:
        a, b = got[at:at + n], want[at:at + n]
        assert np.isfinite(a).all() and np.linalg.norm(a - b) <= 2e-3 * np.linalg.norm(b), (at, n)
        at += n
    assert at == len(got)
    ctx.close()
