"""The proposal network takes its inputs at any 2-byte address: a contiguous view at an odd
element offset gives the logits, loss and gradients of the aligned buffer bit for bit."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("offset", [1, 2, 3])
def test_inputs_off_four_bytes(offset):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    B, n = 64, 64 * 47 * 176 * 2
    x = torch.tensor(sg.Rng(4).uniform(n).astype(np.float32), device="cuda:0").to(torch.bfloat16).view(torch.int16)
    labels = torch.arange(B, dtype=torch.int32, device="cuda:0")
    flat = torch.zeros(n + 8, dtype=torch.int16, device="cuda:0")
    views = [x.view(B, 47, 176, 2), flat[offset:offset + n].view(B, 47, 176, 2)]
    views[1].copy_(views[0])
    assert views[1].data_ptr() % 4 == 2 * (offset % 2)
    got = []
    for v in views:
        ctx = R.Context()
        ctx.proposal_init(3)
        logits = torch.empty((B, 64), device="cuda:0")
        ctx.proposal_forward(v, logits)
        loss = ctx.proposal_train_step(v, labels, 1e-3)
        got.append((logits.cpu().numpy(), loss, ctx.proposal_get(0), ctx.proposal_get(1)))
        ctx.close()
    for a, b in zip(*got):
        assert np.array_equal(a, b)
