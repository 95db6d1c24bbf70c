"""Pairs off 16 bytes are refused before any launch (the solve reads a pair as one 16-byte
load), and the context goes on."""
import numpy as np
import pytest

from pnp_cases import make_pairs, tiny_views

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


def test_pairs_off_16_bytes_are_refused():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    s, Wq, Wr = tiny_views()
    depth, alpha, pairs = make_pairs(s, Wq, Wr)
    depth, alpha = (torch.tensor(np.ascontiguousarray(x), device="cuda:0") for x in (depth, alpha))
    flat = torch.zeros(pairs.size + 4, device="cuda:0")
    ctx = R.Context()
    for k in (1, 2, 3, 4):
        v = flat[k:k + pairs.size].view(-1, 4)
        v.copy_(torch.tensor(pairs))
        if k < 4:
            with pytest.raises(R.RelocError, match="16-byte"):
                ctx.refine_pnp(Wr, s.camera, depth, alpha, v)
        else:
            assert ctx.refine_pnp(Wr, s.camera, depth, alpha, v).n_used == len(pairs)
    ctx.close()
