"""The GEMM's output tiles: several rounds of tiles to a CTA (both TMEM
accumulators in use, the operand ring running on from tile to tile), narrowed
tiles, and the two ways out of the epilogue (16-byte stores; single values
where N or the row stride is not a multiple of 4 or C is not on 16 bytes).
Tolerance: products of BF16 values are exact in FP32, so only the FP32
accumulation rounds, at most K times: |error| <= K 2^-24 sum |a b| <= K 2^-24
|row| |col|."""
import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")


@pytest.mark.parametrize("M,N,K,split,offset", [
    (128 * 152 * 5 + 1, 32, 64, 1, 0),        # five rounds and one row more, narrow tiles
    (128 * 160, 256, 64, 1, 0),               # wide tiles past one round
    (128 * 77 - 3, 512, 128, 1, 0),           # an odd number of rows, two column tiles
    (700, 1024, 192, 1, 0),                   # few rows: the tile is halved until the SMs are covered
    (5000, 33, 64, 1, 0), (5000, 130, 128, 1, 0),
    (300, 64, 128, 1, 1), (300, 64, 128, 2, 3),   # C off the 16-byte boundary
    (40, 16, 64 * 24, 24, 0), (40, 12, 64 * 9, 9, 0)])
def test_every_tile_and_both_stores(M, N, K, split, offset):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    ctx = R.Context()
    r = sg.Rng(M + N)
    A, B = (torch.tensor(r.normal(n * K).reshape(n, K).astype(np.float32)).to(torch.bfloat16).cuda() for n in (M, N))
    bias = torch.tensor(r.normal(N).astype(np.float32), device="cuda:0")
    buf = torch.full((M * N + offset,), float("nan"), device="cuda:0")
    C = buf[offset:].view(M, N)
    ctx.gemm_bf16(A, B, C, bias=bias, relu=True, split_k=split)
    a, b = A.double(), B.double()
    ref = (a @ b.T + bias.double()).clamp(min=0)
    bound = K * 2.0 ** -24 * (a.norm(dim=1)[:, None] * b.norm(dim=1)[None, :] + bias.abs().double())
    assert torch.isfinite(C).all()
    assert bool(((C.double() - ref).abs() <= bound).all())
    assert torch.isnan(buf[:offset]).all()
    ctx.close()
