"""The proposal's backward kernels alone, through their launchers: the ReLU backward with its
bias sums at widths around its thread layout's edges, and the two gradient GEMMs that read
their operands as they lie (MN-major), at N below a tile, past 128 and no multiple of it,
column counts off the tile, and K slices in which the signal's high half ends.

A backward signal is two BF16 terms hi | lo, [rows][2 N].  The products of BF16 values are
exact in FP32, so a GEMM's FP32 sums of K terms are off by at most K 2^-24 sum |a b| <= K
2^-24 |row| |column|; the bias sums of M FP32 terms by M 2^-24 sum |x|.  The split itself is
compared bit for bit."""
import ctypes as C

import numpy as np
import pytest

import scenegen as sg

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

RELU_BACK = "_ZN5reloc16launch_relu_backEPKfiiiiiPK13__nv_bfloat16iiPS2_PfS6_P11CUstream_st"
WEIGHT_GRAD = "_ZN5reloc23launch_gemm_weight_gradEPK13__nv_bfloat16S2_PfiiiiS3_PiP11CUstream_st"
INPUT_GRAD = "_ZN5reloc22launch_gemm_input_gradEPK13__nv_bfloat16S2_PfiiiPiP11CUstream_st"
P, I = C.c_void_p, C.c_int


def launcher(name, types):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2403_11367_gb300 import reloc as R
    f = getattr(R.lib, name)
    f.argtypes, f.restype = types, C.c_int
    return f


def call(f, *args):
    assert f(*[a.data_ptr() if isinstance(a, torch.Tensor) else a for a in args]) == 0
    torch.cuda.synchronize()


def normal(seed, *shape):
    return torch.tensor(sg.Rng(seed).normal(int(np.prod(shape))).reshape(shape).astype(np.float32), device="cuda:0")


def split(x):
    hi = x.to(torch.bfloat16)
    return hi, (x - hi.float()).to(torch.bfloat16)


def signal(seed, rows, n):
    hi, lo = split(normal(seed, rows, n))
    return torch.cat([hi, lo], 1).contiguous(), hi.double() + lo.double()


@pytest.mark.parametrize("M", [1, 37, 3000])
@pytest.mark.parametrize("N", [4, 32, 48, 128, 508, 512, 516, 640, 1000, 1020, 1024, 2048])
def test_relu_back(M, N):
    f = launcher(RELU_BACK, [P, I, I, I, I, I, P, I, I, P, P, P, P])
    d, y = normal(N, M, N), normal(N + 1, M, N).to(torch.bfloat16)
    out = torch.full((M, 2 * N), float("nan"), dtype=torch.bfloat16, device="cuda:0")
    part, db = torch.full((608, N), float("nan"), device="cuda:0"), torch.full((N,), float("nan"), device="cuda:0")
    call(f, d, 0, 0, 0, 0, 0, y, M, N, out, part, db, None)
    x = torch.where(y.float() > 0, d, torch.zeros_like(d))
    hi, lo = split(x)
    assert torch.equal(out[:, :N], hi) and torch.equal(out[:, N:], lo)
    v = hi.double() + lo.double()
    assert bool(((db.double() - v.sum(0)).abs() <= M * 2.0 ** -24 * v.abs().sum(0)).all())


@pytest.mark.parametrize("R,N,Kc,splits", [(64, 32, 64, 1), (192, 32, 64, 3), (192, 136, 200, 1), (320, 200, 96, 2),
                                           (320, 64, 1544, 5), (1088, 128, 320, 2), (64, 1024, 136, 2)])
def test_weight_gradient(R, N, Kc, splits):
    f = launcher(WEIGHT_GRAD, [P, P, P, I, I, I, I, P, P, P])
    dy, v = signal(R + N, R, N)
    x = normal(Kc, R, Kc).to(torch.bfloat16)
    gw = torch.full((N, Kc), float("nan"), device="cuda:0")
    part = torch.full((splits, N, Kc), float("nan"), device="cuda:0")
    status = torch.zeros(4, dtype=torch.int32, device="cuda:0")
    call(f, dy, x, gw, R, N, Kc, splits, part, status, None)
    terms = dy.double().abs()
    mass = (terms[:, :N] + terms[:, N:]).T @ x.double().abs()
    assert int(status[0]) == 0
    assert bool(((gw.double() - v.T @ x.double()).abs() <= 2 * R * 2.0 ** -24 * mass).all())


@pytest.mark.parametrize("R,N,Kc", [(1, 64, 64), (130, 64, 200), (300, 192, 136), (129, 128, 1544), (20000, 64, 576)])
def test_input_gradient(R, N, Kc):
    f = launcher(INPUT_GRAD, [P, P, P, I, I, I, P, P])
    dy, v = signal(R + N, R, N)
    w = normal(Kc, N, Kc).to(torch.bfloat16)
    dx = torch.full((R, Kc), float("nan"), device="cuda:0")
    status = torch.zeros(4, dtype=torch.int32, device="cuda:0")
    call(f, dy, w, dx, R, N, Kc, status, None)
    terms = dy.double().abs()
    mass = (terms[:, :N] + terms[:, N:]) @ w.double().abs()
    assert int(status[0]) == 0
    assert bool(((dx.double() - v @ w.double()).abs() <= 2 * N * 2.0 ** -24 * mass).all())
