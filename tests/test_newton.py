"""The FP64 reciprocals that the PnP solve forms from FP32 seeds (csrc/newton.h), on the
CPU: the exact value rounded once.  1 / x equals the IEEE quotient; 1 / sqrt(x), against
extended precision (64 bits of mantissa or more), lies within half an ulp and what the
reference itself is off.  Seeds up to two FP32 ulps off, as the GPU's may be."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "newton.h"
using namespace reloc;
static double off(float s, int k) { for (; k > 0; --k) s = nextafterf(s, 2 * s); for (; k < 0; ++k) s = nextafterf(s, 0.f); return s; }
extern "C" void recip(const double *x, int n, int k, double *out)
{ for (int i = 0; i < n; ++i) out[i] = newton_recip(x[i], off(1.f / (float)x[i], k)); }
extern "C" void rsqrt_ulps(const double *x, int n, int k, double *ulps)
{
    for (int i = 0; i < n; ++i) {
        const double r = newton_rsqrt(x[i], off(1.f / sqrtf((float)x[i]), k));
        const long double want = 1.0L / sqrtl((long double)x[i]);
        ulps[i] = (double)(fabsl((long double)r - want) / (long double)(nextafter(r, 2 * r) - r));
    }
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("newton")
    (d / "n.cpp").write_text(SRC)
    subprocess.run(["g++", "-O2", "-ffp-contract=off", "-shared", "-fPIC", "-std=c++17",
                    "-I", os.path.join(ROOT, "paper_2403_11367_gb300", "csrc"), str(d / "n.cpp"), "-o", str(d / "n.so")],
                   check=True)
    return ctypes.CDLL(str(d / "n.so"))


@pytest.mark.parametrize("k", [-2, 0, 2])
def test_rounded_once(lib, k):
    x = np.exp(np.random.RandomState(3).uniform(-80.0, 80.0, 200_000))
    dp = ctypes.POINTER(ctypes.c_double)
    out = np.empty_like(x)
    lib.recip(x.ctypes.data_as(dp), len(x), k, out.ctypes.data_as(dp))
    assert np.array_equal(out, 1.0 / x)
    lib.rsqrt_ulps(x.ctypes.data_as(dp), len(x), k, out.ctypes.data_as(dp))
    assert out.max() <= 0.5 + 2.0 ** -9
