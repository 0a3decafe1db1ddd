"""csrc/arith.h against IEEE arithmetic, to the bounds it states: every significand of the divisor and of the
root's argument, over the exponents for which the bounds hold."""
import ctypes as C
import subprocess

import numpy as np
import pytest
import torch

from paper_2406_04008_gb300 import build

pytestmark = pytest.mark.gpu

SRC = """
#include "arith.h"
__global__ void k(int op, const float* a, const float* b, float* out, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) out[i] = op == 0 ? collage::div_normal(a[i], b[i]) : op == 1 ? a[i] / b[i] : collage::rsqrt_normal(b[i]);
}
extern "C" int arith(int op, const float* a, const float* b, float* out, int n) {
  k<<<(n + 255) / 256, 256>>>(op, a, b, out, n);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def build_so(tmp_path_factory):
    def make(src):
        d = tmp_path_factory.mktemp("arith")
        (d / "a.cu").write_text(src)
        so = str(d / "a.so")
        subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-shared", str(d / "a.cu"), "-o", so], check=True)
        return C.CDLL(so)

    return make


@pytest.fixture(scope="module")
def arith(build_so):
    f = build_so(SRC).arith
    f.argtypes = [C.c_int, C.c_void_p, C.c_void_p, C.c_void_p, C.c_int]

    def run(op, a, b):
        b = torch.from_numpy(b).cuda()
        a = torch.from_numpy(a).cuda() if a is not None else b
        out = torch.empty_like(b)
        torch.cuda.synchronize()
        assert f(op, a.data_ptr(), b.data_ptr(), out.data_ptr(), b.numel()) == 0
        return out.cpu().numpy()

    return run


def _floats(significand, exponent):
    return ((exponent + 127).astype(np.uint32) << 23 | significand.astype(np.uint32)).view(np.float32)


@pytest.mark.parametrize("e", [-126, -100, -50, -3, -1, 0, 1, 30, 80, 125])  # exponents of the divisor
def test_quotients_are_ieees(arith, e):
    n = 1 << 23
    rng = np.random.default_rng(e + 200)
    m = np.arange(n)
    b = _floats(m, np.full(n, e))
    lo, hi = max(-100, e - 99), min(126, e + 126)  # |a| and |a / b| of at least 2^-100, the quotient finite
    for a_m in (rng.integers(0, n, n), np.zeros(n, int), m, np.maximum(m - 1, 0)):
        a = _floats(a_m, rng.integers(lo, hi, n)) * rng.choice(np.float32([-1, 1]), n)
        q, ref = arith(0, a, b), arith(1, a, b)
        off = np.abs(q.view(np.int32).astype(np.int64) - ref.view(np.int32))
        assert (off[:-1] == 0).all() and off[-1] <= 1  # (the last significand is all ones)
    assert (arith(0, np.zeros(n, np.float32), b) == 0).all()


@pytest.mark.parametrize("e", [-126, -100, -40, -2, 0, 2, 20, 60, 126])
def test_reciprocal_roots(arith, e):
    for k in (e, e + 1):
        x = _floats(np.arange(1 << 23), np.full(1 << 23, k))
        y, ref = arith(2, None, x).astype(np.float64), 1.0 / np.sqrt(x.astype(np.float64))
        ulp = np.ldexp(1.0, np.floor(np.log2(ref)).astype(int) - 23)
        assert (np.abs(y - ref) <= 0.51 * ulp).all()
