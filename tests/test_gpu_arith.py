"""csrc/arith.h and csrc/trig.h to the bounds they state: quotients and reciprocal roots against IEEE
arithmetic, over every significand of the divisor and of the root's argument and the exponents for which
the bounds hold; rotation entries against longer arithmetic."""
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
        assert (np.abs(y - ref) <= 1.01 * ulp).all()


TRIG = """
#include <vector>
#include "trig.h"
__global__ void k(const float* z, const float* a, float b, const float4* t, float2* s, float2* c, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  float m[2];
  collage::trig_entry(z[i], false, a[i], b, t, m);
  s[i] = make_float2(m[0], m[1]);
  collage::trig_entry(z[i], true, a[i], b, t, m);
  c[i] = make_float2(m[0], m[1]);
}
extern "C" int trig(const float* z, const float* a, float b, float2* s, float2* c, int n) {
  std::vector<float4> h(collage::kTrigSteps / 4 + 1);
  collage::trig_table(h.data());
  float4* t;
  if (cudaMalloc(&t, sizeof(float4) * h.size())) return 1;
  cudaMemcpy(t, h.data(), sizeof(float4) * h.size(), cudaMemcpyHostToDevice);
  k<<<(n + 255) / 256, 256>>>(z, a, b, t, s, c, n);
  const int e = cudaDeviceSynchronize();
  cudaFree(t);
  return e;
}
"""


@pytest.mark.parametrize("b", [1.0, 200.0, 1024.0, 32767.0])  # (a resolution: a float is exact)
def test_rotation_entries_as_exact_as_a_split_double(build_so, b):
    # each entry a b sin z, a b cos z is within half a unit of its low part (2^-48 of a b; the reference and its
    # split add 2^-52), and no further from the exact value on average than the FP64 value split into a pair
    f = build_so(TRIG).trig
    f.argtypes = [C.c_void_p, C.c_void_p, C.c_float, C.c_void_p, C.c_void_p, C.c_int]
    rng = np.random.default_rng(int(b))
    k = rng.integers(-5300000, 5300000, 1 << 16).astype(np.float64)
    mid = (k * (2 * np.pi / 4096)).astype(np.float32)  # beside the table's angles, and half a step from them
    half = ((k + 0.5) * (2 * np.pi / 4096)).astype(np.float32)
    z = np.concatenate([
        mid, half, rng.uniform(-8192, 8192, 1 << 17).astype(np.float32), rng.uniform(-7, 7, 1 << 17).astype(np.float32),
        (10.0 ** rng.uniform(-30, 0, 1 << 15)).astype(np.float32), np.float32(np.pi / 2 * np.arange(-5200, 5200)),
        np.float32([0.0, -0.0, 8192.0, -8192.0, 8191.9995])])
    z = z[np.abs(z) <= 8192]
    a = np.exp(rng.uniform(-3, 3, len(z))).astype(np.float32)
    zt, at = torch.from_numpy(z).cuda(), torch.from_numpy(a).cuda()
    s, c = (torch.empty(len(z), 2, device="cuda") for _ in range(2))
    torch.cuda.synchronize()
    assert f(zt.data_ptr(), at.data_ptr(), b, s.data_ptr(), c.data_ptr(), len(z)) == 0
    assert np.finfo(np.longdouble).nmant >= 63
    ab = a.astype(np.longdouble) * np.longdouble(b)
    for got, fn in ((s, np.sin), (c, np.cos)):
        exact = ab * fn(z.astype(np.longdouble))
        double = a.astype(np.float64) * b * fn(z.astype(np.float64))
        hi = double.astype(np.float32)
        split = hi.astype(np.longdouble) + (double - hi).astype(np.float32)
        m = got.cpu().numpy().astype(np.longdouble)
        err, ref = ((v - exact) / ab for v in (m[:, 0] + m[:, 1], split))
        assert np.abs(err).max() <= 2.0 ** -48
        assert np.sqrt((err ** 2).mean()) <= np.sqrt((ref ** 2).mean())
