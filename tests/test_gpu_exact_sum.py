"""Fixed-point sums over a warp, compiled from their header with a small driver, against
exact sums (fractions: a rounded reference would add its own half a last place)."""
import ctypes as ct
import math
import os
import subprocess
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "exact_sum.cuh"
using namespace rsn;
__global__ void k_pairs(const double2* v, double* out) {
  const double2 w = v[blockIdx.x * 32 + threadIdx.x];
  const double t = warp_sum2_exact(w.x, w.y);
  if (threadIdx.x < 2) out[2 * blockIdx.x + threadIdx.x] = t;
}
__global__ void k_parts(const double2* v, int n, double2* out) {
  const double2 t = warp_sum_parts(v, n);
  out[threadIdx.x] = t;
}
extern "C" int pairs(int warps, const double2* v, double* out) {
  k_pairs<<<warps, 32>>>(v, out);
  return (int)cudaDeviceSynchronize();
}
extern "C" int parts(int n, const double2* v, double2* out) {
  k_parts<<<1, 32>>>(v, n, out);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_0782_gb300 import build
    d = tmp_path_factory.mktemp("sums")
    (d / "sums.cu").write_text(SRC)
    p = subprocess.run([build.nvcc_path(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, "-shared", str(d / "sums.cu"), "-o",
                        str(d / "sums.so")], capture_output=True, text=True)
    assert p.returncode == 0, p.stderr
    return ct.CDLL(str(d / "sums.so"))


def _exact(w):
    return sum((Fraction(float(x)) for x in w), Fraction(0))


def _off(got, exact):
    return abs(float(Fraction(float(got)) - exact))


def _values(kind, shape, r):
    v = r.standard_normal(shape) + 1j * r.standard_normal(shape)
    if kind == "wide":  # many decades, with zeros
        v *= 10.0 ** r.uniform(-30, 30, shape) * (r.random(shape) > 0.2)
    elif kind == "tiny":
        v *= 1e-290
    elif kind == "denormal":
        v *= 1e-310
    elif kind == "huge":  # (sums of 2,000 stay finite)
        v *= 1e303
    elif kind == "ones":  # the largest mantissa, no cancellation
        v = np.full(shape, (2.0 - 2.0 ** -52) * (1 + 1j))
    elif kind == "zero":
        v *= 0.0
    elif kind == "cancel":
        v.reshape(-1)[1::2] = -v.reshape(-1)[: v.size - v.size % 2: 2][: v.reshape(-1)[1::2].size] * (1 + 1e-15)
    return v


KINDS = ["normal", "wide", "tiny", "denormal", "huge", "ones", "zero", "cancel"]


@pytest.mark.parametrize("kind", KINDS)
def test_warp_sums(lib, kind):
    # every value is rounded to 1/32 of the last place of the largest, the total once:
    # half a last place of the largest value (32 times 1/64) and half of the result's;
    # the plain tree (below 2^-950) five roundings
    n = 300
    v = _values(kind, (n, 32), np.random.default_rng(1))
    dev, out = torch.tensor(v, device="cuda"), torch.zeros(2 * n, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.pairs(n, ct.c_void_p(dev.data_ptr()), ct.c_void_p(out.data_ptr())) == 0
    got = out.cpu().numpy().reshape(n, 2)
    for k in range(n):
        for c, w in enumerate((v[k].real, v[k].imag)):
            ref, top = math.fsum(w), np.abs(w).max()
            exact = _exact(w)
            tol = 0.51 * math.ulp(top) + 0.51 * math.ulp(abs(ref)) + (5 * math.ulp(32 * top) if kind in ("tiny", "denormal") else 0.0)
            assert _off(got[k, c], exact) <= tol, (k, c, got[k, c], ref)


@pytest.mark.parametrize("n", [1, 2, 31, 32, 33, 110, 127, 128, 129, 512, 513, 1000, 2000])
@pytest.mark.parametrize("kind", KINDS)
def test_sums_of_parts_are_rounded_once(lib, kind, n):
    # up to 512 values every one is rounded to 2^-guard of the largest one's last place,
    # guard = 9 - ceil(log2 n); of more, what lies below 2^-40 of it is cut off
    each = 2.0 ** -(10 - (n - 1).bit_length()) if n <= 512 else 2.0 ** -40
    v = _values(kind, (n,), np.random.default_rng(n))
    dev, out = torch.tensor(v, device="cuda"), torch.zeros(32, dtype=torch.complex128, device="cuda")
    torch.cuda.synchronize()
    assert lib.parts(n, ct.c_void_p(dev.data_ptr()), ct.c_void_p(out.data_ptr())) == 0
    got = out.cpu().numpy()
    assert np.all(got == got[0])
    for g, w in ((got[0].real, v.real), (got[0].imag, v.imag)):
        ref = math.fsum(w)
        assert _off(g, _exact(w)) <= n * each * math.ulp(np.abs(w).max()) + 0.5001 * math.ulp(abs(ref)), (g, ref)


def test_many_parts(lib):
    n = 1 << 20  # equal values of the largest mantissa: no bit of the 128 may be lost
    v = _values("ones", (n,), np.random.default_rng(0))
    dev, out = torch.tensor(v, device="cuda"), torch.zeros(32, dtype=torch.complex128, device="cuda")
    torch.cuda.synchronize()
    assert lib.parts(n, ct.c_void_p(dev.data_ptr()), ct.c_void_p(out.data_ptr())) == 0
    assert out[0].item() == n * v[0]


@pytest.mark.parametrize("bad", [np.inf, -np.inf, np.nan])
def test_infinities_and_nan(lib, bad):
    for n in (32, 200):
        v = _values("normal", (n,), np.random.default_rng(0))
        v[7] = complex(bad, 0.5)
        dev, out = torch.tensor(v, device="cuda"), torch.zeros(32, dtype=torch.complex128, device="cuda")
        torch.cuda.synchronize()
        assert lib.parts(n, ct.c_void_p(dev.data_ptr()), ct.c_void_p(out.data_ptr())) == 0
        g = out[0].item()
        assert (np.isnan(g.real) if np.isnan(bad) else g.real == bad) and abs(g.imag - math.fsum(v.imag)) <= 1e-12
    o2 = torch.zeros(2, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    assert lib.pairs(1, ct.c_void_p(dev.data_ptr()), ct.c_void_p(o2.data_ptr())) == 0
    g = o2.cpu().numpy()
    assert (np.isnan(g[0]) if np.isnan(bad) else g[0] == bad) and abs(g[1] - math.fsum(v[:32].imag)) <= 1e-12
