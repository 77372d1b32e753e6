"""Accuracy of the block solver's b x b algebra (elimination, Cholesky factor and its
inverse), compiled from its source with a small driver: its errors against extended
precision are no larger than those of textbook Gaussian elimination and Cholesky in
FP64 with every division and square root correctly rounded.  Compared are medians and
upper quartiles over 800 systems, with 10% for the sampling (their spread over draws
is about 3%); a reciprocal in place of divisions, or products fused into the running
value, adds 15% to 45%."""
import ctypes as ct
import os
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "block_kernels.cu"
namespace rsn {
template <int B>
__global__ void t_solve(const double2* M, const double2* Y, double2* X) {
  constexpr int LD = 2 * B + 1;
  __shared__ double2 aug[B * LD];
  __shared__ StepMem<B> sm;
  const int t = threadIdx.x;
  const size_t o = (size_t)blockIdx.x * B * B;
  if (t < B * B) {
    aug[t / B * LD + t % B] = M[o + t];
    aug[t / B * LD + B + t % B] = Y[o + t];
  }
  __syncthreads();
  if (gauss_jordan<B, LD>(aug, sm) && t < B * B) X[o + t] = aug[t / B * LD + B + t % B];
}
template <int B>
__global__ void t_chol(const double2* A, double2* U, double2* Li) {
  __shared__ double2 a[B * B], u[B * B], l[B * B];
  __shared__ StepMem<B> sm;
  const int t = threadIdx.x;
  const size_t o = (size_t)blockIdx.x * B * B;
  if (t < B * B) a[t] = A[o + t];
  __syncthreads();
  if (cholesky_inverse<B>(a, u, l, sm) && t < B * B) U[o + t] = u[t], Li[o + t] = l[t];
}
}  // namespace rsn
extern "C" int solve(int B, int n, const double2* M, const double2* Y, double2* X) {
  if (B == 4) rsn::t_solve<4><<<n, 32>>>(M, Y, X);
  else if (B == 8) rsn::t_solve<8><<<n, 64>>>(M, Y, X);
  else rsn::t_solve<16><<<n, 256>>>(M, Y, X);
  return (int)cudaDeviceSynchronize();
}
extern "C" int chol(int B, int n, const double2* A, double2* U, double2* Li) {
  if (B == 4) rsn::t_chol<4><<<n, 32>>>(A, U, Li);
  else if (B == 8) rsn::t_chol<8><<<n, 64>>>(A, U, Li);
  else rsn::t_chol<16><<<n, 256>>>(A, U, Li);
  return (int)cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_1401_0782_gb300 import build
    d = tmp_path_factory.mktemp("algebra")
    (d / "algebra.cu").write_text(SRC)
    p = subprocess.run([build.nvcc_path(), *build.ARCH, *build.NVCC_FLAGS, "-I", build.CSRC, "-I", os.path.join(ROOT, "include"),
                        "-shared", str(d / "algebra.cu"), "-o", str(d / "algebra.so")], capture_output=True, text=True)
    assert p.returncode == 0, p.stderr
    return ct.CDLL(str(d / "algebra.so"))


def _gpu(f, B, n, ins, n_out):
    dev = [torch.tensor(np.ascontiguousarray(a), device="cuda") for a in ins]
    out = [torch.full((n, B, B), float("nan"), dtype=torch.complex128, device="cuda") for _ in range(n_out)]
    torch.cuda.synchronize()
    assert f(B, n, *(ct.c_void_p(t.data_ptr()) for t in dev + out)) == 0
    return [t.cpu().numpy() for t in out]


def _err(x, ref):
    e = np.sqrt((np.abs(x - ref) ** 2).sum((1, 2)) / (np.abs(ref) ** 2).sum((1, 2))).astype(float)
    return np.quantile(e, [0.5, 0.75])


def _eliminate(M, Y):
    a, n, B = np.concatenate([M, Y], 2), len(M), M.shape[1]
    rows = np.arange(n)
    for k in range(B):
        p = k + np.argmax(np.abs(a[:, k:, k]), 1)
        t = a[:, k].copy()
        a[:, k] = a[rows, p]
        a[rows, p] = t
        for r in range(k + 1, B):
            a[:, r, k + 1:] -= (a[:, r, k] / a[:, k, k])[:, None] * a[:, k, k + 1:]
    X = np.zeros_like(Y)
    for r in range(B - 1, -1, -1):
        v = a[:, r, B:].copy()
        for m in range(r + 1, B):
            v -= a[:, r, m][:, None] * X[:, m]
        X[:, r] = v / a[:, r, r][:, None]
    return X


def _cholesky(A):
    n, B = len(A), A.shape[1]
    Lc, Li = np.zeros_like(A), np.zeros_like(A)
    for k in range(B):
        d = A[:, k, k].real.copy()
        for m in range(k):
            d -= np.abs(Lc[:, k, m] ** 2) if A.dtype != np.complex128 else Lc[:, k, m].real ** 2 + Lc[:, k, m].imag ** 2
        Lc[:, k, k] = np.sqrt(d)
        for r in range(k + 1, B):
            v = A[:, r, k].copy()
            for m in range(k):
                v -= Lc[:, r, m] * Lc[:, k, m].conj()
            Lc[:, r, k] = v / Lc[:, k, k].real
    for j in range(B):
        for r in range(j, B):
            v = np.full(n, 1.0 if r == j else 0.0, A.dtype)
            for m in range(j, r):
                v -= Lc[:, r, m] * Li[:, m, j]
            Li[:, r, j] = v / Lc[:, r, r].real
    return Lc, Li


def _random(B, n, seed):
    r = np.random.default_rng(seed)
    return r, lambda: r.standard_normal((n, B, B)) + 1j * r.standard_normal((n, B, B))


@pytest.mark.parametrize("B", [4, 8, 16])
def test_elimination(lib, B):
    # complex symmetric, mostly diagonal, like P^T A P and Q^T Q of a block; a third of
    # them with rows and columns scaled over two decades
    n = 800
    r, z = _random(B, n, B)
    M = 0.15 * z()
    M = M + M.transpose(0, 2, 1) + np.exp(2j * np.pi * r.random((n, B)))[:, :, None] * np.eye(B)
    s = np.where(np.arange(n)[:, None] % 3 == 0, 10.0 ** r.uniform(-1, 1, (n, B)), 1.0)
    M, Y = M * s[:, :, None] * s[:, None, :], z()
    ref = np.linalg.solve(M, Y).astype(np.clongdouble)
    for _ in range(4):
        res = Y - np.einsum("nij,njk->nik", M.astype(np.clongdouble), ref)
        ref = ref + np.linalg.solve(M, res.astype(complex))
    (X,) = _gpu(lib.solve, B, n, [M, Y], 1)
    got, want = _err(X, ref), _err(_eliminate(M, Y), ref)
    assert np.all(got <= 1.1 * want), (got, want)


@pytest.mark.parametrize("B", [4, 8, 16])
def test_cholesky_and_inverse(lib, B):
    n = 800
    r, z = _random(B, n, 100 + B)
    W = np.eye(B) + 0.2 * z()
    s = np.where(np.arange(n)[:, None] % 3 == 0, 10.0 ** r.uniform(-1, 1, (n, B)), 1.0)
    W = W * s[:, None, :]
    A = np.einsum("nji,njk->nik", W.conj(), W)
    A = 0.5 * (A + A.transpose(0, 2, 1).conj())
    L_ref, Li_ref = _cholesky(A.astype(np.clongdouble))
    U, Li = _gpu(lib.chol, B, n, [A], 2)
    L_tb, Li_tb = _cholesky(A)
    for got, want in ((_err(U.conj().transpose(0, 2, 1), L_ref), _err(L_tb, L_ref)), (_err(Li, Li_ref), _err(Li_tb, Li_ref))):
        assert np.all(got <= 1.1 * want), (got, want)


def test_singular_systems_are_refused(lib):
    M = np.zeros((2, 4, 4), complex)
    M[0] = np.eye(4)
    M[0, 2, 2] = 0.0
    M[1] = np.eye(4) * np.nan
    (X,) = _gpu(lib.solve, 4, 2, [M, M], 1)
    assert np.all(np.isnan(X))
    A = np.stack([np.diag([1.0, 1.0, -1.0, 1.0]), np.ones((4, 4))]).astype(complex)
    U, _ = _gpu(lib.chol, 4, 2, [A], 2)
    assert np.all(np.isnan(U))
