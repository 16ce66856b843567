"""The blocked Cholesky factor and triangular solves of Rayleigh-Ritz, on integers.

L has small integer entries, so A = L L^T, the Schur complements and every partial sum are
integers below 2^53: square roots and quotients are integers too, and a factorisation that takes
correctly rounded roots and quotients returns L itself, a solve its integer solution.  A product
with a rounded reciprocal misses some (49 * (1 / 49) < 1).  The kernels have no entry point of
their own; the test compiles their source with one.  Sizes around the block of 32.
"""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2512_08571_gb300 import build as B
from paper_2512_08571_gb300 import fe_ks as fk

torch = pytest.importorskip("torch")
pytestmark = pytest.mark.gpu

SRC = r"""
#include "fe_ks_rr.cu"
extern "C" int factor(double* A, double* scratch, int n, int* flag) {
  feks::rr_cholesky(A, scratch, n, 0.0, flag, nullptr);
  return cudaDeviceSynchronize();
}
extern "C" int solve(const double* L, double* B, int n, int nr, int trans) {
  if (trans)
    feks::k_rr_trsm<true><<<(nr + 3) / 4, 128>>>(L, B, n, nr);
  else
    feks::k_rr_trsm<false><<<(nr + 3) / 4, 128>>>(L, B, n, nr);
  return cudaDeviceSynchronize();
}
__global__ void k_quotients(const double* x, const double* d, double* q, double* want, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  q[i] = feks::quotient(x[i], d[i], 1.0 / d[i]);
  want[i] = x[i] / d[i];
}
extern "C" int quotients(const double* x, const double* d, double* q, double* want, int n) {
  k_quotients<<<(n + 255) / 256, 256>>>(x, d, q, want, n);
  return cudaDeviceSynchronize();
}
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("rr_factor")
    (d / "t.cu").write_text(SRC)
    out = d / "t.so"
    r = subprocess.run([B._nvcc(), *B.ARCH, *B.FLAGS, "-I" + B.CSRC, "-shared", str(d / "t.cu"), "-o", str(out),
                        fk.LIB_PATH, "-Xlinker", "-rpath", "-Xlinker", os.path.dirname(fk.LIB_PATH), "-lcusolver"],
                       capture_output=True, text=True)
    assert r.returncode == 0, r.stderr
    lib = ctypes.CDLL(str(out))
    vp = ctypes.c_void_p
    lib.factor.argtypes = [vp, vp, ctypes.c_int, vp]
    lib.solve.argtypes = [vp, vp, ctypes.c_int, ctypes.c_int, ctypes.c_int]
    lib.quotients.argtypes = [vp, vp, vp, vp, ctypes.c_int]
    return lib


def test_quotient_is_the_rounded_one(lib):
    """Markstein's theorem: with the rounded reciprocal the corrected quotient is CUDA's x / d bit for bit
    (entries of any size that a factor of a matrix with unit diagonal can meet)."""
    rng = np.random.default_rng(7)
    n = 1 << 20
    x = torch.from_numpy(rng.standard_normal(n) * 10.0 ** rng.uniform(-30, 3, n)).cuda()
    d = torch.from_numpy(rng.uniform(0.5, 2, n) * 10.0 ** rng.uniform(-8, 3, n)).cuda()
    q, want = torch.empty_like(x), torch.empty_like(x)
    assert lib.quotients(x.data_ptr(), d.data_ptr(), q.data_ptr(), want.data_ptr(), n) == 0
    assert torch.equal(q, want)


@pytest.mark.parametrize("n", [1, 5, 31, 32, 33, 64, 96, 130])
def test_integer_factor_and_solves_are_exact(lib, n):
    rng = np.random.default_rng(40 + n)
    L = np.tril(rng.integers(-3, 4, (n, n)), -1) + np.diag(rng.integers(1, 50, n) * 2 + 1)
    dev = lambda a: torch.from_numpy(np.ascontiguousarray(a, dtype=np.float64)).cuda()
    A, scratch = dev(L @ L.T), torch.zeros(32 * 32, dtype=torch.float64, device="cuda")
    flag = torch.zeros(1, dtype=torch.int32, device="cuda")
    assert lib.factor(A.data_ptr(), scratch.data_ptr(), n, flag.data_ptr()) == 0
    assert flag.item() == 0
    assert np.array_equal(np.tril(A.cpu().numpy()), L)
    Z = rng.integers(-9, 10, (n, 7))
    for trans, M in ((0, L), (1, L.T)):
        X = dev(M @ Z)
        assert lib.solve(dev(L).data_ptr(), X.data_ptr(), n, 7, trans) == 0
        assert np.array_equal(X.cpu().numpy(), Z), trans
