"""Direct test of the lane-group Slater inverse group_inverse (wf_device.cuh) at the edges of its
register sizes (8, 16, 32) and group sizes, several matrices per warp where they fit.

Inputs: random orthogonal matrices with rows scaled by powers of two and permuted (condition
number 1 up to an exact scaling, so that pivots off the diagonal are needed), and singular ones
(a zero column).  Gauss-Jordan elimination with partial pivoting on such a matrix leaves
|B A - I| <= c n^2 eps with a small c: 1e-12 is four orders above n^2 eps at n = 32.  ln|det| and
the trace carry the same relative error times n: 1e-11.  A zero column gives sign 0 and a zero
inverse exactly."""
import ctypes
import os
import subprocess
import tempfile

import numpy as np
import pytest

pytestmark = pytest.mark.gpu
torch = pytest.importorskip("torch")

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2207_14715_gb300", "csrc")

PROBE = r"""
#include "wf_device.cuh"
// one warp: m matrices A [m][n][n], L [m][n][n] -> B [m][n][n], det [m][3] (mant, exponent, sign), tr [m]
__global__ void probe(int m, int n, int G, const double* A, const double* L, double* B, double* det, double* tr) {
  __shared__ int perm[32 * 32];
  const int lane = threadIdx.x, ng = 32 / G, g = lane / G;
  for (int u0 = 0; u0 < m; u0 += ng) {
    const int u = u0 + g;
    const bool act = u < m;
    const size_t o = (size_t)(act ? u : 0) * n * n;
    const vbq::GroupDet d = vbq::group_inverse<double>(A + o, n, nullptr, n, G, act, perm + g * n, nullptr, nullptr,
                                                       B + o, L + o, n);
    if (act && lane % G == 0) {
      det[3 * u] = d.mant;
      det[3 * u + 1] = d.ex;
      det[3 * u + 2] = d.sgn;
      tr[u] = d.trace;
    }
    __syncwarp();
  }
}
extern "C" int run(int m, int n, int G, const double* A, const double* L, double* B, double* det, double* tr) {
  const size_t b = sizeof(double) * m * n * n;
  double *dA = nullptr, *dL = nullptr, *dB = nullptr, *dd = nullptr, *dt = nullptr;
  cudaError_t e = cudaMalloc(&dA, b);
  if (e == cudaSuccess) e = cudaMalloc(&dL, b);
  if (e == cudaSuccess) e = cudaMalloc(&dB, b);
  if (e == cudaSuccess) e = cudaMalloc(&dd, 24 * m);
  if (e == cudaSuccess) e = cudaMalloc(&dt, 8 * m);
  if (e == cudaSuccess) e = cudaMemcpy(dA, A, b, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(dL, L, b, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    probe<<<1, 32>>>(m, n, G, dA, dL, dB, dd, dt);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(B, dB, b, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(det, dd, 24 * m, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(tr, dt, 8 * m, cudaMemcpyDeviceToHost);
  cudaFree(dA); cudaFree(dL); cudaFree(dB); cudaFree(dd); cudaFree(dt);
  return (int)e;
}
"""


@pytest.fixture(scope="module")
def lib():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    d = tempfile.mkdtemp(prefix="inverse_probe_")
    src, so = os.path.join(d, "probe.cu"), os.path.join(d, "probe.so")
    with open(src, "w") as f:
        f.write(PROBE)
    subprocess.run([os.environ.get("NVCC", "nvcc"), "-gencode", "arch=compute_103a,code=sm_103a", "-O3",
                    "-std=c++17", "-shared", "-Xcompiler", "-fPIC", "-I", CSRC, src, "-o", so], check=True)
    lib = ctypes.CDLL(so)
    lib.run.argtypes = [ctypes.c_int] * 3 + [ctypes.c_void_p] * 5
    return lib


@pytest.mark.parametrize("n", [1, 2, 3, 4, 7, 8, 9, 15, 16, 17, 24, 31, 32])
def test_inverse(lib, n):
    rng = np.random.default_rng(n)
    m, G = 11, 1 << (n - 1).bit_length()
    A = np.linalg.qr(rng.normal(size=(m, n, n)))[0]
    A = A * 2.0 ** rng.integers(-40, 40, size=(m, n, 1))
    A = np.ascontiguousarray(A[:, rng.permutation(n), :])
    A[4, :, n // 2] = 0.0
    L = rng.normal(size=(m, n, n))
    B, det, tr = np.full((m, n, n), 7.0), np.zeros((m, 3)), np.zeros(m)
    assert lib.run(m, n, G, A.ctypes.data, L.ctypes.data, B.ctypes.data, det.ctypes.data, tr.ctypes.data) == 0
    for u in range(m):
        if u == 4:
            assert det[u, 2] == 0.0 and not B[u].any()
            continue
        assert np.abs(B[u] @ A[u] - np.eye(n)).max() < 1e-12
        sign, ln = np.linalg.slogdet(A[u])
        assert det[u, 2] == sign and 1.0 <= det[u, 0] < 2.0 ** n
        assert abs(np.log(det[u, 0]) + det[u, 1] * np.log(2.0) - ln) < 1e-11 * max(1.0, abs(ln))
        inv = np.linalg.inv(A[u])
        assert abs(tr[u] - np.trace(inv @ L[u])) < 1e-11 * np.abs(inv.T * L[u]).sum()
