"""Direct test of the Slater inverses of wf_device.cuh at the edges of their register sizes (8, 16,
32) and group sizes: the lane-group LU (several matrices per warp where they fit) and the
whole-warp Gauss-Jordan inverse.

Inputs: random orthogonal matrices with rows scaled by powers of two and permuted (condition
number 1 up to an exact scaling, so that pivots off the diagonal are needed), and singular ones
(a zero column).  Elimination with partial pivoting on such a matrix leaves |B A - I| <= c n^2 eps
with a small c: 1e-12 is four orders above n^2 eps at n = 32.  ln|det| carries the same relative
error times n: 1e-11.  A zero column gives sign 0 and a zero inverse exactly."""
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
// one warp: m matrices A [m][n][n] -> B [m][n][n], det [m][3] (mant, exponent, sign)
__global__ void probe_lu(int m, int n, int G, const double* A, const int* idx, double* B, double* det) {
  __shared__ double scr[2 * 32 * 33 + 32 * 9];
  __shared__ int perm[32 * 32];
  const int lane = threadIdx.x, ng = 32 / G, g = lane / G, gl = lane % G, lda = n | 1;
  for (int u0 = 0; u0 < m; u0 += ng) {
    const int u = u0 + g;
    const bool act = u < m;
    const size_t o = (size_t)(act ? u : 0) * n * n;
    double* S = scr + g * n * lda;
    int* p = perm + g * n;
    const vbq::GroupDet d = n <= 8    ? vbq::group_lu8(A + o, n, idx, n, G, act, S, p)
                            : n <= 16 ? vbq::group_lu16(A + o, n, idx, n, G, act, S, p)
                                      : vbq::group_lu_smem(A + o, n, idx, n, G, act, S, scr + n * lda, p);
    if (act && gl < n)
      for (int i = 0; i < n; ++i) B[o + i * n + gl] = S[i * lda + gl];
    if (act && gl == 0) {
      det[3 * u] = d.mant;
      det[3 * u + 1] = d.ex;
      det[3 * u + 2] = d.sgn;
    }
    __syncwarp();
  }
}
__global__ void probe_gj(int m, int n, const double* A, double* B, double* det) {
  __shared__ int perm[32];
  for (int u = 0; u < m; ++u) {
    const size_t o = (size_t)u * n * n;
    const vbq::GroupDet d = vbq::warp_inverse(A + o, n, nullptr, n, perm, B + o);
    if (threadIdx.x == 0) {
      det[3 * u] = d.mant;
      det[3 * u + 1] = d.ex;
      det[3 * u + 2] = d.sgn;
    }
    __syncwarp();
  }
}
extern "C" int run(int gj, int m, int n, int G, const double* A, const int* idx, double* B, double* det) {
  const size_t b = sizeof(double) * m * n * n;
  double *dA = nullptr, *dB = nullptr, *dd = nullptr;
  int* di = nullptr;
  cudaError_t e = cudaMalloc(&dA, b);
  if (e == cudaSuccess) e = cudaMalloc(&dB, b);
  if (e == cudaSuccess) e = cudaMalloc(&dd, 24 * m);
  if (e == cudaSuccess) e = cudaMalloc(&di, 4 * n);
  if (e == cudaSuccess) e = cudaMemcpy(dA, A, b, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemcpy(di, idx, 4 * n, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    if (gj) probe_gj<<<1, 32>>>(m, n, dA, dB, dd);
    else probe_lu<<<1, 32>>>(m, n, G, dA, di, dB, dd);
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemcpy(B, dB, b, cudaMemcpyDeviceToHost);
  if (e == cudaSuccess) e = cudaMemcpy(det, dd, 24 * m, cudaMemcpyDeviceToHost);
  cudaFree(dA); cudaFree(dB); cudaFree(dd); cudaFree(di);
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
    lib.run.argtypes = [ctypes.c_int] * 4 + [ctypes.c_void_p] * 4
    return lib


@pytest.mark.parametrize("n", [1, 2, 3, 4, 7, 8, 9, 15, 16, 17, 24, 31, 32])
@pytest.mark.parametrize("gj", [0, 1])
def test_inverse(lib, n, gj):
    rng = np.random.default_rng(n)
    m, G = 11, 1 << (n - 1).bit_length()
    A = np.linalg.qr(rng.normal(size=(m, n, n)))[0]
    A = A * 2.0 ** rng.integers(-40, 40, size=(m, n, 1))
    A = np.ascontiguousarray(A[:, rng.permutation(n), :])
    A[4, :, n // 2] = 0.0
    idx = np.arange(n, dtype=np.int32) if gj else rng.permutation(n).astype(np.int32)
    B, det = np.full((m, n, n), 7.0), np.zeros((m, 3))
    assert lib.run(gj, m, n, G, A.ctypes.data, idx.ctypes.data, B.ctypes.data, det.ctypes.data) == 0
    for u in range(m):
        if u == 4:
            assert det[u, 2] == 0.0 and not B[u].any()
            continue
        M = A[u][:, idx]
        assert np.abs(B[u] @ M - np.eye(n)).max() < 1e-12
        sign, ln = np.linalg.slogdet(M)
        assert det[u, 2] == sign and 1.0 <= det[u, 0] < 2.0 ** n
        assert abs(np.log(det[u, 0]) + det[u, 1] * np.log(2.0) - ln) < 1e-11 * max(1.0, abs(ln))
