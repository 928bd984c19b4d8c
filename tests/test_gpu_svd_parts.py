"""Parts of the truncated block SVD (csrc/svd_eig.cuh) by themselves, on inputs that no gate brings about on purpose:
a small kernel around each is compiled here."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

from paper_2404_10223_gb300 import build as B

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include <cuda_runtime.h>
#include "svd_eig.cuh"
using namespace tnqe;
struct Warp {                                      // a team of one warp
  __device__ int rank() const { return (int)threadIdx.x; }
  __device__ int size() const { return 32; }
  __device__ void sync() const { __syncwarp(); }
  __device__ float max(float v) const { return warp_max_f(v); }
};
extern __shared__ float4 pool4[];
__global__ void defect_kernel(const float* X, int n, int ld, float* out) {
  const float r = eig_defect<false>(Warp{}, X, n, ld, reinterpret_cast<float*>(pool4));
  if (threadIdx.x == 0) *out = r;
}
__global__ void angles_kernel(const float* X, const float* Rg, int n, int ld, int kc, int kp, const float* lam, float* out) {
  float* R = reinterpret_cast<float*>(pool4);
  double* lk = reinterpret_cast<double*>(R + kp * ld);
  float* lh = reinterpret_cast<float*>(lk + kp);
  float* ek = lh + kp;
  float* l = ek + kp;
  float* T = l + ld;
  for (int x = threadIdx.x; x < kp * ld; x += 32) R[x] = Rg[x];
  for (int x = threadIdx.x; x < n; x += 32) l[x] = lam[x];
  for (int x = threadIdx.x; x < kp; x += 32) {
    lk[x] = lh[x] = x < kc ? lam[x] : 0.f;
    ek[x] = 0.f;
  }
  __syncwarp();
  const float r = eig_angles(Warp{}, X, R, n, ld, kc, kp, lk, lh, ek, l, T);
  if (threadIdx.x == 0) *out = r;
}
static float* up(const float* h, int n) {
  float* d = nullptr;
  cudaMalloc(&d, sizeof(float) * n);
  cudaMemcpy(d, h, sizeof(float) * n, cudaMemcpyHostToDevice);
  return d;
}
extern "C" int run_defect(const float* X, int n, float* out) {
  const int ld = eig_ld(n);
  float *dX = up(X, n * ld), *d = up(out, 1);
  defect_kernel<<<1, 32, n * ld * 4>>>(dX, n, ld, d);
  cudaMemcpy(out, d, 4, cudaMemcpyDeviceToHost);
  cudaFree(dX);
  cudaFree(d);
  return (int)cudaGetLastError();
}
extern "C" int run_angles(const float* X, const float* R, int n, int kc, const float* lam, float* out) {
  const int ld = eig_ld(n), kp = eig_kp(kc);
  float *dX = up(X, n * ld), *dR = up(R, kp * ld), *dl = up(lam, n), *d = up(out, 1);
  angles_kernel<<<1, 32, (kp * ld + 4 * kp + ld + n * kp) * 4>>>(dX, dR, n, ld, kc, kp, dl, d);
  cudaMemcpy(out, d, 4, cudaMemcpyDeviceToHost);
  cudaFree(dX);
  cudaFree(dR);
  cudaFree(dl);
  cudaFree(d);
  return (int)cudaGetLastError();
}
extern "C" int row_stride(int n) { return eig_ld(n); }
"""


@pytest.fixture(scope="module")
def parts(tmp_path_factory):
    d = tmp_path_factory.mktemp("svd_parts")
    src, lib = os.path.join(d, "parts.cu"), os.path.join(d, "parts.so")
    with open(src, "w") as f:
        f.write(SOURCE)
    subprocess.run([B.nvcc()] + B.ARCH + B.COMMON + ["-I" + B.CSRC, "-shared", "-o", lib, src], check=True)
    return ctypes.CDLL(lib)


def p(a):
    return a.ctypes.data_as(ctypes.c_void_p)


def vectors(lib, n):
    """n orthonormal vectors, one per row of the padded stride."""
    X = np.zeros((n, lib.row_stride(n)), dtype=np.float32)
    X[:, :n] = np.linalg.qr(np.random.default_rng(n).normal(size=(n, n)))[0]
    return X


@pytest.mark.parametrize("n", [5, 8, 33])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_vector_that_is_not_finite_is_never_orthonormal(parts, n, bad):
    out = np.zeros(1, dtype=np.float32)
    X = vectors(parts, n)
    assert parts.run_defect(p(X), n, p(out)) == 0 and out[0] < 1e-5
    for row in (0, n // 2, n - 1):
        Y = X.copy()
        Y[row, 0] = bad
        assert parts.run_defect(p(Y), n, p(out)) == 0
        assert out[0] >= 1e29


@pytest.mark.parametrize("n,kc", [(9, 3), (33, 9), (40, 40)])
@pytest.mark.parametrize("bad", [np.nan, np.inf])
def test_a_residual_that_is_not_finite_is_never_converged(parts, n, kc, bad):
    out = np.zeros(1, dtype=np.float32)
    X = vectors(parts, n)
    lam = np.linspace(2.0, 0.1, n, dtype=np.float32)
    R = np.zeros(((kc + 7) // 8 * 8, X.shape[1]), dtype=np.float32)
    assert parts.run_angles(p(X), p(R), n, kc, p(lam), p(out)) == 0 and out[0] == 0.0
    for k in (0, kc // 2, kc - 1):
        Q = R.copy()
        Q[k, n - 1] = bad
        assert parts.run_angles(p(X), p(Q), n, kc, p(lam), p(out)) == 0
        assert out[0] >= 1e29
