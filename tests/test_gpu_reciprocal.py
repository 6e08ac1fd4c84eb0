"""The node update's own reciprocal and square root (lbm_node.cuh) against CUDA's
correctly rounded division and square root, over the exponents that densities,
temperatures and the viscosity laws' denominators reach.

Bounds (relative, u = 2^-53 or 2^-24 the unit roundoff): one Newton (FP32) or cubic
(FP64) step from an estimate of at least 20 (FP64) and 22 (FP32) good bits leaves a
truncation error below u / 8, and the rounding of the last fused multiply-add adds u;
the reference's rounding adds another u: 2.25 u.  The square root also rounds v y once,
which enters with half its weight: 2.75 u."""
import ctypes
import subprocess

import numpy as np
import pytest

from paper_1109_6672_gb300 import build

pytestmark = pytest.mark.gpu

SOURCE = r"""
#include "lbm_node.cuh"
template <class T>
__global__ void probe(int n, const T* v, T* r, T* s, T* r0, T* s0) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  r[i] = lbm::rcp_(v[i]);
  s[i] = lbm::sqrt_(v[i]);
  r0[i] = T(1) / v[i];
  s0[i] = sqrt(v[i]);
}
template <class T>
int run(int n, const T* v, T* out) {
  T *d, *o;
  if (cudaMalloc(&d, 5 * n * sizeof(T)) != cudaSuccess) return 1;
  o = d + n;
  cudaMemcpy(d, v, n * sizeof(T), cudaMemcpyHostToDevice);
  probe<T><<<(n + 255) / 256, 256>>>(n, d, o, o + n, o + 2 * n, o + 3 * n);
  const cudaError_t e = cudaMemcpy(out, o, 4 * n * sizeof(T), cudaMemcpyDeviceToHost);
  cudaFree(d);
  return e != cudaSuccess;
}
extern "C" int run64(int n, const double* v, double* out) { return run<double>(n, v, out); }
extern "C" int run32(int n, const float* v, float* out) { return run<float>(n, v, out); }
"""


@pytest.fixture(scope="module")
def lib(tmp_path_factory):
    d = tmp_path_factory.mktemp("probe")
    (d / "probe.cu").write_text(SOURCE)
    subprocess.run([build.nvcc(), *build.NVCC_FLAGS, *build.ARCH, "-shared", str(d / "probe.cu"),
                    "-o", str(d / "probe.so")], check=True)
    return ctypes.CDLL(str(d / "probe.so"))


@pytest.mark.parametrize("dtype,call,u,span", [(np.float64, "run64", 2.0 ** -53, 300),
                                               (np.float32, "run32", 2.0 ** -24, 60)])
def test_reciprocal_and_square_root(lib, dtype, call, u, span):
    rng = np.random.default_rng(7)
    v = np.concatenate([rng.uniform(0.25, 4.0, 400000),
                        np.exp2(rng.uniform(-span, span, 400000)),
                        np.exp2(np.arange(-span, span + 1.0)),
                        1.0 + u * np.arange(-64, 65)]).astype(dtype)
    out = np.empty((4, v.size), dtype)
    assert getattr(lib, call)(v.size, v.ctypes.data_as(ctypes.c_void_p),
                              out.ctypes.data_as(ctypes.c_void_p)) == 0
    r, s, r0, s0 = out.astype(np.longdouble)
    assert np.abs(r / r0 - 1).max() <= 2.25 * u
    assert np.abs(s / s0 - 1).max() <= 2.75 * u
