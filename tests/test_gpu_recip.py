"""recip_f64 (the FP64 collision's and base chain's 1 / rho) against 1 / v in
extended precision: random densities around 1, over the range that it is stated
for, powers of two and their neighbours.  Bound: half an ulp for the last
rounding and 2^-19 of one for what the two Newton steps leave."""
import ctypes
import subprocess

import numpy as np
import pytest

gpu = pytest.mark.gpu
SRC = r"""
#include "ehd_dev.cuh"
__global__ void k(const double* v, double* x, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) x[i] = ehd::recip_f64(v[i]);
}
extern "C" int recip(const double* v, double* x, int n) {
  double *dv = nullptr, *dx = nullptr;
  cudaError_t e = cudaMalloc(&dv, n * sizeof(double));
  if (e == cudaSuccess) e = cudaMalloc(&dx, n * sizeof(double));
  if (e == cudaSuccess) e = cudaMemcpy(dv, v, n * sizeof(double), cudaMemcpyHostToDevice);
  if (e == cudaSuccess) {
    k<<<(n + 255) / 256, 256>>>(dv, dx, n);
    e = cudaMemcpy(x, dx, n * sizeof(double), cudaMemcpyDeviceToHost);
  }
  cudaFree(dv);
  cudaFree(dx);
  return (int)e;
}
"""


@gpu
def test_recip_f64_half_an_ulp(tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    if np.finfo(np.longdouble).nmant < 63:
        pytest.skip("no extended precision on this host")
    from paper_1812_05711_gb300 import _build
    src, lib = tmp_path / "recip.cu", tmp_path / "recip.so"
    src.write_text(SRC)
    subprocess.run([_build.NVCC, *_build.ARCH, *_build.FLAGS, "-shared", str(src), "-o", str(lib)], check=True)
    rng = np.random.default_rng(5)
    p2 = 2.0 ** np.arange(-990, 990)
    v = np.concatenate([1 + rng.uniform(-0.5, 0.5, 1 << 20), 1 + rng.standard_normal(1 << 20) * 1e-6,
                        rng.uniform(1, 2, 1 << 18) * 2.0 ** rng.integers(-990, 990, 1 << 18),
                        p2, np.nextafter(p2, 0), np.nextafter(p2, np.inf), np.nextafter(np.nextafter(p2, 0), 0)])
    v = np.concatenate([v, -v])
    x = np.empty_like(v)
    f = ctypes.CDLL(str(lib)).recip
    ptr = ctypes.POINTER(ctypes.c_double)
    assert f(v.ctypes.data_as(ptr), x.ctypes.data_as(ptr), ctypes.c_int(v.size)) == 0
    exact = 1 / v.astype(np.longdouble)
    ulp = np.abs(np.spacing(1 / v)).astype(np.longdouble)
    err = np.abs(x.astype(np.longdouble) - exact) / ulp
    print("worst error", float(err.max()), "ulp; not correctly rounded:", int((x != 1 / v).sum()), "of", v.size)
    assert float(err.max()) <= 0.5 + 2.0 ** -19
