"""The FP64 reciprocal of the sweep (Num<double>::rcp in csrc/sweep.cuh): the PTX approximation, whose
relative error is about 2^-20, and one step of Householder's third-order iteration, which cubes it.
With |e| <= 2^-19 the truncation e^3 is at most 2^-57, the rounding of the last operation 2^-53,
and the others are below 2^-70: at most 2^-53 (1 + 2^-4) in all.  Compared with 1/x in long double
(64 or 113 bits) on a small program compiled for this test."""
import ctypes
import subprocess

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

if not torch.cuda.is_available():
    pytest.skip("CUDA device required", allow_module_level=True)

from paper_2101_05886_gb300 import build  # noqa: E402

PROGRAM = r"""
#include "sweep.cuh"
__global__ void k_rcp(const double *x, double *r, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i < n) r[i] = fpk::Num<double>::rcp(x[i]);
}
extern "C" int run_rcp(const double *x_dev, double *r_dev, int n) {
  k_rcp<<<(n + 255) / 256, 256>>>(x_dev, r_dev, n);
  cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? (int)cudaDeviceSynchronize() : (int)e;
}
"""


def test_reciprocal_error(tmp_path):
    src, lib = tmp_path / "rcp.cu", tmp_path / "librcp.so"
    src.write_text(PROGRAM)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-I", build.CSRC, "-shared", str(src), "-o", str(lib)],
                   check=True, capture_output=True)
    rng = np.random.default_rng(11)
    m = np.concatenate([1.0 + rng.random(1 << 18), 1.0 + np.arange(1 << 12) * 2.0 ** -12, 2.0 - np.arange(1, 1 << 12) * 2.0 ** -52,
                        1.0 + np.arange(1 << 12) * 2.0 ** -52])
    e = rng.integers(-1020, 1021, size=m.size)
    e[: m.size // 2] = rng.integers(-40, 41, size=m.size // 2)
    x = np.ldexp(m, e) * rng.choice([-1.0, 1.0], size=m.size)
    xd = torch.as_tensor(x, device="cuda")
    rd = torch.full_like(xd, float("nan"))
    L = ctypes.CDLL(str(lib))
    assert L.run_rcp(ctypes.c_void_p(xd.data_ptr()), ctypes.c_void_p(rd.data_ptr()), ctypes.c_int(x.size)) == 0
    r = rd.cpu().numpy()
    assert np.isfinite(r).all()
    err = np.abs(r.astype(np.longdouble) * x.astype(np.longdouble) - 1)
    assert float(err.max()) <= 2.0 ** -53 * (1 + 2.0 ** -4) + 2.0 ** -62, float(err.max()) * 2.0 ** 53
