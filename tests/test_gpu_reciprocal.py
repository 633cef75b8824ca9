"""The FP64 reciprocal of the collision kernels against the division."""
import ctypes
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SRC = """
#include "lbm_internal.h"
__global__ void k(const double* x, double* y, double* seed, int n) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  y[i] = lbm::rcp_f64(x[i]);
  asm("rcp.approx.ftz.f64 %0, %1;" : "=d"(seed[i]) : "d"(x[i]));
}
extern "C" int run(const double* x, double* y, double* seed, int n) {
  k<<<(n + 255) / 256, 256>>>(x, y, seed, n);
  return (int)cudaDeviceSynchronize();
}
"""


def test_rcp_f64_against_division(tmp_path):
    """Within one unit in the last place of 1 / x for densities of 1e-8 to 1e8:
    one iteration of third order on a seed of relative error e0 leaves e0^3 and
    the rounding of its last multiply-add, half a unit; any e0 below 2^-18 keeps
    the sum below one.  The seed's own error is printed."""
    import torch
    from paper_1904_11792_gb300 import build
    src, lib = tmp_path / "rcp.cu", tmp_path / "rcp.so"
    src.write_text(SRC)
    subprocess.run([build.nvcc(), *build.ARCH, *build.FLAGS, "-shared", "-I", build.INCLUDE, "-I", build.CSRC,
                    str(src), "-o", str(lib), "-lcudart"], check=True)
    rng = np.random.default_rng(11)
    edges = np.concatenate([[v, np.nextafter(v, 0), np.nextafter(v, 9e99)] for v in 2.0 ** np.arange(-26, 27)])
    x = np.concatenate([edges, 10.0 ** rng.uniform(-8, 8, 1 << 21), rng.uniform(0.05, 3.0, 1 << 21)])
    tx = torch.from_numpy(x).cuda()
    y, seed = torch.zeros_like(tx), torch.zeros_like(tx)
    run = ctypes.CDLL(str(lib)).run
    assert run(ctypes.c_void_p(tx.data_ptr()), ctypes.c_void_p(y.data_ptr()), ctypes.c_void_p(seed.data_ptr()),
               x.size) == 0
    want = 1.0 / x
    e0 = np.abs(seed.cpu().numpy() / want - 1.0)
    ulps = np.abs(y.cpu().numpy() - want) / np.spacing(want)
    print("seed error 2^%.2f, result within %g units, %.4f %% not as the division" %
          (np.log2(e0.max()), ulps.max(), 100.0 * (ulps > 0).mean()))
    assert ulps.max() <= 1.0
