"""The FP64 sine and cosine of the quadrature kernels (cis64 in bie_common.cuh) by themselves, over the phases
k R of their use, multiples of pi / 2, and beyond 2^18, where CUDA's function takes over.  The argument's
difference to the multiple of pi / 2 is exact in its first step and rounds once in the second; the two
series are evaluated with one rounding a step, the last ones of the size of the result's: 2 x 2^-53 for
the polynomial and 2^-53 for the difference, 3.4e-16 in all, and numpy's own 1.2e-16."""
import ctypes
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))
SRC = r"""
#include "bie_common.cuh"
__global__ void k(const double* x, int64_t n, double* o) {
  const int64_t i = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (i >= n) return;
  bie::cis64(x[i], o[4 * i], o[4 * i + 1]);
  sincos(x[i], &o[4 * i + 2], &o[4 * i + 3]);
}
extern "C" int run(const double* x, int64_t n, double* o) {
  k<<<(unsigned)((n + 255) / 256), 256>>>(x, n, o);
  return (int)cudaDeviceSynchronize();
}
"""


def test_cis64(tmp_path):
    import torch
    from paper_1706_07919_gb300 import build

    src, so = tmp_path / "cis.cu", tmp_path / "cis.so"
    src.write_text(SRC)
    subprocess.run([build._nvcc(), *build.ARCH, *build.FLAGS, "-I", os.path.join(ROOT, "paper_1706_07919_gb300", "csrc"),
                    "-I", os.path.join(ROOT, "include"), "-shared", str(src), "-o", str(so)], check=True)
    lib = ctypes.CDLL(str(so))
    lib.run.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_void_p]
    rng = np.random.default_rng(1)
    q = np.arange(-4000, 4001) * (np.pi / 2)
    x = np.concatenate([rng.uniform(-np.pi, np.pi, 2 ** 20), rng.uniform(-400, 400, 2 ** 22),
                        rng.uniform(-2.0 ** 18, 2.0 ** 18, 2 ** 22), 10.0 ** rng.uniform(-300, 0, 2 ** 16), q, q * (1 + 2e-16),
                        [0.0, -0.0, 2.0 ** 18, -2.0 ** 18, np.nextafter(2.0 ** 18, 1e9), 1e10, -3e22]])
    xd = torch.tensor(x, device="cuda:0")
    o = torch.empty((len(x), 4), dtype=torch.float64, device="cuda:0")
    torch.cuda.synchronize()
    assert lib.run(xd.data_ptr(), len(x), o.data_ptr()) == 0
    s, c, s0, c0 = o.cpu().numpy().T
    tol = 3.4e-16 + 1.2e-16
    assert np.max(np.abs(s - np.sin(x))) <= tol and np.max(np.abs(c - np.cos(x))) <= tol
    far = np.abs(x) > 2.0 ** 18
    assert far.sum() == 3 and np.array_equal(s[far], s0[far]) and np.array_equal(c[far], c0[far])
    print("largest difference to CUDA's sincos: %.2e, %.2e" % (np.max(np.abs(s - s0)), np.max(np.abs(c - c0))))
    tiny = np.abs(x) < 1e-3  # relative there: no multiple of pi / 2 is taken off
    assert np.all(np.abs(s[tiny] - np.sin(x[tiny])) <= 4.5e-16 * np.abs(x[tiny]))
