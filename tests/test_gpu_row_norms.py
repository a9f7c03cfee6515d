"""Squared norms of FP32 rows (row_sumsq, csrc/vecops.cu) keep the roundings of their FP32
squares and sums: whole numbers below 2^15 (inexact squares and sums of them) give
exact norms."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHIM = r"""
#include "vecops.cuh"
extern "C" void norms(const float* x, long long ld, int k, int n, double* out) {
  tddft::row_sumsq<float>(x, ld, k, n, out, 0);
}
"""


@pytest.mark.parametrize("n", [1, 65, 500, 1023, 1024, 3456, 20001])
def test_exact_squares_add_exactly(n, tmp_path):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()
    from paper_2404_17133_gb300 import build
    src, lib = str(tmp_path / "shim.cu"), str(tmp_path / "libshim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run([build._nvcc()] + build.ARCH + build.FLAGS +
                   ["-I", build.CSRC, "-shared", "-cudart", "shared", src, build.LIBPATH, "-o", lib,
                    "-Xlinker", "-rpath=" + os.path.dirname(build.LIBPATH)], check=True)
    shim = C.CDLL(lib)
    x = np.random.default_rng(n).integers(30000, 32768, (5, n)).astype(np.float64)
    xd = torch.from_numpy(x.astype(np.float32)).cuda()
    out = torch.zeros(5, dtype=torch.float64, device="cuda")
    torch.cuda.synchronize()
    shim.norms(C.c_void_p(xd.data_ptr()), C.c_longlong(n), 5, n, C.c_void_p(out.data_ptr()))
    torch.cuda.synchronize()
    assert np.array_equal(out.cpu().numpy(), (x * x).sum(axis=1))
