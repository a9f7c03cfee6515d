"""Waits of the tensor-core kernels: an mbarrier on which nothing arrives is given up
within WAIT_NS (csrc/tc_ptx.cuh), and a solve whose kernels have reported a
timeout ends at its next read of norms with TDDFT_ERR_CUDA, not after its remaining
iterations.  The wait is made to run out by a barrier that nothing signals, the
report by writing the context's error word from the host: no kernel faults or hangs."""
import ctypes as C
import os
import subprocess

import numpy as np
import pytest

from synth.generator import dipoles, make_config

pytestmark = pytest.mark.gpu

SHIM = r"""
#include "ctx.cuh"
#include "tc_ptx.cuh"
__global__ void k_wait(unsigned long long* out) {
  __shared__ uint64_t bar;
  tddft::mbar_init(&bar, 1);
  const unsigned long long t0 = tddft::global_ns();
  out[0] = tddft::mbar_wait(&bar, 0) ? 1 : 0;
  out[1] = tddft::global_ns() - t0;
}
extern "C" int run_wait(unsigned long long* h) {
  unsigned long long* d = nullptr;
  if (cudaMalloc(&d, 16) != cudaSuccess) return 1;
  k_wait<<<1, 1>>>(d);
  const int rc = cudaMemcpy(h, d, 16, cudaMemcpyDeviceToHost);
  cudaFree(d);
  return rc;
}
extern "C" unsigned long long wait_ns() { return tddft::WAIT_NS; }
extern "C" int set_error_word(void* ctx, int code) {
  return cudaMemcpy(static_cast<tddft::Ctx*>(ctx)->tc_err.p, &code, 4, cudaMemcpyHostToDevice);
}
extern "C" long long launches() { return tddft::g_launches; }
"""


@pytest.fixture(scope="module")
def env(tmp_path_factory):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()
    from paper_2404_17133_gb300 import api, build
    d = tmp_path_factory.mktemp("shim")
    src, lib = str(d / "shim.cu"), str(d / "libshim.so")
    with open(src, "w") as f:
        f.write(SHIM)
    subprocess.run([build._nvcc()] + build.ARCH + build.FLAGS +
                   ["-I", build.CSRC, "-shared", "-cudart", "shared", src, build.LIBPATH, "-o", lib,
                    "-Xlinker", "-rpath=" + os.path.dirname(build.LIBPATH)], check=True)
    shim = C.CDLL(lib)
    shim.wait_ns.restype = C.c_ulonglong
    shim.launches.restype = C.c_longlong
    return api, shim


def test_wait_gives_up_by_time(env):
    _, shim = env
    out = (C.c_ulonglong * 2)()
    assert shim.run_wait(out) == 0
    limit = shim.wait_ns()
    assert out[0] == 0 and limit <= out[1] < 2 * limit, (out[0], out[1], limit)


@pytest.mark.parametrize("precond", ["diag", "rid"])
@pytest.mark.parametrize("kind", ["tda", "rpa", "polar"])
def test_solve_ends_at_a_reported_timeout(env, kind, precond):
    api, shim = env
    p = make_config("tda_small")
    mu = dipoles(1, 3, p.n_ov)
    o = api.default_opts(n_states=5, precond=api.RID if precond == "rid" else api.DIAG)
    s = api.Solver.from_problem(p)
    run = {"tda": lambda: s.solve_tda(o, want_vectors=False), "rpa": lambda: s.solve_rpa(o, want_vectors=False),
           "polar": lambda: s.solve_polar(o, mu, [0.0, 0.05])}[kind]
    try:
        full = run()
        assert full["status"] == api.OK
        assert shim.set_error_word(s.h, 8) == 0
        with pytest.raises(api.TddftError) as e:
            run()
        assert e.value.status == api.ERR_CUDA
        assert shim.launches() < full["stats"]["gpu_launches"] // 3, (shim.launches(), full["stats"])
        again = run()          # the word was cleared
        assert again["status"] == api.OK
        key = "alpha" if kind == "polar" else "omega"
        assert np.array_equal(again[key], full[key])
    finally:
        s.close()
