"""The server's charge bounds the device memory that a request takes, in each arithmetic,
at sizes whose operator intermediates fill their chunks (tensor cores: 4 GB; slices:
1 GB): the pool's high-water mark above its use at server creation, against
tddft_estimate_bytes."""
import time

import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec,tc", [(0, 0), (1, 0), (1, 1)])
@pytest.mark.parametrize("kind", [0, 1])
@pytest.mark.parametrize("shape", [(24, 144, 840, 108), (60, 400, 2000, 360)])
def test_high_water_mark_is_below_the_charge(prec, tc, kind, shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()
    from paper_2404_17133_gb300 import api
    from synth.device import problem_kw
    kw = problem_kw(7, *shape)
    torch.cuda.synchronize()
    o = api.default_opts(n_states=10, precond=api.RID, precision=prec, tensor_cores=tc, max_iter=12)
    srv = api.Server(max_active=1)
    try:
        t = srv.submit(kind, o, create_kw=dict(kw, precisions=1 + prec, dtype=api.F32))
        r, t0 = None, time.time()
        while r is None and time.time() - t0 < 120:
            r = srv.poll(t, timeout_ms=100)
        info = srv.info()
    finally:
        srv.close()
    assert r is not None and r["status"] in (api.OK, api.ERR_NOCONV), r
    used = info["pool_high_bytes"] - info["pool_used_at_create_bytes"]
    print("used %.3f GB, charge %.3f GB" % (used / 1e9, r["charged_bytes"] / 1e9))
    assert used <= r["charged_bytes"], (used, r["charged_bytes"])
