"""Tensor-core solves on many streams at once: the pair kernels (cta_group::2) of one stream
start on SM pairs that other streams' kernels have just left or still share, with their two
CTAs apart in time, and allocate and free their tensor memory there.  Every request
ends, with the result that it has alone."""
import time

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def test_many_streams_of_tensor_core_solves_end():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()
    from paper_2404_17133_gb300 import api
    from synth.device import problem_kw
    shapes = [(8, 40, 240, 36), (13, 70, 415, 63), (24, 120, 720, 108), (31, 190, 600, 144), (40, 200, 500, 180),
              (17, 100, 585, 81)]
    pool = [problem_kw(200 + i, *s) for i, s in enumerate(shapes)]
    torch.cuda.synchronize()
    o = api.default_opts(n_states=6, precond=api.RID, precision=api.MIXED, tensor_cores=1)
    alone = []
    for kw in pool:
        s = api.Solver(**kw, precisions=2, dtype=api.F32)
        try:
            alone.append([s.solve_tda(o, want_vectors=False)["omega"], s.solve_rpa(o, want_vectors=False)["omega"]])
        finally:
            s.close()
    srv = api.Server(max_active=16)
    try:
        reqs = [(i, i % len(pool), (i // len(pool)) % 4 == 3) for i in range(240)]
        tickets = {srv.submit(1 if rpa else 0, o, create_kw=dict(pool[k], precisions=2, dtype=api.F32)): (k, rpa)
                   for _, k, rpa in reqs}
        t0 = time.time()
        while tickets and time.time() - t0 < 120:
            for t in list(tickets):
                r = srv.poll(t, timeout_ms=0)
                if r is not None:
                    k, rpa = tickets.pop(t)
                    assert r["status"] == api.OK, r.get("error")
                    assert np.max(np.abs(r["omega"] - alone[k][1 if rpa else 0])) <= 1e-12
            time.sleep(0.002)
        assert not tickets, "%d requests did not end" % len(tickets)
    finally:
        srv.close()
