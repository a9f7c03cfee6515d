"""Sliced FP64 / FP32 contractions (csrc/slice_gemm.cu) at the edges of their
tiles: K steps (16), k-blocks (32), exact runs (256) and output tiles (128 x 64
or 128), single elements, rows that decay over several decades, powers of two
and non-finite inputs; against the oracle and against the allocation-free
product, whose contractions run on the FP64 / FP32 units.

Tolerances (2-norms): both FP64 references accumulate K = n_aux n_vir terms (at
most 57,600 here) with errors up to sqrt(K) 2^-53 = 2.7e-14 of the result; FP32
(inputs rounded to FP32 first): intermediate, result and Coulomb sums are
rounded to 2^-24 each and the FP32 units accumulate K terms in runs, below
sqrt(K) 2^-24 / 4 = 3.6e-6.
"""
import ctypes as C

import numpy as np
import pytest

from oracle import operators as O
from synth.generator import make_problem

pytestmark = pytest.mark.gpu

TOL = {0: 3e-14, 1: 4e-6}

SHAPES = [(1, 1, 1, 9, 1), (3, 7, 5, 9, 2), (16, 64, 20, 9, 4), (17, 65, 20, 18, 5), (8, 32, 30, 9, 17),
          (33, 257, 12, 27, 3), (24, 144, 400, 27, 4), (10, 40, 300, 9, 10),
          (24, 144, 400, 27, 100), (19, 131, 1031, 27, 53)]


@pytest.fixture(scope="module")
def api():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()
    from paper_2404_17133_gb300 import api as a
    return a


def _rel(a, b):
    return float(np.linalg.norm(a - b) / max(np.linalg.norm(b), 1e-300))


def _as_f32(p):
    for k in ("L_oo", "L_ov", "L_vv"):
        setattr(p, k, getattr(p, k).astype(np.float32).astype(np.float64))
    return p


@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("prec", [0, 1])
def test_products_at_tile_edges(api, shape, prec):
    import torch
    no, nv, na, nr, m = shape
    p = make_problem(no, nv, na, nr, seeds=(40, 41, 42))
    if prec == 1:
        p = _as_f32(p)
    X = np.random.default_rng(no * nv).standard_normal((m, no * nv))
    X = X.astype(np.float32).astype(np.float64)
    s = api.Solver.from_problem(p)
    try:
        for kind in (0, 1) if prec else (0, 1, 2, 3):
            got = s.apply(kind, X, precision=prec)
            got = got if isinstance(got, tuple) else (got,)
            op = O.exact_operator(p) if kind < 2 else O.ris_operator(p)
            ref = op.apb_amb(X) if kind & 1 else (op.tda(X),)
            Xd = torch.from_numpy(X).cuda()
            out = [torch.empty_like(Xd) for _ in got]
            torch.cuda.synchronize()
            st = api.lib().tddft_apply_noalloc(s.h, kind, prec, C.c_void_p(Xd.data_ptr()), m,
                                               C.c_void_p(out[0].data_ptr()),
                                               C.c_void_p(out[1].data_ptr()) if len(out) > 1 else None)
            torch.cuda.synchronize()
            assert st == api.OK
            for g, r, o in zip(got, ref, out):
                assert _rel(g, r) < TOL[prec], (kind, _rel(g, r))
                assert _rel(g, o.cpu().numpy()) < TOL[prec], (kind, _rel(g, o.cpu().numpy()))
    finally:
        s.close()


def test_scales_and_non_finite(api):
    """Powers of two pass through exactly; a zero vector gives zeros; a
    non-finite element makes its own vector's product non-finite and no other."""
    p = make_problem(9, 40, 30, 9, seeds=(50, 51, 52))
    X = np.random.default_rng(3).standard_normal((4, 360))
    s = api.Solver.from_problem(p)
    try:
        for prec in (0, 1):
            base = s.apply(0, X, precision=prec)
            for k in (-40, 30):
                assert np.array_equal(s.apply(0, X * 2.0 ** k, precision=prec), base * 2.0 ** k)
            Y = X.copy()
            Y[1] = 0.0
            Y[2, 7] = np.inf
            Y[3, 11] = np.nan
            out = s.apply(0, Y, precision=prec)
            assert np.array_equal(out[0], base[0]) and not out[1].any()
            assert not np.isfinite(out[2]).any() and not np.isfinite(out[3]).any()
    finally:
        s.close()
