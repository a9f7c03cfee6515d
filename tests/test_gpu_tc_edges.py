"""Tensor-core products (csrc/tc_gemm.cu) at the edges of their tiles: occupied
and virtual spaces of one element, around the 32-row and 256-column blocks of
the vectors' preparation, one and several vectors per stage-1 tile, contraction
lengths above and below what stays resident, one to three output tiles; exact
(FP16 hi + lo) and ris (BF16) operators, TDA and paired, against the oracle.

Tolerances (2-norms).  Exact: factors, vectors and intermediates are split into
22 bits (four errors of 2^-22 at most, with the dropped lo * lo) and FP32 runs of
up to 16,384 terms add sqrt(16384) 2^-25: 4.8e-6.  ris: the oracle gets the rows
as they are stored (BF16); vectors and intermediates are split into 16 bits:
2 * 2^-17 + the FP32 runs: 1.9e-5.
"""
import numpy as np
import pytest

from oracle import operators as O
from synth.generator import make_problem

pytestmark = pytest.mark.gpu

TOL = {0: 4.8e-6, 2: 1.9e-5}

# n_occ, n_vir, n_aux, n_ris, vectors
SHAPES = [(1, 1, 9, 9, 1), (1, 257, 12, 18, 3), (31, 16, 40, 27, 5), (33, 65, 130, 27, 4), (64, 128, 20, 36, 2),
          (65, 300, 12, 18, 2), (3, 520, 30, 27, 9), (161, 33, 9, 9, 3), (40, 161, 16, 36, 7)]


def _bf16(a):
    u = np.ascontiguousarray(a, dtype=np.float32).view(np.uint32)
    u = (u + 0x7fff + ((u >> 16) & 1)) & np.uint32(0xffff0000)
    return u.view(np.float32).astype(np.float64)


@pytest.mark.parametrize("shape", SHAPES)
def test_products_at_tile_edges(shape):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()
    from paper_2404_17133_gb300 import api
    no, nv, na, nr, m = shape
    p = make_problem(no, nv, na, nr, seeds=(70, 71, 72))
    for k in ("Lr_oo", "Lr_ov", "Lr_vv"):
        setattr(p, k, _bf16(getattr(p, k)))
    X = np.random.default_rng(no * nv).standard_normal((m, no * nv))
    s = api.Solver.from_problem(p)
    try:
        for kind, op in ((0, O.exact_operator(p)), (2, O.ris_operator(p))):
            got = (s.apply(kind, X, precision=api.MIXED, tensor_cores=1),)
            got += s.apply(kind + 1, X, precision=api.MIXED, tensor_cores=1)
            for a, b in zip(got, (op.tda(X),) + tuple(op.apb_amb(X))):
                e = float(np.linalg.norm(a - b) / np.linalg.norm(b))
                assert e < TOL[kind], (kind, e)
    finally:
        s.close()
