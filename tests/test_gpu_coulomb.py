"""Coulomb contractions over FP32 and BF16 factor rows (tall_gram, tall_combo in
csrc/skinny.cu) at the edges of their tiles (128 rows, 64-element K steps, 4 to 32
vectors), below their smallest sizes and at every row alignment (16, 8, 4 and 2
bytes): products of the exact (FP32 rows) and ris (BF16 rows) operators against
the oracle.

Tolerance (2-norm): the oracle gets the factors as they are stored (rounded to
FP32 and BF16 first), so what is left is FP32 accumulation of K terms in runs,
below sqrt(K) 2^-24 / 4 (K <= 33,920 here: 2.8e-6), and single roundings.
"""
import numpy as np
import pytest

from oracle import operators as O
from synth.generator import make_problem

pytestmark = pytest.mark.gpu

TOL = 4e-6

# n_occ, n_vir, n_aux, n_ris, vectors (n_occ n_vir: 1023, 1024, 1025, 1026, 1028, 2112, 2100, 4356, 2809)
SHAPES = [(11, 93, 128, 135, 1), (32, 32, 127, 126, 3), (32, 32, 128, 135, 8), (25, 41, 129, 135, 9),
          (27, 38, 257, 144, 17), (4, 257, 130, 261, 33), (8, 264, 300, 135, 41), (3, 700, 131, 135, 40),
          (66, 66, 128, 135, 20), (53, 53, 140, 135, 21)]


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
    p = make_problem(no, nv, na, nr, seeds=(60, 61, 62))
    for k in ("L_oo", "L_ov", "L_vv"):
        setattr(p, k, getattr(p, k).astype(np.float32).astype(np.float64))
    for k in ("Lr_oo", "Lr_ov", "Lr_vv"):
        setattr(p, k, _bf16(getattr(p, k)))
    X = np.random.default_rng(no * nv).standard_normal((m, no * nv)).astype(np.float32).astype(np.float64)
    s = api.Solver.from_problem(p)
    try:
        for kind, op in ((0, O.exact_operator(p)), (2, O.ris_operator(p))):
            got, ref = s.apply(kind, X, precision=api.MIXED), op.tda(X)
            e = float(np.linalg.norm(got - ref) / np.linalg.norm(ref))
            assert e < TOL, (kind, e)
    finally:
        s.close()
