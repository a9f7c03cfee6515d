"""Products without tensor_cores on both sides of the sizes from which the exchange
contractions are sliced (csrc/operator.cu: 2^22 multiply-adds in FP64, 2^28 in
FP32), and sliced products whose contractions are short (K of 1 to 33), against the
oracle.  Tolerances (2-norms) as in test_gpu_slices.py: sqrt(K) 2^-53 for the FP64
sums (K at most 99,000 here: 3.5e-14), sqrt(K) 2^-24 / 4 for the FP32 ones (4.7e-6)."""
import numpy as np
import pytest

from oracle import operators as O
from synth.generator import make_problem

pytestmark = pytest.mark.gpu

TOL = {0: 3.5e-14, 1: 4.7e-6}

# precision, n_occ, n_vir, n_aux, vectors; work = vectors n_aux n_occ n_vir (n_occ + n_vir [+ 2 n_occ])
CASES = [(0, 6, 30, 161, 4), (0, 6, 30, 162, 4),          # 4,173,120 and 4,199,040 (2^22 = 4,194,304)
         (0, 5, 20, 419, 4), (0, 5, 20, 420, 4),
         (1, 16, 90, 439, 4), (1, 16, 90, 440, 4),        # 268,035,840 and 268,646,400 (2^28 = 268,435,456)
         (0, 1, 33, 3000, 40), (0, 2, 9, 4000, 30), (0, 17, 3, 3000, 8), (0, 1, 1, 60000, 40),
         (1, 1, 33, 3000, 80), (1, 2, 40, 2000, 45), (1, 33, 5, 2000, 30), (1, 17, 65, 1000, 5)]


@pytest.mark.parametrize("prec,no,nv,na,m", CASES)
def test_products_against_the_oracle(prec, no, nv, na, m):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()
    from paper_2404_17133_gb300 import api
    p = make_problem(no, nv, na, 9, seeds=(100, 101, 102))
    rnd = (lambda a: a.astype(np.float32).astype(np.float64)) if prec else (lambda a: a)
    for k in ("L_oo", "L_ov", "L_vv"):
        setattr(p, k, rnd(getattr(p, k)))
    X = rnd(np.random.default_rng(na).standard_normal((m, no * nv)))
    s = api.Solver.from_problem(p)
    try:
        op = O.exact_operator(p)
        got = (s.apply(0, X, precision=prec),) + s.apply(1, X, precision=prec)
        for a, b in zip(got, (op.tda(X),) + tuple(op.apb_amb(X))):
            e = float(np.linalg.norm(a - b) / np.linalg.norm(b))
            assert e < TOL[prec], e
    finally:
        s.close()
