"""Sliced FP64 / FP32 products (csrc/slice_gemm.cu) output by output where rows span
decades: two fragments that the factors do not couple, the trial vectors small within
one of them by a factor `eps`.  Every row of a contraction then holds large elements
that meet zeros of the other operand, and the outputs of the small fragment are sums
of small terms alone.  Fragments are contiguous halves of the orbitals or interleaved.

Bound for every output element: 16 roundings of the sum of its terms' absolute
values (2^-53 FP64, 2^-24 FP32; K1 and J are two contractions in a row, each within
a few roundings of that sum, the combination adds three).  The 2-norm sees none of
it: the small fragment's part of a vector is eps of the rest.
"""
import numpy as np
import pytest

from oracle import operators as O
from synth.generator import make_problem

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def api():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()
    from paper_2404_17133_gb300 import api as a
    return a


def _member(n, interleaved):
    """0 or 1 for each orbital (or auxiliary row)."""
    return np.arange(n) % 2 if interleaved else (np.arange(n) >= n // 2).astype(int)


def _fragments(shape, eps, interleaved, f32):
    no, nv, na, m = shape
    p = make_problem(no, nv, na, 9, seeds=(80, 81, 82))
    fo, fv, fp = _member(no, interleaved), _member(nv, interleaved), _member(na, interleaved)
    rng = np.random.default_rng(no * nv + m)
    rnd = (lambda a: a.astype(np.float32).astype(np.float64)) if f32 else (lambda a: a)
    for name, r, c in (("L_oo", fo, fo), ("L_ov", fo, fv), ("L_vv", fv, fv)):
        a = getattr(p, name)
        same = (r[None, :, None] == fp[:, None, None]) & (c[None, None, :] == fp[:, None, None])
        setattr(p, name, rnd(np.where(same, a, 0.0)))
    scale = np.where((fo[:, None] == 1) & (fv[None, :] == 1), eps, 1.0)
    return p, rnd((rng.standard_normal((m, no, nv)) * scale).reshape(m, no * nv))


def _absolute(p):
    """The operator of the terms' absolute values: (A+B) of it has every term added."""
    return O.Operator(p.eps_occ, p.eps_vir, np.abs(p.L_ov), np.abs(p.L_oo), np.abs(p.L_ov), np.abs(p.L_vv), -p.a_x,
                      p.coulomb_factor)


@pytest.mark.parametrize("shape", [(3, 8, 2000, 12), (11, 40, 300, 9), (11, 40, 2100, 24), (24, 144, 400, 25)])
@pytest.mark.parametrize("eps", [1e-4, 1e-8])
@pytest.mark.parametrize("interleaved", [False, True])
@pytest.mark.parametrize("prec", [0, 1])
def test_outputs_of_a_small_fragment(api, shape, eps, interleaved, prec):
    p, X = _fragments(shape, eps, interleaved, prec == 1)
    op, bound = O.exact_operator(p), _absolute(p)
    size = bound.apb_amb(np.abs(X))[0]
    tol = 16 * (2.0 ** -53 if prec == 0 else 2.0 ** -24)
    s = api.Solver.from_problem(p)
    try:
        got = (s.apply(0, X, precision=prec),) + s.apply(1, X, precision=prec)
        for g, r in zip(got, (op.tda(X),) + tuple(op.apb_amb(X))):
            e = np.abs(g - r) / np.maximum(size, 1e-300)
            assert e.max() < tol, (e.max() / tol, np.unravel_index(e.argmax(), e.shape))
    finally:
        s.close()


def test_large_fp32_vectors_stay_finite(api):
    """FP32 rows near the top of the range against small ones: the product is in range."""
    p = make_problem(9, 40, 1000, 9, seeds=(50, 51, 52))
    X = np.random.default_rng(3).standard_normal((16, 360)).astype(np.float32).astype(np.float64)
    s = api.Solver.from_problem(p)
    try:
        base = s.apply(0, X, precision=1)
        assert np.array_equal(s.apply(0, X * 2.0 ** 105, precision=1), base * 2.0 ** 105)
    finally:
        s.close()
