"""The tall Coulomb Gram product (k_tall_gram, csrc/skinny.cu) adds the runs of its long
chunks without rounding: a factor row of whole numbers whose FP32 runs (at most 64
terms of less than 2^18 at these sizes) are exact, whose chunk sums are not (27 bits),
and whose total is small.  Then t is exact, and with one nonzero row so are J
and, the factors being whole numbers below 2^18, the product's Coulomb part."""
import numpy as np
import pytest

from synth.generator import make_problem

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,n_occ,n_vir,vectors", [(1300, 128, 128, 1), (1300, 100, 200, 21), (1290, 97, 181, 8),
                                                      (1300, 128, 130, 40)])
def test_small_total_of_large_chunk_sums(rows, n_occ, n_vir, vectors):
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()
    from paper_2404_17133_gb300 import api
    n_ov = n_occ * n_vir
    p = make_problem(n_occ, n_vir, rows, 9, seeds=(90, 91, 92))
    rng = np.random.default_rng(n_ov)
    half = n_ov // 2
    row = np.zeros(n_ov)
    row[:half] = rng.integers(2 ** 17, 2 ** 18, half)
    row[half:2 * half] = -row[rng.permutation(half)]
    row[0] += 37 - row.sum()                      # the total is 37
    assert row.sum() == 37 and abs(row[0]) < 2 ** 18 + 64
    for k in ("L_oo", "L_vv"):
        setattr(p, k, np.zeros_like(getattr(p, k)))
    p.L_ov = np.zeros_like(p.L_ov)
    p.L_ov[rows // 2] = row.reshape(n_occ, n_vir)
    p.a_x = 0.0
    X = np.ones((vectors, n_ov))
    X[1::2] = -1.0
    s = api.Solver.from_problem(p)
    try:
        got = s.apply(0, X, precision=api.MIXED)
    finally:
        s.close()
    d = (p.eps_vir[None, :] - p.eps_occ[:, None]).reshape(-1)
    want = X * d + p.coulomb_factor * X[:, :1] * 37.0 * row
    np.testing.assert_allclose(got, want, rtol=1e-14)
