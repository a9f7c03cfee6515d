"""PLAIN solves of the medium workload (n_occ 60, n_vir 400, n_aux 2000), whose exchange
and Coulomb contractions are sliced, exact and ris: Casida energies to 1e-6 Ha and
polarizabilities to 1e-6 relative (element by element, floor of tests/parity.py)
against the oracle's stored results, outer iterations within 4 of its counts."""
import json
import os

import numpy as np
import pytest

from synth.generator import CONFIGS, dipoles, make_config
from tests.parity import alpha_excess

pytestmark = pytest.mark.gpu
GOLD = os.path.join(os.path.dirname(__file__), "golden", "rpa_polar_medium.json")


def test_casida_and_polarizability():
    torch = pytest.importorskip("torch")
    if not torch.cuda.is_available():
        pytest.skip("no GPU")
    import __graft_entry__ as g
    g.build()
    from paper_2404_17133_gb300 import api
    with open(GOLD) as f:
        gold = json.load(f)
    p, c = make_config("rpa_polar_medium"), CONFIGS["rpa_polar_medium"]
    mu = dipoles(c["mu_seed"], c["n_dip"], p.n_ov)
    s = api.Solver.from_problem(p, precisions=1)
    try:
        r = s.solve_rpa(api.default_opts(n_states=10, precond=api.RID), want_vectors=False)
        a = s.solve_polar(api.default_opts(precond=api.RID), mu, list(c["omegas"]))
    finally:
        s.close()
    assert r["status"] == api.OK and a["status"] == api.OK
    assert np.max(np.abs(r["omega"] - np.array(gold["rpa"]["omega"]))) < 1e-6
    assert alpha_excess(a["alpha"], np.array(gold["polar"]["alpha"]), 1e-6) <= 1.0
    assert abs(r["stats"]["n_iter"] - gold["rpa"]["n_iter"]) <= 4
    assert abs(a["stats"]["n_iter"] - gold["polar"]["n_iter"]) <= 4
