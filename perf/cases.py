"""Performance cases of the response solver: what a program that uses it has it do.

A program creates a ``Solver`` from a molecule's orbital energies and
density-fitted factors and keeps it, then asks it for operator products (the
step that every Davidson iteration, residual check and user-written iteration is
made of) or for whole solves.  Most cases are therefore single products
(``Solver.apply``: kind 0 A X, kind 1 the pair (A+B)X and (A-B)X, kinds 2 and 3
the same for the ris operator of the preconditioner), over the sizes of the
repository's named workloads and of its served request mix, in each arithmetic
that the options offer; two are whole solves.

``arith`` of a case:
  plain  FP64 factors and products (the default options)
  fp32   MIXED precision on the FP32 units
  tc     MIXED precision on the tensor cores
  fp8    MIXED precision on the tensor cores with the FP8 ris rows (ris kinds)

The C ABI hands every product back in FP64 containers.  MIXED results carry FP32
accuracy, and a program that chose MIXED keeps them as FP32, so those cases
return FP32; PLAIN results stay FP64.
"""
import math

import torch

from paper_2404_17133_gb300 import api

T_CUT = 40.0 / 27.211386245988   # exchange window of the ris operator, Hartree (40 eV)
A_X, C_J = 0.25, 2.0

TDA, PAIR, RIS_TDA, RIS_PAIR = 0, 1, 2, 3


def _product(name, no, nv, aux, ris, kind, arith, m):
    return {"name": name, "do": "apply", "n_occ": no, "n_vir": nv, "n_aux": aux, "n_ris": ris, "kind": kind,
            "arith": arith, "m": m}


def _solve(name, do, no, nv, aux, ris, arith, n_states):
    return {"name": name, "do": do, "n_occ": no, "n_vir": nv, "n_aux": aux, "n_ris": ris, "arith": arith,
            "n_states": n_states}


def listed():
    return [
        # the small named workload with the default options: the guess block of a
        # 5-state TDA solve (5 states + 3); latency and launches count
        _product("small_tda_plain", 10, 40, 200, 90, TDA, "plain", 8),
        # the same molecule in a Casida iteration on the tensor cores (two new
        # directions for each of 5 states)
        _product("small_pair_tc", 10, 40, 200, 90, PAIR, "tc", 10),
        # a typical molecule of the served mix, guess block of a 10-state TDA solve
        _product("served_tda_tc", 24, 144, 840, 108, TDA, "tc", 13),
        # nothing a multiple of anything
        _product("odd_pair_tc", 37, 211, 613, 171, PAIR, "tc", 7),
        # the medium named workload: a full Casida iteration of 10 states
        _product("medium_pair_tc", 60, 400, 2000, 360, PAIR, "tc", 20),
        # the preconditioner's product in the same iteration (BF16 ris rows)
        _product("medium_ris_pair_tc", 60, 400, 8, 360, RIS_PAIR, "tc", 20),
        # MIXED as it comes without the tensor-core option: the guess block
        _product("medium_tda_fp32", 60, 400, 2000, 360, TDA, "fp32", 13),
        # the default precision on the medium workload, half of its states active
        _product("medium_pair_plain", 60, 400, 2000, 360, PAIR, "plain", 10),
        # the large named workload's orbitals and Casida block (20 states), over a
        # slice of its auxiliary rows that spans several of the operator's chunks
        _product("large_pair_tc", 150, 1350, 400, 90, PAIR, "tc", 40),
        # the large workload's preconditioner product on FP8 rows (all ris rows)
        _product("large_ris_tda_fp8", 150, 1350, 8, 1350, RIS_TDA, "fp8", 20),
        # whole solves: the quick start (default options), and a served Casida request
        _solve("solve_tda_small_plain", "solve_tda", 10, 40, 200, 90, "plain", 5),
        _solve("solve_rpa_served_tc", "solve_rpa", 24, 144, 840, 108, "tc", 10),
    ]


def _log_int(rng, lo, hi):
    return int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))


def draw(rng):
    """One more case: occupied orbitals spread over the named workloads' range, 4 to 9 virtuals
    each (as in the served mix) plus an odd remainder, auxiliary counts around 5 per orbital."""
    if rng.random() < 0.15:
        do = rng.choice(["solve_tda", "solve_rpa"])
        arith = rng.choice(["plain", "tc"])
        no = _log_int(rng, 6, 12 if arith == "plain" else 24)
        nv = no * rng.randint(4, 6) + rng.randint(0, 3)
        return {"do": do, "n_occ": no, "n_vir": nv, "n_aux": 5 * (no + nv), "n_ris": 9 * ((no + 1) // 2),
                "arith": arith, "n_states": rng.randint(3, 10)}
    kind = rng.choice([TDA, PAIR, PAIR, RIS_TDA, RIS_PAIR])
    arith = rng.choice(["plain", "fp32", "tc", "tc", "tc"]) if kind < 2 else rng.choice(["tc", "fp8"])
    # the most work that a pass may take, in the units that the arithmetic runs on (FP64 is slow)
    budget = {"plain": 3e11, "fp32": 1.5e12, "tc": 8e12, "fp8": 8e12}[arith]
    no = _log_int(rng, 5, 150)
    nv = min(1350, no * rng.randint(4, 9) + rng.randint(0, 7))
    case = {"do": "apply", "n_occ": no, "n_vir": nv, "n_aux": 8 if kind >= 2 else min(2000, 4 * (no + nv) + rng.randint(0, 99)),
            "n_ris": 9 * (no if kind >= 2 else (no + 1) // 2), "kind": kind, "arith": arith, "m": _log_int(rng, 1, 40)}
    if kind < 2 and case["n_aux"] * float(nv) ** 2 > 8e8:   # a slice of the rows, as in the large listed case
        case["n_aux"] = int(8e8 / float(nv) ** 2)
    while work(case)["flops"] > budget:
        if case["m"] > 4:
            case["m"] = case["m"] * 3 // 4
        elif kind < 2:
            case["n_aux"] = case["n_aux"] * 3 // 4
        else:
            case["n_ris"] = 9 * max(1, case["n_ris"] // 12)
    return case


# ---------------------------------------------------------------------------
# inputs

def _plain(case):
    return case["arith"] == "plain"


def _rows(gen, n, n_mo, scale, dt):
    """n symmetric [n_mo][n_mo] rows, N(0, 1) upper triangles times scale[row]."""
    L = torch.randn((n, n_mo, n_mo), generator=gen, device="cuda", dtype=dt)
    L = torch.triu(L) + torch.triu(L, 1).transpose(1, 2)
    return L.mul_(scale.to(dt).view(-1, 1, 1))


def _inputs(case, seed):
    """The molecule (tddft_create's arrays, on the device) and the trial vectors.

    Exact factors: symmetric rows whose size decays over the auxiliary index, with
    the amplitude of the served mix (it keeps A+B and A-B positive definite at any
    size); ris rows: sqrt(0.9) times the leading exact rows plus a small symmetric
    perturbation, exchange rows every ninth of them.  Trial vectors: unit-norm, with
    the 1/(Delta - shift) weighting that preconditioned residuals have."""
    no, nv, aux, ris = case["n_occ"], case["n_vir"], case["n_aux"], case["n_ris"]
    dt = torch.float64 if _plain(case) else torch.float32
    n_mo = no + nv
    g = torch.Generator(device="cuda")
    g.manual_seed(int(seed) * 7919 + 17)
    rand = lambda n: torch.rand(n, generator=g, device="cuda", dtype=torch.float64)
    eo = torch.sort(-0.8 + 0.5 * rand(no)).values
    ev = torch.sort(0.05 + 1.45 * rand(nv)).values
    rows = max(aux, ris) if case.get("kind", 0) >= 2 else aux   # rows that the decay spans
    d = 0.3 * rows
    s_ref = sum(math.exp(-2.0 * p / 60.0) for p in range(200))
    s_n = sum(math.exp(-2.0 * p / d) for p in range(rows))
    amp = 0.1 * math.sqrt(s_ref / s_n) * min(1.0, 12.5 / math.sqrt(no * nv))
    sig = amp * torch.exp(-torch.arange(max(aux, ris), device="cuda", dtype=torch.float64) / d)
    oo = torch.empty((aux, no, no), device="cuda", dtype=dt)
    ov = torch.empty((aux, no, nv), device="cuda", dtype=dt)
    vv = torch.empty((aux, nv, nv), device="cuda", dtype=dt)
    k_idx = torch.arange(0, ris, 9, device="cuda", dtype=torch.int32)
    r_ov = torch.empty((ris, no, nv), device="cuda", dtype=dt)
    r_oo = torch.empty((k_idx.numel(), no, no), device="cuda", dtype=dt)
    r_vv = torch.empty((k_idx.numel(), nv, nv), device="cuda", dtype=dt)
    chunk = 9 * max(1, int(1e8 / n_mo ** 2) // 9)
    for p0 in range(0, max(aux, ris), chunk):
        p1 = min(max(aux, ris), p0 + chunk)
        L = _rows(g, p1 - p0, n_mo, sig[p0:p1], dt)
        n = min(p1, aux) - p0
        if n > 0:
            oo[p0:p0 + n], ov[p0:p0 + n], vv[p0:p0 + n] = L[:n, :no, :no], L[:n, :no, no:], L[:n, no:, no:]
        n = min(p1, ris) - p0
        if n > 0:
            R = math.sqrt(0.9) * L[:n] + _rows(g, n, n_mo, 0.1 * sig[p0:p0 + n], dt)
            r_ov[p0:p0 + n] = R[:, :no, no:]
            k0, k1 = p0 // 9, (p0 + n + 8) // 9
            r_oo[k0:k1], r_vv[k0:k1] = R[::9, :no, :no], R[::9, no:, no:]
    X = None
    if case["do"] == "apply":
        delta = (ev.view(1, -1) - eo.view(-1, 1)).reshape(1, -1)
        X = torch.randn((case["m"], no * nv), generator=g, device="cuda", dtype=torch.float64) / (delta - 0.9 * delta.min())
        X /= X.norm(dim=1, keepdim=True)
    return dict(eps_occ=eo, eps_vir=ev, L_oo=oo, L_ov=ov, L_vv=vv, Lr_oo=r_oo, Lr_ov=r_ov, Lr_vv=r_vv,
                ris_K_index=k_idx), X


def prepare(case, seed):
    arrays, X = _inputs(case, seed)
    torch.cuda.synchronize()
    stream = torch.cuda.Stream()
    solver = api.Solver(case["n_occ"], case["n_vir"], a_x=A_X, coulomb_factor=C_J, t_cut_ha=T_CUT,
                        precisions=1 if _plain(case) else 2, dtype=api.F64 if _plain(case) else api.F32,
                        stream=stream.cuda_stream, **arrays)
    state = {"case": case, "solver": solver, "stream": stream, "X": X}
    if case["do"] != "apply":
        opts = api.default_opts(n_states=case["n_states"])
        if not _plain(case):
            opts.precision, opts.tensor_cores = api.MIXED, 1
        state["opts"] = opts
    return state


def run(state):
    case, solver = state["case"], state["solver"]
    with torch.cuda.stream(state["stream"]):
        if case["do"] == "apply":
            tc = {"plain": 0, "fp32": 0, "tc": 1, "fp8": 2}[case["arith"]]
            out = solver.apply(case["kind"], state["X"], precision=api.PLAIN if _plain(case) else api.MIXED,
                               tensor_cores=tc)
            out = out if isinstance(out, tuple) else (out,)
            return list(out) if _plain(case) else [o.float() for o in out]
        solve = solver.solve_tda if case["do"] == "solve_tda" else solver.solve_rpa
        omega = solve(state["opts"], want_vectors=False)["omega"]
        return [omega if _plain(case) else omega.astype("float32")]


def _work_exchange(no, nv, rows, m, paired, es):
    """(flops, factor bytes) of the exchange terms over `rows` auxiliary rows."""
    flops = 2.0 * m * rows * (no * no * nv + no * nv * nv)
    size = rows * (no * no + nv * nv)
    if paired:
        flops += 4.0 * m * rows * no * no * nv
        size += rows * no * nv
    return flops, es * size


def work(case):
    """Bytes and flops of one pass: factors and trial vectors read once, results written once."""
    no, nv, aux, ris = case["n_occ"], case["n_vir"], case["n_aux"], case["n_ris"]
    ov = no * nv
    if case["do"] != "apply":
        # a solve of n states takes about 10 products of its block at this accuracy
        m, paired = 10 * case["n_states"] * (1 if case["do"] == "solve_tda" else 2), case["do"] == "solve_rpa"
        f, b = _work_exchange(no, nv, aux, m, paired, 8 if _plain(case) else 4)
        return {"bytes": b + aux * ov * (8 if _plain(case) else 4), "flops": f + 4.0 * m * aux * ov}
    m, paired, is_ris = case["m"], case["kind"] in (PAIR, RIS_PAIR), case["kind"] >= 2
    es_j = 8 if _plain(case) else (2 if is_ris else 4)
    es_k = 1 if case["arith"] == "fp8" else es_j
    nj, nk = (ris, (ris + 8) // 9) if is_ris else (aux, aux)
    f, b = _work_exchange(no, nv, nk, m, paired, es_k)
    f += 4.0 * m * nj * ov
    b += nj * ov * es_j + m * ov * (8 + (2 if paired else 1) * (8 if _plain(case) else 4))
    return {"bytes": b, "flops": f}


# ---------------------------------------------------------------------------
# the same results in 64 bits

def _exact_products(a, X, no, nv, kind):
    L_oo, L_ov, L_vv, J_ov = a["L_oo"], a["L_ov"], a["L_vv"], a["L_ov"]
    eo, ev = a["eps_occ"], a["eps_vir"]
    m, dbl = X.shape[0], torch.float64
    if kind >= 2:
        mo = (eo >= ev[0] - T_CUT).to(dbl)
        mv = (ev <= eo[-1] + T_CUT).to(dbl)
        L_oo, L_vv, J_ov = a["Lr_oo"], a["Lr_vv"], a["Lr_ov"]
        L_ov = J_ov[a["ris_K_index"].long()]
    X3 = X.view(m, no, nv)
    K1, K2 = torch.zeros_like(X3), torch.zeros_like(X3)
    for P in range(L_oo.shape[0]):
        oo, vv, ov = L_oo[P].to(dbl), L_vv[P].to(dbl), L_ov[P].to(dbl)
        if kind >= 2:
            oo, vv, ov = oo * mo * mo.view(-1, 1), vv * mv * mv.view(-1, 1), ov * mv * mo.view(-1, 1)
        Z = torch.matmul(oo, X3)
        K1 += torch.matmul(Z.view(m * no, nv), vv).view(m, no, nv)
        if kind & 1:
            Q = torch.matmul(ov, X3.transpose(1, 2))
            K2 += torch.matmul(Q.reshape(m * no, no), ov).view(m, no, nv)
    J = torch.zeros_like(X)
    for p0 in range(0, J_ov.shape[0], 64):
        rows = J_ov[p0:p0 + 64].to(dbl).view(-1, no * nv)
        J += (X @ rows.T) @ rows
    D = (ev.view(1, -1) - eo.view(-1, 1)).reshape(1, -1) * X
    K1, K2 = K1.view_as(X), K2.view_as(X)
    if kind & 1:
        return [D + 2.0 * C_J * J - A_X * (K1 + K2), D + A_X * (K2 - K1)]
    return [D + C_J * J - A_X * K1]


def _exact_energies(a, no, nv, n, paired):
    oo, ov, vv = (a[k].double() for k in ("L_oo", "L_ov", "L_vv"))
    n_ov, aux = no * nv, ov.shape[0]
    f = ov.view(aux, n_ov)
    J = f.T @ f
    D = torch.diag((a["eps_vir"].view(1, -1) - a["eps_occ"].view(-1, 1)).reshape(-1))
    K1 = (oo.reshape(aux, no * no).T @ vv.reshape(aux, nv * nv)).view(no, no, nv, nv).permute(0, 2, 1, 3).reshape(n_ov, n_ov)
    A = D + C_J * J - A_X * K1
    if not paired:
        return torch.linalg.eigvalsh(A)[:n]
    # (ib|ja) over [i][a][j][b]
    K2 = J.view(no, nv, no, nv).permute(0, 3, 2, 1).reshape(n_ov, n_ov)
    B = C_J * J - A_X * K2
    C = torch.linalg.cholesky(A - B)
    return torch.linalg.eigvalsh(C.T @ (A + B) @ C)[:n].sqrt()


def exact(case, seed):
    arrays, X = _inputs(case, seed)
    no, nv = case["n_occ"], case["n_vir"]
    if case["do"] != "apply":
        return [_exact_energies(arrays, no, nv, min(case["n_states"], no * nv), case["do"] == "solve_rpa")]
    return _exact_products(arrays, X, no, nv, case["kind"])
