"""The calls that users of this library make, at the sizes they make them, for timing one build against another.

Systems are water clusters and core-level molecules with the level structure of ``synth`` (evenly spaced levels, B
normal with sigma 0.6/sqrt(n_aux)), from one molecule to 24, with odd basis sizes beside the 38 virtual and 126
auxiliary functions per water.  B is drawn on the GPU, symmetric in the orbital pair like the generator's, so that the
occupied-virtual block and the target rows agree where they overlap.

A mixed-precision plan computes in BF16 parts and FP32 and hands its results over in float64 arrays; the cases keep
those results as float32, which is the precision such a plan computes in.  An FP64 plan's results stay float64.
"""
import numpy as np
import torch

from paper_2107_10423_gb300 import gw, serve, synth

N_FREQ = 128
ETA = 1e-3
X0 = 0.5


def listed():
    return [
        # a job of the serving stream at its smallest: one molecule, HOMO and LUMO, host arrays in, energies out;
        # plan set-up, allocations and launches count as much as arithmetic
        {"name": "serve_w1", "do": "serve", "prec": "mixed", "n": 1, "n_virt": 38, "n_aux": 126, "targets": "frontier"},
        # a core job of the serving stream (30 % of it): the deepest O1s level, whose residues reach far into the
        # real axis; odd basis sizes
        {"name": "serve_w5_core", "do": "serve", "prec": "mixed", "n": 5, "n_virt": 187, "n_aux": 629,
         "targets": "core"},
        # a whole valence spectrum on a resident plan: screening, many residues and their dense fallback
        {"name": "job_w8_valence", "do": "job", "prec": "mixed", "n": 8, "n_virt": 304, "n_aux": 1008,
         "targets": "valence"},
        # a large cluster of the stream, HOMO and LUMO on a resident plan: the Pi build and the W table dominate
        {"name": "job_w24_frontier", "do": "job", "prec": "mixed", "n": 24, "n_virt": 912, "n_aux": 3024,
         "targets": "frontier"},
        # the imaginary-axis table alone, for the users that keep W and evaluate Sigma themselves; odd sizes
        {"name": "wtable_w10", "do": "wtable", "prec": "mixed", "n": 10, "n_virt": 379, "n_aux": 1259,
         "targets": "valence"},
        # the polarizability matrices at a few frequencies of the caller's
        {"name": "pi_w6", "do": "pi", "prec": "mixed", "n": 6, "n_virt": 228, "n_aux": 757, "n_xi": 8},
        # the core-level batch (ESCA shape, 6 C1s levels): one evaluation of Sigma near the levels, as every step of
        # the QP search makes it; nearly all residues take the dense fallback
        {"name": "core_sigma", "do": "core", "prec": "mixed", "n_virt": 552, "n_aux": 1800, "n_points": 6},
        # a radical cation: two spin channels, targets in both
        {"name": "open_w3", "do": "open", "prec": "mixed", "n": 3, "n_virt": 114, "n_aux": 378},
        # the single water in FP64 by the step tree, the reference calculation of the small systems
        {"name": "fp64_w1_steptree", "do": "steptree", "prec": "fp64", "n": 1, "n_virt": 19, "n_aux": 84,
         "targets": "frontier"},
        # a small cluster in FP64 (the library's default precision), whole valence spectrum
        {"name": "fp64_w4_valence", "do": "job", "prec": "fp64", "n": 4, "n_virt": 152, "n_aux": 504,
         "targets": "valence"},
        # an explicit list of residues in FP64
        {"name": "fp64_w3_residues", "do": "residues", "prec": "fp64", "n": 3, "n_virt": 113, "n_aux": 377,
         "n_rhs": 40},
        # the spectral-decomposition route from the input tensors, as small systems are cross-checked
        {"name": "sd_w2", "do": "sd", "prec": "fp64", "n": 2, "n_virt": 76, "n_aux": 252, "targets": "frontier"},
    ]


def _log(rng, lo, hi):
    return int(round(lo * (hi / lo) ** rng.random()))


def _basis(rng, n):
    """Virtual and auxiliary functions of n waters in basis sets a little smaller or larger than the usual one."""
    return {"n": n, "n_virt": rng.randint(30 * n, 40 * n), "n_aux": rng.randint(105 * n, 126 * n)}


def draw(rng):
    do = rng.choice(["serve", "serve", "job", "job", "wtable", "pi", "core", "open", "fp64", "residues", "sd"])
    if do == "serve":
        return {"do": "serve", "prec": "mixed", "targets": rng.choice(["frontier", "frontier", "core"]),
                **_basis(rng, _log(rng, 1, 10))}
    if do == "job":
        if rng.random() < 0.5:
            return {"do": "job", "prec": "mixed", "targets": "valence", **_basis(rng, _log(rng, 1, 8))}
        return {"do": "job", "prec": "mixed", "targets": "frontier", **_basis(rng, _log(rng, 2, 24))}
    if do == "wtable":
        return {"do": "wtable", "prec": "mixed", "targets": rng.choice(["frontier", "valence"]),
                **_basis(rng, _log(rng, 2, 12))}
    if do == "pi":
        return {"do": "pi", "prec": "mixed", "n_xi": rng.randint(1, 12), **_basis(rng, _log(rng, 1, 10))}
    if do == "core":
        return {"do": "core", "prec": "mixed", "n_virt": _log(rng, 60, 552), "n_aux": _log(rng, 200, 1800),
                "n_points": rng.randint(1, 6)}
    if do == "open":
        return {"do": "open", "prec": rng.choice(["mixed", "mixed", "fp64"]), **_basis(rng, _log(rng, 1, 4))}
    if do == "fp64":
        return {"do": "job", "prec": "fp64", "targets": rng.choice(["frontier", "valence"]),
                **_basis(rng, _log(rng, 1, 4))}
    if do == "residues":
        return {"do": "residues", "prec": "fp64", "n_rhs": _log(rng, 1, 60), **_basis(rng, _log(rng, 1, 4))}
    n = rng.randint(1, 2)
    return {"do": "sd", "prec": "fp64", "targets": "frontier", **_basis(rng, n)}


# ------------------------------------------------------------------------------------------ inputs
def _lin(a, b, n):
    return np.linspace(a, b, n) if n > 1 else np.full(n, (a + b) / 2.0)


def _system(case, seed):
    """Levels, sizes and targets of a case (a ``synth.System``, whose own B generator is not used)."""
    if case["do"] == "core":
        s = synth.esca_like(seed, case["n_virt"], case["n_aux"])
        return s
    n, n_virt = case["n"], case["n_virt"]
    eps = np.concatenate([_lin(-20.6, -20.4, n), _lin(-1.4, -0.4, 4 * n), _lin(0.03, 8.0, n_virt)])
    n_occ = 5 * n
    targets = {"frontier": [n_occ - 1, n_occ], "core": [0],
               "valence": list(range(n, n_occ)) + list(range(n_occ, n_occ + min(10, n_virt)))}
    t = targets[case.get("targets", "frontier")]
    return synth.System(f"water{n}", eps, n_occ, case["n_aux"], 0.6 / np.sqrt(case["n_aux"]), seed,
                        np.array(t, dtype=np.int64), {"n_water": n})


def _tensors(s, seed, n_occ=None, targets=None):
    """B_ia [n_aux, n_occ n_virt] and B_nm [n_targets, n_bas, n_aux] on the GPU, from the seed."""
    g = torch.Generator(device="cuda").manual_seed(int(seed))
    n_occ = s.n_occ if n_occ is None else n_occ
    targets = [int(t) for t in (s.targets if targets is None else targets)]
    n_virt = s.n_bas - n_occ
    kw = dict(generator=g, device="cuda", dtype=torch.float64)
    B = torch.randn(s.n_aux, n_occ, n_virt, **kw) * s.sigma_b
    Bn = torch.randn(len(targets), s.n_bas, s.n_aux, **kw) * s.sigma_b
    for k, t in enumerate(targets):          # (P|ta) of the two blocks is the same number
        if t < n_occ:
            Bn[k, n_occ:] = B[:, t, :].T
        else:
            Bn[k, :n_occ] = B[:, :, t - n_occ].T
    for k, t in enumerate(targets):          # and (P|tu) = (P|ut)
        for j in range(k):
            Bn[k, targets[j]] = Bn[j, t]
    return B.reshape(s.n_aux, n_occ * n_virt), Bn


def _prec(case):
    return gw.GW_PREC_MIXED if case["prec"] == "mixed" else gw.GW_PREC_FP64


def _residue_list(case, s, seed):
    """(target index, state, frequency) triples as a contour's residues have them: inside and beyond the gap."""
    r = np.random.default_rng(seed)
    k = case["n_rhs"]
    return (r.integers(0, len(s.targets), k).astype(np.int32), r.integers(0, s.n_bas, k).astype(np.int32),
            r.uniform(-2.0, 2.0, k))


def _open_spins(case, s):
    """Beta levels 0.05 Ha higher with one electron less; HOMO and LUMO of either spin."""
    oa, ob = s.n_occ, s.n_occ - 1
    return s.eps + 0.05, ob, [oa - 1, oa, ob - 1, ob], [0, 0, 1, 1]


def prepare(case, seed):
    s = _system(case, seed)
    do = case["do"]
    if do == "open":
        eps_b, ob, t, spins = _open_spins(case, s)
        Ba, Bna = _tensors(s, seed, s.n_occ, t[:2])
        Bb, Bnb = _tensors(s, seed + (1 << 20), ob, t[2:])
        Bn = torch.cat([Bna, Bnb])
        plan = gw.Plan.open_shell(s.eps, eps_b, s.n_occ, ob, Ba.cpu().numpy(), Bb.cpu().numpy(), Bn.cpu().numpy(), t,
                                  spins, precision=_prec(case))
        return {"case": case, "plan": plan}
    B, Bn = _tensors(s, seed)
    if do == "serve":
        return {"case": case, "job": serve.Job(0, 0.0, s, B.cpu().numpy(), Bn.cpu().numpy())}
    torch.cuda.synchronize()                 # the plan reads B on a stream of its own
    state = {"case": case, "system": s, "B": B, "Bn": Bn}
    if do == "sd":
        return state
    state["plan"] = gw.Plan(s.eps, s.n_occ, B, Bn, s.targets, precision=_prec(case))
    if do == "core":
        state["points"] = _core_points(case, s)
        state["plan"].screening()            # the table is built once, the search evaluates Sigma many times
    elif do == "pi":
        state["xi"] = _pi_xi(case)
    elif do == "residues":
        state["rhs"] = _residue_list(case, s, seed)
    return state


def _core_points(case, s):
    k = case["n_points"]
    t = np.arange(k, dtype=np.int32) % len(s.targets)
    return t, s.eps[s.targets[t]] - 0.031 * (1 + np.arange(k))


def _pi_xi(case):
    return np.concatenate([[0.0], np.geomspace(0.02, 40.0, case["n_xi"])])[:case["n_xi"]]


# ------------------------------------------------------------------------------------------ one pass
def _out(case, *arrays):
    if case["prec"] == "fp64":
        return list(arrays)
    return [a.astype(np.float32) if a.dtype == np.float64 else a for a in arrays]


def run(state):
    case = state["case"]
    do = case["do"]
    if do == "serve":
        r = serve.run_job(state["job"], precision="mixed", qp="linearised")
        return _out(case, r["e_qp"], r["z"], r["status"])
    if do == "sd":
        s = state["system"]
        with gw.Plan(s.eps, s.n_occ, state["B"], state["Bn"], s.targets) as p:
            return _out(case, *p.sigma_sd(s.eps[s.targets] - 0.05))
    plan = state["plan"]
    if do in ("job", "open"):
        plan.screening()
        return _out(case, *plan.qp_solve(gw.GW_QP_LINEARISED))
    if do == "steptree":
        plan.screening()
        return _out(case, *plan.qp_solve(gw.GW_QP_STEPTREE))
    if do == "wtable":
        plan.screening()
        return _out(case, plan.w_table())
    if do == "pi":
        return _out(case, plan.polarizability(state["xi"]))
    if do == "core":
        return _out(case, *plan.sigma_points(*state["points"]))
    r = plan.residues(*state["rhs"])
    return _out(case, *(r[k] for k in ("w_re", "w_im", "dw_re", "resnorm", "iters", "used_fallback")))


# ------------------------------------------------------------------------------------------ necessary work
def _n_residues(eps, n_occ, omegas):
    return sum(int((eps[:n_occ] > w).sum() + (eps[n_occ:] < w).sum()) for w in omegas)


def work(case):
    """One pass's arithmetic (a multiply-add is 2) and its inputs and outputs.  Pi is a symmetric product; the W table
    a factorisation and a triangular solve per frequency; a residue 26 applications of its operator (25 iterations
    and the right-hand side) and one derivative pass."""
    s = _system(case, 0)
    do, n, K = case["do"], case["n_aux"], s.n_occ * (s.n_bas - s.n_occ)
    n_t = len(s.targets)
    if do == "open":
        K += (s.n_occ - 1) * (s.n_bas - s.n_occ + 1)
        n_t = 4
    b_in = 8 * (n * K + n_t * s.n_bas * n)
    table = (N_FREQ + 1) * (float(n) * n * K + n ** 3 / 3.0 + float(n) * n * n_t * s.n_bas)
    residue = 8.0 * n * K * 26 + 4.0 * n * K
    if do == "pi":
        return {"bytes": 8 * n * K + 8 * case["n_xi"] * n * n, "flops": float(case["n_xi"]) * n * n * K}
    if do == "wtable":
        return {"bytes": b_in + 8 * n_t * s.n_bas * (N_FREQ + 1), "flops": table}
    if do == "core":
        t, om = _core_points(case, s)
        return {"bytes": b_in, "flops": residue * _n_residues(s.eps, s.n_occ, om)}
    if do == "residues":
        return {"bytes": b_in, "flops": residue * case["n_rhs"]}
    if do == "sd":
        # the pair matrix, a symmetric eigenproblem with its vectors, and the pole weights
        return {"bytes": b_in, "flops": 2.0 * n * K * K + 9.0 * float(K) ** 3 + 2.0 * n * K * (K + n_t * s.n_bas)}
    omegas = s.eps[s.targets] if do != "open" else s.eps[[s.n_occ - 1, s.n_occ]].repeat(2)
    evals = 10 if do == "steptree" else 1
    return {"bytes": b_in + 24 * n_t, "flops": table + evals * residue * _n_residues(s.eps, s.n_occ, omegas)}


# ------------------------------------------------------------------------------------------ 64-bit values
MOST_FLOPS = 8e12        # FP64 on this GPU runs at about 1 TFLOP/s


def _grid():
    t, w = np.polynomial.legendre.leggauss(N_FREQ)
    return X0 * (1 + t) / (1 - t), 2 * X0 * w / (1 - t) ** 2


def _exact_table(D, B, rows):
    """b^T [(1 - Pi(i xi))^-1 - 1] b at every grid point, and at 0 in the last column, for the rows b."""
    xi = np.append(_grid()[0], 0.0)
    W = torch.empty(len(rows), len(xi), dtype=torch.float64, device="cuda")
    eye = torch.eye(B.shape[0], dtype=torch.float64, device="cuda")
    b2 = (rows * rows).sum(1)
    for g, x in enumerate(xi):
        L = torch.linalg.cholesky(eye + (B * (4 * D / (D * D + x * x))) @ B.T)
        y = torch.linalg.solve_triangular(L, rows.T, upper=False)
        W[:, g] = (y * y).sum(0) - b2
    return W


def _exact_residue(D, B, b, x):
    """b^T [(1 - Pi(x))^-1 - 1] b and its derivative in x."""
    a1, a2 = (x - D) + 1j * ETA, (-x - D) + 1j * ETA
    c, dc = 2 * (1 / a1 + 1 / a2), 2 * (-1 / a1 ** 2 + 1 / a2 ** 2)
    A = torch.complex(torch.eye(len(b), dtype=torch.float64, device="cuda") - (B * c.real) @ B.T, -(B * c.imag) @ B.T)
    y = torch.linalg.solve(A, b.to(torch.complex128))
    t = torch.complex(B.T @ y.real, B.T @ y.imag)
    return complex((b * y).sum() - (b * b).sum()), complex((dc * t * t).sum())


def _exact_sigma(eps, n_occ, D, B, Bn_t, W_t, omega):
    """Re Sigma_c(omega) and its derivative by contour deformation for one state."""
    xi, wt = (torch.tensor(v, device="cuda") for v in _grid())
    e = torch.tensor(eps, device="cuda")
    a = (omega - e)[:, None]
    dW, x2 = W_t[:, :-1] - W_t[:, -1:], (xi * xi)[None]
    I = float((wt * dW * a / (a * a + x2)).sum()) / np.pi + float((W_t[:, -1] * torch.sign(a[:, 0])).sum()) / 2
    dI = float((wt * dW * (x2 - a * a) / (a * a + x2) ** 2).sum()) / np.pi
    R = dR = 0.0
    for m, em in enumerate(eps):
        d = em - omega if m < n_occ else omega - em
        th = 1.0 if d > 0 else 0.5 if d == 0 else 0.0
        if th:
            w, dw = _exact_residue(D, B, Bn_t[m], em - omega)
            sg = -th if m < n_occ else th
            R, dR = R + sg * w.real, dR - sg * dw.real
    return R - I, dR - dI


def _pairs(eps, n_occ):
    return torch.tensor((eps[None, n_occ:] - eps[:n_occ, None]).reshape(-1), device="cuda")


def _exact_linearised(levels, occ, D, B, Bn, targets, spins):
    W = _exact_table(D, B, Bn.reshape(-1, Bn.shape[2])).reshape(Bn.shape[0], Bn.shape[1], -1)
    e, z = [], []
    for k, (t, sp) in enumerate(zip(targets, spins)):
        eps = levels[sp]
        sg, dsg = _exact_sigma(eps, occ[sp], D, B, Bn[k], W[k], float(eps[t]))
        z.append(1.0 / (1.0 - dsg))
        e.append(float(eps[t]) + z[-1] * sg)
    return [np.array(e), np.array(z), None]


def exact(case, seed):
    do, s = case["do"], _system(case, seed)
    n, K = case["n_aux"], s.n_occ * (s.n_bas - s.n_occ)
    table = 2.0 * (N_FREQ + 1) * n * n * K
    if do == "open":
        eps_b, ob, t, spins = _open_spins(case, s)
        Ba, Bna = _tensors(s, seed, s.n_occ, t[:2])
        Bb, Bnb = _tensors(s, seed + (1 << 20), ob, t[2:])
        D = torch.cat([_pairs(s.eps, s.n_occ), _pairs(eps_b, ob)])
        return _exact_linearised((s.eps, eps_b), (s.n_occ, ob), D, torch.cat([Ba, Bb], 1) * 0.5 ** 0.5,
                                 torch.cat([Bna, Bnb]), t, spins)
    if do == "steptree":
        return None                          # which root a search ends at is not a value of its own
    one = 4.0 * n * n * K + 8.0 / 3.0 * n ** 3
    n_res = {"core": lambda: _n_residues(s.eps, s.n_occ, _core_points(case, s)[1]),
             "residues": lambda: case["n_rhs"]}.get(do, lambda: _n_residues(s.eps, s.n_occ, s.eps[s.targets]))()
    if do == "pi":
        total = 2.0 * case["n_xi"] * n * n * K
    elif do == "wtable":
        total = table
    elif do == "residues":
        total = one * n_res
    elif do == "sd":
        total = 0.0
    else:
        total = table + one * n_res
    if total > MOST_FLOPS:
        return None
    B, Bn = _tensors(s, seed)
    D = _pairs(s.eps, s.n_occ)
    if do == "pi":
        return [torch.stack([-(B * (4 * D / (D * D + x * x))) @ B.T for x in _pi_xi(case)])]
    if do == "wtable":
        return [_exact_table(D, B, Bn.reshape(-1, n)).reshape(len(s.targets), s.n_bas, -1)]
    if do == "residues":
        t, m, x = _residue_list(case, s, seed)
        w = [_exact_residue(D, B, Bn[int(a), int(b)], float(c)) for a, b, c in zip(t, m, x)]
        return [np.array([v[0].real for v in w]), np.array([v[0].imag for v in w]), np.array([v[1].real for v in w]),
                None, None, None]
    if do == "sd":
        r = D.sqrt()
        M = r[:, None] * (torch.diag(D) + 4 * B.T @ B) * r[None]
        lam, T = torch.linalg.eigh(M)
        Om = lam.sqrt()
        V = 2 * (B * r) @ T
        out = []
        for k, t in enumerate(s.targets):
            w2 = (Bn[k] @ V) ** 2 / (2 * Om)
            d = float(s.eps[t]) - 0.05 - torch.tensor(s.eps, device="cuda")[:, None]
            a = torch.cat([d[:s.n_occ] + Om, d[s.n_occ:] - Om])
            q = a * a + ETA * ETA
            out.append((float((w2 * a / q).sum()), -float((w2 * (a * a - ETA * ETA) / (q * q)).sum())))
        return [np.array([v[0] for v in out]), np.array([v[1] for v in out])]
    if do == "core":
        t, om = _core_points(case, s)
        W = _exact_table(D, B, Bn.reshape(-1, n)).reshape(len(s.targets), s.n_bas, -1)
        v = [_exact_sigma(s.eps, s.n_occ, D, B, Bn[int(k)], W[int(k)], float(w)) for k, w in zip(t, om)]
        return [np.array([a[0] for a in v]), np.array([a[1] for a in v])]
    return _exact_linearised((s.eps,), (s.n_occ,), D, B, Bn, s.targets, [0] * len(s.targets))
