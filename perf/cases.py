"""The work a user of this library has it do, as a list of cases that can be timed and checked:
integral matrices of molecules (both precisions, one class or all of them, small and large
grids), a batch of jobs through the serving loop, and the RI 4-index assembly.

``listed()`` names the cases, ``draw(rng)`` gives more of the same ranges, ``prepare`` makes a
case's inputs from a seed, ``run`` is one pass through the public entry points, ``work`` counts
what a pass cannot do without, and ``exact`` is the same result in 64 bits, in plain torch."""
import math

import numpy as np
import torch

import paper_2510_15204_gb300 as P

CHARGE = {"H": 1, "C": 6, "N": 7, "O": 8}

# Shell counts per angular momentum (n = l + 1): basis and auxiliary functions of a heavy atom and
# of hydrogen, and the range the basis exponents are drawn from.  "minimal" is the 1s 2s 2p basis
# with 1s 2s 2p 3d auxiliaries of the diatomic workload, "scan" the single zeta = 1 functions
# (auxiliary l = 3 and l = 5) of the displacement scans.
PATTERNS = {
    "DZ": {"heavy": ((2, 1), (1, 1, 1, 1)), "H": ((2, 1), (1, 1, 1, 1)), "xi": (0.5, 3.0)},
    "TZ": {"heavy": ((3, 2, 1), (5, 4, 3, 2)), "H": ((3, 1), (4, 3, 1)), "xi": (0.3, 12.0)},
    "QZ": {"heavy": ((4, 3, 2, 1), (6, 5, 4, 3, 3)), "H": ((4, 3, 2), (6, 5, 4, 3, 1)), "xi": (0.2, 15.0)},
    "5Z": {"heavy": ((5, 4, 3, 2, 1), (8, 7, 6, 5, 4, 3)), "H": ((5, 4, 3, 2), (8, 7, 6, 5, 4, 3)), "xi": (0.15, 20.0)},
}
ALL, ONE_ELECTRON, COULOMB2 = P.ALL, P.S | P.T | P.V, P.J2


def _integrals(name, formula, basis, grid, precision, mask, **more):
    n_mu, n_nu, n_phi, q_mu, q_nu, q_phi, n_sp = grid
    case = {"name": name, "kind": "integrals", "formula": formula, "basis": basis, "n_mu": n_mu, "n_nu": n_nu,
            "n_phi": n_phi, "q_mu": q_mu, "q_nu": q_nu, "q_phi": q_phi, "n_sp": n_sp, "precision": precision,
            "mask": mask, "uneven": False, "graph": False}
    case.update(more)
    return case


def listed():
    return [
        # the smallest call: a plain FP64 diatomic, 57,600 points
        _integrals("h2_fp64", "HH", "minimal", (15, 10, 6, 4, 4, 4, 3), "fp64", P.S | P.T | P.V | P.J2),
        # the same molecule, every class, replayed from its captured graph: latency and launches
        _integrals("h2_mixed_graph", "HH", "minimal", (15, 10, 6, 4, 4, 4, 3), "mixed", ALL, graph=True),
        # an ordinary molecule in both precisions: bent triatomic, triple-zeta, six grids
        _integrals("triatomic_fp64", "OHH", "TZ", (20, 15, 8, 4, 4, 4, 3), "fp64", ALL),
        _integrals("triatomic_mixed", "OHH", "TZ", (20, 15, 8, 4, 4, 4, 3), "mixed", ALL),
        # one-electron matrices alone (no auxiliary basis read): the SO2-sized study of Table 1
        _integrals("one_electron_fp64", "NOO", "QZ", (26, 32, 14, 4, 4, 4, 3), "fp64", ONE_ELECTRON),
        # pentuple-zeta, dense grid: the precision stress, wide blocks
        _integrals("fivez_diatomic_mixed", "NO", "5Z", (30, 25, 16, 5, 4, 4, 3), "mixed", ALL),
        # the largest: nine atoms, quadruple-zeta, uneven grids per pair, 288 grids
        _integrals("c3h6_mixed", "CCCHHHHHH", "QZ", (30, 20, 8, 4, 4, 4, 3), "mixed", ALL, uneven=True),
        # one point of a displacement scan: 2-centre Coulomb alone on the 80/70/50 grid
        _integrals("scan_point_mixed", "HH", "scan", (80, 70, 50, 4, 4, 4, 3), "mixed", COULOMB2),
        # six jobs of different sizes arriving together at the server: created, submitted, awaited
        {"name": "serve_mixed", "kind": "serve", "formulas": "OHH,CO,HH,CHHO,NHHH,OO", "bases": "TZ,QZ,DZ,DZ,TZ,TZ",
         "n_mu": 20, "n_nu": 15, "n_phi": 8, "q": 4, "n_sp": 3},
        # RI assembly of the triatomic: factor, solve, all (ij|kl); small launches
        {"name": "ri_triatomic", "kind": "ri", "n": 82, "m": 676, "nc": 676, "nd": 676},
        # RI assembly of the nine-atom molecule: factor, solve of all pairs, a 4096 x 4096 block
        {"name": "ri_c3h6", "kind": "ri", "n": 693, "m": 51984, "nc": 4096, "nd": 4096},
        # a tensor-core block of (ij|kl) from a solved B
        {"name": "ri_block_mixed", "kind": "ri_mixed", "n": 693, "m": 51984, "nc": 4096, "nd": 4096},
    ]


def _log_int(rng, lo, hi):
    return min(hi, max(lo, int(round(math.exp(rng.uniform(math.log(lo), math.log(hi)))))))


def draw(rng):
    while True:
        kind = rng.choice(["integrals", "integrals", "integrals", "ri", "ri_mixed", "serve"])
        if kind == "ri" or kind == "ri_mixed":
            n, m = _log_int(rng, 8, 693), _log_int(rng, 30, 51984)
            case = {"kind": kind, "n": n, "m": m, "nc": _log_int(rng, min(m, 20), min(m, 4096)),
                    "nd": _log_int(rng, min(m, 20), min(m, 4096))}
            return case
        if kind == "serve":
            k = rng.randint(2, 6)
            pool = ["HH", "CO", "OO", "OHH", "NHHH", "CHHO", "NO"]
            return {"kind": "serve", "formulas": ",".join(rng.choice(pool) for _ in range(k)),
                    "bases": ",".join(rng.choice(["DZ", "TZ"]) for _ in range(k)), "n_mu": rng.randint(8, 20),
                    "n_nu": rng.randint(6, 15), "n_phi": rng.randint(3, 8), "q": rng.choice([3, 4]), "n_sp": rng.randint(1, 3)}
        precision = rng.choice(["fp64", "mixed", "mixed"])
        natoms = rng.choice([2, 2, 3, 3, 4] if precision == "fp64" else [2, 3, 3, 4, 5, 6])
        formula = "".join(rng.choice("CNO" if k == 0 else "HHCNO") for k in range(natoms))
        case = _integrals("", formula, rng.choice(["DZ", "TZ", "TZ", "QZ", "5Z"]),
                          (_log_int(rng, 8, 50), _log_int(rng, 6, 40), _log_int(rng, 3, 24), rng.choice([3, 4, 4, 5]),
                           rng.choice([3, 4, 4]), rng.choice([3, 4, 4, 5]), rng.randint(1, 4)), precision,
                          rng.choice([ALL, ALL, ALL, ONE_ELECTRON, P.J2 | P.J3, P.S, P.V | P.J3, COULOMB2]))
        case["uneven"], case["graph"] = rng.random() < 0.3, rng.random() < 0.3
        del case["name"]
        terms, points = _terms(case)
        nb, na = _counts(case["formula"], case["basis"])
        rows = 4 * (max(nb) + max(na))  # operand rows of one grid, at most
        if precision == "fp64" and (terms > 4e10 or points > 6e6):
            continue
        if precision == "mixed" and (terms > 1.2e12 or points > 2e7):
            continue
        if points * rows * 8 > 3e10:
            continue
        return case


# ------------------------------------------------------------------------------------- inputs


def _kinds(formula):
    return ["H" if a == "H" else "heavy" for a in formula]


def _counts(formula, basis):
    """Basis and auxiliary functions of each atom."""
    if basis == "minimal":
        return [5] * len(formula), [10] * len(formula)
    if basis == "scan":
        return [1] * len(formula), [7, 11]
    f = lambda c: sum(k * (2 * l + 1) for l, k in enumerate(c))
    return ([f(PATTERNS[basis][k][0]) for k in _kinds(formula)], [f(PATTERNS[basis][k][1]) for k in _kinds(formula)])


def _specs(case, natoms):
    g = [case[k] for k in ("n_mu", "n_nu", "n_phi", "q_mu", "q_nu", "q_phi", "n_sp")]
    if not case["uneven"]:
        return [tuple(g)]
    out = []  # per pair: between half and the whole of n_mu and n_nu
    for p in range(natoms * (natoms - 1) // 2):
        mu = max(2, g[0] - (7 * p + 3) % (g[0] // 2 + 1))
        nu = max(2, g[1] - (5 * p + 2) % (g[1] // 2 + 1))
        out.append((mu, nu) + tuple(g[2:]))
    return out


def _molecule(formula, basis, specs, rng):
    """Atoms placed one by one 1.8 to 2.6 bohr from an earlier one, no pair closer than 1.8, no
    three nearly in line; exponents log-uniform, auxiliary ones even-tempered over the range of
    the summed basis exponents of each angular momentum."""
    n = len(formula)
    while True:
        pos = [rng.normal(scale=0.3, size=3)]
        for _ in range(400):
            if len(pos) == n:
                break
            d = rng.normal(size=3)
            cand = pos[rng.integers(len(pos))] + rng.uniform(1.8, 2.6) * d / np.linalg.norm(d)
            if min(np.linalg.norm(cand - p) for p in pos) < 1.8:
                continue
            line = [np.linalg.norm(np.cross(a - cand, b - cand)) < 0.1 for i, a in enumerate(pos) for b in pos[:i]]
            if not any(line):
                pos.append(cand)
        if len(pos) == n:
            break
    atoms = [(CHARGE[a], tuple(float(x) for x in p)) for a, p in zip(formula, pos)]
    bas, aux = [], []
    for i, k in enumerate(_kinds(formula)):
        if basis == "scan":
            bas.append((i, 1, 0, float(rng.uniform(0.9, 1.1))))
            aux.append((i, 4, 3, float(rng.uniform(0.9, 1.1))) if i == 0 else (i, 6, 5, float(rng.uniform(0.9, 1.1))))
            continue
        if basis == "minimal":
            z, za = np.exp(rng.uniform(math.log(0.5), math.log(3.0), 3)), np.exp(rng.uniform(math.log(0.8), math.log(6.0), 4))
            bas += [(i, nn, l, float(x)) for (nn, l), x in zip(((1, 0), (2, 0), (2, 1)), z)]
            aux += [(i, nn, l, float(x)) for (nn, l), x in zip(((1, 0), (2, 0), (2, 1), (3, 2)), za)]
            continue
        lo, hi = PATTERNS[basis]["xi"]
        mine = []
        for l, c in enumerate(PATTERNS[basis][k][0]):
            mine += [(l, float(z)) for z in sorted(np.exp(rng.uniform(math.log(lo), math.log(hi), c)), reverse=True)]
        bas += [(i, l + 1, l, z) for l, z in mine]
        for big, c in enumerate(PATTERNS[basis][k][1]):
            sums = [z1 + z2 for j, (l1, z1) in enumerate(mine) for l2, z2 in mine[j:] if l1 + l2 == big]
            sums = sums or [z1 + z2 for j, (_, z1) in enumerate(mine) for _, z2 in mine[j:]]
            a, b = min(sums), max(sums)
            a, b = (a, b) if b > 1.01 * a else (a / 1.5, b * 1.5)
            aux += [(i, big + 1, big, float(z)) for z in ([math.sqrt(a * b)] if c == 1 else np.geomspace(b, a, c))]
    return atoms, bas, aux, specs


def _molecules(case, seed):
    """[(atoms, basis, aux, specs)] of a case."""
    rng = np.random.default_rng(seed)
    if case["kind"] == "serve":
        q = case["q"]
        specs = [(case["n_mu"], case["n_nu"], case["n_phi"], q, q, q, case["n_sp"])]
        return [_molecule(f, b, specs, rng) for f, b in zip(case["formulas"].split(","), case["bases"].split(","))]
    return [_molecule(case["formula"], case["basis"], _specs(case, len(case["formula"])), rng)]


def _ri_inputs(case, seed):
    """A symmetric positive definite metric of condition 1e4 and (P|ij) = metric x fit
    coefficients, the pair columns of sizes e^-6 to 1."""
    g = torch.Generator(device="cuda").manual_seed(seed)
    n, m = case["n"], case["m"]
    rnd = lambda *s: torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)
    q, _ = torch.linalg.qr(rnd(n, n))
    ev = torch.exp(math.log(1e4) * torch.rand(n, generator=g, device="cuda", dtype=torch.float64))
    J2 = (q * ev) @ q.T
    J2 = 0.5 * (J2 + J2.T)
    X = rnd(n, m) * torch.exp(-6.0 * torch.rand(1, m, generator=g, device="cuda", dtype=torch.float64))
    return J2.contiguous(), (J2 @ X).contiguous()


_CTX = []


def _context():
    if not _CTX:
        _CTX.append(P.Context(0))
    return _CTX[0]


def prepare(case, seed):
    ctx = _context()
    if case["kind"] == "integrals":
        (mol,) = _molecules(case, seed)
        job = P.Job(ctx, *mol, precision=P.FP64 if case["precision"] == "fp64" else P.MIXED)
        ws, out = job.alloc(case["mask"])
        return {"kind": "integrals", "job": job, "mask": case["mask"], "ws": ws, "out": out,
                "stream": torch.cuda.Stream() if case["graph"] else None}
    if case["kind"] == "serve":
        mols = _molecules(case, seed)
        host = []
        for mol in mols:
            job = P.Job(ctx, *mol, precision=P.MIXED)
            host.append({k: torch.empty(s, dtype=torch.float64).pin_memory() for k, s in job.out_shapes(P.ALL).items()})
        return {"kind": "serve", "ctx": ctx, "mols": mols, "host": host, "server": P.Server(ctx, 12 << 30, 4)}
    J2, J3 = _ri_inputs(case, seed)
    rng = np.random.default_rng(seed + 1)
    c0, d0 = int(rng.integers(0, case["m"] - case["nc"] + 1)), int(rng.integers(0, case["m"] - case["nd"] + 1))
    state = {"kind": case["kind"], "J2": J2, "J3": J3, "block": (c0, case["nc"], d0, case["nd"]),
             "eri": torch.empty((case["nc"], case["nd"]), dtype=torch.float64, device="cuda")}
    if case["kind"] == "ri":
        state["L"], state["B"] = torch.empty_like(J2), torch.empty_like(J3)
    else:
        # B = L^-1 (P|ij) as a program that has solved holds it
        state["B"] = torch.linalg.solve_triangular(torch.linalg.cholesky(J2), J3, upper=False).contiguous()
        need = _mixed_workspace(case["n"], case["nc"], case["nd"])
        state["ws"] = torch.empty(need, dtype=torch.uint8, device="cuda")
    return state


def _mixed_workspace(n, nc, nd):
    import ctypes
    need = ctypes.c_size_t()
    status = P.lib().psq_ri_eri_mixed_workspace(n, nc, nd, ctypes.byref(need))
    if status != 0:
        raise RuntimeError("psq_ri_eri_mixed_workspace: status %d" % status)
    return max(256, need.value)


def run(state):
    if state["kind"] == "integrals":
        job, mask, ws, out, stream = (state[k] for k in ("job", "mask", "ws", "out", "stream"))
        if stream is None:
            return job.compute(mask, ws, out)
        here = torch.cuda.current_stream()
        stream.wait_stream(here)
        job.compute_graph(mask, ws, out, stream)
        here.wait_stream(stream)
        return out
    if state["kind"] == "serve":
        jobs = [P.Job(state["ctx"], *mol, precision=P.MIXED) for mol in state["mols"]]
        tickets = [state["server"].submit(j, P.ALL, h) for j, h in zip(jobs, state["host"])]
        for t in tickets:
            state["server"].wait(t)
        return state["host"]
    c0, nc, d0, nd = state["block"]
    if state["kind"] == "ri":
        L, info = P.ri_factor(state["J2"], L=state["L"])
        state["B"].copy_(state["J3"])
        B = P.ri_solve(L, state["B"])
        return {"L": L, "info": info, "B": B, "eri": P.ri_eri(B, c0, nc, d0, nd, out=state["eri"])}
    return {"eri": P.ri_eri_mixed(state["B"], c0, nc, d0, nd, out=state["eri"], ws=state["ws"])}


# --------------------------------------------------------------------------------------- work


def _terms(case, formula=None, basis=None):
    """Multiply-adds (one per point and integrated element, each element on its one grid) and
    points of an integral job whose third centres all lie inside their grids."""
    formula, basis = formula or case["formula"], basis or case["basis"]
    n = len(formula)
    nb, na = _counts(formula, basis)
    if case["kind"] == "serve":
        g = (case["n_mu"], case["n_nu"], case["n_phi"], case["q"], case["q"], case["q"], case["n_sp"])
        specs, mask = [g], P.ALL
    else:
        specs, mask = _specs(case, n), case["mask"]
    pairs = [(a, b) for a in range(n) for b in range(a + 1, n)]
    base = {}
    fine = {}
    for k, p in enumerate(pairs):
        s = specs[k % len(specs)]
        q3 = s[3] * s[4] * s[5]
        base[p] = s[0] * s[1] * s[2] * q3
        fine[p] = base[p] + 8 * (s[6] ** 3 - 1) * q3
    three = mask & (P.V | P.J3)
    points = sum(base.values()) + (sum(fine[p] * (n - 2) for p in pairs) if three else 0)
    any_base = base[pairs[0]]

    def K(a, b, c):
        s = sorted({a, b, c})
        if len(s) == 1:
            return base.get((min(s[0], (s[0] + 1) % n), max(s[0], (s[0] + 1) % n)), any_base)
        return base[tuple(s)] if len(s) == 2 else fine[(min(a, b), max(a, b))]

    total = 0
    for a in range(n):
        for b in range(a, n):
            nab = nb[a] * nb[b] if a != b else nb[a] * (nb[a] + 1) // 2
            if a != b:  # one-centre overlap and kinetic elements are closed forms
                total += nab * K(a, b, a) * (bool(mask & P.S) + bool(mask & P.T))
            for c in range(n):
                total += nab * K(a, b, c) * (bool(mask & P.V) + na[c] * bool(mask & P.J3))
            if mask & P.J2:
                total += (na[a] * na[b] if a != b else na[a] * (na[a] + 1) // 2) * K(a, b, a)
    return total, points


def _matrix_bytes(formula, basis, mask):
    nb, na = (sum(x) for x in _counts(formula, basis))
    size = [nb * nb] * 3 + [na * na, na * nb * nb]
    return 8 * sum(s for c, s in enumerate(size) if (mask >> c) & 1)


def work(case):
    if case["kind"] == "integrals":
        nb, na = _counts(case["formula"], case["basis"])
        terms, _ = _terms(case)
        return {"bytes": 24 * (sum(nb) + sum(na)) + _matrix_bytes(case["formula"], case["basis"], case["mask"]), "flops": 2 * terms}
    if case["kind"] == "serve":
        each = list(zip(case["formulas"].split(","), case["bases"].split(",")))
        return {"bytes": sum(_matrix_bytes(f, b, P.ALL) for f, b in each), "flops": 2 * sum(_terms(case, f, b)[0] for f, b in each)}
    n, m, nc, nd = case["n"], case["m"], case["nc"], case["nd"]
    if case["kind"] == "ri":
        return {"bytes": 8 * (2 * n * n + 2 * n * m + nc * nd), "flops": n ** 3 // 3 + n * n * m + 2 * n * nc * nd}
    return {"bytes": 8 * (n * (nc + nd) + nc * nd), "flops": 2 * n * nc * nd}


# -------------------------------------------------------------------------------------- exact
# The same quadrature written plainly in 64-bit torch: grids of Section 2, functions of eq 1 and
# eqs 15-16, every element summed on the grid of its distinct centres (Section 4).


def _t(x):
    return torch.as_tensor(np.asarray(x, dtype=np.float64), device="cuda" if torch.cuda.is_available() else "cpu")


def _frame(RA, RB, RC):
    d = RA - RB
    a, M, ez = 0.5 * np.linalg.norm(d), 0.5 * (RA + RB), d / np.linalg.norm(d)
    ex = None
    if RC is not None:
        perp = (RC - M) - ez * np.dot(RC - M, ez)
        if np.linalg.norm(perp) > 1e-10 * a:
            ex = perp / np.linalg.norm(perp)
    if ex is None:
        ex = np.array([1.0, 0, 0]) - ez * ez[0]
        if np.linalg.norm(ex) < 0.5:
            ex = np.array([0, 1.0, 0]) - ez * ez[1]
        ex = ex / np.linalg.norm(ex)
    return a, M, np.stack([ex, np.cross(ez, ex), ez], axis=1)


def _grid(RA, RB, RC, spec):
    """Offsets from A, B (and C) and distances and weights of the points of one grid."""
    n_mu, n_nu, n_phi, q_mu, q_nu, q_phi, n_sp = spec
    a, M, R = _frame(RA, RB, RC)
    mu = 2.3 * a ** 0.25 * np.arctanh(np.arange(n_mu + 1) / (n_mu + 1.0))
    nu, ph = np.pi * np.arange(n_nu + 1) / n_nu, 2 * np.pi * np.arange(n_phi + 1) / n_phi
    touch = set()
    if RC is not None:
        c = R.T @ (RC - M)
        rho = math.hypot(c[0], c[1])
        ra, rb = math.hypot(rho, c[2] - a), math.hypot(rho, c[2] + a)
        mc, vc = math.acosh(max(1.0, (ra + rb) / (2 * a))), math.acos(min(1.0, max(-1.0, (rb - ra) / (2 * a))))
        if mc < mu[-1]:
            assert rho > 1e-6 * a  # the molecules here have no three atoms in line
            i, j = 1 + int(np.argmin(abs(mu[1:-1] - mc))), 1 + int(np.argmin(abs(nu[1:-1] - vc)))
            mu[i], nu[j] = mc, vc
            touch = {(x, y, z) for x in (i - 1, i) for y in (j - 1, j) for z in (0, n_phi - 1)}
    cells = []
    for x in range(n_mu):
        for y in range(n_nu):
            for z in range(n_phi):
                if (x, y, z) not in touch:
                    cells.append((mu[x], mu[x + 1], nu[y], nu[y + 1], ph[z], ph[z + 1]))
    for x, y, z in sorted(touch):
        m, v, f = (np.linspace(e[k], e[k + 1], n_sp + 1) for e, k in ((mu, x), (nu, y), (ph, z)))
        cells += [(m[p], m[p + 1], v[q], v[q + 1], f[r], f[r + 1]) for p in range(n_sp) for q in range(n_sp) for r in range(n_sp)]
    c = _t(np.array(cells))

    def nodes(k, q, shape):
        x, w = np.polynomial.legendre.leggauss(q)
        lo, hi = c[:, 2 * k, None], c[:, 2 * k + 1, None]
        h = 0.5 * (hi - lo)
        v, w = 0.5 * (lo + hi) + h * _t(x), h * _t(w)
        full = (c.shape[0], q_mu, q_nu, q_phi)
        return v.reshape(shape).expand(full).reshape(-1), w.reshape(shape).expand(full).reshape(-1)

    m, wm = nodes(0, q_mu, (-1, q_mu, 1, 1))
    v, wv = nodes(1, q_nu, (-1, 1, q_nu, 1))
    f, wf = nodes(2, q_phi, (-1, 1, 1, q_phi))
    sh, sn, cs = torch.sinh(m), torch.sin(v), torch.cos(v)
    w = wm * wv * wf * a ** 3 * sh * sn * (sh * sh + sn * sn)
    s2m, s2n, c2n = torch.sinh(m / 2) ** 2, torch.sin(v / 2) ** 2, torch.cos(v / 2) ** 2
    xy = torch.stack([a * sh * sn * torch.cos(f), a * sh * sn * torch.sin(f)])
    Rt = _t(R)
    at = {"A": (Rt @ torch.cat([xy, (2 * a * (s2m * cs - s2n))[None]]), 2 * a * (s2m + s2n)),
          "B": (Rt @ torch.cat([xy, (2 * a * (s2m * cs + c2n))[None]]), 2 * a * (s2m + c2n))}
    if RC is not None:
        p = torch.cat([xy, (a * torch.cosh(m) * cs)[None]]) - _t(R.T @ (RC - M))[:, None]
        at["C"] = (Rt @ p, torch.sqrt((p * p).sum(0)))
    return w, at


def _harmonics(lmax, u):
    """Real orthonormal harmonics, no Condon-Shortley phase, {l: (2l+1, k)} with m = -l..l."""
    re, im = [torch.ones_like(u[0])], [torch.zeros_like(u[0])]
    for m in range(1, lmax + 1):
        re.append(u[0] * re[-1] - u[1] * im[-1])
        im.append(u[0] * im[-1] + u[1] * re[-2])
    out = {l: [None] * (2 * l + 1) for l in range(lmax + 1)}
    for m in range(lmax + 1):
        q = {m: torch.full_like(u[0], float(np.prod(np.arange(1, 2 * m, 2))) if m else 1.0)}
        for l in range(m + 1, lmax + 1):
            q[l] = ((2 * l - 1) * u[2] * q[l - 1] - ((l + m - 1) * q[l - 2] if l > m + 1 else 0)) / (l - m)
        for l in range(m, lmax + 1):
            k = math.sqrt((2 * l + 1) / (4 * math.pi) * math.factorial(l - m) / math.factorial(l + m) * (2 if m else 1))
            out[l][l + m] = k * q[l] * re[m]
            if m:
                out[l][l - m] = k * q[l] * im[m]
    return {l: torch.stack(v) for l, v in out.items()}


def _upper_gamma(k, x):
    term, s = torch.ones_like(x), torch.ones_like(x)
    for j in range(1, k):
        term = term * x / j
        s = s + term
    return math.factorial(k - 1) * torch.exp(-x) * s


def _lower_gamma_over(k, x):
    """gamma(k, x) / x^k: the positive series below x = k, (k-1)! - Gamma(k, x) above."""
    xs = torch.clamp(x, max=float(k))
    term = torch.full_like(x, 1.0 / k)
    s = term.clone()
    for j in range(1, 200):
        term = term * xs / (k + j)
        s = s + term
        if j % 16 == 0 and not bool((term > 1e-18 * s).any()):
            break
    return torch.where(x < k, torch.exp(-xs) * s, (math.factorial(k - 1) - _upper_gamma(k, x)) / x ** k)


def _values(shells, d, r, kind):
    """Rows of the functions of one centre: "f" chi, "l" its Laplacian, "v" its Coulomb potential."""
    if not shells:
        return r.new_zeros((0, r.shape[0]))
    Y = _harmonics(max(s[2] for s in shells), d / r)
    rows = []
    for _, n, l, z in shells:
        norm = (2 * z) ** (n + 0.5) / math.sqrt(math.factorial(2 * n))
        x = z * r
        if kind == "v":
            f = 4 * math.pi / (2 * l + 1) * norm * (r ** (n + 1) * _lower_gamma_over(n + l + 2, x)
                                                   + r ** l * _upper_gamma(n - l + 1, x) / z ** (n - l + 1))
        else:
            f = norm * r ** (n - 1) * torch.exp(-x)
            if kind == "l":
                f = f * ((n * (n - 1) - l * (l + 1)) / (r * r) - 2 * n * z / r + z * z)
        rows.append(f[None] * Y[l])
    return torch.cat(rows)


def _one_centre(A, B):
    """Overlap and kinetic element of two functions of one atom, the same l and m."""
    (_, n, l, x), (_, k, _, y) = A, B
    nn = (2 * x) ** (n + 0.5) / math.sqrt(math.factorial(2 * n)) * (2 * y) ** (k + 0.5) / math.sqrt(math.factorial(2 * k))
    I = lambda p: math.factorial(p) / (x + y) ** (p + 1) if p >= 0 else 0.0
    lap = lambda p, z: (p * (p - 1) - l * (l + 1)) * I(n + k - 2) - 2 * p * z * I(n + k - 1) + z * z * I(n + k)
    return nn * I(n + k), -0.25 * nn * (lap(k, y) + lap(n, x))


def _exact_job(atoms, basis, aux, specs, mask):
    n = len(atoms)
    R = [np.array(p) for _, p in atoms]
    bs, au = [[s for s in basis if s[0] == X] for X in range(n)], [[s for s in aux if s[0] == X] for X in range(n)]
    cnt = lambda sh: sum(2 * s[2] + 1 for s in sh)
    ob, oa = np.cumsum([0] + [cnt(s) for s in bs]), np.cumsum([0] + [cnt(s) for s in au])
    sb, sa = [slice(ob[X], ob[X + 1]) for X in range(n)], [slice(oa[X], oa[X + 1]) for X in range(n)]
    near = [min((Y for Y in range(n) if Y != X), key=lambda Y: (np.linalg.norm(R[X] - R[Y]), Y)) for X in range(n)]
    zero = lambda *s: _t(np.zeros(s))
    S, T, V = (zero(ob[-1], ob[-1]) for _ in range(3))
    J2, J3 = zero(oa[-1], oa[-1]), zero(*((oa[-1], ob[-1], ob[-1]) if mask & P.J3 else (1, 1, 1)))

    def grid_of(a, b, c):
        s = sorted({a, b, c})
        if len(s) == 1:
            return (min(s[0], near[s[0]]), max(s[0], near[s[0]]), -1)
        return (s[0], s[1], -1) if len(s) == 2 else (min(a, b), max(a, b), c)

    pairs = [(a, b) for a in range(n) for b in range(a + 1, n)]
    keys = [p + (-1,) for p in pairs] + ([p + (c,) for p in pairs for c in range(n) if c not in p] if mask & (P.V | P.J3) else [])
    for key in keys:
        A, B, C = key
        spec = specs[0] if len(specs) == 1 else specs[pairs.index((A, B))]
        w_all, at_all = _grid(R[A], R[B], R[C] if C >= 0 else None, spec)
        here = {A: "A", B: "B"}
        if C >= 0:
            here[C] = "C"
        for k0 in range(0, w_all.shape[0], 65536):
            w = w_all[k0:k0 + 65536]
            at = {X: (d[:, k0:k0 + 65536], r[k0:k0 + 65536]) for X, (d, r) in ((X, at_all[c]) for X, c in here.items())}
            F = {X: _values(bs[X], *at[X], "f") for X in (A, B)} if mask & ~P.J2 else {}
            U = {X: _values(au[X], *at[X], "v") * w for X in here if C < 0 or X == C} if mask & (P.J2 | P.J3) else {}
            for Y, W in ((A, A), (A, B), (B, B)):
                if Y != W and C < 0:
                    if mask & P.S:
                        S[sb[Y], sb[W]] += (F[Y] * w) @ F[W].T
                    if mask & P.T:
                        LY, LW = _values(bs[Y], *at[Y], "l"), _values(bs[W], *at[W], "l")
                        T[sb[Y], sb[W]] -= 0.25 * ((F[Y] * w) @ LW.T + (LY * w) @ F[W].T)
                for X in here:
                    if grid_of(Y, W, X) != key:
                        continue
                    if mask & P.V:
                        V[sb[Y], sb[W]] -= atoms[X][0] * ((F[Y] * (w / at[X][1])) @ F[W].T)
                    if mask & P.J3:
                        ny, nw = F[Y].shape[0], F[W].shape[0]
                        FF = (F[Y][:, None] * F[W][None]).reshape(ny * nw, -1)
                        J3[sa[X], sb[Y], sb[W]] += (U[X] @ FF.T).reshape(-1, ny, nw)
                if mask & P.J2 and C < 0 and grid_of(Y, W, Y) == key:
                    G = {X: _values(au[X], *at[X], "f") for X in (Y, W)}
                    J2[sa[Y], sa[W]] += 0.5 * (U[Y] @ G[W].T + (U[W] @ G[Y].T).T)
    for Y in range(n):
        for W in range(Y + 1, n):
            for M, s in ((S, sb), (T, sb), (V, sb), (J2, sa)):
                M[s[W], s[Y]] = M[s[Y], s[W]].T
            if mask & P.J3:
                J3[:, sb[W], sb[Y]] = J3[:, sb[Y], sb[W]].transpose(1, 2)
        i = ob[Y]
        for a in bs[Y]:
            j = ob[Y]
            for b in bs[Y]:
                if a[2] == b[2]:
                    s, t = _one_centre(a, b)
                    for m in range(2 * a[2] + 1):
                        S[i + m, j + m], T[i + m, j + m] = s, t
                j += 2 * b[2] + 1
            i += 2 * a[2] + 1
    return {k: v for c, (k, v) in enumerate(zip(P.CLASSES, (S, T, V, J2, J3))) if (mask >> c) & 1}


def exact(case, seed):
    if case["kind"] == "integrals":
        return _exact_job(*_molecules(case, seed)[0], mask=case["mask"])
    if case["kind"] == "serve":
        return [_exact_job(*mol, mask=P.ALL) for mol in _molecules(case, seed)]
    J2, J3 = _ri_inputs(case, seed)
    L = torch.linalg.cholesky(J2)
    B = torch.linalg.solve_triangular(L, J3, upper=False)
    rng = np.random.default_rng(seed + 1)
    c0, d0 = int(rng.integers(0, case["m"] - case["nc"] + 1)), int(rng.integers(0, case["m"] - case["nd"] + 1))
    eri = B[:, c0:c0 + case["nc"]].T @ B[:, d0:d0 + case["nd"]]
    return {"eri": eri} if case["kind"] == "ri_mixed" else {"L": L, "info": None, "B": B, "eri": eri}
