"""Atoms with more shells than the evaluation's tables of one node pair and phi row hold (about 3,070 of a
pair, 380 of a third centre at Q_phi = 16): the shells are taken in ranges.  Every value and element
as in a job that has only some of the shells."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

ATOMS = [(6, (0.1, -0.2, 0.0)), (8, (0.4, 0.3, 2.1)), (1, (1.9, -0.4, 0.6))]


def _many(counts, seed):
    """s shells (and a p and a d shell in front) per atom, exponents in no order."""
    rng = np.random.default_rng(seed)
    out = []
    for a, c in enumerate(counts):
        out += [(a, 2, 1, 0.9 + 0.1 * a), (a, 3, 2, 1.3 + 0.1 * a)][:min(2, c)]
        out += [(a, 1, 0, float(z)) for z in np.exp(rng.uniform(np.log(0.5), np.log(5.0), max(0, c - 2)))]
    return out


def _some(shells):
    """The first and last shells of every atom, and the functions of the whole list that they are."""
    keep, rows, o = [], [], 0
    for a in range(3):
        mine = [s for s in shells if s[0] == a]
        for k, s in enumerate(mine):
            w = 2 * s[2] + 1
            if k < 3 or k >= len(mine) - 2 or k == len(mine) // 2:
                keep.append(s)
                rows += range(o, o + w)
            o += w
    return keep, np.array(rows)


# aux shells per atom, basis shells per atom, spec: a third centre with more than its table's; a pair with more
# than its own in basis and aux functions
@pytest.mark.parametrize("na,nb,spec", [((3, 2, 450), (3, 2, 1), (3, 2, 2, 2, 2, 16, 2)),
                                        ((2, 1700, 1500), (2, 3, 0), (2, 2, 1, 2, 2, 2, 1)),
                                        ((3, 400, 2), (60, 2, 3), (2, 2, 2, 3, 2, 15, 1))])
@pytest.mark.parametrize("precision", [0, 1])
def test_shells_in_ranges(na, nb, spec, precision):
    import torch
    assert torch.cuda.is_available(), "the CUDA path needs a GPU"
    import paper_2510_15204_gb300 as P
    ctx = P.Context(0)
    basis, aux = _many(nb, 1), _many(na, 2)
    (fb, rb), (fa, ra) = _some(basis), _some(aux)
    job, few = synth.Job("many", ATOMS, basis, aux, [spec]), synth.Job("few", ATOMS, fb, fa, [spec])
    J, F = (P.Job.from_synth(ctx, j, precision) for j in (job, few))
    own = lambda sh, f: np.repeat([s[0] for s in sh], [2 * s[2] + 1 for s in sh])
    atom_b, atom_a = own(basis, 0), own(aux, 0)
    # function values: the same bits
    for g in range(J.n_grids()):
        A, B, C, _ = J.grid_info(g)
        for kind in range(4):
            got, want = J.grid_functions(g, kind), F.grid_functions(g, kind)
            on = [A, B] if kind < 2 or C is None else [C]
            at, rows = (atom_b, rb) if kind < 2 else (atom_a, ra)
            pick, o = [], 0
            for X in on:
                mine = np.flatnonzero(at == X)
                pick += [o + int(np.searchsorted(mine, r)) for r in rows if at[r] == X]
                o += len(mine)
            assert got.shape[0] == o
            assert torch.equal(got[pick], want), (g, kind)
    mask = P.J2 if max(na) > 1000 else (P.J3 if precision else P.S | P.V | P.J3)
    ref = oracle.compute(few, mask=mask)
    bound = {"J2": 0.0, "J3": 0.0}
    if precision:
        # mixed: per point 2^-38 of a window's largest factors for each factor's last digit and its value's own
        # error, twice that for the dropped orders and the fold, together below 2^-35 of max |a| max |b|
        for g in range(F.n_grids()):
            w = F.grid_points(g)[3].abs()
            chi, phi, pot = (F.grid_functions(g, k).abs() for k in (0, 2, 3))
            a = w.numel() * 2.0 ** -35 * float((w * pot).max())
            bound["J3"] = max(bound["J3"], a * float(chi.max()) ** 2)
            bound["J2"] = max(bound["J2"], a * float(phi.max()))
    out = J.compute(mask)
    torch.cuda.synchronize()
    for i, k in enumerate(P.CLASSES):
        if not (mask >> i) & 1:
            continue
        got = out[k]
        if k in ("S", "V"):
            got = got[rb][:, rb]
        elif k == "J2":
            got = got[ra][:, ra]
        else:
            got = got[ra][:, rb][:, :, rb]
        err = np.abs(got.cpu().numpy() - ref[k])
        tol = bound[k] if precision else 1e-12 * np.maximum(np.abs(ref[k]), ref["abs" + k])
        assert np.all(err <= tol), (k, float((err / np.where(tol > 0, tol, 1e-300)).max()))
