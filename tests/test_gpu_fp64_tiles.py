"""The plain FP64 path's contraction at the edges of its tiles, against the oracle at the path's bar
(1e-12 of each element's absolute-term sum): basis blocks around the FMA tiles' 16 registers and 31
/ 32 lanes (and the narrow ones that share a warp), aux counts around the 32 columns and pair lists
around the 128 rows of the tensor-core tiles, point counts around its 64-point windows."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

TOL = 1e-12


def _shells(atom, n, rng, lo, hi):
    """Shells of one atom with n functions in all: d, p and s shells, as many as fit."""
    out = []
    while n > 0:
        l = 2 if n >= 9 else (1 if n >= 3 else 0)
        out.append((atom, l + 1, l, float(np.exp(rng.uniform(np.log(lo), np.log(hi))))))
        n -= 2 * l + 1
    return out


@pytest.mark.parametrize("nb,na,spec", [
    ((1, 1), (1, 1), (4, 3, 2, 2, 2, 2, 1)),        # one function each, 192 points
    ((3, 4), (31, 2), (3, 3, 2, 3, 3, 3, 1)),       # 486 points: a short last window
    ((7, 8), (32, 33), (5, 4, 2, 4, 3, 3, 1)),
    ((15, 16), (33, 31), (4, 4, 2, 4, 4, 4, 1)),    # 15 x 16 = 240 pairs, whole windows
    ((16, 17), (5, 64), (4, 3, 3, 3, 4, 3, 1)),
    ((31, 3), (2, 65), (3, 4, 2, 3, 3, 4, 1)),      # 31 rows: the largest whole symmetric tile
    ((32, 33), (9, 1), (3, 3, 2, 4, 3, 3, 1)),
    ((0, 6), (7, 0), (4, 4, 2, 3, 3, 3, 1)),        # an atom without basis, one without aux functions
])
def test_tile_edges_match_oracle(nb, na, spec):
    import torch
    import paper_2510_15204_gb300 as P
    from paper_2510_15204_gb300 import build
    build.build()
    rng = np.random.default_rng(sum(nb) * 100 + sum(na))
    atoms = [(6, (0.1, -0.2, 0.0)), (8, (0.4, 0.3, 2.1)), (1, (1.9, -0.4, 0.6))]
    basis, aux = [], []
    for a in range(3):
        basis += _shells(a, (nb + (4,))[a], rng, 0.4, 4.0)
        aux += _shells(a, (na + (3,))[a], rng, 0.6, 6.0)
    job = synth.Job("tiles", atoms, basis, aux, [spec])
    ref = oracle.compute(job, mask=oracle.ALL)
    J = P.Job.from_synth(P.Context(0), job, P.FP64)
    out = J.compute(oracle.ALL)
    torch.cuda.synchronize()
    for k in P.CLASSES:
        got = out[k].cpu().numpy()
        scale = np.maximum(np.abs(ref[k]), ref["abs" + k])
        err = np.abs(got - ref[k]) / np.where(scale > 0, scale, 1.0)
        assert np.all(err <= TOL), (k, float(err.max()))
