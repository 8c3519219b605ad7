"""A grid with more than 32,767 operand rows (basis functions and their kinetic operands, aux functions, potentials): the
kinetic block of a small atom with one of 16,406 functions, whose shells repeat four exponents, against
the oracle on one shell of each."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("precision", [0, 1])
def test_rows_past_16_bits(precision):
    import torch
    assert torch.cuda.is_available(), "the CUDA path needs a GPU"
    import paper_2510_15204_gb300 as P
    atoms = [(1, (0.0, 0.0, 0.0)), (6, (0.3, 0.4, 1.6))]
    few = [(0, 1, 0, 1.1)] + [(1, 7, 6, z) for z in (1.5, 2.0, 2.7, 3.3)]
    n = 1262
    many = few[:1] + [few[1 + k % 4] for k in range(n)]
    spec = [(3, 3, 2, 3, 3, 3, 1)]
    ref = oracle.compute(synth.Job("few", atoms, few, [], spec), mask=P.T)
    ctx = P.Context(0)
    J = P.Job.from_synth(ctx, synth.Job("many", atoms, many, [], spec), precision)
    ws, out = J.alloc(P.T)
    got = J.compute(P.T, ws, out)["T"]
    J.check(P.T, ws)
    block, mirror = got[0, 1:].cpu().numpy().reshape(n, 13), got[1:, 0].cpu().numpy().reshape(n, 13)
    want = ref["T"][0, 1:].reshape(4, 13)[np.arange(n) % 4]
    if precision == 0:
        tol = 1e-12 * np.maximum(np.abs(want), ref["absT"][0, 1:].reshape(4, 13)[np.arange(n) % 4])
    else:
        # per point 2^-38 of a window's largest factors for each factor's last digit and its value's own error, twice that for
        # the dropped orders and the fold: below 2^-35 of max |w lap chi| max |chi|, and T is half of two sums' mean
        F = P.Job.from_synth(ctx, synth.Job("few", atoms, few, [], spec), precision)
        w = F.grid_points(0)[3].abs()
        tol = w.numel() * 2.0 ** -35 * float((w * F.grid_functions(0, 1).abs()).max()) * float(F.grid_functions(0, 0).abs().max())
    assert np.all(np.abs(block - want) <= tol)
    assert np.all(np.abs(mirror - want) <= tol)
