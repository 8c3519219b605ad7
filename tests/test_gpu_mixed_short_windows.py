"""Mixed contraction where a CTA's work items are ranges of one short window each, formed pair tiles
and packed ones in turn, with aux blocks of different row counts: the A ring then holds chunks of
more windows than the two staged ones, and empties between items of different rows."""
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu

CLASSES = ("S", "T", "V", "J2", "J3")


# points per grid: 32 (one chunk), 48 (two), 108 (four, the last one short), 160 (two windows, the second
# of one chunk), 288 (three windows, the last of one chunk)
@pytest.mark.parametrize("make", [synth.fivez_triatomic, synth.triatomic_oh2])
@pytest.mark.parametrize("spec", [(2, 2, 1, 2, 2, 2, 1), (2, 2, 1, 2, 3, 2, 1), (2, 2, 1, 3, 3, 3, 1), (2, 2, 1, 2, 4, 5, 1),
                                  (2, 2, 2, 4, 3, 3, 1)])
def test_short_windows(make, spec):
    """(P|Q) and (P|ij) within the digits' bound of the FP64 path: per point 2^-38 of a window's largest
    factors for each factor's last digit and for its value's own error, twice that for the dropped orders and
    the fold, together below 2^-35 of max |a| max |b| (a = w V^P; b = chi chi or the aux function).
    The same bits from every pass, and (one-window grids, whose sums are never split) from a job of one class
    alone, where formed and packed tiles do not follow one another."""
    import torch
    assert torch.cuda.is_available(), "the CUDA path needs a GPU"
    import paper_2510_15204_gb300 as P
    job = make(2)
    job.specs = [spec]
    ctx = P.Context(0)
    J64, J = (P.Job.from_synth(ctx, job, p) for p in (P.FP64, P.MIXED))
    bound = {"J2": 0.0, "J3": 0.0}
    for g in range(J64.n_grids()):
        w = J64.grid_points(g)[3].abs()
        chi, aux, pot = (J64.grid_functions(g, k).abs() for k in (0, 2, 3))
        a = w.numel() * 2.0 ** -35 * float((w * pot).max())
        bound["J3"] = max(bound["J3"], a * float(chi.max()) ** 2)
        bound["J2"] = max(bound["J2"], a * float(aux.max()))
    ref = J64.compute(oracle.ALL)
    ws, out = J.alloc(oracle.ALL)
    first = None
    for _ in range(4):
        J.compute(oracle.ALL, ws, out)
        J.check(oracle.ALL, ws)
        got = {k: out[k].clone() for k in CLASSES}
        first = first or got
        for k in CLASSES:
            assert torch.equal(got[k], first[k]), k
    for k in bound:
        assert float((first[k] - ref[k]).abs().max()) <= bound[k], k
    if w.numel() <= 128:
        for i, k in enumerate(CLASSES):
            alone = J.compute(1 << i)
            assert torch.equal(alone[k], first[k]), k
