"""The exact-digit sums where the two factors of a 64-point window are large at different points: every
element keeps the precision of its own terms.

Bound of an (ij|kl) element or a solved right-hand side, from the method: a window of k rows drops
k 2^-60.5 of the product S of its two power-of-two scales (the seven digit products of order 8, 7 x 2^14 x
2^-78 each row, those above, and two truncations of 2^-63), and is only summed that way where its
absolute terms reach 2^-8 S; else it is a chain of k FP64 FMAs.  So k 2^-52.5 of the absolute terms in one case
and k 2^-53 in the other, and a rounding per window of the running sum: below (n + 4) 2^-52 of the
absolute terms in all.  Integrals: the FP64 path's own bar, 1e-12 of an element's absolute terms."""
import numpy as np
import pytest

import oracle
import synth

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "the CUDA path needs a GPU"
    import paper_2510_15204_gb300 as P
    from paper_2510_15204_gb300 import build
    build.build()
    return P


def _shells(counts, lo, hi):
    return [(a, l + 1, l, float(z)) for a in (0, 1) for l, c in enumerate(counts) for z in np.geomspace(hi, lo, c + 1)[:c]]


# (spec, distance, basis and aux shells per l, exponents): cells of 27, 45 and 60 points, so that windows run
# across cells and, where a row of cells ends, from one nucleus to the other; one phi cell; whole
# cells per window with steep functions
CASES = [
    ((10, 8, 4, 3, 3, 3, 1), 6.0, (4, 3, 2, 1), (6, 5, 4, 3, 3), (0.2, 15.0)),
    ((8, 6, 3, 5, 3, 3, 1), 2.2, (5, 4, 3, 2, 1), (4, 3, 3, 3, 3, 3), (0.15, 20.0)),
    ((12, 10, 1, 3, 3, 3, 1), 4.0, (4, 3, 2, 1), (6, 5, 4, 3, 3), (0.2, 15.0)),
    ((6, 5, 3, 3, 4, 5, 1), 8.0, (3, 2, 2), (3, 3, 3, 2, 2, 2, 2), (0.3, 30.0)),
    ((5, 4, 3, 4, 4, 4, 1), 7.0, (3, 2, 2), (3, 3, 3, 2, 2, 2, 2), (0.3, 40.0)),
]


@pytest.mark.parametrize("spec,dist,bas,aux,xi", CASES)
def test_integrals_keep_the_precision_of_their_terms(P, spec, dist, bas, aux, xi):
    import torch
    atoms = [(7, (0.0, 0.0, 0.0)), (8, (0.3 * dist, 0.5 * dist, float(np.sqrt(0.66)) * dist))]
    job = synth.Job("windows", atoms, _shells(bas, *xi), _shells(aux, 1.5 * xi[0], 1.5 * xi[1]), [spec])
    mask = P.J2 | P.J3
    ref = oracle.compute(job, mask=mask)
    out = P.Job.from_synth(P.Context(0), job, P.FP64).compute(mask)
    torch.cuda.synchronize()
    for k in ("J2", "J3"):
        scale = np.maximum(np.abs(ref[k]), ref["abs" + k])
        err = np.abs(out[k].cpu().numpy() - ref[k]) / np.where(scale > 0, scale, 1.0)
        assert np.all(err <= 1e-12), (k, float(err.max()))


def _exact(a, b):
    """a^T b in extended precision, and the sum of the absolute products."""
    a, b = a.astype(np.longdouble), b.astype(np.longdouble)
    return sum(np.outer(x, y) for x, y in zip(a, b)), sum(np.outer(x, y) for x, y in zip(abs(a), abs(b)))


# decay: bits per row by which a column's values fall off from its own largest; scale of all of them
@pytest.mark.parametrize("n", [2, 5, 33, 64, 65, 150])
@pytest.mark.parametrize("decay,scale", [(0.0, 0), (1.0, 0), (6.0, 0), (30.0, 0), (1.0, -500), (0.0, -505), (2.0, 400), (0.0, -970)])
def test_eri_columns_large_at_different_rows(P, n, decay, scale):
    import torch
    rng = np.random.default_rng(n + int(decay))
    m = 150
    at = rng.integers(0, n, m)
    B = rng.standard_normal((n, m)) * 2.0 ** np.maximum(scale - decay * np.abs(np.arange(n)[:, None] - at), -1060.0)
    B[rng.uniform(size=(n, m)) < 0.03] = 0.0
    B[:, 17] = 0.0
    B[:, 23] *= 2.0 ** (600 if scale < 0 else 0)
    got = P.ri_eri(torch.tensor(B, device="cuda"), 3, 140, 0, 70).cpu().numpy()
    ref, terms = _exact(B[:, 3:143], B[:, 0:70])
    err = np.abs(got.astype(np.longdouble) - ref)
    # (products below 2^-1022 round to multiples of 2^-1074)
    bound = (n + 4) * (2.0 ** -52 * terms + np.longdouble(2.0) ** -1074)
    assert np.all(err <= bound), float((err / bound).max())


@pytest.mark.parametrize("n,m", [(40, 9), (97, 300), (161, 2000)])
@pytest.mark.parametrize("span", [0.0, 10.0, 40.0])
def test_solve_with_graded_rows(P, n, m, span):
    """L = D L0 D^-1 with D a diagonal of 2^-span .. 2^span in random order: the solution's rows grow where the
    columns of L shrink."""
    import torch
    rng = np.random.default_rng(n + int(span))
    d = 2.0 ** rng.uniform(-span, span, n)
    L = (np.tril(rng.standard_normal((n, n))) + 4.0 * np.sqrt(n) * np.eye(n)) * d[:, None] / d[None, :]
    R = rng.standard_normal((n, m)) * d[:, None]
    X = P.ri_solve(torch.tensor(L, device="cuda"), torch.tensor(R, device="cuda")).cpu().numpy()
    res = np.abs((L.astype(np.longdouble) @ X.astype(np.longdouble) - R).astype(np.float64))
    assert np.all(res <= (n + 4) * 2.0 ** -52 * (np.abs(L) @ np.abs(X) + np.abs(R)))


def test_last_order_counts(P):
    """Sums of four products that cancel to rounding, between columns of values in [1, 2) (scales 2): what the digits drop
    is 4 x 2^-60.5 S with S = 4, and the joined integer rounds once at 2^-62 S.  The products of the last order kept,
    7, come to about 2^-55 S here."""
    import torch
    rng = np.random.default_rng(7)
    m = 256
    A, B = 1.0 + rng.uniform(size=(4, m)) * 0.99, 1.0 + rng.uniform(size=(4, m)) * 0.99
    B[1:3] *= -1.0
    r = (A[0] * B[0] + A[1] * B[1] + A[2] * B[2]).astype(np.longdouble)
    B[3] = -(r / A[3]).astype(np.float64)
    keep = (np.abs(B[3]) < 1.98)
    both = np.concatenate([A, B], axis=1)
    got = np.diag(P.ri_eri(torch.tensor(both, device="cuda"), 0, m, m, m).cpu().numpy())
    import fractions
    f = fractions.Fraction
    ref = [sum(f(x) * f(y) for x, y in zip(A[:, i], B[:, i])) for i in range(m)]
    err = np.array([float(abs(f(g) - e)) for g, e in zip(got, ref)])
    assert np.all(np.abs(got[keep]) < 2.0 ** -48)
    assert np.all(err[keep] <= 4 * (4 * 2.0 ** -60.5 + 2.0 ** -62) + 2.0 ** -53 * np.abs(got[keep])), float(err[keep].max())
