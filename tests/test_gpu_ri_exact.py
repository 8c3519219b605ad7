"""The exact-digit FP64 products of the RI assembly (psq_ri_eri, psq_ri_solve: eight 8-bit digits per
value and 64-row window on the tensor cores) at the edges of their tiles.

Bound of an (ij|kl) element, from the method: per window of 64 aux rows at most two units of
2^-52 of the product of the power-of-two scales (each below twice the window's largest |value|),
so 2^-49 max|a| max|b|, plus one FP64 rounding per window of the running sum."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def P():
    import torch
    assert torch.cuda.is_available(), "the CUDA path needs a GPU"
    import paper_2510_15204_gb300 as P
    from paper_2510_15204_gb300 import build
    build.build()
    return P


def _bound(a, b):
    out = np.zeros((a.shape[1], b.shape[1]))
    for w in range(0, a.shape[0], 64):
        out += 2.0 ** -49 * np.outer(np.abs(a[w:w + 64]).max(axis=0), np.abs(b[w:w + 64]).max(axis=0))
    return out + (a.shape[0] // 64 + 2) * 2.0 ** -53 * (np.abs(a).T @ np.abs(b))


@pytest.mark.parametrize("n", [1, 31, 32, 33, 63, 64, 65, 127, 129, 200])
@pytest.mark.parametrize("m,blk", [(9, (0, 9, 0, 9)), (333, (1, 127, 3, 33)), (333, (5, 129, 300, 31)), (333, (0, 256, 7, 64))])
@pytest.mark.parametrize("span", [0.0, 3.0, 30.0])
def test_eri_within_the_digit_bound(P, n, m, blk, span):
    import torch
    rng = np.random.default_rng(1000 * n + m + int(span))
    B = rng.standard_normal((n, m)) * np.exp(rng.uniform(-span, span, (n, m)))
    B[rng.uniform(size=(n, m)) < 0.05] = 0.0
    c0, nc, d0, nd = blk
    a, b = B[:, c0:c0 + nc], B[:, d0:d0 + nd]
    got = P.ri_eri(torch.tensor(B, device="cuda"), c0, nc, d0, nd).cpu().numpy()
    ref = (a.astype(np.longdouble)[:, :, None] * b.astype(np.longdouble)[:, None, :]).sum(axis=0)
    err = np.abs((got - ref).astype(np.float64))
    bound = _bound(a, b)
    assert np.all(err <= bound), float((err / np.where(bound > 0, bound, 1)).max())


def test_eri_special_values(P):
    """Infinities, NaN, values near the ends of the FP64 range and constant columns."""
    import torch
    rng = np.random.default_rng(3)
    B = rng.standard_normal((70, 40))
    B[3, 1], B[66, 2], B[10, 5] = np.inf, np.nan, -np.inf
    B[:, 7] = 1e200 * rng.standard_normal(70)
    B[:, 8] = 1e-200 * rng.standard_normal(70)
    B[:, 9] = 0.1
    B[:, 10] = 0.0
    got = P.ri_eri(torch.tensor(B, device="cuda"), 0, 40, 0, 40).cpu().numpy()
    with np.errstate(all="ignore"):
        # the products with a zero column are NaN where the other side is infinite, as in FP64
        ref = np.array([[np.add.reduce(B[:, i] * B[:, j]) for j in range(40)] for i in range(40)])
    assert np.array_equal(np.isnan(got), np.isnan(ref))
    assert np.array_equal(np.isposinf(got), np.isposinf(ref)) and np.array_equal(np.isneginf(got), np.isneginf(ref))
    ok = np.isfinite(ref)
    scale = np.abs(np.where(np.isfinite(B), B, 0)).T @ np.abs(np.where(np.isfinite(B), B, 0))
    assert np.all(np.abs(got - ref)[ok] <= 70 * 2.0 ** -51 * scale[ok] + 1e-300)


@pytest.mark.parametrize("n,m", [(1, 5), (32, 31), (33, 33), (64, 129), (97, 300), (129, 20000), (161, 40001)])
def test_solve_is_backward_stable(P, n, m):
    """L X = R to a few units of the rows' products, as forward substitution gives it: n 2^-52
    |L| |X|, whatever the columns' scales."""
    import torch
    rng = np.random.default_rng(n + m)
    L = np.tril(rng.standard_normal((n, n))) + 4.0 * np.sqrt(n) * np.eye(n)
    R = rng.standard_normal((n, m)) * np.exp(rng.uniform(-20, 20, (1, m)))
    X = P.ri_solve(torch.tensor(L, device="cuda"), torch.tensor(R, device="cuda")).cpu().numpy()
    res = np.abs((L.astype(np.longdouble) @ X.astype(np.longdouble) - R).astype(np.float64)) if n * m < 1e5 else np.abs(L @ X - R)
    assert np.all(res <= (n + 4) * 2.0 ** -52 * (np.abs(L) @ np.abs(X) + np.abs(R)))


@pytest.mark.parametrize("n", [1, 3, 4, 31, 32, 33, 63, 64, 65, 97, 300, 693])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 1000, 2.0 ** -1000])
def test_factor_residual(P, n, scale):
    """|A - L L^T| <= gamma |L| |L|^T: a column sum has at most n products and a subtraction, the reciprocal
    pivot and its use three more roundings, the diagonal's root one."""
    import torch
    rng = np.random.default_rng(n)
    X = rng.standard_normal((n, n + 2)) * np.exp(rng.uniform(-2, 2, (n, 1)))
    A = (X @ X.T + 1e-3 * np.eye(n)) * scale
    A = np.tril(A) + np.tril(A, -1).T
    L, info = P.ri_factor(torch.tensor(A, device="cuda"))
    L = L.cpu().numpy()
    assert int(info.item() if hasattr(info, "item") else info) == 0
    assert np.array_equal(L, np.tril(L)) and np.all(np.diag(L) > 0)
    Ll = (L / np.sqrt(scale)).astype(np.longdouble)
    err = np.abs(Ll @ Ll.T - (A / scale).astype(np.longdouble))
    assert np.all(err <= (n + 8) * 2.0 ** -53 * (np.abs(Ll) @ np.abs(Ll).T))


@pytest.mark.parametrize("n,bad", [(1, 0), (40, 35), (65, 64), (97, 31)])
def test_factor_names_the_first_bad_pivot(P, n, bad):
    import torch
    A = np.eye(n) + 0.01
    A[bad, bad] = -1.0
    _, info = P.ri_factor(torch.tensor(A, device="cuda"))
    assert int(info.item() if hasattr(info, "item") else info) == bad + 1
