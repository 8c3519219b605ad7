"""psq_ri_solve where it changes from the tensor-core kernel to two FP64 launches per block (few columns, many
aux functions), on both sides of the line."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,m", [(1, 1), (16, 3000), (17, 256), (17, 257), (32, 30000), (512, 2), (545, 2), (673, 1), (700, 63), (700, 65), (700, 400), (1025, 257), (1500, 3), (1500, 1400), (2001, 64)])
@pytest.mark.parametrize("span", [0.0, 20.0])
def test_solve_is_backward_stable(n, m, span):
    """L X = R to a few units of the rows' products, as forward substitution gives it."""
    import torch
    assert torch.cuda.is_available(), "the CUDA path needs a GPU"
    import paper_2510_15204_gb300 as P
    rng = np.random.default_rng(n + m)
    d = 2.0 ** rng.uniform(-span, span, n)
    L = (np.tril(rng.standard_normal((n, n))) + 4.0 * np.sqrt(n) * np.eye(n)) * d[:, None] / d[None, :]
    R = rng.standard_normal((n, m)) * d[:, None] * np.exp(rng.uniform(-20, 20, (1, m)))
    X = P.ri_solve(torch.tensor(L, device="cuda"), torch.tensor(R, device="cuda"))
    Lt, Rt = torch.tensor(L, device="cuda"), torch.tensor(R, device="cuda")
    # (residual in FP64: its own rounding, at most (n + 2) 2^-53 of the same terms, is in the bound)
    res = (Lt @ X - Rt).abs()
    terms = Lt.abs() @ X.abs() + Rt.abs()
    assert bool((res <= (n + 4) * 2.0 ** -52 * terms + (n + 2) * 2.0 ** -53 * terms).all())
