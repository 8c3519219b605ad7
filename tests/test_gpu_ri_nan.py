"""NaN of any bit pattern reaches the results of the exact-digit products (psq_ri_eri, psq_ri_solve) as
it does in FP64 arithmetic: numpy's own, the one an FP32 NaN of the GPU widens to, and memory filled
with ones."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

PATTERNS = [0x7FF8000000000000, 0x7FF0000000000001, 0x7FFFFFFFE0000000, 0x7FFFDFC000000000, 0xFFFFFFFFFFFFFFFF]


def _nan(bits):
    return np.array([bits], dtype=np.uint64).view(np.float64)[0]


def _cuda(x):
    """To the device bit by bit (a copy, no arithmetic)."""
    import torch
    return torch.from_numpy(np.ascontiguousarray(x)).cuda()


@pytest.mark.parametrize("bits", PATTERNS)
def test_eri_nan_patterns(bits):
    import torch
    assert torch.cuda.is_available(), "the CUDA path needs a GPU"
    import paper_2510_15204_gb300 as P
    rng = np.random.default_rng(1)
    B = rng.standard_normal((70, 40))
    B[3, 5] = B[66, 30] = _nan(bits)
    got = P.ri_eri(_cuda(B), 0, 40, 0, 40).cpu().numpy()
    want = np.zeros((40, 40), dtype=bool)
    want[[5, 30], :] = True
    want[:, [5, 30]] = True
    assert np.array_equal(np.isnan(got), want)


@pytest.mark.parametrize("bits", PATTERNS)
def test_solve_nan_patterns(bits):
    """n = 70: rows 32 .. 69 take sums of digit products over the rows above them."""
    import torch
    import paper_2510_15204_gb300 as P
    rng = np.random.default_rng(2)
    n, m = 70, 40
    L = np.tril(rng.standard_normal((n, n))) + 20.0 * np.eye(n)
    R = rng.standard_normal((n, m))
    bad = R.copy()
    bad[3, 5] = _nan(bits)  # a right-hand side: its column from row 3 on
    X = P.ri_solve(_cuda(L), _cuda(bad)).cpu().numpy()
    want = np.zeros((n, m), dtype=bool)
    want[3:, 5] = True
    assert np.array_equal(np.isnan(X), want)
    bad = L.copy()
    bad[66, 3] = _nan(bits)  # an element of L: row 66 and what follows from it
    X = P.ri_solve(_cuda(bad), _cuda(R)).cpu().numpy()
    want = np.zeros((n, m), dtype=bool)
    want[66:, :] = True
    assert np.array_equal(np.isnan(X), want)
