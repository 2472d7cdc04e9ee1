"""GPU test of the triangular solve of the stable X: the inverse of R's diagonal blocks
divides by the diagonal, once and rounded once.
"""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


# 1/d rounded, times d, is not 1 for these
@pytest.mark.parametrize("d", [49.0, 98.0, 103.0, 187.0, -49.0, 49.0 * 2.0 ** 500, 49.0 * 2.0 ** -500])
@pytest.mark.parametrize("at,k", [(0, 2), (30, 40), (31, 64), (62, 64), (64, 80)])
def test_quotients_are_rounded_once(d, at, k):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_09417_gb300 import build
    build.build()
    from paper_2310_09417_gb300 import binding as B
    # C = R is upper triangular already: its reflectors are the identity, Q^T A = A, and
    # X(:, k) = R^{-1} e is column at + 1 of the inverse, whose entry `at` is -d / d
    R = torch.eye(k, dtype=torch.float64)
    R[at, at] = R[at, at + 1] = d
    A = torch.cat([R, torch.zeros(k, 3, dtype=torch.float64)], 1)
    A[at + 1, k] = 1.0
    X = B.stable_x(A.cuda().t().contiguous().t(), torch.arange(k, device="cuda")).cpu()
    assert float(X[at, k]) == -1.0
