"""GPU test of Q^T A on the tensor cores (stable X) at the line to the FP64 kernel and at
ragged sizes, and of its answer when A holds a NaN.
"""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_09417_gb300 import build
    build.build()
    from paper_2310_09417_gb300 import binding
    binding.load()
    return binding


def matrix(m, n, scale_columns):
    g = torch.Generator(device="cuda").manual_seed(m + n)
    A = torch.randn(n, m, generator=g, device="cuda", dtype=torch.float64)
    if scale_columns:  # columns from 1e-150 to 1e150: their exponents travel apart from the digits
        A *= (10.0 ** (torch.arange(n, device="cuda", dtype=torch.float64) * (300.0 / n) - 150.0))[:, None]
    return A.t()


# the tensor cores take k >= 16 with m n k >= 16e6
@pytest.mark.parametrize("m,n,k", [(4000, 2000, 15), (4000, 2000, 16), (1001, 999, 16), (1001, 999, 17),
                                   (4099, 129, 40), (300, 3001, 65), (129, 8000, 129)])
@pytest.mark.parametrize("scaled", [False, True])
def test_stable_x(B, m, n, k, scaled):
    A = matrix(m, n, scaled)
    g = torch.Generator(device="cuda").manual_seed(k)
    J = torch.randperm(n, generator=g, device="cuda")[:k]
    X = B.stable_x(A, J)
    s = A.abs().amax(0)  # compare per column, the skeleton's own scale divided out
    C = (A[:, J] / s[J]).contiguous()
    Q, R = torch.linalg.qr(C)
    ref = torch.linalg.solve_triangular(R, Q.t() @ (A / s), upper=True)
    got = X * s[J][:, None] / s[None, :]
    cond = float(torch.linalg.cond(C))
    # two orthogonal reductions of length m and a triangular solve, each within a small
    # multiple of m^(1/2) k 2^-53 of the scaled columns, amplified by cond(C)
    tol = 8.0 * cond * k * m ** 0.5 * 2.0 ** -53
    assert float(torch.linalg.norm(got - ref)) <= tol * float(torch.linalg.norm(ref))


def test_nan_stays_visible(B):
    A = matrix(4000, 500, False)
    J = torch.arange(32, device="cuda")
    A[17, 400] = float("nan")
    X = B.stable_x(A, J)
    assert bool(X[:, 400].isnan().all())
    assert bool(X[:, :400].isfinite().all()) and bool(X[:, 401:].isfinite().all())
