"""GPU tests of what follows the pivots of one block: the quotients by the pivot (a
reciprocal and two FMAs, or a division at the ends of the exponent range) and the new
block of the interpolation matrix at the edges of its kernels' tiles.
"""
import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

from test_gpu_parity import dev, dev_cm  # noqa: E402


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_09417_gb300 import build
    build.build()
    from paper_2310_09417_gb300 import binding
    binding.load()
    return binding


@pytest.mark.parametrize("e", [-700, -499, 499, 700])
def test_quotients_do_not_depend_on_the_scale(B, e):
    # a power of two changes no bit of the factorisation, but the ends of the exponent
    # range take the division where the middle takes the reciprocal
    rng = np.random.default_rng(4)
    k, n = 64, 3001
    A = rng.standard_normal((k, n))
    A[:, ::7] *= 2.0 ** -30
    Om = dev(np.eye(k), torch.float64)
    a = B.id_fixed_rank(dev_cm(A, torch.float64), k, k, omega=Om)
    b = B.id_fixed_rank(dev_cm(A * 2.0 ** e, torch.float64), k, k, omega=Om)
    assert torch.equal(a.J, b.J)
    assert torch.equal(a.X, b.X)


# FP64: groups of one, two and four columns (by the number of rows); FP32: 32 rows a CTA,
# two columns a lane
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
@pytest.mark.parametrize("n", [70, 129, 1300, 2500, 5000])
@pytest.mark.parametrize("k,block", [(1, 1), (5, 5), (33, 33), (64, 64), (66, 64), (65, 128)])
def test_interpolation_of_one_block(B, dtype, n, k, block):
    rng = np.random.default_rng(n + k)
    A = rng.standard_normal((max(k, 2), n)).astype(np.float32).astype(np.float64)
    Om = np.eye(max(k, 2))
    g = B.id_fixed_rank(dev_cm(A, dtype), k, max(k, 2), block=block, omega=dev(Om, dtype))
    J = g.J.cpu().numpy()
    C = A[:k, J]
    ref = np.linalg.solve(C, A[:k])
    eps = 2.0 ** -53 if dtype == torch.float64 else 2.0 ** -24
    # LU with partial pivoting: a small multiple of k eps cond(C), normwise
    tol = 16.0 * k * eps * np.linalg.cond(C)
    assert np.linalg.norm(g.X.double().cpu().numpy() - ref) <= tol * np.linalg.norm(ref)
