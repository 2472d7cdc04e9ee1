"""GPU test of the QR panel where a reflector's scale lies near the ends of the range
(v is formed before the update there) and inside it, and mixed within one panel: the
stable X of A D is D's rescaling of A's.
"""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k", [(300, 80, 33), (65, 40, 40), (1500, 64, 2)])
@pytest.mark.parametrize("exponents", [(0,), (293, 295, 297, 299), (-302, -304, -306, -308), (-450, 0, 450)])
def test_stable_x_of_scaled_columns(m, n, k, exponents):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_09417_gb300 import build
    build.build()
    from paper_2310_09417_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(m + k)
    A = torch.randn(n, m, generator=g, device="cuda", dtype=torch.float64)
    e = torch.tensor([exponents[i % len(exponents)] for i in range(n)], device="cuda", dtype=torch.float64)
    J = torch.arange(k, device="cuda")
    C = A[:k].t()
    Q, R = torch.linalg.qr(C)
    ref = torch.linalg.solve_triangular(R, Q.t() @ A.t(), upper=True)
    got = B.stable_x((A * torch.exp2(e)[:, None]).t(), J)
    got = got * torch.exp2(e[:k])[:, None]  # exact: powers of two
    got = got / torch.exp2(e)[None, :]
    cond = float(torch.linalg.cond(C))
    # two orthogonal reductions of length m and a triangular solve, each within a small
    # multiple of m^(1/2) k 2^-53 of the scaled columns, amplified by cond(C)
    tol = 8.0 * cond * k * m ** 0.5 * 2.0 ** -53
    assert float(torch.linalg.norm(got - ref)) <= tol * float(torch.linalg.norm(ref))
