"""GPU test of the FP64 product kernel at the edges of its 32 x 32 tiles, 16-deep
steps and split-K partials: the plain FP64 sketch against FP64 torch.
"""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m", [1, 15, 17, 64, 333, 5001])
@pytest.mark.parametrize("n,rows", [(1, 1), (31, 33), (32, 32), (33, 31), (97, 64), (1000, 7)])
def test_sketch(m, n, rows):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_09417_gb300 import build
    build.build()
    from paper_2310_09417_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(m + n + rows)
    A = torch.randn(n, m, generator=g, device="cuda", dtype=torch.float64).t()
    Om = torch.randn(rows, m, generator=g, device="cuda", dtype=torch.float64)
    G = B.id_sketch(A, Om)
    ref = (Om @ A).t()
    bound = 2.0 * m * 2.0 ** -53 * (Om.abs() @ A.abs()).t()  # each side's rounding
    assert bool(((G - ref).abs() <= bound).all())
