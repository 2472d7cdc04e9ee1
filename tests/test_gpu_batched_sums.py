"""GPU test that a batch's norms and error estimates are the same bits whatever tile height
the batched kernel runs with (the tuner picks it by time), and near the 64-bit values.
"""
import os

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

SIZES = [(700, 300), (65, 33), (33, 129), (1, 40), (40, 1), (513, 127), (90, 4001), (257, 64), (8, 8), (3000, 128)]


@pytest.mark.parametrize("block", [5, 16, 32])
@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_same_bits_with_every_tile(dtype, block):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_09417_gb300 import build
    build.build()
    from paper_2310_09417_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(block)
    As = []
    for m, n in SIZES:
        r = min(m, n, 20)
        At = torch.randn(n, r, generator=g, device="cuda", dtype=torch.float64) @ torch.randn(
            r, m, generator=g, device="cuda", dtype=torch.float64)
        At += 1e-3 * torch.randn(n, m, generator=g, device="cuda", dtype=torch.float64)
        At = torch.nn.functional.pad(At, (0, 1 if n == 1 or m == 1 else 0)).to(dtype)  # a stride of its own
        As.append(At.t()[:m])
    want = None
    try:
        for cfg in ("32x1", "32x2", "64x1", "64x2") + (("128x1", "128x2") if dtype == torch.float32 else ()):
            os.environ["RANDID_BATCHED_CONFIG"] = cfg
            got = [(r.norm_A, r.est_err, r.k, r.status) for r in B.id_batched(As, 1e-2, block=block, seed=3, k_max=60)]
            want = want or got
            assert got == want, cfg
    finally:
        os.environ.pop("RANDID_BATCHED_CONFIG", None)
    for A, (norm, est, k, status) in zip(As, want):
        ref = float(torch.linalg.norm(A.double()))
        # 2048 sums of at most a few hundred squares, then a tree
        assert abs(norm - ref) <= 1e-13 * ref
