"""GPU tests of the LUPP panel at the sizes where its blocks change shape: more rows
per block than threads, rows that no longer fit in shared memory, one block, and
panels narrower than a warp.

With Omega = I the sketch is Y = A, so J must be the oracle's LUPP of A^T; every
pivot is chosen among candidates of all blocks.
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


@pytest.mark.parametrize("k,n", [
    (6, 45001),    # about 300 rows per block: a thread holds two rows
    (64, 65003),   # FP64 rows of a block exceed shared memory
    (33, 20),      # fewer columns than the sketch has rows: one block
    (128, 700),    # the widest panel
    (2, 40),
])
def test_pivots_match_the_oracle(B, orc, k, n):
    rng = np.random.default_rng(k + n)
    A = rng.standard_normal((k, n))
    r = min(k, n)
    g = B.id_fixed_rank(dev_cm(A, torch.float64), r, k, block=min(k, 128), omega=dev(np.eye(k), torch.float64))
    o = orc.id_fixed_rank(A, np.eye(k), r)
    assert np.array_equal(g.J.cpu().numpy(), o["J"])


@pytest.mark.parametrize("dtype", [torch.float64, torch.float32])
def test_equal_candidates_of_one_block_go_to_the_smallest_column(B, dtype):
    # |A(0, :)| is 1 everywhere but at two columns whose rows lie in one block, the later
    # one held by a thread with a lower number than the earlier one's
    n, k = 45001, 2
    A = np.ones((k, n))
    A[1] = np.arange(n) / n
    A[0, [7, 258]] = 2.0, -2.0
    g = B.id_fixed_rank(dev_cm(A, dtype), k, k, omega=dev(np.eye(k), dtype))
    assert int(g.J[0]) == 7
