"""The waits without a counter or a barrier of one CTA: the LUPP panel's poll for the other
blocks' candidates and the mbarrier wait of a CTA pair.  Each gives up after its bounded
time (4 s), the call returns ID_ERR_TIMEOUT and the context stays usable.  No fault, trap
or unbounded wait is involved.  The file is named to be collected last."""
import time

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("which", [2, 3], ids=["panel_poll", "pair_mbarrier"])
def test_unsatisfied_wait_times_out_and_the_context_survives(which):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_09417_gb300 import build
    build.build()
    from paper_2310_09417_gb300 import binding as B
    g = torch.Generator(device="cuda").manual_seed(1)
    A = (torch.randn(200, 32, generator=g, device="cuda", dtype=torch.float64)
         @ torch.randn(32, 300, generator=g, device="cuda", dtype=torch.float64)).t()
    want = B.id_adaptive(A, 1e-8, block=16, seed=1)
    t0 = time.perf_counter()
    assert B.selftest_timeout(which) == B.ERR_TIMEOUT
    assert 3.0 < time.perf_counter() - t0 < 60.0
    got = B.id_adaptive(A, 1e-8, block=16, seed=1)
    assert got.status == B.OK and torch.equal(got.J, want.J) and torch.equal(got.X, want.X)
