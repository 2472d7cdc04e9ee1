"""GPU tests of the adaptive loop where it is launched one round ahead of its stop test:
stops at every distance from the rank cap and from n, against the loop that waits for
every round (profile=True), and a non-finite A found with a round queued behind it.
"""
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu

BLOCK = 32
TYPE = {"f64": torch.float64, "f64emu": torch.float64, "f32": torch.float32, "f32emu": torch.float32,
        "bf16": torch.bfloat16}
TOL = {"f64": 1e-8, "f64emu": 1e-8, "f32": 1e-3, "f32emu": 1e-3, "bf16": 1e-1}


@pytest.fixture(scope="module")
def B():
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_09417_gb300 import build
    build.build()
    from paper_2310_09417_gb300 import binding
    binding.load()
    return binding


def low_rank(prec, m, n, r):
    g = torch.Generator(device="cuda").manual_seed(1000 * r + n)
    At = torch.randn(n, r, generator=g, device="cuda", dtype=torch.float64) @ torch.randn(
        r, m, generator=g, device="cuda", dtype=torch.float64)
    return At.to(TYPE[prec]).t()


def call(B, prec, A, **kw):
    sp = {"f64emu": B.F64_EMU, "f32emu": B.F32_EMU}.get(prec)
    return B.id_adaptive(A, TOL[prec], block=BLOCK, seed=5, sketch_prec=sp, **kw)


def assert_same(a, b):
    assert (a.k, a.status, a.rounds, a.passes) == (b.k, b.status, b.rounds, b.passes)
    assert (a.est_err, a.norm_A, list(a.trace)) == (b.est_err, b.norm_A, list(b.trace))
    assert torch.equal(a.J, b.J) and torch.equal(a.X, b.X)


# blocks of the matrix's rank, of the cap (0: none), and n: a stop one round before the cap
# (at the first and at a later test), two before it, at it, the cap without a stop; a stop
# in the round before n, at n, and n reached without one
@pytest.mark.parametrize("rank,cap,n", [(1, 2, 300), (2, 3, 300), (4, 5, 300), (1, 3, 300), (3, 3, 300), (4, 3, 300),
                                        (1, 1, 300), (2, 0, 96), (1, 0, 96), (3, 0, 96), (2, 0, 80), (1, 0, 33),
                                        (1, 0, 32), (1, 0, 20)])
@pytest.mark.parametrize("per_pass", [0, 1, 3])
@pytest.mark.parametrize("prec", list(TYPE))
def test_same_as_the_loop_that_waits(B, prec, per_pass, rank, cap, n):
    A = low_rank(prec, 400, n, min(rank * BLOCK, n))
    kw = dict(k_max=cap * BLOCK or None, blocks_per_pass=per_pass)
    assert_same(call(B, prec, A, **kw), call(B, prec, A, profile=True, **kw))


# the FP64 re-solve works through the list of columns outside the skeleton
@pytest.mark.parametrize("rank,cap", [(1, 2), (2, 3), (1, 3), (3, 3), (4, 3)])
def test_resolved_columns(B, rank, cap):
    A = low_rank("f32", 400, 300, rank * BLOCK)
    a = call(B, "f32", A, k_max=cap * BLOCK, x_solve_f64=2)
    assert_same(a, call(B, "f32", A, k_max=cap * BLOCK, x_solve_f64=2, profile=True))
    if rank < cap:  # a larger cap changes nothing
        assert_same(a, call(B, "f32", A, k_max=(cap + 3) * BLOCK, x_solve_f64=2))


@pytest.mark.parametrize("bad", [float("nan"), float("inf")])
@pytest.mark.parametrize("cap", [0, 1, 2])
@pytest.mark.parametrize("prec", list(TYPE))
def test_nonfinite_with_rounds_queued(B, prec, cap, bad):
    A = low_rank(prec, 400, 300, 4 * BLOCK)
    before = call(B, prec, A, k_max=cap * BLOCK or None)
    hurt = A.t().clone().t()
    hurt[17, 250] = bad
    for kw in ({}, {"x_solve_f64": 1}):
        with pytest.raises(B.IDError) as e:
            call(B, prec, hurt, k_max=cap * BLOCK or None, **kw)
        assert e.value.code == B.ERR_NONFINITE
    assert_same(before, call(B, prec, A, k_max=cap * BLOCK or None))
