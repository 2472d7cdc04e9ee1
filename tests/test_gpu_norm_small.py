"""GPU test of ||A||_F of FP32 matrices whose squares lie so low that a square's rounding
error has bits below the smallest FP32 number, alone and beside larger entries.
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


def matrix(m, n, exps):
    # one value repeated (its square's error would add up) times powers of two
    g = torch.Generator(device="cuda").manual_seed(m + n)
    e = torch.tensor(exps, device="cuda")[torch.randint(0, len(exps), (n, m), generator=g, device="cuda")]
    return torch.ldexp(torch.full((n, m), 1.0 + 2.0 ** -12 + 2.0 ** -23, device="cuda"), e).t()


EXPS = [(-49,), (-50,), (-51,), (-52,), (-55,), (-58,), (-62,), (-63,), (-64,), (-70,), (-51, -62, -75, -130),
        (-52, -53), (0, -60), (-49, -58), (53, -60), (54, 53)]


@pytest.mark.parametrize("exps", EXPS, ids=str)
@pytest.mark.parametrize("m,n", [(4099, 33), (127, 9)])
def test_norm_of_one_matrix(B, m, n, exps):
    A = matrix(m, n, exps)
    ref = float(torch.linalg.norm(A.double() * 2.0 ** 60)) * 2.0 ** -60
    for sp in (None, B.F32_EMU):
        got = B.id_fixed_rank(A, 2, 4, seed=3, sketch_prec=sp).norm_A
        # at most about 70 squares per thread and two tree sums: below 100 * 2^-53 on either side
        assert abs(got - ref) <= 1e-13 * ref


@pytest.mark.parametrize("exps", EXPS, ids=str)
def test_norm_in_a_batch(B, exps):
    As = [matrix(m, n, exps) for m, n in ((300, 40), (65, 33), (1000, 7))]
    for A, r in zip(As, B.id_batched(As, 0.5, block=8, seed=1)):
        ref = float(torch.linalg.norm(A.double() * 2.0 ** 60)) * 2.0 ** -60
        # groups of 64 squares, each to 2^-45 relative, and sums of a few hundred groups in FP64
        assert abs(r.norm_A - ref) <= 1e-13 * ref
