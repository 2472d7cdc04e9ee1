"""GPU tests of ||A||_F and the finiteness check at the edges of the norm kernels:
odd sizes, columns off 16-byte boundaries, zeros, magnitudes whose squares leave the
FP32 range, and a single NaN or Inf anywhere.
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


PREC = {"f64": torch.float64, "f64emu": torch.float64, "f32": torch.float32, "bf16": torch.bfloat16,
        "fp8": torch.bfloat16}


def matrix(prec, m, n, kind):
    g = torch.Generator(device="cuda").manual_seed(m * 7 + n)
    x = torch.randn(n, m, generator=g, device="cuda", dtype=torch.float64)
    if kind == "zeros":
        x[:, ::3] = 0.0
        x[n // 2] = 0.0
    elif kind == "wide" and prec != "fp8":  # squares below and above the normal FP32 range
        x *= torch.tensor([1e-30, 1.0, 1e25, 1e-3], device="cuda", dtype=torch.float64)[
            torch.randint(0, 4, (n, m), generator=g, device="cuda")]
    ld = -(-m // 8) * 8 if prec in ("bf16", "fp8") else m
    At = torch.zeros((n, ld), dtype=PREC[prec], device="cuda")
    At[:, :m] = x.to(PREC[prec])
    return At[:, :m].t()


def call(B, prec, A, k=2, l=4):
    sp = {"f64emu": B.F64_EMU}.get(prec)
    return B.id_fixed_rank(B.quantize_fp8(A) if prec == "fp8" else A, k, l, seed=3, sketch_prec=sp)


@pytest.mark.parametrize("kind", ["plain", "zeros", "wide"])
@pytest.mark.parametrize("m,n", [(5, 9), (127, 33), (4099, 65), (20003, 7), (33000, 311)])
@pytest.mark.parametrize("prec", list(PREC))
def test_norm(B, prec, m, n, kind):
    A = matrix(prec, m, n, kind)
    g = call(B, prec, A)
    if prec == "fp8":
        q = B.quantize_fp8(A)
        A = q.data.float().double() * q.scale.double().repeat_interleave(128, 0)[:m]
    x = A.double().abs()
    s = float(x.max())
    ref = s * float(torch.linalg.norm(x / s))
    # at most about 70 squares per thread and two tree sums: below 100 * 2^-53 on either side
    assert abs(g.norm_A - ref) <= 1e-13 * ref


@pytest.mark.parametrize("bad", [float("nan"), float("inf"), -float("inf")])
@pytest.mark.parametrize("at", [0, 1, 4098, 4095])
@pytest.mark.parametrize("prec", ["f64", "f64emu", "f32", "bf16"])
def test_nonfinite_is_refused(B, prec, at, bad):
    A = matrix(prec, 4099, 5, "plain")
    A[at, 3] = bad
    with pytest.raises(B.IDError) as e:
        call(B, prec, A)
    assert e.value.code == -101
