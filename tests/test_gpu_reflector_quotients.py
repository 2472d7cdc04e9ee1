"""GPU test of the Householder reflector of the QR: tau and the scale of v are quotients
rounded once, so a column whose norm is a whole number gives the same bits as exact
arithmetic rounded at each step.
"""
from fractions import Fraction

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def expected(a, b, nrm):
    """X = R^{-1} Q^T c of the column c = (a, b), |c| = nrm, rounded step by step."""
    beta = -nrm if a >= 0 else nrm
    dx = beta - a
    tau, v = float(Fraction(dx, beta)), float(Fraction(b) * Fraction(float(Fraction(-1, dx))))
    q1 = float(1 - Fraction(tau))
    q2 = -float(Fraction(tau) * Fraction(v))
    m = float(Fraction(float(Fraction(q1) * a)) + Fraction(q2) * b)
    return float(Fraction(float(Fraction(1, beta))) * Fraction(m))


@pytest.mark.parametrize("e", [0, 280, -280, 310, -310])  # beyond 2^300: v is formed before the update
def test_whole_norms(e):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_09417_gb300 import build
    build.build()
    from paper_2310_09417_gb300 import binding as B
    J = torch.zeros(1, dtype=torch.int64, device="cuda")
    for p in range(2, 12):
        for q in range(1, p):
            for a, b in ((p * p - q * q, 2 * p * q), (2 * p * q, p * p - q * q), (q * q - p * p, 2 * p * q)):
                c = torch.tensor([[a, b]], dtype=torch.float64, device="cuda") * 2.0 ** e
                got = float(B.stable_x(c.t(), J)[0, 0])
                assert got == expected(a, b, p * p + q * q), (a, b)
