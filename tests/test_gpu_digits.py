"""GPU test of the digit slicing of the tensor-core paths at its edges: rounding
ties, carries through every digit, entries far below their column's largest, the
ends of the exponent range, subnormals and zeros.  With rows of the identity as
Omega the sketch returns what the digits hold, F 2^(e - w) with F the entry rounded
to w = 55 (FP64) or 23 (FP32) bits below 2^e, e the column's exponent: exact.
"""
import math
from fractions import Fraction

import numpy as np
import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


def columns(single):
    rng = np.random.default_rng(8)
    p, lo, top, w = (24, -149, 127, 23) if single else (53, -1074, 1023, 55)
    m = 96
    out = []
    for e in (0, 1, -37, top, lo + p, lo + 3):  # the column's largest entry is in [2^e, 2^(e+1))
        frac = 1.0 + rng.integers(0, 2 ** (p - 1), m) / 2.0 ** (p - 1)
        drop = np.minimum(rng.integers(0, w + 6, m), e - lo)
        drop[0] = 0
        v = np.ldexp(frac, (e - drop).astype(int))
        # ties and runs of ones: an odd multiple of half the digits' unit, 2^d - unit
        u = math.ldexp(1.0, max(e + 1 - w - 1, lo))
        v[1:9] = [u, 3 * u, 5 * u, 7 * u, 255 * u, 257 * u, 127 * u, 129 * u]
        v[9] = math.ldexp(2.0 - 2.0 ** (1 - p), e) if e >= lo + p else v[0]  # all ones
        v[10:12] = 0.0
        v *= rng.choice([-1.0, 1.0], m)
        out.append(v.astype(np.float32) if single else v)
    out.append(np.zeros(m, out[0].dtype))
    return np.stack(out, axis=1)


def held(x, e, w):
    if x == 0.0:
        return 0.0
    q = Fraction(float(x)) * (Fraction(2) ** (w - e))
    return math.ldexp(float(round(q)), e - w)  # round: to even


@pytest.mark.parametrize("single", [False, True])
@pytest.mark.parametrize("rows", [1, 96])
def test_digits_hold_the_rounded_entry(single, rows):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_09417_gb300 import build
    build.build()
    from paper_2310_09417_gb300 import binding as B
    A = columns(single)
    m, n = A.shape
    w = 23 if single else 55
    Om = np.eye(m, dtype=A.dtype)[:rows]
    Ad = torch.from_numpy(np.ascontiguousarray(A.T)).cuda().t()
    G = B.id_sketch(Ad, torch.from_numpy(Om).cuda(), sketch_prec=B.F32_EMU if single else B.F64_EMU).cpu().numpy()
    ref = np.zeros((n, rows), A.dtype)
    for j in range(n):
        amax = float(np.abs(A[:, j]).max())
        e = math.frexp(amax)[1] if amax else 0
        with np.errstate(over="ignore"):  # an entry that rounds up to the end of the FP32 range
            ref[j] = [held(A[r, j], e, w) for r in range(rows)]
    np.testing.assert_array_equal(G, ref)
