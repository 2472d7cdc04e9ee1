"""GPU test of the stable X and the CUR middle factor of a matrix whose rows are in two
units: a block of X must be as accurate as its own rows allow, whatever the other unit.
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


def graded(m, n, k, unit):
    """A = C X with C = diag(C1, unit C2) its first k columns; the scaled blocks and X."""
    g = torch.Generator(device="cuda").manual_seed(m + n + k)

    def randn(*s):
        return torch.randn(*s, generator=g, device="cuda", dtype=torch.float64)
    m1, k1 = m // 2, k // 2
    C1, C2 = randn(m1, k1), randn(m - m1, k - k1)
    C = torch.block_diag(C1, C2)
    X = torch.cat([torch.eye(k, device="cuda", dtype=torch.float64), randn(k, n - k)], 1)
    A = C @ X
    A[m1:] *= unit  # a power of two
    return A.t().contiguous().t(), X, (C1, C2)


def parts(M, k):
    return M[:k // 2], M[k // 2:]


# forming A rounds each entry by at most about k 2^-53 of |C||X|, and the QR and the product
# add a small multiple of m^(1/2) k 2^-53, all relative to the rows' own unit and amplified
# by the block's condition
def bound(m, k, C):
    return 8.0 * float(torch.linalg.cond(C)) * k * m ** 0.5 * 2.0 ** -53


@pytest.mark.parametrize("unit", [2.0 ** 13, 2.0 ** 27, 2.0 ** 40])
@pytest.mark.parametrize("m,n,k", [(4000, 500, 16), (1001, 999, 34), (260, 90, 12)])
def test_stable_x(B, m, n, k, unit):
    A, X, Cs = graded(m, n, k, unit)
    got = B.stable_x(A, torch.arange(k, device="cuda"))
    for g, x, C in zip(parts(got, k), parts(X, k), Cs):
        assert float(torch.linalg.norm(g - x)) <= bound(m, k, C) * float(torch.linalg.norm(x))


@pytest.mark.parametrize("unit", [2.0 ** 13, 2.0 ** 40])
@pytest.mark.parametrize("m,n,k", [(4000, 500, 16), (1001, 999, 34)])
def test_cur_middle(B, m, n, k, unit):
    # R = [A(first rows of each unit)] = diag(C1(:k/2), unit C2(:k/2)) X, so
    # C^+ A R^+ = diag(C1(:k/2)^-1, C2(:k/2)^-1 / unit): graded by columns, compared by columns
    A, X, (C1, C2) = graded(m, n, k, unit)
    h, m1 = k // 2, m // 2
    Iq = torch.cat([torch.arange(h, device="cuda"), m1 + torch.arange(k - h, device="cuda")])
    U = B.cur_middle(A, Iq, torch.arange(k, device="cuda"), B.CUR_PSEUDOINVERSE)
    ref = torch.block_diag(torch.linalg.inv(C1[:h]), torch.linalg.inv(C2[:k - h]) / unit)
    amp = float(torch.linalg.cond(C1[:h])) * float(torch.linalg.cond(C2[:k - h]))
    # the first unit's rows of U against its own columns; R's rows in two units and its QR
    # bring in cond(R's blocks) in place of one unit's alone
    err = float(torch.linalg.norm(U[:h, :h] - ref[:h, :h]))
    assert err <= 8.0 * amp * bound(m, k, C1) * float(torch.linalg.norm(ref[:h, :h]))


def test_workspace_does_not_grow_with_a(B):
    import ctypes as C
    for m, n, k in ((4000, 2000, 96), (40000, 10000, 64)):
        A = torch.empty(1, device="cuda", dtype=torch.float64).expand(n, m).t()
        mat = B.IdMatrix(A.data_ptr(), B.F64, m, n, m, None)
        nb = C.c_size_t(0)
        for name, args in (("id_stable_x_workspace_size", (k,)), ("cur_middle_workspace_size", (k, 0))):
            assert getattr(B.load(), name)(C.byref(mat), *args, C.byref(nb)) == 0
            # panels, Q, M, X and their split sums: a few hundred doubles per row and column of A at most
            assert nb.value <= 8 * 64 * (m + n) * k + (64 << 20), (name, m, n, k, nb.value)
