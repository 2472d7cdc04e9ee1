"""id_fixed_rank_noalloc just under its buffer's size: problems whose matrices take nearly
64 MiB fit beside the words that the panel's blocks exchange, and give what the call with
a workspace gives.  The file is named to be collected last."""
import ctypes

import pytest

torch = pytest.importorskip("torch")

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("prec", ["f32emu", "fp8"])
def test_largest_problems(prec):
    if not torch.cuda.is_available():
        pytest.skip("no CUDA device")
    from paper_2310_09417_gb300 import build
    build.build()
    from paper_2310_09417_gb300 import binding as B
    f = B.load().id_fixed_rank_noalloc
    f.argtypes = [ctypes.c_void_p, ctypes.c_int64, ctypes.c_int64, ctypes.c_void_p, ctypes.c_void_p, ctypes.c_void_p]
    f.restype = ctypes.c_int
    size, l, block = (2000, 120, 128) if prec == "f32emu" else (2200, 200, 32)
    k = 100
    g = torch.Generator(device="cuda").manual_seed(7)
    A = torch.randn(size, size, generator=g, device="cuda").t()
    sp = B.F32_EMU if prec == "f32emu" else None
    if prec == "fp8":
        A = B.quantize_fp8(B.colmajor_padded(A.to(torch.bfloat16), 8))
    ref = B.id_fixed_rank(A, k, l, block=block, seed=3, sketch_prec=sp)
    opts = B._opts(A, block=block, tol=0.0, relative=False, k_max=k, k0=0, blocks_per_pass=1, seed=3, omega=None,
                   profile=False, sketch_prec=sp)
    assert B.workspace_size(A, opts, l) > (64 << 20) - (1 << 20)
    J = torch.full((k,), -1, dtype=torch.int64, device="cuda")
    Xb = torch.zeros((size, k), dtype=torch.float32, device="cuda")
    res = B.IdResult()
    res.J, res.X, res.ldx = J.data_ptr(), Xb.data_ptr(), k
    rc = f(ctypes.byref(B._matrix(A)), k, l, ctypes.byref(opts), ctypes.byref(res),
           torch.cuda.current_stream().cuda_stream)
    assert rc == B.OK, B.status_string(rc)
    assert torch.equal(J, ref.J) and torch.equal(Xb.t(), ref.X)
