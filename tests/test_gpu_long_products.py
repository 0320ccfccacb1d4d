"""Products whose sums the pair tiles add up in several passes (more than 2048
terms), with ragged rows, columns and last passes, against float64.

Tolerance (relative Frobenius): two bf16 planes leave x1 y1 and the third planes,
2^-16 of a term each; the tensor cores truncate at most 2 x 2048 / 16 additions
of a pass, 2^-24 each, one-sided: 1.5e-5 + 1.5e-5, rounded up to 4e-5."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("m,n,k", [(129, 128, 2048), (300, 250, 2080), (256, 384, 4160), (130, 64, 6200)])
def test_against_float64(m, n, k):
    torch = pytest.importorskip("torch")
    from paper_2306_09257_gb300 import apf, build
    build.build_lib()
    L = apf.load_library()
    f = ctypes.c_void_p
    L.apf_debug_cgemm.argtypes = [f, ctypes.c_int, ctypes.c_int, ctypes.c_int] + [f] * 6 + [ctypes.c_int]
    g = torch.Generator(device="cuda").manual_seed(m + n + k)
    A = torch.randn(m, k, dtype=torch.complex64, device="cuda", generator=g)
    B = torch.randn(k, n, dtype=torch.complex64, device="cuda", generator=g)
    p = [t.contiguous() for z in (A, B) for t in (z.real, z.imag)]
    C = [torch.empty(m, n, device="cuda") for _ in range(2)]
    s = apf.Solver(0, "mixed")
    rc = L.apf_debug_cgemm(s._h, m, n, k, *[t.data_ptr() for t in p + C], 2)
    assert rc == 0, L.apf_last_error(s._h)
    ref = A.to(torch.complex128) @ B.to(torch.complex128)
    got = C[0].double() + 1j * C[1].double()
    assert (torch.linalg.norm(got - ref) / torch.linalg.norm(ref)).item() < 4e-5
