"""What the tensor cores truncate from a sum must not grow with its length: a
long product, summed in parts of at most 16 blocks of 64 terms, is as accurate as
one of 1024 terms.

Operands of one sign that bf16 holds exactly, and real, so that nothing but the
truncation of the running sum is left: it is one-sided and proportional to the
number of additions to one accumulator (64 for 1024 terms).  A quarter more is
allowed for the parts' own sum in float32 (at most 16 additions, rounded)."""
import ctypes

import pytest

pytestmark = pytest.mark.gpu


def error(torch, planes, m, n, k):
    from paper_2306_09257_gb300 import apf, build
    build.build_lib()
    L = apf.load_library()
    f = ctypes.c_void_p
    L.apf_debug_cgemm.argtypes = [f, ctypes.c_int, ctypes.c_int, ctypes.c_int] + [f] * 6 + [ctypes.c_int]
    g = torch.Generator(device="cuda").manual_seed(k)
    A = (0.5 + 0.5 * torch.rand(m, k, device="cuda", generator=g)).bfloat16().float()
    B = (0.5 + 0.5 * torch.rand(k, n, device="cuda", generator=g)).bfloat16().float()
    Z = [torch.zeros_like(A), torch.zeros_like(B)]
    C = [torch.empty(m, n, device="cuda") for _ in range(2)]
    s = apf.Solver(0, "mixed")
    rc = L.apf_debug_cgemm(s._h, m, n, k, *[t.data_ptr() for t in (A, Z[0], B, Z[1], *C)], planes)
    assert rc == 0, L.apf_last_error(s._h)
    ref = A.double() @ B.double()
    assert C[1].abs().max().item() == 0.0
    return (torch.linalg.norm(C[0].double() - ref) / torch.linalg.norm(ref)).item()


@pytest.mark.parametrize("planes", [2, 3])
@pytest.mark.parametrize("m,n,k", [(256, 256, 4096), (300, 250, 8192), (129, 128, 2080)])
def test_as_accurate_as_a_short_one(planes, m, n, k):
    torch = pytest.importorskip("torch")
    assert error(torch, planes, m, n, k) <= 1.25 * error(torch, planes, m, n, 1024)
