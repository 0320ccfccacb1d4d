"""The diagonal-block inverses (64 x 64 and 128 x 128) against float64."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def invert(torch, X):
    from paper_2306_09257_gb300 import apf, build
    build.build_lib()
    L = apf.load_library()
    f = ctypes.c_void_p
    L.apf_debug_inv32.argtypes = [f, ctypes.c_int, f, f, ctypes.c_int]
    n = X.shape[0]
    s = apf.Solver(0, "mixed")
    s.set_grid(n, 8 + 2 * 4 + 4, 4, 4, 8.0)
    s.set_eps(np.full((1, n), 1.5), 2.25, 1.0)
    s.set_channels([0], [0])
    re, im = X.real.float().contiguous(), X.imag.float().contiguous()
    rc = L.apf_debug_inv32(s._h, n, re.data_ptr(), im.data_ptr(), n)
    assert rc == 0, L.apf_last_error(s._h)
    return re.double() + 1j * im.double()


def noise(torch, n, seed, scale):
    P = torch.randn(n, n, dtype=torch.complex128, generator=torch.Generator(device="cpu").manual_seed(seed))
    return (P + P.T) * scale


@pytest.mark.parametrize("n", [64, 128])
@pytest.mark.parametrize("shift", [1, 9, 31])
def test_permuted_pivots(n, shift):
    """The 32 x 32 diagonal blocks have their large elements off the diagonal, so
    that every pivot is found in another row: condition number below 2, float32
    elimination of n columns within n * 2^-24 * 4."""
    torch = pytest.importorskip("torch")
    X = noise(torch, n, shift, 0.1 / n ** 0.5)
    for b in range(0, n, 32):
        for i in range(32):
            X[b + i, b + (shift - i) % 32] += 1.0 + 0.5j
    X = X.cuda()
    ref = torch.linalg.inv(X)
    err = (torch.linalg.norm(invert(torch, X) - ref) / torch.linalg.norm(ref)).item()
    assert err < n * 2.0 ** -24 * 4, err


@pytest.mark.parametrize("n", [64, 128])
def test_singular_leading_block(n):
    """The leading 32 x 32 block is zero while the whole is well conditioned: the
    block elimination must notice and pivoting over all rows take over (condition
    number below 2; same bound)."""
    torch = pytest.importorskip("torch")
    X = noise(torch, n, n, 0.02 / n ** 0.5)
    X[:32, :32] = 0.0
    for i in range(n):
        X[i, (i + n // 2) % n] += 1.0
    X = X.cuda()
    ref = torch.linalg.inv(X)
    err = (torch.linalg.norm(invert(torch, X) - ref) / torch.linalg.norm(ref)).item()
    assert err < n * 2.0 ** -24 * 4, err
