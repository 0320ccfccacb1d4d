"""The 128 x 128 diagonal-block inverse against float64."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("shift", [1, 9, 31])
def test_diagonal_block_with_permuted_pivots(shift):
    """128 x 128 block whose 32 x 32 diagonal blocks have their large elements
    off the diagonal, so that every pivot is found in another row: condition
    number below 2, float32 elimination of 128 columns within 128 * 2^-24 * 4."""
    torch = pytest.importorskip("torch")
    from paper_2306_09257_gb300 import apf, build
    build.build_lib()
    L = apf.load_library()
    f = ctypes.c_void_p
    L.apf_debug_inv32.argtypes = [f, ctypes.c_int, f, f, ctypes.c_int]
    n = 128
    g = torch.Generator(device="cpu").manual_seed(shift)
    P = torch.randn(n, n, dtype=torch.complex128, generator=g) * (0.1 / n ** 0.5)
    X = P + P.T
    for b in range(4):
        for i in range(32):
            X[32 * b + i, 32 * b + (shift - i) % 32] += 1.0 + 0.5j
    X = X.cuda()
    s = apf.Solver(0, "mixed")
    s.set_grid(n, 8 + 2 * 4 + 4, 4, 4, 8.0)
    s.set_eps(np.full((1, n), 1.5), 2.25, 1.0)
    s.set_channels([0], [0])
    re, im = X.real.float().contiguous(), X.imag.float().contiguous()
    rc = L.apf_debug_inv32(s._h, n, re.data_ptr(), im.data_ptr(), 128)
    assert rc == 0, L.apf_last_error(s._h)
    ref = torch.linalg.inv(X)
    err = (torch.linalg.norm(re.double() + 1j * im.double() - ref) / torch.linalg.norm(ref)).item()
    assert err < 128 * 2.0 ** -24 * 4, err
