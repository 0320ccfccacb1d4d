"""The recursive inverse of a complex-symmetric block against float64, every
quadrant of the result (the upper right one is written by transposed stores).

Tolerance (Frobenius, relative to the whole inverse): L levels of four products,
each with a relative error of 2^-16 (two bf16 planes) independent of the others
and at most 2 x 3 x K / 16 additions truncated at 2^-24, K the largest block;
the blocks' own float32 inverses, 4 x 128 x 2^-24; condition number below 2."""
import ctypes

import numpy as np
import pytest

pytestmark = pytest.mark.gpu


def symmetric(torch, n, seed, scale):
    g = torch.Generator(device="cuda").manual_seed(seed)
    P = torch.randn(n, n, dtype=torch.complex128, device="cuda", generator=g) * (scale / n ** 0.5)
    return P + P.T


def check(torch, X, leaf, levels, planes=2):
    """X inverted with `leaf` as the hook takes it; returns the number of diagonal blocks that fell back."""
    from paper_2306_09257_gb300 import apf, build
    build.build_lib()
    L = apf.load_library()
    f = ctypes.c_void_p
    L.apf_debug_inv32.argtypes = [f, ctypes.c_int, f, f, ctypes.c_int]
    n = X.shape[0]
    s = apf.Solver(0, "mixed")
    s.set_elimination(planes, True)
    s.set_grid(n, 8 + 2 * 4 + 4, 4, 4, 8.0)
    s.set_eps(np.full((1, n), 1.5), 2.25, 1.0)
    s.set_channels([0], [0])
    re, im = X.real.float().contiguous(), X.imag.float().contiguous()
    rc = L.apf_debug_inv32(s._h, n, re.data_ptr(), im.data_ptr(), leaf)
    assert rc == 0, L.apf_last_error(s._h)
    ref = torch.linalg.inv(X)
    tol = 2 * ((4 * levels) ** 0.5 * 2.0 ** -16 + (6 * n / 32 + 512) * 2.0 ** -24)
    norm, h = torch.linalg.norm(ref).item(), n // 2
    err = re.double() + 1j * im.double() - ref
    for r in (0, h):
        for c in (0, h):
            e = torch.linalg.norm(err[r:r + h, c:c + h]).item() / norm
            assert e < tol, (r, c, e, tol)
    return s.stats()["leaf_fallbacks"]


@pytest.mark.parametrize("n,leaf", [(16, 8), (64, 32), (128, 16), (256, 32), (256, 100032), (512, 8), (64, 2)])
def test_blocks_below_64(n, leaf):
    """Blocks narrower than the 64 columns of a k block: the products must not read their neighbours."""
    torch = pytest.importorskip("torch")
    X = symmetric(torch, n, n + leaf, 0.2)
    X[range(n), range(n)] += 2.0 + 0.5j
    check(torch, X, leaf, int(np.log2(n / max(8, leaf % 1000))))


@pytest.mark.parametrize("planes", [2, 3])
@pytest.mark.parametrize("leaf", [128, 100128])
def test_pair_tiles(leaf, planes):
    """n = 4096: the products of the top level have 2048 terms and rows and run on two-CTA tiles, with beta input,
    the symmetric walk over the tiles, and float32, split and transposed outputs."""
    torch = pytest.importorskip("torch")
    n = 4096
    X = symmetric(torch, n, leaf, 0.2)
    X[range(n), range(n)] += 2.0 + 0.5j
    check(torch, X, leaf, 5, planes)


@pytest.mark.parametrize("n,leaf", [(128, 64), (256, 128), (512, 128)])
def test_fallback_replaces_the_split_form(n, leaf):
    """The first 32 x 32 block is zero while the leading diagonal block is well conditioned: its cluster inverse is
    rejected after its split form has been written, and the products of the levels above read what pivoting over all
    rows writes over it."""
    torch = pytest.importorskip("torch")
    X = symmetric(torch, n, n, 0.1)
    X[range(leaf, n), range(leaf, n)] += 1.0
    i = torch.arange(leaf)
    X[i, (i + leaf // 2) % leaf] += 1.0
    X[:32, :32] = 0.0
    assert check(torch, X, leaf, int(np.log2(n / leaf))) == 1
