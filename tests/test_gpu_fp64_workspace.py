"""Device memory of the float64 mode: the inverses of the slab rows, one block of
scratch and the columns' buffers.  The second chain of the elimination works in
memory that is there anyway."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("h", [2, 3, 6])
def test_workspace(h):
    from paper_2306_09257_gb300 import apf
    n = 512
    s = apf.Solver(0, "fp64")
    s.set_grid(n, 60 + h, 12, 12, 21.0)
    s.set_eps(np.full((h, n), 1.5), 2.25, 1.0)
    s.set_channels()
    n_in, n_out = (len(m) for m in s.channels())
    ncol = n_in + n_out
    blocks = 16 * n * n * (h + 1)
    # fields, two buffers of one row, the gradient's and the reflection block's columns
    columns = 16 * n * (h * max(ncol, 2 * n_in) + 2 * ncol + h * n_out + n_in)
    rest = 8 * h * n + 48 * n_in * n_out + 256 * (n + 60 + h + ncol)
    assert s.stats()["workspace_bytes"] <= blocks + columns + rest
