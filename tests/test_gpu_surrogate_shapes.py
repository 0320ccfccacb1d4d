"""Surrogate kernels at the edges of their tiles: single channels and samples,
odd widths, mode counts around the 32-pair and 64-mode chunks, positions that
are no multiple of a block's, batches that take the one-output kernels and either
block width of the tiled ones; forward and every gradient against the float64 reference.

Tolerance: float32 sums of up to n x width terms (relative error of the order of
sqrt(16384) x 2^-24 = 8e-6) through three or four layers: 5e-5 forward, 2e-4 on
each parameter group's gradient."""
import numpy as np
import pytest

from oracle import surrogate_ref as R

pytestmark = pytest.mark.gpu

# n, in_ch, width, modes, layers, n_out, batch
SHAPES = [(64, 1, 1, 1, 1, 1, 1), (64, 2, 9, 32, 2, 3, 5), (192, 5, 7, 31, 3, 2, 3), (320, 12, 33, 65, 2, 5, 2),
          (256, 20, 54, 33, 2, 7, 1), (1024, 12, 48, 64, 2, 5, 66), (512, 3, 16, 130, 2, 1, 9), (960, 3, 53, 37, 2, 2, 6)]


@pytest.mark.parametrize("shape", SHAPES)
def test_against_reference(shape):
    from paper_2306_09257_gb300 import surrogate as SG
    n, ci, c, m, layers, no, B = shape
    cfg = dict(in_ch=ci, width=c, modes=m, layers=layers, n_out=no)
    rng = np.random.default_rng(n + c + m)
    p = SG.init_params(7, ci, c, m, layers, no)
    p = (1.5 * p + 0.02 * rng.normal(size=p.size)).astype(np.float32)
    sno = SG.Surrogate(n=n, max_batch=B, **cfg)
    sno.set_params(p)
    x = rng.uniform(1.0, 2.25, size=(B, ci, n)).astype(np.float32)
    t = rng.uniform(0, 0.5, size=(B, no)).astype(np.float32)
    loss_ref, g_ref, y_ref = R.loss_and_grads(p, x.astype(np.float64), t.astype(np.float64), **cfg)
    y = sno.forward(x).cpu().numpy()
    assert np.linalg.norm(y - y_ref) <= 5e-5 * np.linalg.norm(y_ref)
    g, loss = sno.gradients(x, t)
    assert abs(loss - loss_ref) <= 1e-4 * abs(loss_ref)
    off = 0
    for name, s in SG.param_layout(ci, c, m, layers, no):
        k = int(np.prod(s))
        a, b = g[off:off + k], g_ref[off:off + k]
        assert np.linalg.norm(a - b) <= 2e-4 * np.linalg.norm(b) + 1e-7, name
        off += k
