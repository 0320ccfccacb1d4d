"""A sample's predicted efficiencies do not depend on the samples that share its
call: the same bits alone (one-output kernels), among a few and among many
(both block widths of the tiled kernels), at odd widths and mode counts and
where n / 4 lies inside and at the start of a warp's positions."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

# n, in_ch, width, modes, layers, n_out, batches
SHAPES = [(1024, 12, 48, 64, 3, 5, (8, 64)), (320, 5, 33, 31, 2, 3, (30, 130)), (64, 2, 9, 32, 2, 1, (470, 500)),
          (448, 1, 54, 129, 2, 2, (20, 140))]


@pytest.mark.parametrize("shape", SHAPES)
def test_same_bits_in_every_batch(shape):
    torch = pytest.importorskip("torch")
    from paper_2306_09257_gb300 import surrogate as SG
    n, ci, c, m, layers, no, batches = shape
    rng = np.random.default_rng(n + m)
    p = SG.init_params(3, ci, c, m, layers, no)
    p = (1.5 * p + 0.02 * rng.normal(size=p.size)).astype(np.float32)
    sno = SG.Surrogate(n=n, in_ch=ci, width=c, modes=m, layers=layers, n_out=no, max_batch=max(batches))
    sno.set_params(p)
    x = torch.as_tensor(rng.uniform(1.0, 2.25, size=(max(batches), ci, n)).astype(np.float32), device="cuda")
    whole = {b: sno.forward(x[:b].contiguous()) for b in batches}
    for i in (0, 1, batches[0] - 1):
        alone = sno.forward(x[i:i + 1].contiguous())[0]
        for b in batches:
            assert torch.equal(alone, whole[b][i]), (i, b, (alone - whole[b][i]).abs().max().item())
