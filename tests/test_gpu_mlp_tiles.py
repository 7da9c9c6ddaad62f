"""The training kernel's row tiles (128 rows, persistent blocks) against the
oracle's FP64 gradient: one row, both sides of a tile's edge, a ragged last
tile, more tiles than resident blocks, and arrays that start off a 16-byte
boundary.  Bars: those of the plain
gradient test (2e-4 of the largest entry, loss 1e-5): an entry is an FP32 sum
of at most 2,048 rows in a thread's registers and one atomic a block, whose
error is at most 2,048 x 2^-24 = 1.2e-4 of the sum of its absolute terms."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("rows,shift", [(1, 0), (127, 0), (128, 1), (129, 0), (1000, 3), (40001, 0)])
def test_gradient_tiles(rows, shift):
    import torch

    import paper_1709_10010_gb300 as pwh
    from oracle import mlp as om
    from paper_1709_10010_gb300 import build, learned
    build.build()
    s = pwh.System(np.diag([6.0] * 3), ecut_ha=2.0)
    rng = np.random.default_rng([rows, shift])
    p = (learned.init_params(3) + 0.05 * rng.standard_normal(pwh.MLP_PARAMS)).astype(np.float32)
    F = rng.standard_normal((rows, 4)).astype(np.float32)
    y = rng.standard_normal(rows).astype(np.float32)
    w = rng.uniform(0.1, 1.0, rows).astype(np.float32)

    def dev(a):  # the same values, `shift` floats into an allocation
        buf = torch.zeros(a.size + shift, dtype=torch.float32, device="cuda")
        buf[shift:] = torch.from_numpy(a.reshape(-1)).cuda()
        return buf[shift:].view(a.shape)

    loss, g = s.mlp_loss_grad(dev(p), dev(F), dev(y), dev(w))
    args = [a.astype(np.float64) for a in (p, F, y, w)]
    lo, go = om.loss(*args), om.grad(*args)
    assert abs(float(loss.item()) - lo) <= 1e-5 * lo
    assert np.abs(g.cpu().numpy() - go).max() <= 2e-4 * np.abs(go).max()
