"""The FP64 H of a cubic box at every edge with compiled double-float passes against
the oracle: their index maps (prime-factor and four-step) and the choice of the
operations, spheres as wide as the edge allows, ragged last blocks of sticks.  Bar as
for the other FP64 H tests: 1e-12 of the largest element."""
import numpy as np
import pytest

from oracle import basis as ob
from oracle import hamiltonian as oh
from paper_1709_10010_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [30, 36, 40, 48, 50, 60, 72, 80, 90, 96, 120, 144])
def test_fp64_h_at_compiled_edges(n):
    import torch

    import paper_1709_10010_gb300 as pwh
    from paper_1709_10010_gb300 import build
    build.build()
    m = (n - 1) // 4
    cell = syn.make_cell(n, 10.0, 1, 2 * 0.5 * (2 * np.pi / 10.0 * (m + 0.2)) ** 2, 1)
    b = ob.sphere(cell.lattice, cell.kpoint, cell.ecut_ha, fft=(n, n, n))
    assert np.abs(b.miller).max() == m
    v = np.random.default_rng(n).standard_normal((n, n, n))
    beta, D = syn.projectors(cell, b.miller), syn.d_diagonal(cell)
    s = pwh.System(cell.lattice, cell.kpoint, cell.ecut_ha, fft=(n, n, n))
    s.set_potential(v)
    s.set_projectors(beta, D)
    psi = syn.initial_bands(n, b.npw, 2)
    out = s.apply_h(torch.from_numpy(psi).cuda()).cpu().numpy()
    s.close()
    ref = oh.apply_h(b, v, beta, D, psi)
    assert np.abs(out - ref).max() <= 1e-12 * np.abs(ref).max()
