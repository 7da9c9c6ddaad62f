"""FP64 passes by axis (boxes that are not cubic) against the oracle: every
compiled edge at least once, in each of the three directions for some, with an
edge that has no compiled transform among them (the runtime plans), more rows
and columns than a block's 16 lines and ragged last blocks; the density and the
exchange operator on such a box.  Bars as for the cubic boxes: 1e-12 of the
largest element."""
import numpy as np
import pytest

from oracle import basis as ob
from oracle import exx as ox
from oracle import hamiltonian as oh
from oracle import scf as osc
from paper_1709_10010_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

BOXES = [(20, 24, 30), (144, 20, 32), (36, 40, 48), (24, 54, 60), (64, 32, 72), (30, 80, 20), (20, 90, 96),
         (100, 24, 108), (32, 30, 120), (128, 36, 24), (54, 20, 18), (64, 64, 64), (50, 20, 24)]


def system(fft, nproj_atoms=1):
    import torch

    import paper_1709_10010_gb300 as pwh
    from paper_1709_10010_gb300 import build
    build.build()
    # a skewed cell whose spheres reach the largest Miller index each edge allows
    m = [(n - 1) // 4 for n in fft]
    lat = np.array([[1.0, 0.0, 0.0], [0.2, 1.0, 0.0], [0.0, -0.1, 1.0]]) * (2.0 * np.array(m) - 1.0)[:, None]
    cell = syn.make_cell(3, lat, nproj_atoms, 2 * 0.5 * (np.pi) ** 2 * 0.8, 1, (0.1, -0.2, 0.05))
    b = ob.sphere(cell.lattice, cell.kpoint, cell.ecut_ha, fft=fft)
    assert all(4 * np.abs(b.miller[:, d]).max() + 1 <= fft[d] for d in range(3))
    s = pwh.System(cell.lattice, cell.kpoint, cell.ecut_ha, fft=fft)
    return torch, s, cell, b


@pytest.mark.parametrize("fft", BOXES)
def test_h_by_axes(fft):
    torch, s, cell, b = system(fft)
    v = np.random.default_rng(1).standard_normal(fft)
    beta, D = syn.projectors(cell, b.miller), syn.d_diagonal(cell)
    s.set_potential(v)
    s.set_projectors(beta, D)
    psi = syn.initial_bands(2, b.npw, 3)
    out = s.apply_h(torch.from_numpy(psi).cuda()).cpu().numpy()
    ref = oh.apply_h(b, v, beta, D, psi)
    assert np.abs(out - ref).max() <= 1e-12 * np.abs(ref).max()


@pytest.mark.parametrize("fft", [(24, 36, 20), (20, 18, 30)])
def test_density_and_exchange_by_axes(fft):
    torch, s, cell, b = system(fft)
    psi = syn.initial_bands(4, b.npw, 5)
    psi /= np.linalg.norm(psi, axis=1, keepdims=True)
    occ = np.array([2.0, 1.0, 0.5, 2.0, 0.25])
    rho = s.density(torch.from_numpy(psi).cuda(), occ).cpu().numpy()
    ref = osc.density(b.miller, fft, psi, occ, cell.volume)
    assert np.abs(rho - ref).max() <= 1e-12 * np.abs(ref).max()
    out = s.exx_apply(torch.from_numpy(psi).cuda(), occ, torch.from_numpy(psi[:2]).cuda()).cpu().numpy()
    ref = ox.exchange(b, cell.lattice, psi, occ, psi[:2])
    assert np.abs(out - ref).max() <= 1e-12 * np.abs(ref).max()
