"""The FP64 eigensolver on matrices of very small and very large elements, on both sides
of the size from which the refinement runs: as accurate as at unit scale.  Bar: the
target of the sweeps, off-diagonal elements of 1e-13 of the largest, twice."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [200, 257, 300])
@pytest.mark.parametrize("scale", [1.0, 2.0 ** 40, 2.0 ** 41, 1e30, 1e36, 2.0 ** -20, 2.0 ** -21, 1e-12, 1e-20, 1e-24,
                                   1e-30, 1e-36, 1e-40, 1e-60])
def test_eigh_scale(n, scale):
    import torch

    import paper_1709_10010_gb300 as pwh
    from paper_1709_10010_gb300 import build
    build.build()
    s = pwh.System(np.diag([6.0] * 3), ecut_ha=2.0)
    rng = np.random.default_rng(n)
    B = rng.standard_normal((n, n)) + 1j * rng.standard_normal((n, n))
    H = B + B.conj().T
    ref = np.linalg.eigvalsh(H)
    theta, C = s.subspace_eigh(torch.from_numpy(np.ascontiguousarray((H * scale).T)).cuda(), n)[:2]
    s.sync()
    theta, C = theta.cpu().numpy() / scale, C.cpu().numpy().T
    top = np.abs(ref).max()
    assert np.abs(theta - ref).max() <= 2e-13 * top
    assert np.abs(C.conj().T @ C - np.eye(n)).max() <= 2e-13
    assert np.abs(H @ C - C * theta).max() <= 2e-13 * top
