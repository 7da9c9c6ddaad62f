"""The FP64 eigensolver's refined path (n >= 256: one sweep in FP32 pairs, then
refinement by products) at its first sizes, with odd sizes (a padding player in
the sweep), exact clusters, and matrices so small that the FP32 stage and the
pairs see only zeros: the FP64 sweeps behind the refinement then do it all.
"""
import numpy as np
import pytest

from paper_1709_10010_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu

# backward stable: eigenvalues, orthonormality and residuals to a few n eps of
# the largest |eigenvalue|; n <= 321, eps 2.2e-16, factor 8
BAR = 8 * 321 * 2.2e-16


@pytest.fixture(scope="module")
def env():
    import torch
    import paper_1709_10010_gb300 as pwh
    from paper_1709_10010_gb300 import build
    build.build()
    return torch, pwh.System(np.diag([6.0] * 3), ecut_ha=2.0)


def matrix(kind, n):
    H = syn.random_hermitian(n, n)
    if kind == "pairs":  # every level twice, the last alone when n is odd
        q = np.linalg.qr(H)[0]
        H = (q * (np.arange(n) // 2 / n)) @ q.conj().T
    elif kind == "blocks":  # uncoupled blocks with equal spectra
        m = n // 3
        H = np.kron(np.eye(3), H[:m, :m])
        H = np.pad(H, (0, n - 3 * m))
    return (H + H.conj().T) / 2


@pytest.mark.parametrize("kind,n,scale", [
    ("random", 255, 1.0), ("random", 256, 1.0), ("random", 321, 1.0), ("pairs", 256, 1.0),
    ("pairs", 257, 1.0), ("blocks", 289, 1.0), ("random", 257, 2.0 ** -160), ("random", 256, 2.0 ** 80)])
def test_refined_eigh(env, kind, n, scale):
    torch, s = env
    H = matrix(kind, n)
    theta, C = s.subspace_eigh(torch.from_numpy(np.ascontiguousarray((H * scale).T)).cuda(), n)
    s.sync()
    w = theta.cpu().numpy() / scale
    V = C.cpu().numpy().T
    ref = np.linalg.eigvalsh(H)
    top = np.abs(ref).max()
    assert np.abs(w - ref).max() < BAR * top
    assert np.abs(V.conj().T @ V - np.eye(n)).max() < BAR
    assert np.abs(H @ V - V * w).max() < BAR * top
