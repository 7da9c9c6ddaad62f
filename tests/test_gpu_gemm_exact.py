"""Products of integers by the residue GEMM are the exact integers: the operands'
integers, the residues and their sum are exact, and the reconstruction, within 2^-61
of the value, is rounded once, so a result that FP64 holds comes out as it is (the
fraction's own error, 2^-91 |a| |b|, is far below 1 here).  Sums of one sign,
of random signs down to small results and to zero, both forms, K on both sides of an exact
chunk."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("K", [419, 961, 2000])
@pytest.mark.parametrize("conj_a", [True, False])
@pytest.mark.parametrize("kind", ["ones", "small", "thousands", "cancel"])
def test_integer_products_are_exact(K, conj_a, kind):
    import torch

    import paper_1709_10010_gb300 as pwh
    from paper_1709_10010_gb300 import build
    build.build()
    s = pwh.System(np.diag([6.0] * 3), ecut_ha=2.0)
    M, N = 301, 203
    rng = np.random.default_rng([K, int(conj_a)])
    top = {"ones": 1, "small": 3, "thousands": 1000, "cancel": 1000}[kind]
    draw = lambda *sh: rng.integers(-top if kind != "ones" else 1, top + 1, sh)
    ar, ai, br, bi = draw(M, K), draw(M, K), draw(K, N), draw(K, N)
    if kind == "ones":
        ai[:], bi[:] = 0, 0
        br[rng.integers(0, K, N), np.arange(N)] = 0      # sums of K and K - 1 ones
    if kind == "cancel":                                 # every element is zero
        ar, ai, br, bi = (np.concatenate(p) for p in ((ar.T, ar.T), (ai.T, ai.T), (br, -br), (bi, -bi)))
        ar, ai = ar.T, ai.T
    re, im = ar @ br - ai @ bi, ar @ bi + ai @ br
    A = ar + 1j * ai
    A = A.conj().T if conj_a else A
    dev = lambda X: torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
    C = s.gemm(dev(A), dev(br + 1j * bi), conj_a=conj_a)
    s.sync()
    C = C.cpu().numpy().T
    assert np.array_equal(C.real, re) and np.array_equal(C.imag, im)


def test_opposite_results_have_the_same_bits():
    """B^H A is the conjugate transpose of A^H B bit for bit, also where the elements
    are so small against the norms (here 2^-53 of them) that the fraction is cut off."""
    import torch

    import paper_1709_10010_gb300 as pwh
    from paper_1709_10010_gb300 import build
    build.build()
    s = pwh.System(np.diag([6.0] * 3), ecut_ha=2.0)
    M, K = 260, 1000
    rng = np.random.default_rng(8)
    draw = lambda top, *sh: rng.integers(-top, top + 1, sh) + 1j * rng.integers(-top, top + 1, sh)
    X, Y = draw(2 ** 26, K, M), draw(2 ** 26, K, M)
    X[0] = draw(1000, M)
    D = np.zeros((K, M), dtype=complex)
    D[0] = draw(3, M)
    A, B = np.concatenate((X, X)), np.concatenate((Y, D - Y))     # A^H B = X^H D
    dev = lambda Z: torch.from_numpy(np.ascontiguousarray(Z.T)).cuda()
    C = s.gemm(dev(A), dev(B), conj_a=True).cpu().numpy().T
    E = s.gemm(dev(B), dev(A), conj_a=True).cpu().numpy().T
    s.sync()
    norm = np.linalg.norm(A, axis=0)[:, None] * np.linalg.norm(B, axis=0)
    assert np.all(np.abs(C - X.conj().T @ D) <= 2.0 ** -90 * norm)    # 2^-91 for each part
    assert np.array_equal(E, C.conj().T)
