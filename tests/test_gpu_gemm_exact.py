"""Products of integers by the residue GEMM are the exact integers: the operands'
integers, the residues and their sum are exact, and the reconstruction, within 2^-61
of the value, is rounded once, so a result that FP64 holds comes out as it is (the
fraction's own error, 2^-94 |a| |b|, is far below 1 here).  Sums of one sign,
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
