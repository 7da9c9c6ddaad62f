"""A^H B by the residue GEMM where real and imaginary parts differ in size: each part
of the result keeps its own accuracy, as in FP64 arithmetic.

Bar: a part of a column is rounded to integers with an error of at most sqrt(2 K)
2^-61 of its norm (test_gpu_gemm_mod.py), up to 2^4 more where both parts share an
exponent, and each real product and their sum are rounded to FP64: for Re C, with
|.| the columns' norms, (|Re a| |Re b| + |Im a| |Im b|) (sqrt(2 K) 2^-56 + 2^-51),
for Im C the same with the crossed norms."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("ga,gb", [(1.0, 1.0), (2.0 ** -4, 1.0), (2.0 ** -7, 2.0 ** 5), (1e-10, 1.0), (1.0, 1e-12),
                                   (1e-10, 1e-10), (1e-30, 1e30), (1e40, 1.0), (0.0, 1e-8)])
def test_parts_keep_their_accuracy(ga, gb):
    import torch

    import paper_1709_10010_gb300 as pwh
    from paper_1709_10010_gb300 import build
    build.build()
    s = pwh.System(np.diag([6.0] * 3), ecut_ha=2.0)
    M, N, K = 203, 151, 1500
    rng = np.random.default_rng(3)
    ar, br = rng.standard_normal((K, M)), rng.standard_normal((K, N))
    ai, bi = ga * rng.standard_normal((K, M)), gb * rng.standard_normal((K, N))
    bi[:, ::3] *= 2.0 ** -9                             # columns of both kinds
    dev = lambda X: torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
    C = s.gemm(dev(ar + 1j * ai), dev(br + 1j * bi), conj_a=True)
    s.sync()
    C = C.cpu().numpy().T[:25, :25]
    L = lambda X: X[:, :25].astype(np.longdouble)
    mul = lambda X, Y: np.einsum("km,kn->mn", L(X), L(Y))
    nrm = lambda X, Y: np.outer(np.linalg.norm(X[:, :25], axis=0), np.linalg.norm(Y[:, :25], axis=0))
    eps = np.sqrt(2 * K) * 2.0 ** -56 + 2.0 ** -51
    re, im = mul(ar, br) + mul(ai, bi), mul(ar, bi) - mul(ai, br)
    assert np.all(np.abs(C.real - re) <= eps * (nrm(ar, br) + nrm(ai, bi)))
    assert np.all(np.abs(C.imag - im) <= eps * (nrm(ar, bi) + nrm(ai, br)))
