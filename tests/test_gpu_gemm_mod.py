"""The FP64-equivalent GEMM by residues (pwh_subspace_gemm, FP64, at least 2e8
flops) at the places where its form can go wrong: both sides of a 256-row tile
and of a 32-wide tile column, K on both sides of a 960-wide exact chunk, several
K ranges, values whose residues add up with one sign (the largest exact sums),
rows of very different scale, exact zeros, infinities.

Bar: an operand row is rounded to integers with 2-norm between 2^61 and 2^62,
an error of 2-norm at most sqrt(2 K) / 2, so an element is off by at most
2 (sqrt(2 K) / 2) 2^-61 = sqrt(2 K) 2^-61 of |a| |b| plus its FP64 rounding;
the reference sums K products in FP64: 2 sqrt(K) 2^-53 |a| |b| with random
signs.  (The norm itself is bounded to a factor 2 by its exponent: 2^-60.)"""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(255, 130, 960, True), (257, 129, 961, True), (256, 16, 6000, True), (513, 97, 1921, True),
          (256, 128, 1100, False), (2049, 33, 500, False), (300, 500, 480, False),
          (40, 1, 700000, True), (70000, 2, 300, False)]


@pytest.fixture(scope="module")
def env():
    import torch

    import paper_1709_10010_gb300 as pwh
    from paper_1709_10010_gb300 import build
    build.build()
    return torch, pwh.System(np.diag([6.0] * 3), ecut_ha=2.0)


def product(env, A, B, conj_a, **kw):
    torch, s = env
    dev = lambda X: torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
    C = s.gemm(dev(A), dev(B), conj_a=conj_a, **kw)
    s.sync()
    return C.cpu().numpy().T


def norms(X):
    """2-norms of the columns, without overflow or underflow of the squares."""
    m = np.maximum(np.abs(X).max(axis=0), 1e-290)
    return np.linalg.norm(X / m, axis=0) * m


def check(env, A, B, conj_a):
    op = A.conj().T if conj_a else A
    K = B.shape[0]
    C, ref = product(env, A, B, conj_a), op @ B
    norm = norms(op.T)[:, None] * norms(B)[None, :]
    bar = norm * (2.0 ** -60 * np.sqrt(2 * K) + 2 * np.sqrt(K) * 2.0 ** -53) + 2.0 ** -52 * np.abs(ref)
    assert np.all(np.abs(C - ref) <= bar), float((np.abs(C - ref) / np.maximum(norm, 1e-300)).max())


@pytest.mark.parametrize("M,N,K,conj_a", SHAPES)
def test_edges(env, M, N, K, conj_a):
    if 8.0 * M * N * K < 2e8:
        K = K * int(np.ceil(2e8 / (8.0 * M * N * K)))
    rng = np.random.default_rng([M, N, K])
    z = lambda *s: rng.standard_normal(s) + 1j * rng.standard_normal(s)
    check(env, z(K, M) if conj_a else z(M, K), z(K, N), conj_a)


@pytest.mark.parametrize("kind", ["one", "alternating", "scales", "tiny"])
def test_values(env, kind):
    rng = np.random.default_rng(5)
    M, N, K = 300, 200, 2000
    A = np.ones((K, M), dtype=complex)
    B = np.ones((K, N), dtype=complex) * (1 - 1j)
    if kind == "alternating":
        A[::2] *= -1
    elif kind != "one":
        A = rng.standard_normal((K, M)) * np.exp(rng.uniform(-200, 200, M)) + 0j
        B = rng.standard_normal((K, N)) * np.exp(-np.arange(K) / 20.0)[:, None] + 0j
        if kind == "tiny":
            A, B = A * 1e-300 / np.abs(A).max(), B * 1e290
    check(env, A, B, True)


def test_zeros_and_nonfinite(env):
    rng = np.random.default_rng(6)
    A = rng.standard_normal((1500, 300)) + 1j * rng.standard_normal((1500, 300))
    A[:, 7] = 0
    B = A[:, :200].copy()
    B[3, 5], B[9, 11] = np.nan, np.inf
    C = product(env, A, B, True)
    good = [j for j in range(200) if j not in (5, 11)]
    assert np.all(np.isfinite(C[:, good])) and not np.any(np.isfinite(C[:, [5, 11]].real))
    assert np.all(C[7, good] == 0) and np.all(C[:, 7] == 0)
    assert np.all(np.diag(C[:200])[good].imag == 0)      # Gram matrix: exactly real diagonal
    R = product(env, A.real + 0j, B[:, good].real + 0j, True)
    assert np.all(R.imag == 0)                            # real data stays real
