"""FP64 products on the FP64 pipe at the tile shapes and K splits that their
cost model picks (small squares, narrow and short ones, long reductions, one
row or column, ragged edges), with row scaling left to the H tests.  Bar as for
the solver's GEMM: 4e-15 sqrt(K) max|A| max|B|, against numpy complex128."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("M,N,K", [(15, 17, 16), (16, 16, 31), (33, 15, 47), (32, 16, 1503), (1503, 16, 32),
                                   (1, 200, 900), (200, 1, 900), (65, 63, 257), (129, 33, 100), (700, 9, 40),
                                   (40, 40, 3000), (54, 18, 1503)])
@pytest.mark.parametrize("conj_a", [False, True])
def test_small_products(M, N, K, conj_a):
    import torch

    import paper_1709_10010_gb300 as pwh
    from paper_1709_10010_gb300 import build
    build.build()
    s = pwh.System(np.diag([6.0] * 3), ecut_ha=2.0)
    rng = np.random.default_rng([M, N, K, int(conj_a)])
    z = lambda *sh: rng.standard_normal(sh) + 1j * rng.standard_normal(sh)
    A, B, C0 = z(K, M) if conj_a else z(M, K), z(K, N), z(M, N)
    dev = lambda X: torch.from_numpy(np.ascontiguousarray(X.T)).cuda()
    Ct = dev(C0)
    s.gemm(dev(A), dev(B), Ct, conj_a=conj_a, alpha=1.5, beta=-1j)
    s.sync()
    ref = 1.5 * ((A.conj().T if conj_a else A) @ B) - 1j * C0
    bar = 1.5 * 4e-15 * np.sqrt(K) * np.abs(A).max() * np.abs(B).max() + 4e-15 * np.abs(C0).max()
    assert np.abs(Ct.cpu().numpy().T - ref).max() <= bar
