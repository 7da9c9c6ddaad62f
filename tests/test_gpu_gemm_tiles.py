"""FP64 products on the FP64 pipe at every tile of the cost model (test_gemm_plan.py checks
that these shapes reach all seven), ragged edges, split and unsplit, both forms, with
outputs of several million elements and more columns than a grid of narrow tiles
holds; the timer says that the FP64 pipe ran them.  Bar as for the other FP64 products:
4e-15 sqrt(K) max|A| max|B|, against numpy complex128."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu

SHAPES = [(878, 1321, 1), (17801, 18, 2), (6890, 67, 1), (6318, 1, 83), (189, 638, 5), (2501, 71, 16),
          (33, 15, 47), (129, 33, 100), (145, 143, 150), (600, 500, 64), (2000003, 3, 4), (3, 1200007, 3)]


@pytest.mark.parametrize("M,N,K", SHAPES)
@pytest.mark.parametrize("conj_a", [False, True])
def test_fp64_pipe_tiles(M, N, K, conj_a):
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
    s.set_kernel_timing(True)
    s.gemm(dev(A), dev(B), Ct, conj_a=conj_a, alpha=1.5, beta=-1j)
    s.sync()
    assert {k for k, v in s.kernel_times().items() if v["launches"]} == {"cgemm_fp64"}
    ref = 1.5 * ((A.conj().T if conj_a else A) @ B) - 1j * C0
    bar = 1.5 * 4e-15 * np.sqrt(K) * np.abs(A).max() * np.abs(B).max() + 4e-15 * np.abs(C0).max()
    assert np.abs(Ct.cpu().numpy().T - ref).max() <= bar
