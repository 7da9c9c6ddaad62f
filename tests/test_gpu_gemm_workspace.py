"""The residue GEMM in several K segments and pieces: the bits of a smaller product
that runs in one, and a workspace within its caps (3 GiB of operand residues, 1 GiB of
the result's, norms) whatever the sizes, in place of one that grew with K and with
the output."""
import numpy as np
import pytest

pytestmark = pytest.mark.gpu


@pytest.fixture(scope="module")
def env():
    import torch

    import paper_1709_10010_gb300 as pwh
    from paper_1709_10010_gb300 import build
    build.build()
    return torch, pwh


# (3 segments of A^H B; 2 of A B; row pieces of a tall A B; column pieces of a short one)
@pytest.mark.parametrize("M,N,K,conj_a", [(1500, 1500, 40000, True), (700, 5000, 9000, False),
                                          (200000, 300, 200, False), (64, 30000, 2500, False)])
def test_segments_and_pieces_give_the_same_bits(env, M, N, K, conj_a):
    torch, pwh = env
    s = pwh.System(np.diag([6.0] * 3), ecut_ha=2.0)
    g = torch.Generator(device="cuda").manual_seed(M + K)
    rnd = lambda *sh: torch.view_as_complex(torch.randn(*sh, 2, generator=g, device="cuda", dtype=torch.float64))
    A = rnd(M, K) if conj_a else rnd(K, M)     # stored by columns
    B = rnd(N, K)
    C = s.gemm(A, B, conj_a=conj_a)
    s.sync()
    m0, n0, m, n = M // 3, N // 2 + 1, min(1000, M - M // 3), min(400, N // 2 - 1)
    sub = (A[m0:m0 + m] if conj_a else A[:, m0:m0 + m]).contiguous()
    D = s.gemm(sub, B[n0:n0 + n].contiguous(), conj_a=conj_a)
    s.sync()
    assert torch.equal(torch.view_as_real(C[n0:n0 + n, m0:m0 + m]), torch.view_as_real(D))


@pytest.mark.parametrize("M,N,K,conj_a", [(400000, 800, 16, False), (1500, 1500, 400000, True)])
def test_workspace_stays_within_the_caps(env, M, N, K, conj_a):
    torch, pwh = env
    s = pwh.System(np.diag([6.0] * 3), ecut_ha=2.0)
    A = torch.zeros((M, K) if conj_a else (K, M), dtype=torch.complex128, device="cuda")
    B = torch.zeros((N, K), dtype=torch.complex128, device="cuda")
    C = torch.empty((N, M), dtype=torch.complex128, device="cuda")
    s.sync()
    torch.cuda.synchronize()
    free = torch.cuda.mem_get_info()[0]
    s.gemm(A, B, C, conj_a=conj_a)
    s.sync()
    used = free - torch.cuda.mem_get_info()[0]
    assert 0 < used <= (4 << 30) + (300 << 20)
