"""A band's H does not depend on how many bands are applied with it: one, a few and many
bands take other launch shapes (reordering, blocks of the FP32 plane pass), and each
band has to come out with the same bits, in every order of leading dimension."""
import numpy as np
import pytest

from paper_1709_10010_gb300 import synthetic as syn

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n", [30, 48, 50, 60, 90, 96, 120])
@pytest.mark.parametrize("precision", ["mixed", "fp64"])
def test_band_alone_and_among_others(n, precision):
    import torch

    import paper_1709_10010_gb300 as pwh
    from paper_1709_10010_gb300 import build
    build.build()
    m = (n - 1) // 4
    s = pwh.System(np.diag([10.0] * 3), ecut_ha=0.5 * (2 * np.pi / 10.0 * (m + 0.2)) ** 2, fft=(n, n, n),
                   precision=precision)
    s.set_potential(np.random.default_rng(n).standard_normal((n, n, n)))
    nb = 361 // n + 3                                   # more than 360 planes
    psi = torch.from_numpy(syn.initial_bands(n, s.npw, nb)).cuda()
    ref = s.apply_h(psi)
    s.sync()
    for k in (1, 3, nb - 1):
        out = s.apply_h(psi[nb - k:].contiguous())
        s.sync()
        assert torch.equal(torch.view_as_real(out), torch.view_as_real(ref[nb - k:])), k
    # bands with a longer leading dimension
    wide = torch.zeros((nb, s.npw + 5), dtype=torch.complex128, device="cuda")
    wide[:, :s.npw] = psi
    out = s.apply_h(wide[:, :s.npw])
    s.sync()
    s.close()
    assert torch.equal(torch.view_as_real(out), torch.view_as_real(ref))
