"""Real cubic grids in two passes: every edge that has the kernels, each
direction and normalisation, spectra that are not Hermitian in the self-mirrored
columns, grids of very different size in one batch, and both sides of the batch
from which 64^3 and 128^3 take the persistent inverse.

Bar: 5e-6 relative L2 per grid, the FP32 path's."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2006_08435_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 5e-6


@pytest.mark.parametrize("n", [48, 60, 64, 72, 80, 90, 96, 100, 108, 120, 128])
def test_two_pass_real_grids(cuda, n):
    from paper_2006_08435_gb300 import irfft3d, rfft3d
    r = np.ascontiguousarray(synth.uniform_grids(n, 2, seed=n).real.astype(np.float32))
    r *= np.array([1.0, 1e-3], dtype=np.float32)[:, None, None, None]
    ref = oracle.rdft3d(r.astype(np.float64))
    h = synth.uniform_grids((n, n, n // 2 + 1), 2, seed=n + 1)
    h *= np.array([1.0, 1e3], dtype=np.float32)[:, None, None, None]
    back = oracle.irdft3d(h.astype(np.complex128), n)
    rd, hd = torch.from_numpy(r).cuda(), torch.from_numpy(h).cuda()
    for norm, s in (("none", 1.0), ("by_n", n ** -3.0), ("ortho", n ** -1.5)):
        f = rfft3d(rd, norm=norm).cpu().numpy()
        g = irfft3d(hd, norm=norm).cpu().numpy()
        for b in range(2):
            assert oracle.rel_l2(f[b], s * ref[b]) <= TOL
            assert oracle.rel_l2(g[b], s * back[b]) <= TOL
    assert np.array_equal(rd.cpu().numpy(), r) and np.array_equal(hd.cpu().numpy(), h)


@pytest.mark.parametrize("n,batch", [(64, 99), (64, 100), (128, 47), (128, 48)])
def test_inverse_of_either_kernel(cuda, n, batch):
    """The same grids on both sides of the rule, with and without the Hartree
    weights, against the complex transform of the Hermitian extension's real part."""
    from paper_2006_08435_gb300 import irfft3d, rfft3d
    from paper_2006_08435_gb300.hartree import gradient_from_half_spectrum, seed_from_half_spectrum
    gen = torch.Generator(device="cuda").manual_seed(n)
    r = torch.randn((batch, n, n, n), device="cuda", generator=gen)
    f = rfft3d(r)
    back = irfft3d(f, norm="by_n")
    g = torch.randn(batch, dtype=torch.float64, device="cuda", generator=gen)
    grad = gradient_from_half_spectrum(f, 7.0, g)
    ref = irfft3d(seed_from_half_spectrum(f, 7.0, g))
    assert torch.equal(grad, ref)
    for b in (0, batch // 2, batch - 1):
        assert float((back[b] - r[b]).norm() / r[b].norm()) <= TOL
