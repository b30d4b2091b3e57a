"""Errors of the real and the two-pass transforms against FP64 on the workloads'
inputs (pairs of densities, single orbitals): at most those of the kernels that
these transforms ran on before, which are the bars (measured on the same inputs
with the pair scheme and the fused kernels, 2% added)."""
import numpy as np
import pytest
import torch

from paper_2006_08435_gb300 import synth

pytestmark = pytest.mark.gpu

# edge: relative L2 error times 1e7, forward and inverse
REAL = {36: (1.336, 1.396), 80: (1.383, 1.474), 108: (1.636, 1.705)}
COMPLEX = {48: (1.498, 1.519), 80: (1.467, 1.469)}
# edge: of eight densities, forth and back (the pair scheme's other kernel)
ROUND = {96: 2.182}


def rel(got, ref):
    return np.linalg.norm((got - ref).ravel()) / np.linalg.norm(ref.ravel())


def real_errors(n):
    from paper_2006_08435_gb300 import irfft3d, rfft3d
    rho = np.stack([synth.hartree_density(n, seed=s)[0] for s in (1, 2)]).astype(np.float32)
    ref = np.fft.rfftn(rho.astype(np.float64), axes=(1, 2, 3))
    fwd = rel(rfft3d(torch.from_numpy(rho).cuda()).cpu().numpy(), ref)
    half = ref.astype(np.complex64)
    back = np.fft.irfftn(half.astype(np.complex128), s=(n, n, n), axes=(1, 2, 3))
    inv = rel(irfft3d(torch.from_numpy(half).cuda(), norm="by_n").cpu().numpy(), back)
    return fwd, inv


def complex_errors(n):
    """The mean over three orbitals, one at a time."""
    from paper_2006_08435_gb300 import fft3d
    fwd = inv = 0.0
    for seed in (1, 2, 3):
        x = synth.gaussian_sum_grids(n, 1, seed=seed)
        xd, xr = torch.from_numpy(x).cuda(), x.astype(np.complex128)
        fwd += rel(fft3d(xd).cpu().numpy(), np.fft.fftn(xr, axes=(1, 2, 3))) / 3
        back = np.fft.ifftn(xr, axes=(1, 2, 3), norm="forward")
        inv += rel(fft3d(xd, inverse=True).cpu().numpy(), back) / 3
    return fwd, inv


def round_trip_error(n):
    from paper_2006_08435_gb300 import irfft3d, rfft3d
    rho = np.stack([synth.hartree_density(n, seed=s)[0] for s in range(8)]).astype(np.float32)
    back = irfft3d(rfft3d(torch.from_numpy(rho).cuda()), norm="by_n").cpu().numpy()
    return rel(back, rho.astype(np.float64))


@pytest.mark.parametrize("n", sorted(REAL))
def test_real_errors(cuda, n):
    for got, bar in zip(real_errors(n), REAL[n]):
        assert got <= bar * 1e-7


@pytest.mark.parametrize("n", sorted(COMPLEX))
def test_complex_errors(cuda, n):
    for got, bar in zip(complex_errors(n), COMPLEX[n]):
        assert got <= bar * 1e-7


@pytest.mark.parametrize("n", sorted(ROUND))
def test_round_trip_errors(cuda, n):
    assert round_trip_error(n) <= ROUND[n] * 1e-7
