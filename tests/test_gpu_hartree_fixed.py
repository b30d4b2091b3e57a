"""Hartree energies are FP64 values of FP32 spectra and keep their bits: energies of
densities of exact binary fractions, at edges whose general transforms run in
another order of sums, against the values of the stage-by-stage passes that these
energies were first computed with."""
import pytest
import torch

pytestmark = pytest.mark.gpu

GOLDEN = {
    75: ["0x1.55de314b4fd28p+3", "0x1.55eef4353e6dap+3"],
    81: ["0x1.2d637d3ad2d2fp+3"],
    100: ["0x1.7c1fb1d2a7c09p+2", "0x1.7c1f6108e510ap+2", "0x1.7c1f2f81765b0p+2"],
    486: ["0x1.04a4f5d1c5cdbp-2"],
    500: ["0x1.ef788341c108ap-3"],
    512: ["0x1.d914b18356796p-3"],
}


def density(n, batch):
    i = torch.arange(n, device="cuda")
    rho = (37 * i[:, None, None] + 101 * i[None, :, None] + 53 * i) % 1009
    return torch.stack([((rho + 5 * b) % 1009).to(torch.float32) / 1024 for b in range(batch)])


def energies(n, batch):
    from paper_2006_08435_gb300 import hartree_energy
    return [e.hex() for e in hartree_energy(density(n, batch), 10.0).cpu().tolist()]


@pytest.mark.parametrize("n", sorted(GOLDEN))
def test_energies_keep_their_bits(cuda, n):
    assert energies(n, len(GOLDEN[n])) == GOLDEN[n]
