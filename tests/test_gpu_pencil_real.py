"""Real grids on the pencil passes (every even edge above 2 without a
dedicated kernel): small and large edges, odd widths of half spectra, spectra
that are not Hermitian, grids of very different size in one batch, and a
batch that runs as two chains of chunks.

Bar: 5e-6 relative L2 per grid, the FP32 path's."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2006_08435_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 5e-6
EDGES = sorted(2 ** a * 3 ** b * 5 ** c for a in range(10) for b in range(6) for c in range(4)
               if 2 <= 2 ** a * 3 ** b * 5 ** c <= 512)


@pytest.mark.parametrize("n", [e for e in EDGES if e % 2 == 0 and 4 <= e <= 60
                               and e not in (16, 32)])
def test_real_grids_of_every_small_edge(cuda, n):
    """Half spectra and back (the inverse on half spectra that are not
    Hermitian in the self-mirrored columns), three grids of very different
    size: each grid's error is relative to itself."""
    from paper_2006_08435_gb300 import irfft3d, rfft3d
    r = np.ascontiguousarray(synth.uniform_grids(n, 3, seed=n).real.astype(np.float32))
    r *= np.array([1.0, 1e-3, 1e3], dtype=np.float32)[:, None, None, None]
    f = rfft3d(torch.from_numpy(r).cuda()).cpu().numpy()
    ref = oracle.rdft3d(r.astype(np.float64))
    h = synth.uniform_grids((n, n, n // 2 + 1), 3, seed=n + 1)
    hd = torch.from_numpy(h).cuda()
    g = irfft3d(hd, norm="by_n").cpu().numpy()
    back = oracle.irdft3d(h.astype(np.complex128), n) / float(n) ** 3
    for b in range(3):
        assert oracle.rel_l2(f[b], ref[b]) <= TOL
        assert oracle.rel_l2(g[b], back[b]) <= TOL
    assert np.array_equal(hd.cpu().numpy(), h)


@pytest.mark.parametrize("n", [150, 162, 250, 500])
def test_real_round_trip_and_samples_of_large_edges(cuda, n):
    from paper_2006_08435_gb300 import irfft3d, rfft3d
    r = np.ascontiguousarray(synth.uniform_grids(n, 1, seed=n).real.astype(np.float32))
    rd = torch.from_numpy(r).cuda()
    f = rfft3d(rd)
    pts = [(0, 0, 0), (n // 2, n // 2, n // 2), (1, n - 1, n // 2), (n - 3, 5, 7), (n // 3, 1, 0)]
    ref = np.array(oracle.dft3d_points(r[0].astype(np.complex128), pts))
    got = np.array([f[0, z, y, x].item() for z, y, x in pts])
    assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= TOL
    b = irfft3d(f, norm="by_n").cpu().numpy()
    assert oracle.rel_l2(b[0], r[0]) <= TOL


def test_real_two_chains(cuda):
    """A real batch above 40 MB of half spectra, odd count: the same bits as
    one grid per call, in both directions."""
    from paper_2006_08435_gb300 import RealPlan
    n, batch = 90, 15
    gen = torch.Generator(device="cuda").manual_seed(6)
    r = torch.randn((batch, n, n, n), device="cuda", generator=gen)
    f = torch.empty((batch, n, n, n // 2 + 1), dtype=torch.complex64, device="cuda")
    ref, back, refb = torch.empty_like(f), torch.empty_like(r), torch.empty_like(r)
    RealPlan(n, batch).execute(r, f)
    RealPlan(n, batch, inverse=True, norm="by_n").execute(f, back)
    p1, q1 = RealPlan(n, 1), RealPlan(n, 1, inverse=True, norm="by_n")
    for b in range(batch):
        p1.execute(r[b], ref[b])
        q1.execute(f[b], refb[b])
    assert torch.equal(f, ref) and torch.equal(back, refb)
    assert oracle.rel_l2(back.cpu().numpy(), r.cpu().numpy()) <= TOL


@pytest.mark.parametrize("n,batch", [(18, 3), (48, 5), (80, 9), (90, 2), (96, 8), (100, 1)])
def test_fixed_spectra_and_the_energy_taken_from_them(cuda, n, batch):
    """RealPlan.fixed against the oracle (pairs of grids of equal size, so the
    same bar holds), and hartree_energy's value is bit for bit the one of its
    spectrum."""
    from paper_2006_08435_gb300 import RealPlan, hartree_energy
    from paper_2006_08435_gb300.hartree import energy_from_half_spectrum
    r = np.ascontiguousarray(synth.uniform_grids(n, batch, seed=n).real.astype(np.float32))
    rd = torch.from_numpy(r).cuda()
    f = torch.empty((batch, n, n, n // 2 + 1), dtype=torch.complex64, device="cuda")
    p = RealPlan.fixed(n, batch)
    p.execute(rd, f)
    assert p.device_status() == 0
    for b in (0, batch - 1):
        assert oracle.rel_l2(f[b].cpu().numpy(), oracle.rdft3d(r[b].astype(np.float64))) <= TOL
    assert torch.equal(hartree_energy(rd, 10.0), energy_from_half_spectrum(f, 10.0))
