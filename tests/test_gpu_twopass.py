"""The two-pass kernels of cubic edges (general path): every edge they are built
for, both directions, out of place and in place, one grid and a batch that runs
as two chains of chunks, against the FP64 oracle.

Bar: 5e-6 relative L2 per grid, the FP32 path's."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2006_08435_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 5e-6
EDGES = [48, 60, 64, 72, 80, 90, 96, 100, 108, 128]


@pytest.mark.parametrize("n", EDGES)
@pytest.mark.parametrize("inverse", [False, True])
def test_two_passes_against_oracle(cuda, monkeypatch, n, inverse):
    from paper_2006_08435_gb300 import Plan
    monkeypatch.setenv("FFT3D_VARIANT", "10")
    batch = 3
    x = torch.from_numpy(synth.uniform_grids(n, batch, seed=n)).cuda()
    p = Plan(n, n, n, batch, inverse=inverse, norm="by_n" if inverse else "none")
    assert p.variant == 10
    y = torch.empty_like(x)
    p.execute(x, y)
    scale = 1.0 / n ** 3 if inverse else 1.0
    for b in (0, batch - 1):
        ref = oracle.dft3d(x[b].cpu().numpy().astype(np.complex128), 1 if inverse else -1) * scale
        assert oracle.rel_l2(y[b].cpu().numpy(), ref) <= TOL
    z = x.clone()
    p.execute(z, z)  # the cluster form
    assert torch.equal(z, y)


@pytest.mark.parametrize("n,batch", [(48, 77), (90, 11), (128, 7)])
def test_two_chains_equal_one_grid_at_a_time(cuda, monkeypatch, n, batch):
    from paper_2006_08435_gb300 import Plan
    monkeypatch.setenv("FFT3D_VARIANT", "10")
    gen = torch.Generator(device="cuda").manual_seed(n)
    x = torch.randn((batch, n, n, n), dtype=torch.complex64, device="cuda", generator=gen)
    one, p = Plan(n, n, n, 1), Plan(n, n, n, batch)
    ref, y = torch.empty_like(x), torch.empty_like(x)
    for b in range(batch):
        one.execute(x[b], ref[b])
    p.execute(x, y)
    assert torch.equal(y, ref)
    for _ in range(20):  # in place, back to back
        y.copy_(x)
        p.execute(y, y)
        assert torch.equal(y, ref)


@pytest.mark.parametrize("shape,batch", [((64, 128, 96), 4), ((50, 75, 45), 6), ((45, 100, 32), 5),
                                         ((80, 96, 128), 3), ((90, 120, 135), 2), ((40, 36, 160), 9),
                                         ((75, 75, 75), 3), ((60, 162, 54), 5), ((128, 64, 50), 4)])
@pytest.mark.parametrize("inverse", [False, True])
def test_boxes_against_oracle(cuda, shape, batch, inverse):
    """Boxes on the two-pass kernels: run-time y steps, x tiles cut off at the
    edge, and the in-place form."""
    from paper_2006_08435_gb300 import Plan
    nz, ny, nx = shape
    x = torch.from_numpy(synth.uniform_grids(shape, batch, seed=sum(shape))).cuda()
    p = Plan(nx, ny, nz, batch, inverse=inverse, norm="ortho")
    y = torch.empty_like(x)
    p.execute(x, y)
    for b in (0, batch - 1):
        ref = oracle.dft3d(x[b].cpu().numpy().astype(np.complex128), 1 if inverse else -1)
        assert oracle.rel_l2(y[b].cpu().numpy(), ref / np.sqrt(nx * ny * nz)) <= TOL
    z = x.clone()
    p.execute(z, z)
    assert torch.equal(z, y)
