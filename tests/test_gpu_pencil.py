"""The pencil passes of the general path: every plannable edge on each axis,
tile remainders, batches that run as two chains of chunks, grids beyond the
chunk budget, and a captured graph with forked chains.

Bar: 5e-6 relative L2 per grid, the FP32 path's (two register codelets of at
most 32 points and one twiddle per axis: a few FP32 roundings more or less than
the other FP32 kernels)."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2006_08435_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 5e-6
EDGES = sorted(2 ** a * 3 ** b * 5 ** c for a in range(10) for b in range(6) for c in range(4)
               if 2 <= 2 ** a * 3 ** b * 5 ** c <= 512)


def _complex(shape, batch, seed):
    return torch.from_numpy(synth.uniform_grids(shape, batch, seed=seed)).cuda()


@pytest.mark.parametrize("inverse", [False, True])
@pytest.mark.parametrize("axis", [0, 1, 2])
def test_every_edge_on_every_axis(cuda, axis, inverse):
    """(n, 3, 4) and its rotations, two grids: rows, y and z pencils of every
    plannable edge, partial tiles."""
    from paper_2006_08435_gb300 import Plan
    for n in EDGES:
        shape = [4, 3, 4]
        shape[2 - axis] = n  # (nz, ny, nx)
        nz, ny, nx = shape
        if nx == ny == nz and nx in (16, 32, 48, 64, 80, 96, 128):
            continue
        x = _complex(tuple(shape), 2, seed=n)
        y = torch.empty_like(x)
        Plan(nx, ny, nz, 2, inverse=inverse).execute(x, y)
        ref = oracle.dft3d(x.cpu().numpy().astype(np.complex128), 1 if inverse else -1)
        for b in range(2):
            assert oracle.rel_l2(y[b].cpu().numpy(), ref[b]) <= TOL, (n, axis)


@pytest.mark.parametrize("shape,batch", [((75, 60, 45), 27), ((64, 100, 90), 12), ((192, 160, 250), 3)])
def test_two_chains_equal_one_grid_at_a_time(cuda, shape, batch):
    """Batches above 40 MB (two chains; odd counts, a shorter last chunk) and
    grids beyond the chunk budget: the same bits as one grid per call, out of
    place, in place, and replayed from a captured graph."""
    from paper_2006_08435_gb300 import Plan
    nz, ny, nx = shape
    gen = torch.Generator(device="cuda").manual_seed(5)
    x = torch.randn((batch,) + shape, dtype=torch.complex64, device="cuda", generator=gen)
    one, p = Plan(nx, ny, nz, 1), Plan(nx, ny, nz, batch)
    ref = torch.empty_like(x)
    for b in range(batch):
        one.execute(x[b], ref[b])
    y = torch.empty_like(x)
    p.execute(x, y)
    assert torch.equal(y, ref)
    z = x.clone()
    p.execute(z, z)
    assert torch.equal(z, ref)
    s = torch.cuda.Stream()
    s.wait_stream(torch.cuda.current_stream())
    g = torch.cuda.CUDAGraph()
    y.zero_()
    with torch.cuda.graph(g, stream=s):
        p.execute(x, y, stream=s)
    for _ in range(2):
        y.zero_()
        g.replay()
        torch.cuda.synchronize()
        assert torch.equal(y, ref)
