"""The two-pass boxes at every y step and number of groups they have: pass 1
takes B points per thread, chosen at run time, and pass 2 is a kernel of its own for
each number of groups A (ny = A B).  The rule that sends a box to them (passes.cu,
twopass_box.cuh) is restated here, so that a shape that falls out of it shows.

Bar: 5e-6 relative L2 per grid, the FP32 path's."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2006_08435_gb300 import synth

TOL = 5e-6
RADICES = [32, 30, 27, 25, 24, 20, 18, 16, 15, 12, 10]
CODELETS = {1, 2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32}
NX = {32, 36, 40, 45, 48, 50, 54, 60, 64, 72, 75, 80, 81, 90, 96, 100, 108, 120, 125, 128, 135, 144,
      150, 160}
# (nz, ny, nx): every B, A = 2 .. 6, columns that end inside a tile, odd nx
SHAPES = [(128, 20, 96), (128, 24, 75), (128, 30, 64), (120, 32, 64), (120, 36, 60), (120, 40, 54),
          (80, 72, 45), (75, 81, 45), (50, 125, 45), (54, 160, 50), (75, 75, 128), (120, 60, 81),
          (128, 64, 100), (45, 150, 72), (75, 96, 32), (90, 108, 36), (60, 100, 48), (48, 162, 40)]


def route(nz, ny, nx):
    """(A, B) of the two passes of a box, or None."""
    for b in RADICES:
        if ny % b == 0 and 2 <= ny // b <= 6:
            a = ny // b
            split = any(nz % z == 0 and z in CODELETS and nz // z in CODELETS and nz // z <= 20
                        for z in range(2, 36 // a + 1))
            fits = 8 * 16 * a * nz <= 72 * 1024
            ok = nz * a >= 220 and b * nx >= 800 and nx in NX and nz in NX and split and fits
            return (a, b) if ok else None
    return None


def test_the_shapes_cover_the_kernels():
    taken = [route(*s) for s in SHAPES]
    assert None not in taken
    assert {b for _, b in taken} == set(RADICES)
    assert {a for a, _ in taken} == {2, 3, 4, 5, 6}


@pytest.mark.gpu
@pytest.mark.parametrize("shape", SHAPES)
@pytest.mark.parametrize("inverse", [False, True])
def test_box_shapes_against_oracle(cuda, shape, inverse):
    from paper_2006_08435_gb300 import Plan
    nz, ny, nx = shape
    x = torch.from_numpy(synth.uniform_grids(shape, 2, seed=sum(shape))).cuda()
    p = Plan(nx, ny, nz, 2, inverse=inverse, norm="ortho")
    y = torch.empty_like(x)
    p.execute(x, y)
    for b in (0, 1):
        ref = oracle.dft3d(x[b].cpu().numpy().astype(np.complex128), 1 if inverse else -1)
        assert oracle.rel_l2(y[b].cpu().numpy(), ref / np.sqrt(nx * ny * nz)) <= TOL
    z = x.clone()
    p.execute(z, z)
    assert torch.equal(z, y)
