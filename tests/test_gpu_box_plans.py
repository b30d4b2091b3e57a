"""Box plans of one nx and several ny alive at once: pass 1 of the two-pass boxes
is one kernel for every ny, so nothing a plan sets on it may take from another.

Bar: 5e-6 relative L2 per grid, the FP32 path's."""
import numpy as np
import pytest
import torch

from oracle import oracle
from paper_2006_08435_gb300 import synth

pytestmark = pytest.mark.gpu

TOL = 5e-6


@pytest.mark.parametrize("inverse", [False, True])
def test_plans_of_one_nx_side_by_side(cuda, inverse):
    from paper_2006_08435_gb300 import Plan
    shapes = [(64, 128, 96), (64, 100, 96)]  # 32 rows per block, then 25
    plans, xs, refs = [], [], []
    for nz, ny, nx in shapes:
        x = synth.uniform_grids((nz, ny, nx), 1, seed=ny)
        refs.append(oracle.dft3d(x[0].astype(np.complex128), 1 if inverse else -1))
        xs.append(torch.from_numpy(x).cuda())
        plans.append(Plan(nx, ny, nz, 1, inverse=inverse))
    for i in (0, 1, 0):
        y = torch.empty_like(xs[i])
        plans[i].execute(xs[i], y)
        assert oracle.rel_l2(y[0].cpu().numpy(), refs[i]) <= TOL
        z = xs[i].clone()
        plans[i].execute(z, z)
        assert torch.equal(z, y)
