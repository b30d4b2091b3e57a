"""Default plans on the general path whose in-place executes run the ticket kernel
(batches where two passes in place are slower): in place the bits are those of a
plan forced to that kernel, out of place those of the general path.  Mixed plans: the
same grids in place and out of place agree within twice the FP32 path's bar."""
import pytest
import torch

pytestmark = pytest.mark.gpu

TOL = 5e-6


def grids(batch, n, seed):
    gen = torch.Generator(device="cuda").manual_seed(seed)
    return torch.randn((batch, n, n, n), dtype=torch.complex64, device="cuda", generator=gen)


@pytest.mark.parametrize("n,batch,ticket", [(32, 163, 13), (32, 240, 13), (80, 55, 13), (128, 13, 6)])
def test_in_place_runs_the_ticket_kernel(cuda, monkeypatch, n, batch, ticket):
    from paper_2006_08435_gb300 import Plan
    x = grids(batch, n, n)
    plan = Plan(n, n, n, batch, norm="ortho")
    assert plan.variant == 10
    forced = {}
    for v in (10, ticket):
        monkeypatch.setenv("FFT3D_VARIANT", str(v))
        forced[v] = Plan(n, n, n, batch, norm="ortho")
        assert forced[v].variant == v
    a, b = torch.empty_like(x), torch.empty_like(x)
    plan.execute(x, a)
    forced[10].execute(x, b)
    assert torch.equal(a, b)
    for _ in range(2):
        a.copy_(x)
        b.copy_(x)
        plan.execute(a, a)
        forced[ticket].execute(b, b)
        assert torch.equal(a, b)
    assert plan.device_status() == 0
    # forced to the general path, in place stays there
    a.copy_(x)
    forced[10].execute(a, a)
    forced[10].execute(x, b)
    assert torch.equal(a, b)


@pytest.mark.parametrize("n,count", [(96, 25), (96, 27), (128, 13)])
def test_mixed_in_place(cuda, n, count):
    from paper_2006_08435_gb300 import MixedPlan
    dims = [16, 64] + [n] * count + [16]
    plan = MixedPlan(dims)
    gen = torch.Generator(device="cuda").manual_seed(count)
    x = torch.randn(plan.total_points, dtype=torch.complex64, device="cuda", generator=gen)
    y, z = torch.empty_like(x), x.clone()
    plan.execute(x, y)
    plan.execute(z, z)
    for g in range(len(dims)):
        a, b = (t[plan.offsets[g]:plan.offsets[g + 1]] for t in (y, z))
        assert torch.linalg.vector_norm(a - b) <= 2 * TOL * torch.linalg.vector_norm(a)
    assert plan.device_status() == 0
