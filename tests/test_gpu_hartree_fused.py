"""The Hartree gradient in one weighted inverse transform against its two steps
(seed kernel, inverse transform), which it repeats operation by operation: the
same bits, for every family of real kernels, batches above and below one chunk,
and a spectrum whose m = 0 bin is not finite (it has weight 0)."""
import pytest
import torch

pytestmark = pytest.mark.gpu


@pytest.mark.parametrize("n,batch", [(16, 5), (32, 3), (64, 4), (128, 3), (10, 2), (48, 70), (90, 3),
                                     (96, 14), (100, 1), (216, 1)])
def test_weighted_inverse_is_seed_then_inverse(cuda, n, batch):
    from paper_2006_08435_gb300 import irfft3d
    from paper_2006_08435_gb300.hartree import gradient_from_half_spectrum, seed_from_half_spectrum
    gen = torch.Generator(device="cuda").manual_seed(n)
    f = torch.randn((batch, n, n, n // 2 + 1), dtype=torch.complex64, device="cuda", generator=gen)
    f[0, 0, 0, 0] = complex(float("inf"), float("nan"))
    g = torch.randn(batch, dtype=torch.float64, device="cuda", generator=gen)
    keep = f.clone()
    got = gradient_from_half_spectrum(f, 9.5, g)
    ref = irfft3d(seed_from_half_spectrum(f, 9.5, g))
    assert torch.isfinite(ref).all()
    assert torch.equal(got, ref)
    assert torch.equal(torch.view_as_real(f)[1:], torch.view_as_real(keep)[1:])


def test_weighted_inverse_rejects_other_plans(cuda):
    from paper_2006_08435_gb300 import RealPlan
    from paper_2006_08435_gb300 import _lib as L
    n = 64
    f = torch.zeros((1, n, n, n // 2 + 1), dtype=torch.complex64, device="cuda")
    out = torch.empty((1, n, n, n), device="cuda")
    g = torch.ones(1, dtype=torch.float64, device="cuda")

    def call(plan, cell=10.0):
        return L.lib().fft3d_real_execute_hartree(plan._h, f.data_ptr(), cell, g.data_ptr(),
                                                  out.data_ptr(), 0)
    assert call(RealPlan(n, 1)) == L.FFT3D_ERR_INVALID_ARG
    assert call(RealPlan(n, 1, inverse=True, norm="by_n")) == L.FFT3D_ERR_INVALID_ARG
    assert call(RealPlan(n, 1, inverse=True), 0.0) == L.FFT3D_ERR_INVALID_ARG
    assert call(RealPlan(n, 1, precision="split_fp16", inverse=True)) == \
        L.FFT3D_ERR_UNSUPPORTED_PRECISION
