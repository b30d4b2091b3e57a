"""Real plans refuse what their batch of complex grids would: more than 2^40 points
in all (two grids to a complex one), before the GPU is touched."""
import ctypes

import pytest

from paper_2006_08435_gb300 import _lib as L


@pytest.mark.parametrize("n,batch", [(100, 1 << 24), (480, 1 << 24), (512, 1 << 15)])
@pytest.mark.parametrize("direction", [L.FFT3D_FORWARD, L.FFT3D_INVERSE])
def test_too_many_points(fft3d_lib, n, batch, direction):
    h = ctypes.c_void_p()
    rc = fft3d_lib.fft3d_real_plan_create(n, batch, L.FFT3D_FP32, direction, L.FFT3D_NORM_NONE,
                                          ctypes.byref(h))
    assert rc == L.FFT3D_ERR_INVALID_ARG and not h.value


@pytest.mark.parametrize("n,batch", [(100, 1 << 24), (512, 1 << 15)])
def test_too_many_points_fixed(fft3d_lib, n, batch):
    h = ctypes.c_void_p()
    rc = fft3d_lib.fft3d_real_plan_create_fixed(n, batch, ctypes.byref(h))
    assert rc == L.FFT3D_ERR_INVALID_ARG and not h.value


@pytest.mark.parametrize("n,batch,code", [(64, 1, L.FFT3D_ERR_UNSUPPORTED_SIZE),   # a fused edge
                                          (7, 1, L.FFT3D_ERR_UNSUPPORTED_SIZE),
                                          (75, 0, L.FFT3D_ERR_INVALID_ARG),
                                          (405, 1 << 15, L.FFT3D_ERR_INVALID_ARG)])
def test_fixed_complex_plans_validate_before_device(fft3d_lib, n, batch, code):
    h = ctypes.c_void_p()
    assert fft3d_lib.fft3d_plan_create_fixed(n, batch, ctypes.byref(h)) == code and not h.value
