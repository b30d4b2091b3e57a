"""The prime-factor register DFTs (csrc/primefactor.cuh), compiled as host code by
nvcc and run on the CPU: every radix of the kernels that use them, forward and
inverse, against numpy.fft in FP64.  The index maps and constants are compile-time,
so a wrong one shows here without a GPU.

Bar: 1e-6 of the largest output, a few FP32 roundings (6e-8 each) over at most
five steps of additions."""
import os
import subprocess

import numpy as np
import pytest

RADICES = [2, 3, 4, 5, 6, 8, 9, 10, 12, 15, 16, 18, 20, 24, 25, 27, 30, 32]

SRC = r"""
#include <cmath>
#include <cstdio>
#include "primefactor.cuh"
using namespace fft3d;

template <int R, int DIR>
void one() {
  float2 v[R];
  for (int n = 0; n < R; ++n)
    v[n] = make_float2((float)std::cos(0.7 * n + 0.3), (float)std::sin(1.3 * n - 0.2));
  pf::transform<R, DIR>(v);
  std::printf("%d %d", R, DIR);
  for (int n = 0; n < R; ++n) std::printf(" %.9e %.9e", v[n].x, v[n].y);
  std::printf("\n");
}
template <int... R>
void all() {
  (one<R, -1>(), ...);
  (one<R, 1>(), ...);
}
int main() {
  all<RADICES>();
  return 0;
}
"""


@pytest.fixture(scope="module")
def output(tmp_path_factory):
    from paper_2006_08435_gb300 import build as B
    cc = B.nvcc()
    if not cc or not os.path.exists(cc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("primefactor")
    src, exe = d / "host.cu", d / "host"
    src.write_text(SRC.replace("RADICES", ", ".join(map(str, RADICES))))
    csrc = os.path.join(os.path.dirname(B.__file__), "csrc")
    subprocess.run([cc, "-std=c++17", "-O2", "-I", csrc, str(src), "-o", str(exe)], check=True,
                   capture_output=True)
    out = subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout
    res = {}
    for line in out.strip().splitlines():
        f = line.split()
        res[int(f[0]), int(f[1])] = np.array(f[2:], dtype=np.float64).view(np.complex128)
    return res


@pytest.mark.parametrize("radix", RADICES)
@pytest.mark.parametrize("sign", [-1, 1])
def test_prime_factor_dft(output, radix, sign):
    n = np.arange(radix)
    v = (np.cos(0.7 * n + 0.3).astype(np.float32) + 1j * np.sin(1.3 * n - 0.2).astype(np.float32))
    ref = np.fft.fft(v) if sign < 0 else np.fft.ifft(v, norm="forward")
    assert np.abs(output[radix, sign] - ref).max() <= 1e-6 * np.abs(ref).max()
