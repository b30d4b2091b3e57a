"""The pencil passes' building blocks without a GPU: the register transforms
of their steps, and the two-step split of every plannable edge, compiled as host
code from the kernels' own headers and compared with numpy.fft."""
import os
import subprocess

import numpy as np
import pytest

RADICES = [16, 18, 20, 24, 25, 27, 30, 32]

SRC = r"""
#include <cmath>
#include <cstdio>
#include "pencil.cuh"
using namespace fft3d;

template <int R, int DIR>
void one() {
  float2 v[R];
  for (int n = 0; n < R; ++n)
    v[n] = make_float2((float)std::cos(0.7 * n + 0.3), (float)std::sin(1.3 * n - 0.2));
  pc::transform<R, DIR>(v);
  std::printf("dft %d %d", R, DIR);
  for (int n = 0; n < R; ++n) std::printf(" %.9e %.9e", v[n].x, v[n].y);
  std::printf("\n");
}
template <int R>
void both() {
  one<R, -1>();
  one<R, 1>();
}
int main() {
  both<16>(); both<18>(); both<20>(); both<24>(); both<25>(); both<27>(); both<30>(); both<32>();
  for (int n = 0; n <= kAxisMaxLen + 1; ++n)
    if (pc::smooth(n))
      std::printf("split %d %d %d %d\n", n, pc::split_a(n, pc::kStrided), pc::split_a(n, pc::kContig),
                  (int)(pc::codelet(n / pc::split_a(n, pc::kStrided)) &&
                        pc::codelet(n / pc::split_a(n, pc::kContig)) &&
                        pc::codelet(pc::split_a(n, pc::kStrided)) &&
                        pc::codelet(pc::split_a(n, pc::kContig))));
  return 0;
}
"""


@pytest.fixture(scope="module")
def host_output(tmp_path_factory):
    from paper_2006_08435_gb300 import build as B
    cc = B.nvcc()
    if not cc or not os.path.exists(cc):
        pytest.skip("nvcc not available")
    d = tmp_path_factory.mktemp("pencil")
    src = d / "pencil_host.cu"
    exe = d / "pencil_host"
    src.write_text(SRC)
    csrc = os.path.join(os.path.dirname(B.__file__), "csrc")
    inc = os.path.join(os.path.dirname(os.path.dirname(B.__file__)), "include")
    subprocess.run([cc, "-std=c++17", "-O2", "--expt-relaxed-constexpr", "-gencode",
                    "arch=compute_103a,code=sm_103a", "-I", csrc, "-I", inc, str(src), "-o",
                    str(exe)], check=True, capture_output=True)
    return subprocess.run([str(exe)], check=True, capture_output=True, text=True).stdout


def test_transforms_of_the_steps(host_output):
    seen = 0
    for line in host_output.splitlines():
        f = line.split()
        if f[0] != "dft":
            continue
        r, sign = int(f[1]), int(f[2])
        vals = np.array([float(t) for t in f[3:]]).reshape(r, 2)
        n = np.arange(r)
        x = np.cos(0.7 * n + 0.3).astype(np.float32).astype(np.float64) + \
            1j * np.sin(1.3 * n - 0.2).astype(np.float32).astype(np.float64)
        ref = np.fft.fft(x) if sign < 0 else np.fft.ifft(x) * r
        got = vals[:, 0] + 1j * vals[:, 1]
        assert np.linalg.norm(got - ref) / np.linalg.norm(ref) <= 1e-6, (r, sign)
        seen += 1
    assert seen == 2 * len(RADICES)


def test_every_plannable_edge_splits_into_two_steps(host_output):
    edges = []
    for line in host_output.splitlines():
        f = line.split()
        if f[0] != "split":
            continue
        n, a, c, ok = (int(t) for t in f[1:])
        assert a >= 1 and c >= 1 and n % a == 0 and n % c == 0 and ok == 1, line
        edges.append(n)
    want = sorted(2 ** a * 3 ** b * 5 ** c for a in range(10) for b in range(6) for c in range(4)
                  if 2 <= 2 ** a * 3 ** b * 5 ** c <= 512)
    assert [e for e in edges if e <= 512] == want
