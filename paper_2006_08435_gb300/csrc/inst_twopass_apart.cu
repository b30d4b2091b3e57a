// The two-pass kernels (twopass.cuh) on the grids of mixed-edge plans.
#include "twopass.cuh"

namespace fft3d {
TwoPassKernel two_pass_apart_kernel_info(int L, int dir) {
  switch (L) {
    case 128: return tp::entry_of<128, true>(dir);
    case 96: return tp::entry_of<96, true>(dir);
    case 80: return tp::entry_of<80, true>(dir);
    case 64: return tp::entry_of<64, true>(dir);
    case 48: return tp::entry_of<48, true>(dir);
    default: return TwoPassKernel{};
  }
}
}  // namespace fft3d
