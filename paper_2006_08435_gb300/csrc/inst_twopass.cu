// The two-pass kernels (twopass.cuh) on packed batches.
#include "twopass.cuh"

namespace fft3d {
TwoPassKernel two_pass_kernel_info(int L, int dir) {
  switch (L) {
    case 128: return tp::entry_of<128, false>(dir);
    case 108: return tp::entry_of<108, false>(dir);
    case 100: return tp::entry_of<100, false>(dir);
    case 96: return tp::entry_of<96, false>(dir);
    case 90: return tp::entry_of<90, false>(dir);
    case 80: return tp::entry_of<80, false>(dir);
    case 72: return tp::entry_of<72, false>(dir);
    case 64: return tp::entry_of<64, false>(dir);
    case 60: return tp::entry_of<60, false>(dir);
    case 48: return tp::entry_of<48, false>(dir);
    default: return TwoPassKernel{};
  }
}
}  // namespace fft3d
