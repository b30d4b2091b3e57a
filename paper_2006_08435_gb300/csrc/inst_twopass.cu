// The two-pass kernels (twopass.cuh).
#include "twopass.cuh"

namespace fft3d {
TwoPassKernel two_pass_kernel_info(int L, int dir) {
  switch (L) {
    case 128: return tp::entry_of<128>(dir);
    case 100: return tp::entry_of<100>(dir);
    case 96: return tp::entry_of<96>(dir);
    case 80: return tp::entry_of<80>(dir);
    case 64: return tp::entry_of<64>(dir);
    case 108: return tp::entry_of<108>(dir);
    case 90: return tp::entry_of<90>(dir);
    case 72: return tp::entry_of<72>(dir);
    case 60: return tp::entry_of<60>(dir);
    case 48: return tp::entry_of<48>(dir);
    default: return TwoPassKernel{};
  }
}
}  // namespace fft3d
