// Two-pass real transforms (twopass_real.cuh), every other edge.
#include "twopass_real.cuh"

namespace fft3d {
RealPassKernel real_pass_kernel_unit1(int n, int dir);

RealPassKernel real_pass_kernel_info(int n, int dir) {
  switch (n) {
    case 48: return tpr::entry<48>(dir);
    case 64: return tpr::entry<64>(dir);
    case 80: return tpr::entry<80>(dir);
    case 96: return tpr::entry<96>(dir);
    case 108: return tpr::entry<108>(dir);
    case 128: return tpr::entry<128>(dir);
    default: return real_pass_kernel_unit1(n, dir);
  }
}
}  // namespace fft3d
