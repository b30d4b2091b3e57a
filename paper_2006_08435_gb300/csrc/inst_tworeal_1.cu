// Two-pass real transforms (twopass_real.cuh), every other edge.
#include "twopass_real.cuh"

namespace fft3d {
RealPassKernel real_pass_kernel_unit1(int n, int dir) {
  switch (n) {
    case 60: return tpr::entry<60>(dir);
    case 72: return tpr::entry<72>(dir);
    case 90: return tpr::entry<90>(dir);
    case 100: return tpr::entry<100>(dir);
    case 120: return tpr::entry<120>(dir);
    default: return RealPassKernel{};
  }
}
}  // namespace fft3d
