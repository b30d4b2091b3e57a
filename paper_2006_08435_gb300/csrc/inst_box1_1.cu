// Pass 1 of the two-pass boxes (twopass_box.cuh), every other edge.
#include "twopass_box.cuh"

namespace fft3d {
BoxKernel box1_kernel_unit1(int nx, int dir) {
  switch (nx) {
    case 36: return tp::box1_entry<36>(dir);
    case 45: return tp::box1_entry<45>(dir);
    case 50: return tp::box1_entry<50>(dir);
    case 60: return tp::box1_entry<60>(dir);
    case 72: return tp::box1_entry<72>(dir);
    case 80: return tp::box1_entry<80>(dir);
    case 90: return tp::box1_entry<90>(dir);
    case 100: return tp::box1_entry<100>(dir);
    case 120: return tp::box1_entry<120>(dir);
    case 128: return tp::box1_entry<128>(dir);
    case 144: return tp::box1_entry<144>(dir);
    case 160: return tp::box1_entry<160>(dir);
    default: return BoxKernel{};
  }
}
}  // namespace fft3d
