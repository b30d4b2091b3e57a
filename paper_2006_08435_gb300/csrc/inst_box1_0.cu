// Pass 1 of the two-pass boxes (twopass_box.cuh), every other edge.
#include "twopass_box.cuh"

namespace fft3d {
BoxKernel box1_kernel_unit0(int nx, int dir) {
  switch (nx) {
    case 32: return tp::box1_entry<32>(dir);
    case 40: return tp::box1_entry<40>(dir);
    case 48: return tp::box1_entry<48>(dir);
    case 54: return tp::box1_entry<54>(dir);
    case 64: return tp::box1_entry<64>(dir);
    case 75: return tp::box1_entry<75>(dir);
    case 81: return tp::box1_entry<81>(dir);
    case 96: return tp::box1_entry<96>(dir);
    case 108: return tp::box1_entry<108>(dir);
    case 125: return tp::box1_entry<125>(dir);
    case 135: return tp::box1_entry<135>(dir);
    case 150: return tp::box1_entry<150>(dir);
    default: return BoxKernel{};
  }
}
}  // namespace fft3d
