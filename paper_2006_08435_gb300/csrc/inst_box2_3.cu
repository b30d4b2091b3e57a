// Pass 2 of the two-pass boxes (twopass_box.cuh), 3 groups.
#include "twopass_box.cuh"

namespace fft3d {
BoxKernel box2_kernel_a3(int nz, int dir) {
  switch (nz) {
    case 32: return tp::box2_entry<3, 32>(dir);
    case 36: return tp::box2_entry<3, 36>(dir);
    case 40: return tp::box2_entry<3, 40>(dir);
    case 45: return tp::box2_entry<3, 45>(dir);
    case 48: return tp::box2_entry<3, 48>(dir);
    case 50: return tp::box2_entry<3, 50>(dir);
    case 54: return tp::box2_entry<3, 54>(dir);
    case 60: return tp::box2_entry<3, 60>(dir);
    case 64: return tp::box2_entry<3, 64>(dir);
    case 72: return tp::box2_entry<3, 72>(dir);
    case 75: return tp::box2_entry<3, 75>(dir);
    case 80: return tp::box2_entry<3, 80>(dir);
    case 81: return tp::box2_entry<3, 81>(dir);
    case 90: return tp::box2_entry<3, 90>(dir);
    case 96: return tp::box2_entry<3, 96>(dir);
    case 100: return tp::box2_entry<3, 100>(dir);
    case 108: return tp::box2_entry<3, 108>(dir);
    case 120: return tp::box2_entry<3, 120>(dir);
    case 125: return tp::box2_entry<3, 125>(dir);
    case 128: return tp::box2_entry<3, 128>(dir);
    case 135: return tp::box2_entry<3, 135>(dir);
    case 144: return tp::box2_entry<3, 144>(dir);
    case 150: return tp::box2_entry<3, 150>(dir);
    case 160: return tp::box2_entry<3, 160>(dir);
    default: return BoxKernel{};
  }
}
}  // namespace fft3d
