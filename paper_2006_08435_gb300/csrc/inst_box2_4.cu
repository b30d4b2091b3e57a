// Pass 2 of the two-pass boxes (twopass_box.cuh), 4 groups.
#include "twopass_box.cuh"

namespace fft3d {
BoxKernel box2_kernel_a4(int nz, int dir) {
  switch (nz) {
    case 32: return tp::box2_entry<4, 32>(dir);
    case 36: return tp::box2_entry<4, 36>(dir);
    case 40: return tp::box2_entry<4, 40>(dir);
    case 45: return tp::box2_entry<4, 45>(dir);
    case 48: return tp::box2_entry<4, 48>(dir);
    case 50: return tp::box2_entry<4, 50>(dir);
    case 54: return tp::box2_entry<4, 54>(dir);
    case 60: return tp::box2_entry<4, 60>(dir);
    case 64: return tp::box2_entry<4, 64>(dir);
    case 72: return tp::box2_entry<4, 72>(dir);
    case 75: return tp::box2_entry<4, 75>(dir);
    case 80: return tp::box2_entry<4, 80>(dir);
    case 81: return tp::box2_entry<4, 81>(dir);
    case 90: return tp::box2_entry<4, 90>(dir);
    case 96: return tp::box2_entry<4, 96>(dir);
    case 100: return tp::box2_entry<4, 100>(dir);
    case 108: return tp::box2_entry<4, 108>(dir);
    case 120: return tp::box2_entry<4, 120>(dir);
    case 125: return tp::box2_entry<4, 125>(dir);
    case 128: return tp::box2_entry<4, 128>(dir);
    case 135: return tp::box2_entry<4, 135>(dir);
    case 144: return tp::box2_entry<4, 144>(dir);
    case 150: return tp::box2_entry<4, 150>(dir);
    case 160: return tp::box2_entry<4, 160>(dir);
    default: return BoxKernel{};
  }
}
}  // namespace fft3d
