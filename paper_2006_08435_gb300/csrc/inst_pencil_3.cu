// Pencil kernels (pencil.cuh) of the plannable edges of rank 3 modulo 8.
#include "pencil.cuh"

namespace fft3d {
PencilKernel pencil_kernel_unit3(int L, int dir, int kind) {
  return pc::unit_kernel<3>(L, dir, kind);
}
}  // namespace fft3d
