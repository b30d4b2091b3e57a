// Pencil kernels (pencil.cuh) of the plannable edges of rank 7 modulo 8.
#include "pencil.cuh"

namespace fft3d {
PencilKernel pencil_kernel_unit7(int L, int dir, int kind) {
  return pc::unit_kernel<7>(L, dir, kind);
}
}  // namespace fft3d
