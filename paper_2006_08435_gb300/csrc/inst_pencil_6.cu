// Pencil kernels (pencil.cuh) of the plannable edges of rank 6 modulo 8.
#include "pencil.cuh"

namespace fft3d {
PencilKernel pencil_kernel_unit6(int L, int dir, int kind) {
  return pc::unit_kernel<6>(L, dir, kind);
}
}  // namespace fft3d
