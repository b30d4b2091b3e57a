// Lookup and launch of the two-pass box kernels (twopass_box.cuh).
#include "twopass_box.cuh"

namespace fft3d {
BoxKernel box1_kernel_unit0(int, int);
BoxKernel box1_kernel_unit1(int, int);
BoxKernel box2_kernel_a2(int, int);
BoxKernel box2_kernel_a3(int, int);
BoxKernel box2_kernel_a4(int, int);
BoxKernel box2_kernel_a5(int, int);
BoxKernel box2_kernel_a6(int, int);

BoxKernel box1_kernel_info(int nx, int dir) {
  const BoxKernel k = box1_kernel_unit0(nx, dir);
  return k.func ? k : box1_kernel_unit1(nx, dir);
}
BoxKernel box2_kernel_info(int A, int nz, int dir) {
  switch (A) {
    case 2: return box2_kernel_a2(nz, dir);
    case 3: return box2_kernel_a3(nz, dir);
    case 4: return box2_kernel_a4(nz, dir);
    case 5: return box2_kernel_a5(nz, dir);
    case 6: return box2_kernel_a6(nz, dir);
    default: return BoxKernel{};
  }
}
cudaError_t launch_box(const BoxKernel& k, unsigned grid, size_t smem, int cluster,
                       const BoxArgs& a, cudaStream_t s) {
  return tp::launch_dependent(k.func, grid, k.threads, smem, cluster, a, s);
}
}  // namespace fft3d
