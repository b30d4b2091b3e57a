// The two-pass transform (twopass.cuh) of boxes nx x ny x nz: pass 1 compiled
// per nx, with the points B per thread of its y step chosen at run time, pass 2
// per (A, nz), ny = A B.  Packed batches; in place with clusters of A blocks.
// What bounds it and why the steps are split as they are: see twopass.cuh.
// GB300, us, two passes / three: 96 x 128 x 64, 64 grids 215 / 264; 128 x 96 x
// 80 x 16 78 / 88; 75^3 x 20 46 / 59; 135 x 128 x 90 x 4 33.5 / 42; 120^3 x 16 143 /
// 190 (two passes with tiles of 16 columns of one row k2).
#pragma once

#include "twopass.cuh"

namespace fft3d {
namespace tp {

// x: AX points apart in the first step (AX lanes of a warp read one run), the
// first of the order whose partner is a codelet too; 10 .. 16 before more, which
// leaves the first step too few points (90 x 90 x 90 x 38 by 18 / 15: 174 / 150 us).
constexpr int box_ax(int L) {
  const int order[] = {16, 15, 12, 10, 20, 18, 24, 25, 27, 30, 32, 9, 8};
  for (int a : order)
    if (L % a == 0 && L / a >= 2 && L / a <= 16 && pc::codelet(L / a)) return a;
  return 0;
}
// z: AZ points of each of the A rows in one thread's second step, at most 36
// in all, and at most 20 in the first step (54 x 81 x 125 with 25: slower than
// three passes).
constexpr int box_az(int A, int L) {
  for (int az = 2; az * A <= 36; ++az)
    if (L % az == 0 && pc::codelet(az) && pc::codelet(L / az) && L / az <= 20) return az;
  return 0;
}

template <int LX>
struct BoxX {
  static constexpr int AX = box_ax(LX), BX = LX / AX;
  static constexpr Layout rows = row_layout(32, AX, BX, LX);  // (any number of rows)
  static constexpr int PD = rows.PD, RP = rows.RP;
  static_assert(sizeof(float2) * 32 * RP <= 48 * 1024, "32 rows within the default limit");
  static constexpr int T = LX <= 64 ? 64 : (LX + 31) / 32 * 32;
  // threads for 32 rows, whose shared memory leaves few blocks: a warp more where
  // that keeps the lanes of the first step busy (96 x 128 x 64 x 64 231 -> 213 us,
  // 60 x 128 x 72 x 40 119 -> 107, 90 x 128 x 96 x 20 123 -> 112; not for 64 x 128 x 64 x
  // 40, a ninth of them idle, 96 -> 99, nor for fewer rows, 108 x 96 x 100 104 -> 110)
  // and BX is even (odd, 80 x 128 x 64 x 40 117 -> 120, 125 x 128 x 96 x 10 80 -> 85)
  static constexpr int T32 =
      AX >= 15 && BX % 2 == 0 && (32 * AX + T + 31) / (T + 32) * (T + 32) * 10 <= 32 * AX * 11 ? T + 32 : T;
};
constexpr int kBoxW = 16;  // columns of a pass-2 block
template <int A, int LZ>
struct BoxZ {
  static constexpr int AZ = box_az(A, LZ), BZ = LZ / AZ, W = kBoxW;
  static constexpr bool uniform = W * A % 32 == 0;
  static constexpr int ZR = AZ * A * W, ZP = ZR;  // W = 16: a half-warp is one row
  static constexpr int T = (W * BZ + 31) / 32 * 32;
  static constexpr size_t smem = sizeof(float2) * (size_t)BZ * ZP;
};

// y step of pass 1 for one column: x[j * RP], j < B.
template <int B, int DIR>
__device__ __forceinline__ void box_y(const float2* x, int RP, float2* o, int nx, const float2* ty,
                                      int A, int n1, uint64_t pol) {
  float2 v[B];
#pragma unroll
  for (int j = 0; j < B; ++j) v[j] = x[j * RP];
  pc::transform<B, DIR>(v);
#pragma unroll
  for (int k = 0; k < B; ++k) stg(o + k * nx, k ? twiddle<DIR>(v[k], ty[k * A + n1]) : v[k], pol);
}

template <int LX, int DIR>
__global__ void __launch_bounds__(BoxX<LX>::T32) box1_kernel(const __grid_constant__ BoxArgs a) {
  using D = BoxX<LX>;
  constexpr int AX = D::AX, BX = D::BX;
  const int T = blockDim.x;  // D::T or D::T32
  extern __shared__ __align__(16) float2 sm[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int A = a.A, B = a.B;
  const unsigned zz = pc::fdiv(blockIdx.x, a.divA);  // plane
  const int n1 = (int)(blockIdx.x - zz * A);
  const uint64_t once = l2_policy(kEvictFirst), keep = l2_policy(kEvictLast);
  const size_t plane = (size_t)zz * A * B * LX;
  const float2* src = a.in + plane + (size_t)n1 * LX;
  float2* dst = a.out + plane + (size_t)n1 * B * LX;
  asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll 1
  for (int e = threadIdx.x; e < B * AX; e += T) {
    const int j = e / AX, m = e % AX;
    const float2* s = src + j * A * LX + m;
    float2 v[BX];
#pragma unroll
    for (int i = 0; i < BX; ++i) v[i] = ldg(s + AX * i, once);
    pc::transform<BX, DIR>(v);
    float2* x = sm + j * D::RP;
#pragma unroll
    for (int k = 0; k < BX; ++k) x[slot(D::PD, BX * m + k)] = k ? twiddle<DIR>(v[k], __ldg(a.tx + k * AX + m)) : v[k];
  }
  if (a.in_place) {  // the cluster's A blocks read and write the same plane
    __syncwarp();
    asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");
  }
  __syncthreads();
#pragma unroll 1
  for (int e = threadIdx.x; e < B * BX; e += T) {
    const int k = (int)pc::fdiv((unsigned)e, a.divB);
    float2* x = sm + (e - k * B) * D::RP;
    float2 v[AX];
#pragma unroll
    for (int i = 0; i < AX; ++i) v[i] = x[slot(D::PD, BX * i + k)];
    pc::transform<AX, DIR>(v);
#pragma unroll
    for (int i = 0; i < AX; ++i) x[slot(D::PD, BX * i + k)] = v[i];
  }
  if (a.in_place) {
    __syncwarp();
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  }
  __syncthreads();
  const int kx = threadIdx.x;
  if (kx < LX) {
    const float2* x = sm + slot(D::PD, kx);
    float2* o = dst + kx;
    switch (B) {
      case 10: box_y<10, DIR>(x, D::RP, o, LX, a.ty, A, n1, keep); break;
      case 12: box_y<12, DIR>(x, D::RP, o, LX, a.ty, A, n1, keep); break;
      case 15: box_y<15, DIR>(x, D::RP, o, LX, a.ty, A, n1, keep); break;
      case 16: box_y<16, DIR>(x, D::RP, o, LX, a.ty, A, n1, keep); break;
      case 18: box_y<18, DIR>(x, D::RP, o, LX, a.ty, A, n1, keep); break;
      case 20: box_y<20, DIR>(x, D::RP, o, LX, a.ty, A, n1, keep); break;
      case 24: box_y<24, DIR>(x, D::RP, o, LX, a.ty, A, n1, keep); break;
      case 25: box_y<25, DIR>(x, D::RP, o, LX, a.ty, A, n1, keep); break;
      case 27: box_y<27, DIR>(x, D::RP, o, LX, a.ty, A, n1, keep); break;
      case 30: box_y<30, DIR>(x, D::RP, o, LX, a.ty, A, n1, keep); break;
      case 32: box_y<32, DIR>(x, D::RP, o, LX, a.ty, A, n1, keep); break;
      default: break;
    }
  }
}

template <int A, int LZ, int DIR>
__global__ void __launch_bounds__(BoxZ<A, LZ>::T) box2_kernel(const __grid_constant__ BoxArgs a) {
  using D = BoxZ<A, LZ>;
  constexpr int AZ = D::AZ, BZ = D::BZ, W = D::W, T = D::T;
  extern __shared__ __align__(16) float2 sm[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const int nc = a.B * a.nx;  // columns (k2, x) of a group
  const unsigned g = pc::fdiv(blockIdx.x, a.divt);
  const int c0 = (int)(blockIdx.x - g * a.tiles) * W, cols = min(W, nc - c0);
  const uint64_t once = l2_policy(kEvictFirst);
  const long long pl = (long long)A * nc;
  float2* base = a.out + (long long)g * pl * LZ + c0;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  constexpr int N1 = W * A * AZ;
#pragma unroll 1
  for (int it = 0; it < (N1 + T - 1) / T; ++it) {
    const int e = threadIdx.x + it * T;
    if (N1 % T && e >= N1) break;
    const int q = e % W, n1 = e / W % A;
    int m1 = e / (W * A);
    if constexpr (D::uniform) m1 = __shfl_sync(0xffffffffu, m1, 0);
    if (q >= cols) continue;
    const float2* s = base + m1 * pl + n1 * nc + q;
    float2 v[BZ];
#pragma unroll
    for (int i = 0; i < BZ; ++i) v[i] = ldg(s + (long long)(AZ * i) * pl, once);
    pc::transform<BZ, DIR>(v);
    float2* x = sm + (m1 * A + n1) * W + q;
#pragma unroll
    for (int k = 0; k < BZ; ++k) {
      const float2 w = D::uniform ? a.tz[k * AZ + m1] : __ldg(a.tzg + k * AZ + m1);
      x[k * D::ZP] = k ? twiddle<DIR>(v[k], w) : v[k];
    }
  }
  __syncthreads();
  const int q = threadIdx.x % W, kz2 = threadIdx.x / W;
  if (kz2 < BZ && q < cols) {
    const float2* x = sm + kz2 * D::ZP + q;
    float2 v[A][AZ];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) {
#pragma unroll
      for (int m = 0; m < AZ; ++m) v[n1][m] = x[(m * A + n1) * W];
      pc::transform<AZ, DIR>(v[n1]);
    }
    float2* o = base + kz2 * pl + q;
#pragma unroll
    for (int k = 0; k < AZ; ++k) {
      float2 u[A];
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) u[n1] = v[n1][k];
      pc::transform<A, DIR>(u);
#pragma unroll
      for (int k1 = 0; k1 < A; ++k1)
        stg(o + (long long)(BZ * k) * pl + k1 * nc, a.do_scale ? cscale(u[k1], a.scale) : u[k1],
            once);
    }
  }
}

inline cudaError_t launch_dependent(const void* fn, unsigned grid, int threads, size_t smem,
                                    int cluster, const BoxArgs& a, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  cfg.stream = s;
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  void* args[] = {const_cast<BoxArgs*>(&a)};
  return cudaLaunchKernelExC(&cfg, fn, args);
}

template <int LX>
BoxKernel box1_entry(int dir) {
  using D = BoxX<LX>;
  return BoxKernel{dir < 0 ? (const void*)&box1_kernel<LX, -1> : (const void*)&box1_kernel<LX, 1>,
                   D::T, sizeof(float2) * (size_t)D::RP, D::AX, D::T32};
}
template <int A, int LZ>
BoxKernel box2_entry(int dir) {
  if constexpr (box_az(A, LZ) != 0) {
    using D = BoxZ<A, LZ>;
    if constexpr (D::smem <= 72 * 1024)  // three blocks per multiprocessor
      return BoxKernel{dir < 0 ? (const void*)&box2_kernel<A, LZ, -1> : (const void*)&box2_kernel<A, LZ, 1>,
                       D::T, D::smem, D::AZ};
  }
  return BoxKernel{};
}

}  // namespace tp
}  // namespace fft3d
