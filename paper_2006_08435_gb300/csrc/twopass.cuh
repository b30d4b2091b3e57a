// A cubic L^3 transform in two passes of small blocks, for the edges whose
// y axis splits into A groups that one thread can hold (see Cfg).
//
// With y = n1 + A j and ky = k2 + B k1 (L = A B, A small):
//   pass 1, block (grid, z, n1): the B rows y = n1 + A j: x transform (two
//     register steps with one exchange in shared memory), then per column the
//     B-point DFT over j in one thread, times W_L^(n1 k2), stored to row
//     k2 + B n1 of plane z;
//   pass 2, block (grid, k2, W columns): the rows k2 + B n1 of every z: first
//     step of the z transform from global memory to shared memory, then one
//     thread per (column, kz2) holds its points of all A rows, finishes the z
//     transforms and the A-point DFT over n1, and stores rows k2 + B k1, the
//     same rows it read.
// A grid crosses L2 twice (32 bytes per point; the separate passes of
// pencil.cuh 48), which with HBM's own fills and write-backs is what bounds
// both: 48 and 64 bytes per point at the 13.8 TB/s that a copy from and to HBM
// reaches there (64^3 x 256: 233 us; measured 283).  The rest is L1: wavefronts
// of short runs and of bank conflicts.  Hence at least 16 lanes along x in the
// first step of pass 1 (AX; 128^3 x 32 with 8 columns and 8 lanes 434 us, with 16
// and 16 338), W >= 16 columns in pass 2, pitches searched at compile time for
// the three access patterns of pass 1, and twiddles that are the same for a
// whole warp read from the kernel's parameters (constant bank).  Splits per
// edge from a sweep; the next best lies 1-5% behind.  Measured, us, two passes /
// three: 64^3 x 12 16.8 / 21.5, x 64 74.6 / 90.3; 96^3 x 8 33.6 / 44.2; 128^3 x 2
// 23.6 / 27.5, x 8 78.7 / 92.7; 100^3 x 16 86 / 94; 60^3 x 80 89 / 98.  At 120, 144
// and 160 no split gains more than the tiles' size costs.
//
// In place, the A blocks of a plane read rows that the others write: they run
// as a cluster and store after a cluster barrier behind everybody's loads.
#pragma once

#include <cuda_runtime.h>

#include "codelets.cuh"
#include "internal.h"
#include "pencil.cuh"

namespace fft3d {
namespace tp {

using pc::l2_policy;
using pc::ldg;
using pc::stg;
using pc::transform;
using pc::twiddle;

// Splits of an edge: y into A groups of B; x and z into two register steps,
// BX (BZ) points first, AX (AZ) apart, then AX (AZ); W columns in pass 2.
template <int L>
struct Cfg;
#define FFT3D_TP(L_, A_, AX_, AZ_, W_)                                  \
  template <>                                                           \
  struct Cfg<L_> {                                                      \
    static constexpr int L = L_, A = A_, B = L_ / A_;                   \
    static constexpr int AX = AX_, BX = L_ / AX_, AZ = AZ_, BZ = L_ / AZ_; \
    static constexpr int W = W_;                                        \
  };
FFT3D_TP(48, 3, 16, 4, 16)
FFT3D_TP(60, 3, 20, 6, 20)
FFT3D_TP(64, 4, 16, 4, 16)
FFT3D_TP(72, 3, 24, 6, 24)
FFT3D_TP(80, 4, 16, 8, 16)
FFT3D_TP(90, 3, 18, 9, 18)
FFT3D_TP(96, 4, 16, 8, 16)
FFT3D_TP(100, 4, 20, 5, 20)
FFT3D_TP(108, 6, 18, 6, 18)
FFT3D_TP(128, 4, 16, 8, 16)
#undef FFT3D_TP

// Bank conflicts (extra wavefronts per half-warp of 8-byte accesses) of the
// three access patterns of pass 1 for slots (row j, k2, m) at j RP + k2 AP + m.
constexpr int conflicts(int AX, int BX, int L, int AP, int RP) {
  int total = 0;
  for (int pat = 0; pat < 3; ++pat)
    for (int h = 0; h < 4; ++h) {
      int n[16] = {}, worst = 0;
      for (int l = 0; l < 16; ++l) {
        const int e = h * 16 + l;
        const int at = pat == 0 ? e / AX * RP + e % AX
                     : pat == 1 ? e / BX * RP + e % BX * AP
                                : e % L % BX * AP + e % L / BX;
        const int c = ++n[at % 16];
        worst = c > worst ? c : worst;
      }
      total += worst - 1;
    }
  return total;
}
struct Pitch {
  int AP, RP;
};
constexpr Pitch best_pitch(int AX, int BX, int L) {
  Pitch best{AX, AX * BX};
  int least = 1 << 20;
  for (int ap = AX; ap < AX + 4; ++ap)
    for (int rp = ap * BX; rp < ap * BX + 16; ++rp) {
      const int c = 64 * conflicts(AX, BX, L, ap, rp) + rp - AX * BX;
      if (c < least) {
        least = c;
        best = Pitch{ap, rp};
      }
    }
  return best;
}

template <int L>
struct Dims : Cfg<L> {
  using C = Cfg<L>;
  // pass 1: row j at j * RP, point (k2, n1) of it at k2 * AP + n1
  static constexpr Pitch pitch = best_pitch(C::AX, C::BX, L);
  static constexpr int AP = pitch.AP, RP = pitch.RP;
  static constexpr int T1 = (L + 31) / 32 * 32;
  static constexpr size_t smem1 = sizeof(float2) * (size_t)C::B * RP;
  // pass 2: point (kz2, m1, n1) of column q at kz2 * ZP + (m1 * A + n1) * W + q
  static constexpr bool uniform = C::W * C::A % 32 == 0;  // m1 the same for a warp
  static constexpr int ZR = C::AZ * C::A * C::W;
  static constexpr int ZP = ZR % 16 == 0 ? ZR + 8 : ZR;
  static constexpr int T2 = (C::W * C::BZ + 31) / 32 * 32;
  static constexpr size_t smem2 = sizeof(float2) * (size_t)C::BZ * ZP;
};

// Where grid g of a launch lies (plan data first: it may be read before the
// launch it depends on is done; the callers' pointer arrays may not).
template <bool APART>
struct GridAt {
  size_t off;
  int pg;
  __device__ __forceinline__ GridAt(const TwoPassArgs& a, unsigned g, size_t points)
      : off(g * points), pg(0) {
    if constexpr (APART) {
      pg = a.first + (int)g;
      if (a.map) pg = a.map[pg];
      off = (size_t)a.off[pg];
    }
  }
  __device__ __forceinline__ const float2* in(const TwoPassArgs& a) const {
    return APART && a.in_ptrs ? a.in_ptrs[pg] : a.in + off;
  }
  __device__ __forceinline__ float2* out(const TwoPassArgs& a) const {
    return APART && a.out_ptrs ? a.out_ptrs[pg] : a.out + off;
  }
};

template <int L, int DIR, bool INPLACE, bool APART>
__global__ void __launch_bounds__(Dims<L>::T1) pass1_kernel(const __grid_constant__ TwoPassArgs a) {
  using D = Dims<L>;
  constexpr int A = D::A, B = D::B, AX = D::AX, BX = D::BX, T = D::T1;
  extern __shared__ __align__(16) float2 sm[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const unsigned zz = blockIdx.x / A, g = zz / L;  // plane, grid
  const int n1 = (int)(blockIdx.x - zz * A);
  const uint64_t once = l2_policy(kEvictFirst), keep = l2_policy(kEvictLast);
  const GridAt<APART> at(a, g, (size_t)L * L * L);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  const size_t plane = (size_t)(zz - g * L) * L * L;
  const float2* src = at.in(a) + plane + (size_t)n1 * L;
  float2* dst = at.out(a) + plane + (size_t)n1 * B * L;
  // x, first step: item (row j, m) -> points m + AX i
  constexpr int N1 = B * AX;
#pragma unroll 1
  for (int it = 0; it < (N1 + T - 1) / T; ++it) {
    const int e = threadIdx.x + it * T;
    if (N1 % T && e >= N1) break;
    const int j = e / AX, m = e % AX;
    const float2* s = src + j * (A * L) + m;
    float2 v[BX];
#pragma unroll
    for (int i = 0; i < BX; ++i) v[i] = ldg(s + AX * i, once);
    transform<BX, DIR>(v);
    float2* x = sm + j * D::RP + m;
#pragma unroll
    for (int k = 0; k < BX; ++k)
      x[k * D::AP] = k ? twiddle<DIR>(v[k], __ldg(a.tx + k * AX + m)) : v[k];
  }
  if constexpr (INPLACE) {
    // the cluster's A blocks read and write the same plane
    __syncwarp();
    asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");
  }
  __syncthreads();
  // x, second step, in place: item (row j, k2)
  constexpr int N2 = B * BX;
#pragma unroll 1
  for (int it = 0; it < (N2 + T - 1) / T; ++it) {
    const int e = threadIdx.x + it * T;
    if (N2 % T && e >= N2) break;
    float2* x = sm + e / BX * D::RP + e % BX * D::AP;
    float2 v[AX];
#pragma unroll
    for (int i = 0; i < AX; ++i) v[i] = x[i];
    transform<AX, DIR>(v);
#pragma unroll
    for (int i = 0; i < AX; ++i) x[i] = v[i];
  }
  if constexpr (INPLACE) {
    __syncwarp();
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  }
  __syncthreads();
  // y: column kx = k2 + BX k1, its B points of this group
  if (threadIdx.x < L) {
    const int kx = threadIdx.x;
    const float2* x = sm + kx % BX * D::AP + kx / BX;
    float2 v[B];
#pragma unroll
    for (int j = 0; j < B; ++j) v[j] = x[j * D::RP];
    transform<B, DIR>(v);
    float2* o = dst + kx;
#pragma unroll
    for (int k = 0; k < B; ++k)
      stg(o + k * L, k ? twiddle<DIR>(v[k], a.ty[k * A + n1]) : v[k], keep);
  }
}

template <int L, int DIR, bool APART>
__global__ void __launch_bounds__(Dims<L>::T2) pass2_kernel(const __grid_constant__ TwoPassArgs a) {
  using D = Dims<L>;
  constexpr int A = D::A, B = D::B, AZ = D::AZ, BZ = D::BZ, W = D::W, T = D::T2;
  constexpr long long LL = (long long)L * L;
  extern __shared__ __align__(16) float2 sm[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const unsigned xt = blockIdx.x % (L / W), r = blockIdx.x / (L / W);
  const unsigned k2 = r % B, g = r / B;
  const uint64_t once = l2_policy(kEvictFirst);
  const GridAt<APART> at(a, g, (size_t)LL * L);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  float2* base = at.out(a) + (long long)k2 * L + xt * W;
  // z, first step: item (m1, n1, q) -> planes m1 + AZ i
  constexpr int N1 = W * A * AZ;
#pragma unroll 1
  for (int it = 0; it < (N1 + T - 1) / T; ++it) {
    const int e = threadIdx.x + it * T;
    if (N1 % T && e >= N1) break;
    const int q = e % W, n1 = e / W % A;
    const int m1 = D::uniform ? __shfl_sync(0xffffffffu, e / (W * A), 0) : e / (W * A);
    const float2* s = base + m1 * LL + n1 * (B * L) + q;
    float2 v[BZ];
#pragma unroll
    for (int i = 0; i < BZ; ++i) v[i] = ldg(s + (long long)(AZ * i) * LL, once);
    transform<BZ, DIR>(v);
    float2* x = sm + (m1 * A + n1) * W + q;
#pragma unroll
    for (int k = 0; k < BZ; ++k)
      x[k * D::ZP] = k ? twiddle<DIR>(v[k], (D::uniform ? a.tz[k * AZ + m1] : __ldg(a.tzg + k * AZ + m1))) : v[k];
  }
  __syncthreads();
  // z, second step, and y: item (kz2, q)
  constexpr int N2 = W * BZ;
  const int e = threadIdx.x;
  if (N2 % T == 0 || e < N2) {
    const int q = e % W, kz2 = e / W;
    const float2* x = sm + kz2 * D::ZP + q;
    float2 v[A][AZ];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) {
#pragma unroll
      for (int m = 0; m < AZ; ++m) v[n1][m] = x[(m * A + n1) * W];
      transform<AZ, DIR>(v[n1]);
    }
    float2* o = base + kz2 * LL + q;
#pragma unroll
    for (int k = 0; k < AZ; ++k) {
      float2 u[A];
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) u[n1] = v[n1][k];
      transform<A, DIR>(u);
#pragma unroll
      for (int k1 = 0; k1 < A; ++k1)
        stg(o + (long long)(BZ * k) * LL + k1 * (B * L), a.do_scale ? cscale(u[k1], a.scale) : u[k1],
            once);
    }
  }
}

template <int L, int DIR, bool APART>
cudaError_t launch(const TwoPassArgs& a, int grids, bool in_place, cudaStream_t s) {
  using D = Dims<L>;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = D::A;
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.stream = s;
  cfg.gridDim = dim3((unsigned)grids * L * D::A, 1, 1);
  cfg.blockDim = dim3(D::T1, 1, 1);
  cfg.dynamicSmemBytes = D::smem1;
  cfg.numAttrs = in_place ? 2 : 1;
  const cudaError_t e = in_place ? cudaLaunchKernelEx(&cfg, &pass1_kernel<L, DIR, true, APART>, a)
                                 : cudaLaunchKernelEx(&cfg, &pass1_kernel<L, DIR, false, APART>, a);
  if (e != cudaSuccess) return e;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3((unsigned)grids * D::B * (L / D::W), 1, 1);
  cfg.blockDim = dim3(D::T2, 1, 1);
  cfg.dynamicSmemBytes = D::smem2;
  return cudaLaunchKernelEx(&cfg, &pass2_kernel<L, DIR, APART>, a);
}

template <int L, int DIR, bool APART>
TwoPassKernel entry() {
  using D = Dims<L>;
  TwoPassKernel k;
  k.launch = &launch<L, DIR, APART>;
  k.func[0] = (const void*)&pass1_kernel<L, DIR, false, APART>;
  k.func[1] = (const void*)&pass1_kernel<L, DIR, true, APART>;
  k.func[2] = (const void*)&pass2_kernel<L, DIR, APART>;
  k.smem[0] = k.smem[1] = D::smem1;
  k.smem[2] = D::smem2;
  k.A = D::A;
  k.AX = D::AX;
  k.AZ = D::AZ;
  return k;
}
template <int L, bool APART>
TwoPassKernel entry_of(int dir) {
  return dir < 0 ? entry<L, -1, APART>() : entry<L, 1, APART>();
}

}  // namespace tp
}  // namespace fft3d
