// A cubic L^3 transform in two passes of small blocks, for the edges whose
// y axis splits into A groups that one thread can hold (see Cfg).
//
// With y = n1 + A j and ky = k2 + B k1 (L = A B, A small):
//   pass 1, block (grid, z, n1): the B rows y = n1 + A j: x transform (two
//     register steps with one exchange in shared memory), then per column the
//     B-point DFT over j in one thread, times W_L^(n1 k2), stored to row
//     k2 + B n1 of plane z;
//   pass 2, block (grid, W of the B L columns (k2, x)): the rows k2 + B n1 of
//     every z: first step of the z transform from global memory to shared memory,
//     then one thread per (column, kz2) holds its points of all A rows, finishes
//     the z transforms and the A-point DFT over n1, and stores rows k2 + B k1, the
//     same points it read.
// A grid crosses L2 twice (32 bytes per point; the separate passes of
// pencil.cuh 48).  Neither HBM nor L2 bounds that: at the 12.5 TB/s of L2-resident
// copies 64^3 x 106 would take 71 us, of HBM's one round trip 66; measured 119, with
// L2 at 24-29% and HBM at 22-28% (pass 1) and below 1% (pass 2: the intermediate
// stays in L2).  L1 does (50-80%), and latency: short runs, bank conflicts, loads in
// flight, the ramp and drain of a chunk's launch.  Hence runs of 64 bytes and more
// in the first step of pass 1, shared rows whose strided accesses do not conflict
// (row_layout), columns taken 16 at a time across the rows k2 (whatever L is, full
// and aligned to 128 bytes where B L is a multiple of 16), and
// twiddles that are the same for a whole warp read from the kernel's parameters
// (constant bank; of x they stay in the first step: in the second, where lanes
// run along the rows, 96 x 128 x 64 x 64 took 257 us for 231).
// Splits per edge from a sweep; the next best lies 1-5% behind.  us, three passes /
// two passes with padded rows of their own splits / now: 60^3 x 129 - / 140 / 123;
// 72^3 x 75 - / 135 / 120; 80^3 x 54 - / 129 / 118; 90^3 x 38 - / 174 / 137; 108^3 x 22
// - / 155 / 129; 100^3 x 16 94 / 86 / 79; 48^3 x 400 - / 191 / 169; 64^3 x 64 90.3 / 74.6 /
// 72.4; 96^3 x 31 - / 126 / 124; 128^3 x 8 92.7 / 78.7 / 80.5.
//
// In place, the A groups of a plane read rows that the others write.  Where their
// rows take at most 56 KB they are one block (four fit a multiprocessor);
// above, they run as a cluster of blocks and store after a cluster barrier behind
// everybody's loads.  us in place, cluster / one block: 48^3 x 253 158 / 116, 60^3 x
// 129 178 / 135, 64^3 x 106 156 / 120, 80^3 x 54 140 / 134, 96^3 x 31 139 / 144, 128^3 x
// 32 317 / 379.
//
// Steps by prime factors (Cfg::PF; primefactor.cuh) for the errors: one orbital of
// 80^3 1.52e-7 -> 1.41e-7, 48^3 1.50 -> 1.38; 48^3 x 198 in place 85.7 -> 82.1 us, x 4
// 6.9 -> 6.5, the others within 1%.
#pragma once

#include <cuda_runtime.h>

#include "codelets.cuh"
#include "internal.h"
#include "pencil.cuh"
#include "primefactor.cuh"

namespace fft3d {
namespace tp {

using pc::l2_policy;
using pc::ldg;
using pc::stg;
using pc::twiddle;

// The R-point transform of a step, by prime factors (primefactor.cuh) if PF.
template <int R, int DIR, bool PF>
FFT3D_HD void transform(float2* v) {
  if constexpr (PF) pf::transform<R, DIR>(v);
  else pc::transform<R, DIR>(v);
}

// Splits of an edge: y into A groups of B; x and z into two register steps,
// BX (BZ) points first, AX (AZ) apart, then AX (AZ); T threads of pass 1; PF: the
// steps by prime factors, where that is no slower.
template <int L>
struct Cfg;
#define FFT3D_TP(L_, A_, AX_, AZ_, T_, PF_)                             \
  template <>                                                           \
  struct Cfg<L_> {                                                      \
    static constexpr int L = L_, A = A_, B = L_ / A_;                   \
    static constexpr int AX = AX_, BX = L_ / AX_, AZ = AZ_, BZ = L_ / AZ_; \
    static constexpr int T1 = T_, W = 16; /* W: columns of a pass-2 block */ \
    static constexpr bool PF = PF_;                                     \
  };
FFT3D_TP(48, 3, 8, 4, 64, true)
FFT3D_TP(60, 4, 12, 4, 64, false)
FFT3D_TP(64, 4, 16, 4, 64, false)
FFT3D_TP(72, 3, 12, 6, 96, true)
FFT3D_TP(80, 4, 16, 4, 96, true)
FFT3D_TP(90, 5, 15, 6, 160, false)
FFT3D_TP(96, 4, 16, 8, 192, true)
FFT3D_TP(100, 5, 10, 5, 128, true)
FFT3D_TP(108, 4, 12, 9, 128, false)
FFT3D_TP(128, 4, 16, 8, 128, false)
#undef FFT3D_TP

// Rows in shared memory for an x transform in two register steps, P lanes of Q
// points first, then Q of P: row j at j RP, its points in natural order (k + Q m
// the output k of lane m), with one slot left free after every PD where PD is not
// 0.  Each step's items read and write one set of slots, and columns lie side by
// side.  The layout is the one of least extra wavefronts per half-warp of 8-byte
// accesses in the two strided patterns: items (j, m) at j RP + m Q, and items
// (k, j) with lanes along j at j RP + k (whose twiddles are the same for a row's
// worth of lanes).
struct Layout {
  int PD, RP;
};
FFT3D_HD constexpr int slot(int PD, int p) { return PD ? p + p / PD : p; }
constexpr Layout row_layout(int B, int P, int Q, int points) {
  Layout best{0, 0};
  int least = 1 << 20;
  int lcm = 16;
  while (lcm % Q) lcm += 16;
  for (int o = 0; o < (Q % 2 ? 1 : 2); ++o) {
    const int PD = o ? lcm : 0;
    for (int rp = slot(PD, points - 1) + 1, i = 0; i < 16; ++i, ++rp) {
      int total = 0;
      for (int pat = 0; pat < 2; ++pat)
        for (int h = 0; h < 8; ++h) {
          int n[16] = {}, worst = 0;
          for (int l = 0; l < 16; ++l) {
            const int e = h * 16 + l;
            const int at = pat == 0 ? e / P * rp + slot(PD, e % P * Q) : e % B * rp + e / B;
            const int c = ++n[at % 16];
            worst = c > worst ? c : worst;
          }
          total += worst - 1;
        }
      if (total * 64 + i < least) {
        least = total * 64 + i;
        best = Layout{PD, rp};
      }
    }
  }
  return best;
}

template <int L>
struct Dims : Cfg<L> {
  using C = Cfg<L>;
  static constexpr Layout rows = row_layout(C::B, C::AX, C::BX, L);
  static constexpr int PD = rows.PD, RP = rows.RP;
  using C::T1;
  static constexpr size_t smem1 = sizeof(float2) * (size_t)C::B * RP;
  static constexpr bool MERGED = C::A * smem1 <= 56 * 1024;  // in place: see above
  // pass 2: point (kz2, m1, n1) of column q at kz2 * ZP + (m1 * A + n1) * W + q
  static constexpr int NC = C::B * L, TILES = (NC + C::W - 1) / C::W;  // columns (k2, x)
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
__global__ void __launch_bounds__(Dims<L>::T1 * (INPLACE && Dims<L>::MERGED ? Dims<L>::A : 1))
    pass1_kernel(const __grid_constant__ TwoPassArgs a) {
  using D = Dims<L>;
  constexpr int A = D::A, B = D::B, AX = D::AX, BX = D::BX, T = D::T1;
  extern __shared__ __align__(16) float2 rows[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr bool M = INPLACE && D::MERGED;
  // plane, grid; group n1 of y and this thread of it
  const unsigned zz = M ? blockIdx.x : blockIdx.x / A, g = zz / L;
  const int n1 = M ? (int)threadIdx.x / T : (int)(blockIdx.x - zz * A);
  const int tid = M ? (int)threadIdx.x % T : (int)threadIdx.x;
  float2* const sm = rows + (M ? n1 * (B * D::RP) : 0);
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
    const int e = tid + it * T;
    if (N1 % T && e >= N1) break;
    const int j = e / AX, m = e % AX;
    const float2* s = src + j * (A * L) + m;
    float2 v[BX];
#pragma unroll
    for (int i = 0; i < BX; ++i) v[i] = ldg(s + AX * i, once);
    transform<BX, DIR, D::PF>(v);
    float2* x = sm + j * D::RP;
#pragma unroll
    for (int k = 0; k < BX; ++k) x[slot(D::PD, BX * m + k)] = k ? twiddle<DIR>(v[k], __ldg(a.tx + k * AX + m)) : v[k];
  }
  if constexpr (INPLACE && !M) {
    // the cluster's A blocks read and write the same plane
    __syncwarp();
    asm volatile("barrier.cluster.arrive.aligned;" ::: "memory");
  }
  __syncthreads();
  // x, second step, in place: item (k2, row j)
  constexpr int N2 = B * BX;
#pragma unroll 1
  for (int it = 0; it < (N2 + T - 1) / T; ++it) {
    const int e = tid + it * T;
    if (N2 % T && e >= N2) break;
    const int k = e / B;
    float2* x = sm + e % B * D::RP;
    float2 v[AX];
#pragma unroll
    for (int i = 0; i < AX; ++i) v[i] = x[slot(D::PD, BX * i + k)];
    transform<AX, DIR, D::PF>(v);
#pragma unroll
    for (int i = 0; i < AX; ++i) x[slot(D::PD, BX * i + k)] = v[i];
  }
  if constexpr (INPLACE && !M) {
    __syncwarp();
    asm volatile("barrier.cluster.wait.aligned;" ::: "memory");
  }
  __syncthreads();
  // y: column kx = k2 + BX k1, its B points of this group
  if (tid < L) {
    const int kx = tid;
    const float2* x = sm + slot(D::PD, kx);
    float2 v[B];
#pragma unroll
    for (int j = 0; j < B; ++j) v[j] = x[j * D::RP];
    transform<B, DIR, D::PF>(v);
    float2* o = dst + kx;
#pragma unroll
    for (int k = 0; k < B; ++k)
      stg(o + k * L, k ? twiddle<DIR>(v[k], a.ty[k * A + n1]) : v[k], keep);
  }
}

template <int L, int DIR, bool APART>
__global__ void __launch_bounds__(Dims<L>::T2) pass2_kernel(const __grid_constant__ TwoPassArgs a) {
  using D = Dims<L>;
  constexpr int A = D::A, AZ = D::AZ, BZ = D::BZ, W = D::W, T = D::T2;
  constexpr long long LL = (long long)L * L;
  extern __shared__ __align__(16) float2 sm[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  constexpr int NC = D::NC;
  const unsigned g = blockIdx.x / D::TILES;
  const int c0 = (int)(blockIdx.x - g * D::TILES) * W;  // first column (k2, x)
  const int cols = min(W, NC - c0);
  const uint64_t once = l2_policy(kEvictFirst);
  const GridAt<APART> at(a, g, (size_t)LL * L);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  float2* base = at.out(a) + c0;
  // z, first step: item (m1, n1, q) -> planes m1 + AZ i
  constexpr int N1 = W * A * AZ;
#pragma unroll 1
  for (int it = 0; it < (N1 + T - 1) / T; ++it) {
    const int e = threadIdx.x + it * T;
    if (N1 % T && e >= N1) break;
    const int q = e % W, n1 = e / W % A;
    const int m1 = D::uniform ? __shfl_sync(0xffffffffu, e / (W * A), 0) : e / (W * A);
    if (NC % W && q >= cols) continue;
    const float2* s = base + m1 * LL + n1 * NC + q;
    float2 v[BZ];
#pragma unroll
    for (int i = 0; i < BZ; ++i) v[i] = ldg(s + (long long)(AZ * i) * LL, once);
    transform<BZ, DIR, D::PF>(v);
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
    if (NC % W && q >= cols) return;
    const float2* x = sm + kz2 * D::ZP + q;
    float2 v[A][AZ];
#pragma unroll
    for (int n1 = 0; n1 < A; ++n1) {
#pragma unroll
      for (int m = 0; m < AZ; ++m) v[n1][m] = x[(m * A + n1) * W];
      transform<AZ, DIR, D::PF>(v[n1]);
    }
    float2* o = base + kz2 * LL + q;
#pragma unroll
    for (int k = 0; k < AZ; ++k) {
      float2 u[A];
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) u[n1] = v[n1][k];
      transform<A, DIR, D::PF>(u);
#pragma unroll
      for (int k1 = 0; k1 < A; ++k1)
        stg(o + (long long)(BZ * k) * LL + k1 * NC, a.do_scale ? cscale(u[k1], a.scale) : u[k1],
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
  const bool merged = in_place && D::MERGED;
  cfg.attrs = attr;
  cfg.numAttrs = in_place && !merged ? 2 : 1;
  cfg.stream = s;
  cfg.gridDim = dim3((unsigned)grids * L * (merged ? 1 : D::A), 1, 1);
  cfg.blockDim = dim3(D::T1 * (merged ? D::A : 1), 1, 1);
  cfg.dynamicSmemBytes = D::smem1 * (merged ? D::A : 1);
  const cudaError_t e = in_place ? cudaLaunchKernelEx(&cfg, &pass1_kernel<L, DIR, true, APART>, a)
                                 : cudaLaunchKernelEx(&cfg, &pass1_kernel<L, DIR, false, APART>, a);
  if (e != cudaSuccess) return e;
  cfg.numAttrs = 1;
  cfg.gridDim = dim3((unsigned)grids * D::TILES, 1, 1);
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
  k.smem[0] = D::smem1;
  k.smem[1] = D::smem1 * (D::MERGED ? D::A : 1);
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
