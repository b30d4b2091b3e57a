// Real cubic grids of even edge N in two passes of small blocks (the forms of
// twopass.cuh on rows of L = N / 2 complex points and half spectra of HX = L + 1
// columns; y = n1 + A j, ky = k2 + B k1, N = A B):
//   forward, pass 1, block (grid, z, n1): the B rows y = n1 + A j: complex x
//     transform, split into the real rows' HX bins as the y step reads them, the
//     B-point DFT over j of a column in one thread, times W_N^(n1 k2), to row
//     k2 + B n1 of plane z; pass 2, block (grid, W of the B HX columns (k2, kx)):
//     z transforms of its A rows and the A-point DFT over n1, in place.
//   inverse, pass 1: the same pass 2 from the half spectra to the workspace, the
//     DFT going over k1 (optionally times the Hartree weights as it reads);
//     pass 2, block (grid, z, n1): times W_N^(-n1 k2) and the B-point DFT over k2
//     of a column in one thread, then the rows: half bins to complex points and
//     the x transform.
// The spectrum crosses L2 once less than in the pencil passes, and stays there in
// between (HBM at 27-30% in the pass on its side, 1% in the other).  Neither HBM (96^3 x
// 32, one direction: 34 us) nor L2 (20-32%) bounds it: the row kernels are bound by L1
// (70-73%), in wavefronts of shared memory and of twiddles: hence the row layout of
// twopass.cuh, which hardly an access conflicts in, and lanes along the rows in the
// steps whose twiddles are then one address for a warp (96^3 x 32, with padded runs and
// lanes along the columns: forward 77.5, inverse 98.1 us; now 63.8 and 77.6).  The column
// kernels wait for loads.  The B HX columns of a group lie side by side, so a block of
// the column kernel takes 16 of them whatever HX is.
// Splits per edge from a sweep over A, P, AZ and threads; the next best lies 1-5%
// behind.  us, pencil passes / two passes (these replayed from a graph), forward and
// inverse: 48^3 x 300 114.5 / 74.1, 122.2 / 81.9; 60^3 x 200 150.0 / 109.2, 165.3 / 112.7;
// 80^3 x 60 102.2 / 71.2, 108.3 / 78.6; 96^3 x 32 93.4 / 63.5, 100.1 / 77.1; 100^3 x 40
// 132.3 / 103.6, 140.9 / 111.0; 120^3 x 24 148.3 / 100.3, 148.0 / 113.4; one grid: within
// 1.5 us (48^3 8.5 / 6.6, 96^3 11.5 / 9.8, 100^3 10.1 / 11.2).  96^3 has AZ = 8 for its
// errors: eight densities forth and back 2.19e-7 with 6, 2.12e-7 with 8 (forward
// 65.1 / 63.8 us).
#pragma once

#include "hartree.cuh"
#include "twopass.cuh"

namespace fft3d {
namespace tpr {

using pc::l2_policy;
using pc::ldg;
using pc::stg;
using pc::twiddle;
using tp::slot;

// A groups of the y axis; x as P lanes of Q points, z as AZ BZ (first step BZ);
// PF: the rows' steps by prime factors (the columns' always).
template <int N>
struct Split;
#define FFT3D_TPR(N_, A_, P_, AZ_, T_, PF_)                  \
  template <>                                             \
  struct Split<N_> {                                      \
    static constexpr int A = A_, P = P_, AZ = AZ_, T = T_; \
    static constexpr bool PF = PF_;                        \
  };
FFT3D_TPR(48, 3, 8, 4, 32, true)
FFT3D_TPR(60, 3, 6, 4, 64, true)
FFT3D_TPR(64, 2, 16, 4, 64, true)
FFT3D_TPR(72, 3, 6, 6, 64, true)
FFT3D_TPR(80, 5, 8, 4, 64, true)
FFT3D_TPR(90, 5, 9, 6, 64, false)
FFT3D_TPR(96, 4, 8, 8, 64, true)
FFT3D_TPR(100, 4, 10, 5, 96, true)
FFT3D_TPR(108, 6, 9, 6, 64, true)
FFT3D_TPR(120, 5, 12, 6, 96, true)
FFT3D_TPR(128, 4, 16, 8, 96, true)
#undef FFT3D_TPR

template <int N>
struct Dims {
  static constexpr int L = N / 2, HX = L + 1;
  static constexpr int A = Split<N>::A, B = N / A;
  static constexpr bool PF = Split<N>::PF;
  static constexpr int P = Split<N>::P, Q = L / P, AZ = Split<N>::AZ, BZ = N / AZ;
  static_assert(A * B == N && P * Q == L && AZ * BZ == N, "splits");
  static constexpr tp::Layout rows = tp::row_layout(B, P, Q, HX);
  static constexpr int PD = rows.PD, RP = rows.RP;
  static constexpr int T1 = Split<N>::T;
  static constexpr size_t smem1 = sizeof(float2) * (size_t)B * RP;
  // columns: point (kz2, m1, n1) of column q at kz2 ZP + (m1 A + n1) W + q
  static constexpr int W = 16, NC = B * HX, TILES = (NC + W - 1) / W;
  static constexpr bool uniform = W * A % 32 == 0;
  static constexpr int ZP = AZ * A * W;
  static constexpr int T2 = (W * BZ + 31) / 32 * 32;
  static constexpr size_t smem2 = sizeof(float2) * (size_t)BZ * ZP;
  static constexpr long long PL = (long long)N * HX;  // points of a plane of spectra
};

template <int N>
__global__ void __launch_bounds__(Dims<N>::T1) rows_fwd_kernel(const __grid_constant__ RealPassArgs a) {
  using D = Dims<N>;
  constexpr int A = D::A, B = D::B, L = D::L, P = D::P, Q = D::Q, T = D::T1;
  constexpr int PD = D::PD;
  extern __shared__ __align__(16) float2 sm[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const unsigned zz = blockIdx.x / A;  // plane
  const int n1 = (int)(blockIdx.x - zz * A);
  const uint64_t once = l2_policy(kEvictFirst), keep = l2_policy(kEvictLast);
  const float2* src = a.in + (size_t)zz * N * L + n1 * L;
  float2* dst = a.out + (size_t)zz * D::PL + n1 * (B * D::HX);
  asm volatile("griddepcontrol.wait;" ::: "memory");
  // x, first step: item (j, m), the points m + P i
#pragma unroll 2
  for (int e = threadIdx.x; e < B * P; e += T) {
    const int j = e / P, m = e % P;
    const float2* s = src + j * (A * L) + m;
    float2 v[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] = ldg(s + P * i, once);
    tp::transform<Q, -1, D::PF>(v);
    float2* x = sm + j * D::RP;
#pragma unroll
    for (int k = 0; k < Q; ++k) x[slot(PD, m * Q + k)] = k ? twiddle<-1>(v[k], __ldg(a.tx + k * P + m)) : v[k];
  }
  __syncthreads();
  // second step, in place: item (k, j), lanes along j
#pragma unroll 1
  for (int e = threadIdx.x; e < B * Q; e += T) {
    const int k = e / B;
    float2* x = sm + e % B * D::RP;
    float2 v[P];
#pragma unroll
    for (int i = 0; i < P; ++i) v[i] = x[slot(PD, Q * i + k)];
    tp::transform<P, -1, D::PF>(v);
#pragma unroll
    for (int i = 0; i < P; ++i) x[slot(PD, Q * i + k)] = v[i];
  }
  __syncthreads();
#pragma unroll 1
  for (int kx = threadIdx.x; kx < D::HX; kx += T) {
    // X[k] = (Z[k] + conj Z[L-k]) / 2 - i W_N^k (Z[k] - conj Z[L-k]) / 2, Z[L] = Z[0]
    const int k = kx == L ? 0 : kx, mk = k == 0 ? 0 : L - k;
    const float2 *xu = sm + slot(PD, k), *xm = sm + slot(PD, mk);
    const float2 w = __ldg(a.twr + kx);
    float2 v[B];
#pragma unroll
    for (int j = 0; j < B; ++j) {
      const float2 u = xu[j * D::RP], m = xm[j * D::RP];
      const float2 E = make_float2(0.5f * (u.x + m.x), 0.5f * (u.y - m.y));
      const float2 O = make_float2(0.5f * (u.y + m.y), 0.5f * (m.x - u.x));
      v[j] = cadd(E, cmul_tw<-1>(O, w));
    }
    tp::transform<B, -1, D::PF>(v);
    float2* o = dst + kx;
#pragma unroll
    for (int i = 0; i < B; ++i)
      stg(o + i * D::HX, i ? twiddle<-1>(v[i], a.ty[i * A + n1]) : v[i], keep);
  }
}

template <int N>
__global__ void __launch_bounds__(Dims<N>::T1) rows_inv_kernel(const __grid_constant__ RealPassArgs a) {
  using D = Dims<N>;
  constexpr int A = D::A, B = D::B, L = D::L, P = D::P, Q = D::Q, T = D::T1;
  constexpr int PD = D::PD;
  extern __shared__ __align__(16) float2 sm[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const unsigned zz = blockIdx.x / A;
  const int n1 = (int)(blockIdx.x - zz * A);
  const uint64_t once = l2_policy(kEvictFirst);
  const float2* src = a.work + (size_t)zz * D::PL + n1 * (B * D::HX);
  float2* dst = a.out + (size_t)zz * N * L + n1 * L;
  asm volatile("griddepcontrol.wait;" ::: "memory");
#pragma unroll 1
  for (int kx = threadIdx.x; kx < D::HX; kx += T) {
    float2 v[B];
#pragma unroll
    for (int i = 0; i < B; ++i) v[i] = ldg(src + i * D::HX + kx, once);
#pragma unroll
    for (int i = 1; i < B; ++i) v[i] = twiddle<1>(v[i], a.ty[i * A + n1]);
    tp::transform<B, 1, D::PF>(v);
    float2* x = sm + slot(PD, kx);
#pragma unroll
    for (int j = 0; j < B; ++j) x[j * D::RP] = v[j];
  }
  __syncthreads();
  // Z[k] = 2 E + i 2 O, 2 E = X[k] + conj X[L-k], 2 O = (X[k] - conj X[L-k])
  // W_N^-k, and its mirror Z[L-k] = conj(2 E) + i conj(2 O): item (n, j), lanes
  // along j, makes and transforms the points n + Q i and their mirrors, in
  // place.  Of X[0] and X[L] only the real parts count.
#pragma unroll 1
  for (int e = threadIdx.x; e < B * (Q / 2 + 1); e += T) {
    const int n = e / B;
    float2* x = sm + e % B * D::RP;
    float2 u[P], m[P];
#pragma unroll
    for (int i = 0; i < P; ++i) {
      u[i] = x[slot(PD, n + Q * i)];
      m[i] = x[slot(PD, L - n - Q * i)];
    }
    if (n == 0) u[0].y = m[0].y = 0.0f;
#pragma unroll
    for (int i = 0; i < P; ++i) {
      const float2 s = make_float2(u[i].x + m[i].x, u[i].y - m[i].y);
      const float2 d = make_float2(u[i].x - m[i].x, u[i].y + m[i].y);
      const float2 t = cmul_tw<1>(d, __ldg(a.twr + n + Q * i));
      u[i] = make_float2(s.x - t.y, s.y + t.x);
      m[i] = make_float2(s.x + t.y, t.x - s.y);
    }
    tp::transform<P, 1, D::PF>(u);
#pragma unroll
    for (int k = 0; k < P; ++k)
      x[slot(PD, n + Q * k)] = k ? twiddle<1>(u[k], __ldg(a.tx + n * P + k)) : u[k];
    if (n != 0 && 2 * n != Q) {
      float2 v[P];
#pragma unroll
      for (int i = 0; i < P; ++i) v[i] = m[P - 1 - i];
      tp::transform<P, 1, D::PF>(v);
#pragma unroll
      for (int k = 0; k < P; ++k)
        x[slot(PD, Q - n + Q * k)] = k ? twiddle<1>(v[k], __ldg(a.tx + (Q - n) * P + k)) : v[k];
    }
  }
  __syncthreads();
  // second step: item (j, k), lanes along k: the real points 2 (k + P i), + 1
  const float sc = a.do_scale ? a.scale : 1.0f;
#pragma unroll 2
  for (int e = threadIdx.x; e < B * P; e += T) {
    const int j = e / P, k = e % P;
    const float2* x = sm + j * D::RP;
    float2 v[Q];
#pragma unroll
    for (int i = 0; i < Q; ++i) v[i] = x[slot(PD, Q * k + i)];
    tp::transform<Q, 1, D::PF>(v);
    float2* o = dst + j * (A * L) + k;
#pragma unroll
    for (int i = 0; i < Q; ++i) stg(o + P * i, cscale(v[i], sc), once);
  }
}

// Forward: a.out in place, scaled; inverse: a.in to a.work.
template <int N, int DIR, bool WEIGHT>
__global__ void __launch_bounds__(Dims<N>::T2) cols_kernel(const __grid_constant__ RealPassArgs a) {
  using D = Dims<N>;
  constexpr int A = D::A, AZ = D::AZ, BZ = D::BZ, W = D::W, T = D::T2, NC = D::NC;
  constexpr long long PL = D::PL;
  extern __shared__ __align__(16) float2 sm[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const unsigned g = blockIdx.x / D::TILES, c0 = (blockIdx.x - g * D::TILES) * W;
  const uint64_t once = l2_policy(kEvictFirst), keep = l2_policy(DIR < 0 ? kEvictFirst : kEvictLast);
  const int cols = min(W, NC - (int)c0);
  const size_t at = (size_t)g * PL * N + c0;
  const float2* src = (DIR < 0 ? a.out : a.in) + at;
  float2* dst = (DIR < 0 ? a.out : a.work) + at;
  asm volatile("griddepcontrol.wait;" ::: "memory");
  float scale = 0.0f;
  if constexpr (WEIGHT) scale = (float)(a.weight.s * a.weight.grad[g]);
  constexpr int N1 = W * A * AZ;
#pragma unroll 1
  for (int it = 0; it < (N1 + T - 1) / T; ++it) {
    const int e = threadIdx.x + it * T;
    if (N1 % T && e >= N1) break;
    const int q = e % W, n1 = e / W % A;
    int m1 = e / (W * A);
    if constexpr (D::uniform) m1 = __shfl_sync(0xffffffffu, m1, 0);
    if (q >= cols) continue;
    const float2* s = src + m1 * PL + n1 * NC + q;
    float2 v[BZ];
#pragma unroll
    for (int i = 0; i < BZ; ++i) v[i] = ldg(s + (long long)(AZ * i) * PL, once);
    if constexpr (WEIGHT) {
      const int c = (int)c0 + q, kx = c % D::HX, my = signed_index(c / D::HX + D::B * n1, N);
      const float xy = (float)(kx * kx + my * my);
#pragma unroll
      for (int i = 0; i < BZ; ++i) {
        const float mz = (float)signed_index(m1 + AZ * i, N);
        v[i] = weighted(v[i], scale, fmaf(mz, mz, xy));
      }
    }
    tp::transform<BZ, DIR, true>(v);
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
      tp::transform<AZ, DIR, true>(v[n1]);
    }
    float2* o = dst + kz2 * PL + q;
#pragma unroll
    for (int k = 0; k < AZ; ++k) {
      float2 u[A];
#pragma unroll
      for (int n1 = 0; n1 < A; ++n1) u[n1] = v[n1][k];
      tp::transform<A, DIR, true>(u);
#pragma unroll
      for (int k1 = 0; k1 < A; ++k1)
        stg(o + (long long)(BZ * k) * PL + k1 * NC,
            DIR < 0 && a.do_scale ? cscale(u[k1], a.scale) : u[k1], keep);
    }
  }
}

inline cudaError_t launch_dependent(const void* fn, unsigned grid, int threads, size_t smem,
                                    const RealPassArgs& a, cudaStream_t s) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  cfg.stream = s;
  cfg.gridDim = dim3(grid, 1, 1);
  cfg.blockDim = dim3((unsigned)threads, 1, 1);
  cfg.dynamicSmemBytes = smem;
  void* args[] = {const_cast<RealPassArgs*>(&a)};
  return cudaLaunchKernelExC(&cfg, fn, args);
}

template <int N>
cudaError_t launch_fwd(const RealPassArgs& a, int grids, cudaStream_t s) {
  using D = Dims<N>;
  const cudaError_t e = launch_dependent((const void*)&rows_fwd_kernel<N>, (unsigned)grids * N * D::A,
                                         D::T1, D::smem1, a, s);
  return e != cudaSuccess ? e
                          : launch_dependent((const void*)&cols_kernel<N, -1, false>,
                                             (unsigned)grids * D::TILES, D::T2, D::smem2, a, s);
}
template <int N>
cudaError_t launch_inv(const RealPassArgs& a, int grids, cudaStream_t s) {
  using D = Dims<N>;
  const void* cols = a.weight.grad ? (const void*)&cols_kernel<N, 1, true>
                                   : (const void*)&cols_kernel<N, 1, false>;
  const cudaError_t e =
      launch_dependent(cols, (unsigned)grids * D::TILES, D::T2, D::smem2, a, s);
  return e != cudaSuccess ? e
                          : launch_dependent((const void*)&rows_inv_kernel<N>,
                                             (unsigned)grids * N * D::A, D::T1, D::smem1, a, s);
}

template <int N>
RealPassKernel entry(int dir) {
  using D = Dims<N>;
  static_assert(real_kernels(N), "the pencil passes leave this edge out");
  RealPassKernel k;
  k.launch = dir < 0 ? &launch_fwd<N> : &launch_inv<N>;
  k.func[0] = dir < 0 ? (const void*)&rows_fwd_kernel<N> : (const void*)&rows_inv_kernel<N>;
  k.func[1] = dir < 0 ? (const void*)&cols_kernel<N, -1, false> : (const void*)&cols_kernel<N, 1, false>;
  k.func[2] = dir < 0 ? nullptr : (const void*)&cols_kernel<N, 1, true>;
  k.smem[0] = D::smem1;
  k.smem[1] = k.smem[2] = D::smem2;
  k.A = D::A;
  k.AX = D::P;
  k.AZ = D::AZ;
  return k;
}

}  // namespace tpr
}  // namespace fft3d
