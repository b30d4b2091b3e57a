// Register-first 1D transforms of pencils for every edge L, 2 <= L <= 512,
// with prime factors 2, 3, 5: the passes of the general path (the 1D FFTs
// along x, then y, then z of the paper's section "Approach").
//
// L = A * B, both register codelets.  With
// n = n1 + A n2 and k = k2 + B k1:
//   phase 1: thread (pencil, n1) loads the B points n1 + A n2 straight from
//            global memory into registers, DFT_B, times W_L^(n1 k2), to
//            shared memory;
//   phase 2: thread (pencil, k2) reads its A values, DFT_A, and stores the
//            outputs k2 + B k1 straight to global memory, in natural order.
// One round trip through shared memory (16 bytes per point) and one barrier
// per tile, every index of a butterfly a compile-time constant; B loads of
// every thread are in flight at once.  The kernels before staged a tile by
// cp.async and ran two or more in-place stages and a digit-reversed read
// there (32 bytes and more of shared-memory traffic per point, run-time
// radices): 96 x 128 x 64, 64 grids 524 -> 412 us by the kernels alone, 261
// with the launches and chunks of passes.cu; 256^3 x 4 827 -> 396; 100^3 x
// 16 174 -> 94.  A pass is bound by latency and its launch: L2-resident ones of 50 MB
// take 16 us of which a copy kernel takes 12 (its ramp and drain 4); L2 is at 17-34%,
// L1 at 47-59%, HBM at 37% where x reads it and 58% in the z pass of 256^3, whose
// grid exceeds L2.
//
// A block waits for nothing but its predecessor launch: passes are
// programmatic dependent launches (launch_dependents at the start, wait
// before the first read), so a pass's blocks are resident when the pass
// before it drains (96 x 128 x 64, 64 grids, one chain: 412 -> 372 us).
// L2 policies: inputs read once and final outputs evict first, the
// intermediate last (256^3 x 4 455 -> 418 us, small ones 1-2%).
//
// Strided pencils (y and z): lanes are consecutive pencils.  The pencils of
// a pass are numbered p = o * nx + x and start at o * so + x, so that a run
// of lanes crosses row ends without idle lanes whatever nx is (the half
// spectra of real grids have n/2 + 1 columns); the z pass takes a whole
// plane as one row (nx = plane, so = grid).  Contiguous pencils (x): lanes
// are consecutive n1 (loads) and k2 (stores) of a row.
//
// Real rows of n = 2 L points (kinds kR2C, kC2R) are contiguous pencils of
// z[m] = r[2m] + i r[2m+1] with Z[k] = E[k] + i O[k], E and O the transforms
// of the even and odd samples, X[k] = E[k] + W_n^k O[k], k = 0 .. L.  The
// split needs Z[k] and Z[L-k], which are outputs of the phase-2 items k2 and
// B - k2: one thread takes both and splits in registers.  The inverse undoes
// the split as it starts, one thread taking the points of n1 and A - n1.
// These rows are staged: copied in with cp.async and out as whole runs, at an
// odd pitch, and the lanes of a warp are rows -- no bank conflicts, one n1 or
// k2 (one branch of the split, one twiddle) per half-warp, where lanes along
// the row took 5 to 8 short runs per access and both branches (10 grids of
// 96^3: L1 wavefronts of the forward x pass 5.0 -> 2.9 M, 21.5 -> 15.6 us; the
// three passes of 96^3 x 32 forward 107 -> 93, inverse 106 -> 101 us; 100^3 x 16 64 ->
// 55, 60 -> 59).  Complex rows do better without (256^3 x 4 419 us, staged 489).
#pragma once

#include <cuda_runtime.h>

#include <utility>

#include "codelets.cuh"
#include "internal.h"
#include "primefactor.cuh"

namespace fft3d {
namespace pc {

enum {
  kStrided = 0,
  kContig = 1,
  kR2C = 2,
  kC2R = 3,
  kWeighted = 4,
  kStridedReal = 5,
  kStridedFixed = 6,
  kContigFixed = 7
};
constexpr bool strided(int kind) {
  return kind == kStrided || kind == kWeighted || kind == kStridedReal || kind == kStridedFixed;
}
constexpr bool contig(int kind) { return kind == kContig || kind == kContigFixed; }
// Complex kinds of the fixed plans, at the edges where the general ones have another
// order of sums.
constexpr bool fixed(int kind) { return kind == kStridedFixed || kind == kContigFixed; }
constexpr bool fixed_edge(int L) { return L == 486 || L == 500 || L == 512; }

constexpr bool smooth(int n) {
  if (n < 2) return false;
  while (n % 2 == 0) n /= 2;
  while (n % 3 == 0) n /= 3;
  while (n % 5 == 0) n /= 5;
  return n == 1;
}
// Lengths of a step's transform in registers (transform below).
constexpr bool codelet(int r) {
  return r == 1 || r == 2 || r == 3 || r == 4 || r == 5 || r == 6 || r == 8 || r == 9 || r == 10 ||
         r == 12 || r == 15 || r == 16 || r == 18 || r == 20 || r == 24 || r == 25 || r == 27 ||
         r == 30 || r == 32;
}
// The factor A of the split; B = L / A.
// Edges without a fused kernel: B is the first radix of the edge's mixed-radix
// plan (fft3d_axis_digit_map: the largest of 16, 15, 12, 10, 9, 8, ...) where
// the rest is a codelet (all but 486, 500 and 512). The sums, twiddles and order
// are then those of the plan's decimation-in-frequency stages, and the bits
// those of the stage-by-stage passes before: the Hartree energy is returned
// in FP64 and keeps its value (486, 500 and 512: by kinds of the fixed plans' own,
// three stages with two of them in one thread).
// Fused edges, whose Hartree spectra come from other kernels, 486, 500, 512, and real
// rows: the closest pair, the larger factor in the phase that holds one
// transform per thread (64^3 x 4 12.2 us, with 16 * 4 16.8; 48^3 x 12 12.0,
// with 16 * 3 16.2; 512^3 1060, with 16 * 2 * 16 1255).
// Pencils of a codelet's length stay in one thread (no exchange), rows only
// below 16 points (real ones up to 6): the lanes of a warp share longer ones.
constexpr int first_radix(int L) {
  const int radices[] = {16, 15, 12, 10, 9, 8, 6, 5, 4, 3, 2};
  for (int r : radices)
    if (L % r == 0) return r;
  return 0;
}
constexpr int split_a(int L, int kind) {
  const bool real = kind == kR2C || kind == kC2R;
  const bool closest = real || L == 16 || L == 32 || L == 48 || L == 64 || L == 80 || L == 96 || L == 512;
  if (fixed(kind)) return L / first_radix(L);
  if (codelet(L) && L <= (real ? 6 : contig(kind) ? 15 : 32)) return 1;
  int a = L / first_radix(L);
  if (!closest && codelet(a)) return a;
  int best = 0;
  for (a = 1; a * a <= L; ++a)
    if (L % a == 0 && codelet(a) && codelet(L / a)) best = a;
  return kind == kC2R ? L / best : best;
}
// Threads of a block: the multiple of 32 up to 512 that leaves the fewest
// lanes idle over the two phases (n1 items of work w1, then n2 of w2), at
// most four items per thread and phase.
constexpr int block_threads(int n1, int w1, int n2, int w2) {
  int best = 0;
  long best_cost = 0;
  const int need = n1 > n2 ? n1 : n2;
  for (int t = 512; t >= 128; t -= 32) {
    if (t - 31 > need && t > 128) continue;
    const int i1 = (n1 + t - 1) / t, i2 = (n2 + t - 1) / t;
    if (i1 > 4 || i2 > 4) continue;
    const long cost = (long)t * ((long)i1 * w1 + (long)i2 * w2);
    if (!best || cost * 100 < best_cost * 98) {
      best = t;
      best_cost = cost;
    }
  }
  return best ? best : 512;
}
// Pencils per block: 16 (a 128-byte run of columns) at the long edges, more
// at the short ones, about 2048 points.
constexpr int tile_pencils(int L, int A) {
  if (A == 1) return 64;
  int w = 16;
  while (w < 64 && 2 * w * L <= 2048) w *= 2;
  return w;
}

// Registers a thread may use (complex kinds), so that the compiler aims at
// 32 warps and more: 256^3 x 4 419 -> 395, 100^3 x 16 102 -> 94 us.
constexpr int reg_budget(int B) { return B <= 8 ? 48 : B <= 12 ? 56 : B <= 16 ? 64 : 96; }

template <int L, int KIND>
struct Cfg {
  static constexpr int A = split_a(L, KIND), B = L / A;
  static constexpr bool REAL = KIND == kR2C || KIND == kC2R;
  static constexpr int W = tile_pencils(L, A);
  // items of the two phases (real rows: mirrored pairs where the split is)
  static constexpr int N1 = W * (KIND == kC2R && A > 1 ? A / 2 + 1 : A);
  static constexpr int N2 = A == 1 ? 0 : W * (KIND == kR2C ? B / 2 + 1 : B);
  static constexpr int T = block_threads(N1, KIND == kC2R ? 2 * B : B, N2, KIND == kR2C ? 2 * A : A);
  static constexpr int I1 = (N1 + T - 1) / T, I2 = (N2 + T - 1) / T;
  // rows: exchange slot of (pencil, k2, n1), odd pitch of k2 (and of real rows)
  static constexpr int AP = A | 1, RP = REAL ? B * AP | 1 : B * AP;
  static constexpr int exchange = A == 1 ? 0 : strided(KIND) ? W * L : W * RP;
  // real rows: points of a staged row in and out, odd pitch; one buffer (two
  // for one-step rows, whose threads read and write it in the same phase)
  static constexpr int IR = KIND == kC2R ? L + 1 : L, OR = KIND == kR2C ? L + 1 : L;
  static constexpr int SP = (L + 1) | 1;
  static constexpr int out_at = A == 1 ? W * SP : 0;
  static constexpr size_t smem = sizeof(float2) * (size_t)(exchange + (REAL ? out_at + W * SP : 0));
  static constexpr int blocks =
      (strided(KIND) || contig(KIND)) && !fixed(KIND) ? 65536 / (T * reg_budget(A > B ? A : B)) : 1;
  static_assert(A >= 1, "no split into two codelets");
  static_assert(strided(KIND) || contig(KIND) || L <= 256, "real rows hold 2 L points");
};

// a * w (forward) or a * conj w, w a forward table twiddle.  The order of the
// fused operations is written out: left to the compiler it differs from one
// kernel to the next, and results are to keep their bits.
template <int DIR>
FFT3D_HD float2 twiddle(float2 a, float2 w) {
  const float s = DIR < 0 ? w.y : -w.y;
  return make_float2(fmaf(a.x, w.x, -(a.y * s)), fmaf(a.y, w.x, a.x * s));
}

// The R-point transform of a step.  Above 16 points (but 32, which only fused
// edges and 512 have, unless PLAN) R = R1 * R2 with R1 = first_radix(R): the two decimation-
// in-frequency stages of the mixed-radix plan in registers, R1 points R2
// apart, the twiddles W_R^(j k) as the table has them, then R2 points.
template <int R, int DIR, bool PLAN = false>
FFT3D_HD void transform(float2* v) {
  if constexpr (R <= 16 || (R == 32 && !PLAN)) {
    DFT<R, DIR>::run(v);
  } else {
    constexpr int R1 = first_radix(R), R2 = R / R1;
    float2 t[R2][R1];
    static_for<0, R2>([&](auto J) {
      constexpr int j = decltype(J)::value;
      static_for<0, R1>([&](auto I) { t[j][decltype(I)::value] = v[j + R2 * decltype(I)::value]; });
      DFT<R1, DIR>::run(t[j]);
      static_for<1, R1>([&](auto K) {
        constexpr int k = decltype(K)::value;
        if constexpr (j > 0)
          t[j][k] = twiddle<DIR>(t[j][k], make_float2((float)turn_cos(j * k, R), (float)-turn_sin(j * k, R)));
      });
    });
    static_for<0, R1>([&](auto K) {
      constexpr int k = decltype(K)::value;
      float2 u[R2];
      static_for<0, R2>([&](auto J) { u[decltype(J)::value] = t[decltype(J)::value][k]; });
      DFT<R2, DIR>::run(u);
      static_for<0, R2>([&](auto M) { v[k + R1 * decltype(M)::value] = u[decltype(M)::value]; });
    });
  }
}

__device__ __forceinline__ unsigned fdiv(unsigned n, FastDiv d) {
  return (unsigned)(((unsigned long long)__umulhi(n, d.mul) + n) >> d.shift);
}

// L2 policy of a pass's loads or stores (kEvictNormal, kEvictFirst, kEvictLast).
__device__ __forceinline__ uint64_t l2_policy(int which) {
  uint64_t n, f, l;
  asm volatile("createpolicy.fractional.L2::evict_normal.b64 %0, 1.0;" : "=l"(n));
  asm volatile("createpolicy.fractional.L2::evict_first.b64 %0, 1.0;" : "=l"(f));
  asm volatile("createpolicy.fractional.L2::evict_last.b64 %0, 1.0;" : "=l"(l));
  return which == kEvictFirst ? f : which == kEvictLast ? l : n;
}
__device__ __forceinline__ float2 ldg(const float2* p, uint64_t pol) {
  float2 v;
  asm volatile("ld.global.L2::cache_hint.v2.f32 {%0, %1}, [%2], %3;"
               : "=f"(v.x), "=f"(v.y) : "l"(p), "l"(pol));
  return v;
}
__device__ __forceinline__ void stg(float2* p, float2 v, uint64_t pol) {
  asm volatile("st.global.L2::cache_hint.v2.f32 [%0], {%1, %2}, %3;"
               ::"l"(p), "f"(v.x), "f"(v.y), "l"(pol) : "memory");
}

// `rows` consecutive rows of R points, packed at g, to pitch P at s, and back.
template <int R, int P, int T>
__device__ __forceinline__ void rows_in(float2* s, const float2* g, int rows, uint64_t pol) {
  for (int u = threadIdx.x; u < rows * R; u += T)
    asm volatile("cp.async.ca.shared.global.L2::cache_hint [%0], [%1], 8, %2;"
                 ::"r"((uint32_t)__cvta_generic_to_shared(s + u / R * P + u % R)), "l"(g + u), "l"(pol)
                 : "memory");
  asm volatile("cp.async.wait_all;" ::: "memory");
}
template <int R, int P, int T>
__device__ __forceinline__ void rows_out(float2* g, const float2* s, int rows, float sc, uint64_t pol) {
#pragma unroll 4
  for (int u = threadIdx.x; u < rows * R; u += T) stg(g + u, cscale(s[u / R * P + u % R], sc), pol);
}

// Half spectrum of a real row of 2 L points from Z: X[k] = E + W_n^k O and
// X[L-k] = conj(E - W_n^k O), E = (Z[k] + conj Z[L-k]) / 2,
// O = -i (Z[k] - conj Z[L-k]) / 2.  z[k1] = Z[k2 + B k1]; mz holds the
// mirrors: mz[A-1-k1] = Z[L-k2-B k1], or, for k2 = 0, z itself with
// Z[L - B k1] = z[(A - k1) % A].  A = 1 (L = B): z and mz are the row.
template <int L, int A>
__device__ __forceinline__ void split(const float2* twr, float2* dst, const float2* z,
                                      const float2* mz, int k2) {
  constexpr int B = L / A, N = A == 1 ? L : A, S = A == 1 ? 1 : B;
#pragma unroll
  for (int k1 = 0; k1 < N; ++k1) {
    const int k = k2 + S * k1;
    const float2 u = z[k1], m = k2 == 0 ? z[(N - k1) % N] : mz[N - 1 - k1];
    const float2 E = make_float2(0.5f * (u.x + m.x), 0.5f * (u.y - m.y));
    const float2 O = make_float2(0.5f * (u.y + m.y), 0.5f * (m.x - u.x));
    const float2 t = cmul_tw<-1>(O, __ldg(twr + k));
    dst[k] = cadd(E, t);
    dst[L - k] = make_float2(E.x - t.x, t.y - E.y);
  }
}

// The kinds of real grids take the prime-factor forms, whose errors are smaller;
// those of complex grids keep the order of the sums (see split_a).
template <int R, int DIR, int KIND>
__device__ __forceinline__ void step(float2* v) {
  if constexpr (KIND == kStrided || contig(KIND) || fixed(KIND)) transform<R, DIR, fixed(KIND)>(v);
  else pf::transform<R, DIR>(v);
}

template <int L, int DIR, int KIND>
__global__ void __launch_bounds__(Cfg<L, KIND>::T, Cfg<L, KIND>::blocks) pencil_kernel(const PencilArgs a) {
  using C = Cfg<L, KIND>;
  constexpr int A = C::A, B = C::B, W = C::W, T = C::T;
  extern __shared__ __align__(16) float2 sm[];
  asm volatile("griddepcontrol.launch_dependents;" ::: "memory");
  const unsigned p0 = blockIdx.x * (unsigned)W;
  const float sc = a.scale;
  const uint64_t pin = l2_policy(a.pol_in), pout = l2_policy(a.pol_out);
  asm volatile("griddepcontrol.wait;" ::: "memory");

  const int np = (int)min((unsigned)W, a.np - p0);  // pencils of this block
  // first point of pencil c of the block
  auto base = [&](int c) -> long long {
    const unsigned p = p0 + (unsigned)c;
    if constexpr (strided(KIND)) {
      const unsigned o = fdiv(p, a.divn);
      return (long long)o * a.so + (long long)(p - o * a.nx);
    } else {
      return (long long)p * L;
    }
  };
  float2* const st = sm + C::exchange;  // staged real rows in
  float2* const so = st + C::out_at;    // and out
  if constexpr (C::REAL) {
    rows_in<C::IR, C::SP, T>(st, a.in + (size_t)p0 * C::IR, np, pin);
    __syncthreads();
  }

  // phase 1
#pragma unroll 1
  for (int it = 0; it < C::I1; ++it) {
    const int e = threadIdx.x + it * T;
    if (e >= C::N1) break;
    const int c = contig(KIND) ? e / A : e % W, n1 = contig(KIND) ? e % A : e / W;
    if (c >= np) continue;
    if constexpr (KIND == kC2R) {
      // Z[k] = 2 E + i 2 O and Z[L-k] = conj(2 E) + i conj(2 O) with
      // 2 E = X[k] + conj X[L-k], 2 O = (X[k] - conj X[L-k]) W_n^-k: the item
      // of n1 makes the points n1 + A j and their mirrors, A - n1 + A j (its
      // own points for n1 = 0 and A / 2).  Of X[0] and X[L] only the real
      // parts count.
      const float2* row = st + c * C::SP;
      float2 u[B], m[B];
#pragma unroll
      for (int j = 0; j < B; ++j) {
        u[j] = row[n1 + A * j];
        m[j] = row[L - n1 - A * j];
      }
      if (n1 == 0) u[0].y = m[0].y = 0.0f;
#pragma unroll
      for (int j = 0; j < B; ++j) {
        const float2 s = make_float2(u[j].x + m[j].x, u[j].y - m[j].y);
        const float2 d = make_float2(u[j].x - m[j].x, u[j].y + m[j].y);
        const float2 t = cmul_tw<1>(d, __ldg(a.twr + n1 + A * j));
        u[j] = make_float2(s.x - t.y, s.y + t.x);
        m[j] = make_float2(s.x + t.y, t.x - s.y);
      }
      step<B, DIR, KIND>(u);
      if constexpr (A > 1) {
        float2* x = sm + c * C::RP;
#pragma unroll
        for (int k = 0; k < B; ++k)
          x[k * C::AP + n1] = k ? twiddle<DIR>(u[k], __ldg(a.tw + k * A + n1)) : u[k];
        if (n1 != 0 && 2 * n1 != A) {
          float2 v[B];
#pragma unroll
          for (int j = 0; j < B; ++j) v[j] = m[B - 1 - j];
          step<B, DIR, KIND>(v);
          const int n2 = A - n1;
#pragma unroll
          for (int k = 0; k < B; ++k)
            x[k * C::AP + n2] = k ? twiddle<DIR>(v[k], __ldg(a.tw + k * A + n2)) : v[k];
        }
      } else {
#pragma unroll
        for (int k = 0; k < B; ++k) so[c * C::SP + k] = u[k];
      }
    } else {
      float2 v[B];
      if constexpr (KIND == kR2C) {
        const float2* row = st + c * C::SP + n1;
#pragma unroll
        for (int j = 0; j < B; ++j) v[j] = row[A * j];
      } else {
        const long long pi = strided(KIND) ? a.pi : 1, step = A * pi;
        const float2* src = a.in + base(c) + n1 * pi;
#pragma unroll
        for (int j = 0; j < B; ++j) v[j] = ldg(src + j * step, pin);
        if constexpr (KIND == kWeighted) {
          // pencil -> (grid, ky, kx); its points are kz = n1 + A j
          const unsigned p = p0 + (unsigned)c, o = fdiv(p, a.divn), r = p - o * a.nx;
          const int ky = (int)fdiv(r, a.divh), kx = (int)r - ky * a.hx;
          const int my = signed_index(ky, a.n);
          const float xy = (float)(kx * kx + my * my);
          const float scale = (float)(a.weight.s * a.weight.grad[o]);
#pragma unroll
          for (int j = 0; j < B; ++j) {
            const float mz = (float)signed_index(n1 + A * j, L);
            v[j] = weighted(v[j], scale, fmaf(mz, mz, xy));
          }
        }
      }
      step<B, DIR, KIND>(v);
      if constexpr (A > 1) {
#pragma unroll
        for (int k = 0; k < B; ++k) {
          const float2 y = k ? twiddle<DIR>(v[k], __ldg(a.tw + k * A + n1)) : v[k];
          sm[strided(KIND) ? (k * A + n1) * W + c : c * C::RP + k * C::AP + n1] = y;
        }
      } else if constexpr (KIND == kR2C) {
        split<L, 1>(a.twr, so + c * C::SP, v, v, 0);
      } else {
        float2* dst = a.out + base(c);
        const long long ostep = strided(KIND) ? a.pi : 1;
#pragma unroll
        for (int k = 0; k < B; ++k) stg(dst + k * ostep, a.do_scale ? cscale(v[k], sc) : v[k], pout);
      }
    }
  }

  // phase 2
  if constexpr (A > 1) {
    __syncthreads();
#pragma unroll 1
    for (int it = 0; it < C::I2; ++it) {
      const int e = threadIdx.x + it * T;
      if (e >= C::N2) break;
      const int c = contig(KIND) ? e / B : e % W, k2 = contig(KIND) ? e % B : e / W;
      if (c >= np) continue;
      float2 v[A];
#pragma unroll
      for (int j = 0; j < A; ++j)
        v[j] = sm[strided(KIND) ? (k2 * A + j) * W + c : c * C::RP + k2 * C::AP + j];
      step<A, DIR, KIND>(v);
      if constexpr (KIND == kR2C) {
        float2* row = so + c * C::SP;
        // the mirrors of this item's outputs are those of B - k2
        if (k2 == 0 || 2 * k2 == B) {
          split<L, A>(a.twr, row, v, v, k2);
        } else {
          float2 w[A];
#pragma unroll
          for (int j = 0; j < A; ++j) w[j] = sm[c * C::RP + (B - k2) * C::AP + j];
          step<A, DIR, KIND>(w);
          split<L, A>(a.twr, row, v, w, k2);
        }
      } else if constexpr (KIND == kC2R) {
        float2* row = so + c * C::SP + k2;
#pragma unroll
        for (int k = 0; k < A; ++k) row[B * k] = v[k];
      } else {
        const long long pi = strided(KIND) ? a.pi : 1, step = B * pi;
        float2* dst = a.out + base(c) + k2 * pi;
        if (a.do_scale) {
#pragma unroll
          for (int k = 0; k < A; ++k) v[k] = cscale(v[k], sc);
        }
#pragma unroll
        for (int k = 0; k < A; ++k) stg(dst + k * step, v[k], pout);
      }
    }
  }

  if constexpr (C::REAL) {
    __syncthreads();
    rows_out<C::OR, C::SP, T>(a.out + (size_t)p0 * C::OR, so, np, a.do_scale ? sc : 1.0f, pout);
  }
}

template <int L, int DIR, int KIND>
cudaError_t launch(const PencilArgs& a, cudaStream_t s) {
  using C = Cfg<L, KIND>;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((a.np + C::W - 1) / C::W, 1, 1);
  cfg.blockDim = dim3(C::T, 1, 1);
  cfg.dynamicSmemBytes = C::smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, &pencil_kernel<L, DIR, KIND>, a);
}

template <int L, int DIR, int KIND>
PencilKernel entry() {
  using C = Cfg<L, KIND>;
  PencilKernel k;
  k.launch = &launch<L, DIR, KIND>;
  k.func = (const void*)&pencil_kernel<L, DIR, KIND>;
  k.A = C::A;
  k.smem = C::smem;
  k.width = C::W;
  return k;
}

template <int L>
PencilKernel entry_of(int dir, int kind) {
  if (kind == kStrided) return dir < 0 ? entry<L, -1, kStrided>() : entry<L, 1, kStrided>();
  if constexpr (fixed_edge(L)) {
    if (kind == kStridedFixed && dir < 0) return entry<L, -1, kStridedFixed>();
    if (kind == kContigFixed && dir < 0) return entry<L, -1, kContigFixed>();
  }
  if constexpr (L % 2 == 0 && !real_kernels(L)) {
    if (kind == kWeighted && dir > 0) return entry<L, 1, kWeighted>();
    if (kind == kStridedReal) return dir < 0 ? entry<L, -1, kStridedReal>() : entry<L, 1, kStridedReal>();
  }
  if (kind == kContig) return dir < 0 ? entry<L, -1, kContig>() : entry<L, 1, kContig>();
  if constexpr (L <= 256 && !real_kernels(2 * L)) {
    if (kind == kR2C && dir < 0) return entry<L, -1, kR2C>();
    if (kind == kC2R && dir > 0) return entry<L, 1, kC2R>();
  }
  return PencilKernel{};
}

// The plannable edges are shared out over kUnits translation units by their
// rank, so that they compile in parallel.
constexpr int kUnits = 8;
constexpr int rank_of(int L) {
  int r = 0;
  for (int n = 2; n < L; ++n) r += smooth(n);
  return r;
}
template <int UNIT, int L>
void pick(int want, int dir, int kind, PencilKernel& k) {
  if constexpr (smooth(L) && rank_of(L) % kUnits == UNIT)
    if (L == want) k = entry_of<L>(dir, kind);
}
template <int UNIT, int... I>
PencilKernel unit_kernel(int L, int dir, int kind, std::integer_sequence<int, I...>) {
  PencilKernel k;
  (pick<UNIT, I>(L, dir, kind, k), ...);
  return k;
}
template <int UNIT>
PencilKernel unit_kernel(int L, int dir, int kind) {
  return unit_kernel<UNIT>(L, dir, kind, std::make_integer_sequence<int, kAxisMaxLen + 1>{});
}

}  // namespace pc
}  // namespace fft3d
