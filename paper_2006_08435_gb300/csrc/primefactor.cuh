// Register DFTs by the prime-factor algorithm (Good 1958, Thomas 1963) where the
// radix has coprime factors, for the kernels that need not keep the order of
// the codelets (codelets.cuh): with R = R1 R2 coprime, n = R2 n1 + R1 n2 and
// k = R2 t2 k1 + R1 t1 k2 (mod R; R2 t2 = 1 mod R1, R1 t1 = 1 mod R2),
//   X[k] = sum_n1 W_R1^(n1 k1) sum_n2 W_R2^(n2 k2) v[n]:
// no twiddles between the two steps, so neither their operations nor their
// roundings.  Radix 3 adds sqrt(3)/2 times the difference in one rounding.
// Prime powers are the codelets' four steps.
//
// Relative L2 errors against FP64, pairs of densities, with the codelets / with
// these / of the pair scheme before the real kernels: forward 80^3 1.41 / 1.35 / 1.36e-7,
// 96^3 1.51 / 1.43 / 1.56, 108^3 1.67 / 1.56 / 1.60, 200^3 1.61 / 1.50 / 1.62; inverse 108^3
// 1.77 / 1.59 / 1.67; one orbital of 80^3 1.52 / 1.41, on the fused kernels 1.44.  The
// passes are bound by L1 and L2, so times hardly move: real 96^3 x 27 forward
// 56.3 / 56.4 us, 72^3 x 64 66.1 / 63.6, 216^3 x 4 153.0 / 150.4; complex 48^3 x 198 in place
// 85.7 / 82.1.  Slower, and left on the codelets: complex 108^3 x 17 98.2 / 115
// (fewer registers, a block more per multiprocessor and that much less L1), 90^3 x
// 30 107.2 / 109.7, 60^3 in place 1-7%, boxes 96 x 128 x 64 x 64 212 / 222, one real grid of
// 90^3 7.8 / 9.4 (rows).
#pragma once

#include "codelets.cuh"

namespace fft3d {
namespace pf {

// The smaller of two coprime factors of R above 1 (a power of 2 first), or 0.
constexpr int coprime(int R) {
  int p2 = 1, r = R;
  while (r % 2 == 0) {
    r /= 2;
    p2 *= 2;
  }
  if (p2 > 1) return r > 1 ? p2 : 0;
  int p3 = 1;
  while (r % 3 == 0) {
    r /= 3;
    p3 *= 3;
  }
  return p3 > 1 && r > 1 ? p3 : 0;
}
constexpr int inverse_mod(int a, int m) {
  for (int t = 1; t < m; ++t)
    if (a * t % m == 1) return t;
  return 1;
}

template <int R, int DIR>
FFT3D_HD void transform(float2* v) {
  constexpr int C = coprime(R);
  if constexpr (R == 3) {
    constexpr float h3 = 0.86602540378443864676f;
    const float2 a = v[0], t1 = cadd(v[1], v[2]), t2 = mul_i<DIR>(csub(v[1], v[2]));
    const float2 m = fma2(make_float2(-0.5f, -0.5f), t1, a);
    v[0] = cadd(a, t1);
    v[1] = fma2(make_float2(h3, h3), t2, m);
    v[2] = fma2(make_float2(-h3, -h3), t2, m);
  } else if constexpr (C != 0) {
    constexpr int R1 = C, R2 = R / C;
    constexpr int e1 = R2 * inverse_mod(R2, R1) % R, e2 = R1 * inverse_mod(R1, R2) % R;
    float2 t[R1][R2];
    static_for<0, R1>([&](auto I) {
      constexpr int n1 = decltype(I)::value;
      static_for<0, R2>([&](auto J) {
        constexpr int n2 = decltype(J)::value;
        t[n1][n2] = v[(R2 * n1 + R1 * n2) % R];
      });
      transform<R2, DIR>(t[n1]);
    });
    static_for<0, R2>([&](auto J) {
      constexpr int k2 = decltype(J)::value;
      float2 u[R1];
      static_for<0, R1>([&](auto I) { u[decltype(I)::value] = t[decltype(I)::value][k2]; });
      transform<R1, DIR>(u);
      static_for<0, R1>([&](auto I) {
        constexpr int k1 = decltype(I)::value;
        v[(e1 * k1 + e2 * k2) % R] = u[k1];
      });
    });
  } else if constexpr (R == 9 || R == 25 || R == 27) {
    constexpr int R1 = R == 25 ? 5 : 3, R2 = R / R1;
    float2 t[R1][R2];
    static_for<0, R1>([&](auto I) {
      constexpr int n1 = decltype(I)::value;
      static_for<0, R2>([&](auto J) {
        constexpr int n2 = decltype(J)::value;
        t[n1][n2] = v[n1 + R1 * n2];
      });
      transform<R2, DIR>(t[n1]);
      static_for<1, R2>([&](auto J) {
        constexpr int k2 = decltype(J)::value;
        t[n1][k2] = twc<n1 * k2, R, DIR>(t[n1][k2]);
      });
    });
    static_for<0, R2>([&](auto J) {
      constexpr int k2 = decltype(J)::value;
      float2 u[R1];
      static_for<0, R1>([&](auto I) { u[decltype(I)::value] = t[decltype(I)::value][k2]; });
      transform<R1, DIR>(u);
      static_for<0, R1>([&](auto I) { v[k2 + R2 * decltype(I)::value] = u[decltype(I)::value]; });
    });
  } else {
    DFT<R, DIR>::run(v);
  }
}

}  // namespace pf
}  // namespace fft3d
