// Host side of the general path's 1D plans: division constants, and the
// decimation-in-frequency stages and digit reversal of an edge.
#include "fft3d.h"
#include "internal.h"

namespace fft3d {

static constexpr int kRadices[] = {16, 15, 12, 10, 9, 8, 6, 5, 4, 3, 2};

// n / d for n < 2^32 with a multiplier and a shift (Granlund and Montgomery,
// "Division by invariant integers using multiplication", 1994:
// m = floor(2^32 (2^l - d) / d) + 1 with l = ceil(log2 d), q = (hi(n m) + n) >> l).
FastDiv make_fastdiv(unsigned d) {
  FastDiv f{1u, 0};
  if (d <= 1) {
    f.mul = 1u;  // hi(n * 1) = 0: q = n
    return f;
  }
  int l = 0;
  while ((1ull << l) < d) ++l;
  f.shift = l;
  f.mul = (unsigned)(((1ull << 32) * ((1ull << l) - d)) / d + 1);
  return f;
}

int axis_stages(int L, int* radix) {
  if (L < 2 || L > kAxisMaxLen) return 0;
  int n = 0, rem = L;
  while (rem > 1) {
    int r = 0;
    for (int c : kRadices)
      if (rem % c == 0) {
        r = c;
        break;
      }
    if (!r || n == kAxisMaxStages) return 0;
    radix[n++] = r;
    rem /= r;
  }
  return n;
}

void axis_positions(int L, int nst, const int* radix, int* pos) {
  for (int K = 0; K < L; ++K) {
    int rem = K, span = L, p = 0;
    for (int t = 0; t < nst; ++t) {
      span /= radix[t];
      p += (rem % radix[t]) * span;
      rem /= radix[t];
    }
    pos[K] = p;
  }
}

}  // namespace fft3d

extern "C" int fft3d_axis_digit_map(int n, int* nstages, int* radix, int* pos) {
  if (!nstages || !radix || !pos) return FFT3D_ERR_NULL_PTR;
  int r[fft3d::kAxisMaxStages];
  const int s = fft3d::axis_stages(n, r);
  if (!s) return FFT3D_ERR_UNSUPPORTED_SIZE;
  for (int t = 0; t < s; ++t) radix[t] = r[t];
  *nstages = s;
  fft3d::axis_positions(n, s, r, pos);
  return FFT3D_SUCCESS;
}
