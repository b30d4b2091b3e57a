// The general path's schedule: a 3D transform as one pencil pass per axis
// (pencil.cuh), or in two passes where there are kernels for the lengths (cubic
// edges twopass.cuh, boxes twopass_box.cuh, real grids twopass_real.cuh), over
// chunks of grids -- or, for a grid beyond the chunk budget, ranges of its planes
// for x and y -- whose intermediate stays in L2 from one pass to the next.
//
// Three passes move 48 bytes per point through L2 (in-place copies of
// 37 .. 75 MB run at 12.5 TB/s there once started), but a launch of a few
// tens of MB spends about 4 us of its 12 ramping up and draining.  Two things
// hide that: the passes of a chunk are programmatic dependent launches
// (pencil.cuh), and from 40 MB on the chunks alternate between two chains, the
// caller's stream and a side stream of the plan, so that one chain's ramp and
// drain, and its reads from HBM, fall into the other's L2 passes.  96 x 128 x
// 64, 64 grids: 412 us one chain, plain launches; 312 us with both (261 us
// with the present pencil kernels).  Three chains, or larger chunks: slower.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <vector>

#include "internal.h"

namespace fft3d {

PencilKernel pencil_kernel_unit0(int, int, int);
PencilKernel pencil_kernel_unit1(int, int, int);
PencilKernel pencil_kernel_unit2(int, int, int);
PencilKernel pencil_kernel_unit3(int, int, int);
PencilKernel pencil_kernel_unit4(int, int, int);
PencilKernel pencil_kernel_unit5(int, int, int);
PencilKernel pencil_kernel_unit6(int, int, int);
PencilKernel pencil_kernel_unit7(int, int, int);

PencilKernel pencil_kernel_info(int L, int dir, int kind) {
  using Fn = PencilKernel (*)(int, int, int);
  const Fn units[] = {pencil_kernel_unit0, pencil_kernel_unit1, pencil_kernel_unit2,
                      pencil_kernel_unit3, pencil_kernel_unit4, pencil_kernel_unit5,
                      pencil_kernel_unit6, pencil_kernel_unit7};
  for (Fn f : units) {
    const PencilKernel k = f(L, dir, kind);
    if (k.launch) return k;
  }
  return PencilKernel{};
}

namespace {

// W_n^m = exp(-2 pi i m / n), FP64 rounded to nearest FP32.
float2 root(long long m, int n) {
  const double a = 2.0 * 3.14159265358979323846 * (double)(m % n) / (double)n;
  return make_float2((float)std::cos(a), (float)(-std::sin(a)));
}

}  // namespace

void two_pass_twiddles(int A, int AX, int AZ, int lx, int L, TwoPassArgs& a,
                       std::vector<float2>& tab) {
  for (int i = 0; i < L; ++i) {
    a.ty[i] = root((long long)(i / A) * (i % A), L);
    a.tz[i] = root((long long)(i / AZ) * (i % AZ), L);
  }
  for (int i = 0; i < lx; ++i) tab.push_back(root((long long)(i / AX) * (i % AX), lx));
  tab.insert(tab.end(), a.tz, a.tz + L);
}

int two_pass_prepare(const TwoPassKernel& k, int L, TwoPassArgs& a, std::vector<float2>& tab) {
  for (int i = 0; i < 3; ++i)
    if (k.smem[i] > 48 * 1024 &&
        cudaFuncSetAttribute(k.func[i], cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)k.smem[i]) != cudaSuccess) {
      cudaGetLastError();
      return FFT3D_ERR_CUDA;
    }
  a = TwoPassArgs{};
  two_pass_twiddles(k.A, k.AX, k.AZ, L, L, a, tab);
  return FFT3D_SUCCESS;
}

int AxisPasses::create(PassKind kind_, int nx_, int ny_, int nz_, int batch_, int dir, float scale_,
                       int do_scale_, int l2_bytes, bool fixed) {
  kind = kind_;
  nx = nx_;
  ny = ny_;
  nz = nz_;
  batch = batch_;
  scale = scale_;
  do_scale = do_scale_;
  const int lx = kind == kPassC2C ? nx : nx / 2;
  hx = kind == kPassC2C ? nx : nx / 2 + 1;
  const int len[3] = {lx, ny, nz};
  const int kx = kind == kPassC2C ? 1 : kind == kPassR2C ? 2 : 3;
  two = TwoPassKernel{};
  if (kind == kPassC2C && nx == ny && ny == nz && !fixed) two = two_pass_kernel_info(nx, dir);
  std::vector<float2> tab;
  size_t off[3] = {}, off_r = 0;
  if (two.launch) {
    const int rc = two_pass_prepare(two, nx, two_args, tab);
    if (rc) return rc;
    two_args.scale = scale;
    two_args.do_scale = do_scale;
  }
  real = RealPassKernel{};
  if (kind != kPassC2C && nx == ny && ny == nz) real = real_pass_kernel_info(nx, dir);
  if (real.launch) {
    for (int i = 0; i < 3; ++i)
      if (real.func[i] && real.smem[i] > 48 * 1024 &&
          cudaFuncSetAttribute(real.func[i], cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)real.smem[i]) != cudaSuccess) {
        cudaGetLastError();
        return FFT3D_ERR_CUDA;
      }
    real_args = RealPassArgs{};
    two_pass_twiddles(real.A, real.AX, real.AZ, lx, nx, real_args, tab);
    real_args.scale = scale;
    real_args.do_scale = do_scale;
  }
  // a box: ny = A B with B points per thread, A as small as it goes
  box[0] = box[1] = BoxKernel{};
  if (kind == kPassC2C && !two.launch && !fixed) {
    int A = 0;
    static_assert(6 * 32 <= kTwoPassMaxLen, "ny = A B");
    const int radices[] = {32, 30, 27, 25, 24, 20, 18, 16, 15, 12, 10};
    for (int B : radices)
      if (!A && ny % B == 0 && ny / B >= 2 && ny / B <= 6) A = ny / B;
    // enough blocks in one grid to fill the GPU, of enough points (45 x 75 x 50,
    // 150 blocks: 2 grids 13.0 us, three passes 8.6, though 40 grids 40.5 and
    // 46.0; 36^3, rows of 18 * 36 points: 68 us for 200 grids, three passes 54).
    // The batch has no say: a grid's bits are the same alone and in a batch.
    if (A && (nz * A < 220 || ny / A * nx < 800)) A = 0;
    if (A) {
      box[0] = box1_kernel_info(nx, dir);
      box[1] = box2_kernel_info(A, nz, dir);
    }
    if (!box[0].func || !box[1].func) {
      box[0] = box[1] = BoxKernel{};
    } else {
      // (the limit belongs to the kernel, which plans of several ny share: pass 1,
      // whose rows are the plan's, stays below the default and leaves it alone)
      if (box[1].smem > 48 * 1024 &&
          cudaFuncSetAttribute(box[1].func, cudaFuncAttributeMaxDynamicSharedMemorySize,
                               (int)box[1].smem) != cudaSuccess) {
        cudaGetLastError();
        return FFT3D_ERR_CUDA;
      }
      if (ny / A == 32) box[0].threads = box[0].threads32;
      BoxArgs& b = box_args;
      b = BoxArgs{};
      b.A = A;
      b.B = ny / A;
      b.nx = nx;
      b.tiles = (b.B * nx + 15) / 16;
      b.divA = make_fastdiv((unsigned)b.A);
      b.divB = make_fastdiv((unsigned)b.B);
      b.divt = make_fastdiv((unsigned)b.tiles);
      b.scale = scale;
      b.do_scale = do_scale;
      for (int i = 0; i < ny; ++i) b.ty[i] = root((long long)(i / A) * (i % A), ny);
      const int ax = box[0].split, az = box[1].split;
      for (int i = 0; i < nz; ++i) b.tz[i] = root((long long)(i / az) * (i % az), nz);
      for (int i = 0; i < nx; ++i) tab.push_back(root((long long)(i / ax) * (i % ax), nx));
      tab.insert(tab.end(), b.tz, b.tz + nz);
    }
  }
  // the pencil passes, where no two passes take their place
  for (int a = 0; a < 3 && !two.launch && !real.launch && !box[0].func; ++a) {
    k[a] = PencilKernel{};
    if (fixed) k[a] = pencil_kernel_info(len[a], dir, a == 0 ? 7 : 6);
    if (!k[a].launch)
      k[a] = pencil_kernel_info(len[a], dir, a == 0 ? kx : kind == kPassC2C ? 0 : 5);
    if (!k[a].launch) return FFT3D_ERR_UNSUPPORTED_SIZE;
    if (k[a].smem > 48 * 1024 &&
        cudaFuncSetAttribute(k[a].func, cudaFuncAttributeMaxDynamicSharedMemorySize,
                             (int)k[a].smem) != cudaSuccess) {
      cudaGetLastError();
      return FFT3D_ERR_CUDA;
    }
    off[a] = tab.size();
    const int A = k[a].A, B = len[a] / A;
    if (A > 1)
      for (int k2 = 0; k2 < B; ++k2)
        for (int n1 = 0; n1 < A; ++n1) tab.push_back(root((long long)n1 * k2, len[a]));
  }
  kw = PencilKernel{};
  if (kind == kPassC2R && !real.launch) {
    kw = pencil_kernel_info(nz, dir, 4);
    if (kw.launch && kw.smem > 48 * 1024 &&
        cudaFuncSetAttribute(kw.func, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kw.smem) !=
            cudaSuccess) {
      cudaGetLastError();
      return FFT3D_ERR_CUDA;
    }
  }
  off_r = tab.size();
  if (kind != kPassC2C)
    for (int m = 0; m <= lx; ++m) tab.push_back(root(m, nx));
  if (tab.empty()) tab.push_back(make_float2(1.0f, 0.0f));
  if (cudaMalloc(&d_tab, sizeof(float2) * tab.size()) != cudaSuccess) {
    cudaGetLastError();
    d_tab = nullptr;
    return FFT3D_ERR_ALLOC;
  }
  if (cudaMemcpy(d_tab, tab.data(), sizeof(float2) * tab.size(), cudaMemcpyHostToDevice) !=
      cudaSuccess) {
    cudaGetLastError();
    return FFT3D_ERR_CUDA;
  }
  for (int a = 0; a < 3; ++a) tw[a] = d_tab + off[a];
  twr = d_tab + off_r;
  two_args.tx = d_tab;
  two_args.tzg = d_tab + nx;
  box_args.tx = d_tab;
  box_args.tzg = d_tab + nx;
  real_args.tx = d_tab;
  real_args.tzg = d_tab + lx;
  real_args.twr = twr;

  // Chunk budget: the intermediates of the chunks in flight within 40% of L2
  // (complex grids: 96 x 128 x 64 x 64 261 us, 60%: 270), 60% for real
  // grids, whose other side is half as large (96^3 x 32 forward 111 -> 107,
  // 160^3 x 4 65 -> 61 us), and for two passes (128^3 x 32: 40% 338, 55% 297,
  // 70% 297, 85% 312; 64^3 x 256: 297, 295, 298, 316).  One chain below 40 MB, where the fork and join
  // cost more than the overlap gives (64^3, one chain / two: 8 grids 18.9 /
  // 20.7 us, 16 grids 27.8 / 27.9, 24 grids 38.8 / 35.3).
  const long long pp = (long long)hx * ny;
  const double plane_bytes = 8.0 * (double)pp, grid_bytes = plane_bytes * nz;
  const double l2 = (double)l2_bytes;
  chains = batch >= 2 && grid_bytes * batch > 40.0 * 1048576.0 ? kMaxChains : 1;
  const double budget = (kind == kPassC2C && !two.launch && !box[0].func ? 0.4 : 0.6) * l2 / chains;
  // a pass's pencils stay below 2^31
  const long long most = std::max({(long long)ny * nz, (long long)nz * hx, pp});
  const long long cap = std::max(1LL, (1LL << 30) / most);
  chunk = std::max(1LL, std::min({(long long)(budget / grid_bytes), (long long)batch, cap}));
  long long nchunks = (batch + chunk - 1) / chunk;
  nchunks = std::min<long long>(batch, (nchunks + chains - 1) / chains * chains);
  chunk = (batch + nchunks - 1) / nchunks;
  sub = chunk * nz;
  // a grid beyond the budget: x and y over planes of 30% of L2 (256^3 x 4
  // with planes of 15 / 30 / 50%: 671 / 603 / 534 us one chain, 477 two)
  if (grid_bytes > budget)
    sub = std::max(1LL, std::min((long long)nz, (long long)(0.3 * l2 / plane_bytes)));
  if (chains > 1) {
    mu = new (std::nothrow) std::mutex();
    if (!mu) return FFT3D_ERR_ALLOC;
    if (cudaEventCreateWithFlags(&fork, cudaEventDisableTiming) != cudaSuccess ||
        cudaEventCreateWithFlags(&join, cudaEventDisableTiming) != cudaSuccess ||
        cudaStreamCreateWithFlags(&side, cudaStreamNonBlocking) != cudaSuccess) {
      cudaGetLastError();
      return FFT3D_ERR_CUDA;
    }
  }
  return FFT3D_SUCCESS;
}

void AxisPasses::destroy() {
  if (side) cudaStreamDestroy(side);
  if (join) cudaEventDestroy(join);
  if (fork) cudaEventDestroy(fork);
  delete mu;
  cudaFree(d_tab);
  side = nullptr;
  join = fork = nullptr;
  mu = nullptr;
  d_tab = nullptr;
}

long long AxisPasses::work_points() const { return chains * chunk * hx * ny * nz; }

// The passes of grids g .. g + chunk - 1 (work: one chunk of spectra, kPassC2R).
cudaError_t AxisPasses::chunk_passes(long long g, const void* in, void* out, float2* work,
                                     cudaStream_t s, const HartreeWeight* weight) const {
  const long long pp = (long long)hx * ny;  // complex points of a plane
  if (two.launch) {
    const long long m = std::min(chunk, batch - g);
    TwoPassArgs a = two_args;
    a.in = static_cast<const float2*>(in) + g * pp * nz;
    a.out = static_cast<float2*>(out) + g * pp * nz;
    return two.launch(a, (int)m, in == out, s);
  }
  if (real.launch) {
    const long long m = std::min(chunk, batch - g);
    const long long real_pts = (long long)nx / 2 * ny * nz, spec_pts = pp * nz;
    RealPassArgs a = real_args;
    a.in = static_cast<const float2*>(in) + g * (kind == kPassR2C ? real_pts : spec_pts);
    a.out = static_cast<float2*>(out) + g * (kind == kPassR2C ? spec_pts : real_pts);
    a.work = work;
    if (weight) {
      a.weight = *weight;
      a.weight.grad += g;
    }
    return real.launch(a, (int)m, s);
  }
  if (box[0].func) {
    const long long m = std::min(chunk, batch - g);
    BoxArgs a = box_args;
    a.in = static_cast<const float2*>(in) + g * pp * nz;
    a.out = static_cast<float2*>(out) + g * pp * nz;
    a.in_place = in == out;
    const cudaError_t e = launch_box(box[0], (unsigned)(m * nz * a.A), box[0].smem * a.B,
                                     a.in_place ? a.A : 1, a, s);
    return e != cudaSuccess ? e
                            : launch_box(box[1], (unsigned)(m * a.tiles), box[1].smem, 1, a, s);
  }
  // contiguous rows of `planes` planes
  auto x_pass = [&](const float2* src, float2* dst, long long planes) {
    PencilArgs a{};
    a.in = src;
    a.out = dst;
    a.tw = tw[0];
    a.twr = twr;
    a.np = (unsigned)(planes * ny);
    a.nx = 1;
    a.divn = make_fastdiv(1);
    a.scale = scale;
    a.do_scale = kind == kPassC2R && do_scale;
    a.pol_in = kEvictFirst;
    a.pol_out = kind == kPassC2R ? kEvictFirst : kEvictLast;
    return k[0].launch(a, s);
  };
  auto y_pass = [&](float2* dat, long long planes) {
    PencilArgs a{};
    a.in = dat;
    a.out = dat;
    a.tw = tw[1];
    a.np = (unsigned)(planes * hx);
    a.nx = (unsigned)hx;
    a.divn = make_fastdiv((unsigned)hx);
    a.so = pp;
    a.pi = hx;
    a.pol_in = kEvictNormal;
    a.pol_out = kEvictLast;
    return k[1].launch(a, s);
  };
  auto z_pass = [&](const float2* src, float2* dst, long long grids) {
    PencilArgs a{};
    a.in = src;
    a.out = dst;
    a.tw = tw[2];
    a.np = (unsigned)(grids * pp);
    a.nx = (unsigned)pp;
    a.divn = make_fastdiv((unsigned)pp);
    a.so = pp * nz;
    a.pi = pp;
    a.scale = scale;
    a.do_scale = kind != kPassC2R && do_scale;
    a.pol_in = kEvictFirst;
    a.pol_out = kind == kPassC2R ? kEvictLast : kEvictFirst;
    if (weight) {
      a.weight = *weight;
      a.weight.grad += g;
      a.n = nz;
      a.hx = hx;
      a.divh = make_fastdiv((unsigned)hx);
      return kw.launch(a, s);
    }
    return k[2].launch(a, s);
  };
  // complex points of one grid on the x pass's two sides
  const long long real_pts = (long long)nx / 2 * ny * nz, spec_pts = pp * nz;
  const long long m = std::min(chunk, batch - g);
  cudaError_t e;
  if (kind == kPassC2R) {
    const float2* src = static_cast<const float2*>(in) + g * spec_pts;
    float2* dst = static_cast<float2*>(out) + g * real_pts;
    if ((e = z_pass(src, work, m)) != cudaSuccess) return e;
    for (long long z = 0; z < m * nz; z += sub) {
      const long long pl = std::min(sub, m * nz - z);
      float2* to = dst + z * ny * (nx / 2);
      if ((e = y_pass(work + z * pp, pl)) != cudaSuccess) return e;
      if ((e = x_pass(work + z * pp, to, pl)) != cudaSuccess) return e;
    }
  } else {
    const long long in_pts = kind == kPassC2C ? spec_pts : real_pts;
    const float2* src = static_cast<const float2*>(in) + g * in_pts;
    float2* dst = static_cast<float2*>(out) + g * spec_pts;
    for (long long z = 0; z < m * nz; z += sub) {
      const long long pl = std::min(sub, m * nz - z);
      const float2* from = src + z * (in_pts / nz);
      if ((e = x_pass(from, dst + z * pp, pl)) != cudaSuccess) return e;
      if ((e = y_pass(dst + z * pp, pl)) != cudaSuccess) return e;
    }
    if ((e = z_pass(dst, dst, m)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t AxisPasses::execute(const void* in, void* out, float2* work, cudaStream_t s,
                                const HartreeWeight* weight) const {
  cudaError_t e = cudaSuccess;
  if (chains == 1) {
    for (long long g = 0; g < batch && e == cudaSuccess; g += chunk)
      e = chunk_passes(g, in, out, work, s, weight);
    return e;
  }
  // the events are recorded and waited for under a lock: executes of one
  // plan from several threads keep their own order
  std::lock_guard<std::mutex> lock(*mu);
  if ((e = cudaEventRecord(fork, s)) != cudaSuccess) return e;
  if ((e = cudaStreamWaitEvent(side, fork, 0)) != cudaSuccess) return e;
  int c = 0;
  for (long long g = 0; g < batch && e == cudaSuccess; g += chunk, c ^= 1)
    e = chunk_passes(g, in, out, work && c ? work + chunk * hx * ny * nz : work, c ? side : s, weight);
  // the side stream is joined even when a launch failed
  cudaError_t j = cudaEventRecord(join, side);
  if (j == cudaSuccess) j = cudaStreamWaitEvent(s, join, 0);
  return e == cudaSuccess ? j : e;
}

}  // namespace fft3d
