// Host/device structures shared by the planner (plan.cu) and the kernel
// translation units.  Not part of the public C ABI.
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <mutex>
#include <vector>

#include "fft3d.h"
#include "hartree.cuh"

namespace fft3d {

// Device status word values (sticky until read by fft3d_get_device_status).
constexpr unsigned kStatusOk = 0u;
constexpr unsigned kStatusTimeout = 1u;

// Default limit of one inter-block wait (nanoseconds of %globaltimer).
constexpr long long kDefaultWaitNs = 2000000000LL;

// One run of consecutive work items: all plane items (phase 0: x then y
// transform of plane z = i) or all slab items (phase 1: z transform of the
// slab y = i) of one grid.  Items [start, start + n) of the global ticket
// sequence, i = ticket - start.
struct SchedBlock {
  int grid;
  int phase;
  int start;
  int n;  // edge of that grid (cubic), also the number of items
};

struct FusedArgs {
  const float2* in;             // packed input base (unused when in_ptrs)
  float2* out;                  // packed output base (unused when out_ptrs)
  const float2* const* in_ptrs; // device array of per-grid inputs, or null
  float2* const* out_ptrs;      // device array of per-grid outputs, or null
  const long long* grid_off;    // per-grid element offsets, or null (g * n^3)
  const int* grid_map;          // local grid -> plan grid index, or null (identity)
  const SchedBlock* blocks;
  int nblocks;
  int total_items;
  const float2* twiddles;       // concatenated tables in kernel size order
  unsigned* work;               // [0] ticket, [1 + g] plane items done for grid g
  unsigned* status;             // sticky status word
  float scale;                  // output scale of the last pass
  int do_scale;
  long long timeout_ns;
  const uint32_t* mma_frag;     // tensor-core B fragments (split precisions), or null
  int ngrids;                   // grids of the launch unit
  float2* aux;                  // a kernel's own workspace (real grids: Nyquist columns), or null
};
static_assert(sizeof(FusedArgs) == 128, "tensor maps behind it keep their 128-byte lines");

// Arguments of the weighted real inverse kernels.  (A type of their own: two more
// words in FusedArgs moved the tensor maps behind it off their 128-byte lines in the
// parameters: split precision 128^3 x 32 355 -> 375 us.)
struct alignas(128) WeightedArgs : FusedArgs {
  HartreeWeight weight;
};

using LaunchFn = cudaError_t (*)(const FusedArgs&, int grid, cudaStream_t);
// Launch of a unit of a mixed-edge plan on packed buffers with per-grid
// tensor maps (at most kMixMaps grids, passed with the launch): host_off[l]
// = element offset of the unit's grid l.
constexpr int kMixMaps = 32;
using LaunchMapsFn = cudaError_t (*)(const FusedArgs&, const long long* host_off, int grid,
                                     cudaStream_t);

struct KernelInfo {
  LaunchFn launch = nullptr;
  const void* func = nullptr;   // for occupancy / attributes
  int threads = 0;
  size_t smem = 0;              // dynamic shared memory bytes
  int twiddle_entries = 0;      // complex entries in the concatenated table
  int sizes[8] = {0};           // edges handled, in table order
  int nsizes = 0;
  int items_in_flight = 1;      // work items a block holds at once (schedule lag)
  int prec = 0;                 // 0 FP32, else fft3d_precision of the tensor-core kinds
  int cluster = 0;              // > 0: cluster kernel of this many blocks per cluster
  int tw_l1 = 0;                // twiddle table split n = l1 * (n / l1); 0: item_l1(n, prec)
  int phase_items = 0;          // work items per phase of a grid; 0: the grid's edge
  int umma_b = 0;               // mma_frag holds the tcgen05 B table (tcgen.cuh), not mma.sync fragments
  int uses_work = 1;            // 0: no ticket counters (nothing to clear before a launch)
  LaunchMapsFn launch_maps = nullptr;  // mixed-edge units on packed buffers (tensor-map kernels)
  const void* func_maps = nullptr;     // its kernel
  // real inverse kernels: the input times the weight
  cudaError_t (*launch_weighted)(const WeightedArgs&, int grid, cudaStream_t) = nullptr;
  const void* func_weighted = nullptr;
};

// ---------------------------------------------------------------- general path
// Passes for any edge 2..kAxisMaxLen with prime factors 2, 3, 5 (passes.cu).
constexpr int kAxisMaxLen = 512;
constexpr int kGeneralVariant = 10;  // plan variant of the general path
constexpr int kFixedVariant = 11;    // three passes in the order of the mixed-radix plan (internal)
constexpr int kAxisMaxStages = 12;

// n / d = (hi32(n * mul) + n) >> shift for every n < 2^32 (make_fastdiv).
struct FastDiv {
  unsigned mul;
  int shift;
};
FastDiv make_fastdiv(unsigned d);

int axis_stages(int L, int* radix);                              // 0: not plannable
void axis_positions(int L, int nst, const int* radix, int* pos);  // pos[K], K < L

// Register-first pencil passes (pencil.cuh).  np pencils; strided kind:
// pencil p starts at (p / nx) * so + p % nx, its points pi apart; the other
// kinds: rows packed back to back.  tw[k * A + n1] = W_L^(n1 k) (k < L / A);
// real rows: twr[k] = W_2L^k, k <= L.
enum { kEvictNormal = 0, kEvictFirst = 1, kEvictLast = 2 };
struct PencilArgs {
  const float2* in;  // may equal out (complex kinds)
  float2* out;
  const float2* tw;
  const float2* twr;
  unsigned np, nx;
  FastDiv divn;  // by nx
  long long so, pi;
  float scale;
  int do_scale;
  int pol_in, pol_out;  // L2 policies of the loads and the stores
  // weighted kind: spectra of n^3 grids, rows of hx points, times weight / |m|^2
  HartreeWeight weight;
  FastDiv divh;  // by hx
  int n, hx;
};
struct PencilKernel {
  cudaError_t (*launch)(const PencilArgs&, cudaStream_t) = nullptr;
  const void* func = nullptr;
  int A = 0, width = 0;  // split L = A * B; pencils per block
  size_t smem = 0;
};
// kind: 0 strided, 1 rows, 2 real rows of 2 L points forward (dir -1), 3 the
// same inverse (dir 1), 4 strided with weights (dir 1, even L), 5 strided for the
// half spectra of real grids (even L), 6 and 7 strided and rows in the order of the
// mixed-radix plan (dir -1, where kinds 0 and 1 have another); launch is null for an edge
// that is not plannable.
PencilKernel pencil_kernel_info(int L, int dir, int kind);

// Two-pass transforms of cubic edges (twopass.cuh).  tx, ty, tz: W_L^(n1 k) at
// [k * split + n1] for the splits AX, A and AZ.
constexpr int kTwoPassMaxLen = 192;  // = 6 * 32: ny = A B of a box
struct TwoPassArgs {
  const float2* in;  // may equal out
  float2* out;
  const float2 *tx, *tzg;
  float2 ty[kTwoPassMaxLen], tz[kTwoPassMaxLen];
  float scale;
  int do_scale;
  // grids that do not lie back to back (two_pass_apart_kernel_info): grid i is
  // plan grid map[first + i] (map null: first + i), at element off[.] of in and
  // out or at the pointers of the arrays
  const long long* off;
  const int* map;
  const float2* const* in_ptrs;
  float2* const* out_ptrs;
  int first;
};
struct TwoPassKernel {
  // passes 1 and 2 of `grids` grids; in_place: some output may overlie its input
  cudaError_t (*launch)(const TwoPassArgs&, int grids, bool in_place, cudaStream_t) = nullptr;
  const void* func[3] = {};  // pass 1, pass 1 in place, pass 2
  size_t smem[3] = {};
  int A = 0, AX = 0, AZ = 0;
};
TwoPassKernel two_pass_kernel_info(int L, int dir);        // launch null: none
TwoPassKernel two_pass_apart_kernel_info(int L, int dir);  // for mixed-edge plans
// The twiddles of splits A, AX, AZ of axes of L (x: lx) points: ty and tz into a,
// tx and tzg appended to tab (lx + L entries: a.tx and a.tzg are set once tab is
// on the device).
void two_pass_twiddles(int A, int AX, int AZ, int lx, int L, TwoPassArgs& a,
                       std::vector<float2>& tab);
int two_pass_prepare(const TwoPassKernel& k, int L, TwoPassArgs& a, std::vector<float2>& tab);

// Two-pass real transforms (twopass_real.cuh).
struct RealPassArgs : TwoPassArgs {
  const float2* twr;     // W_N^k, k <= N / 2
  float2* work;          // inverse: the grids' spectra between the passes
  HartreeWeight weight;  // inverse: grad null: none
};
struct RealPassKernel {
  cudaError_t (*launch)(const RealPassArgs&, int grids, cudaStream_t) = nullptr;
  const void* func[3] = {};
  size_t smem[3] = {};
  int A = 0, AX = 0, AZ = 0;
};
RealPassKernel real_pass_kernel_info(int n, int dir);  // launch null: none
// Edges whose real grids always run on these or, at 16 and 32, on a whole grid per
// block: no pencil passes are compiled for them.
constexpr bool real_kernels(int n) {
  return n == 16 || n == 32 || n == 48 || n == 60 || n == 64 || n == 72 || n == 80 || n == 90 ||
         n == 96 || n == 100 || n == 108 || n == 120 || n == 128;
}

// Two-pass transforms of boxes (twopass_box.cuh): ny = A B.
struct BoxArgs {
  const float2* in;
  float2* out;
  int in_place;  // out == in: pass 1 runs in clusters of A blocks
  const float2 *tx, *tzg;
  float2 ty[kTwoPassMaxLen], tz[kTwoPassMaxLen];
  int A, B, nx, tiles;  // tiles: pass-2 blocks of a grid, 16 of its B nx columns each
  FastDiv divA, divB, divt;
  float scale;
  int do_scale;
};
struct BoxKernel {
  const void* func = nullptr;
  int threads = 0;
  size_t smem = 0;  // pass 1: per row
  int split = 0;    // AX or AZ
  int threads32 = 0;  // pass 1: threads for 32 rows
};
BoxKernel box1_kernel_info(int nx, int dir);         // func null: none
BoxKernel box2_kernel_info(int A, int nz, int dir);
cudaError_t launch_box(const BoxKernel& k, unsigned grid, size_t smem, int cluster, const BoxArgs& a,
                       cudaStream_t s);

// A 3D transform as three pencil passes or two (passes.cu): complex grids (x, y,
// z, out of place or in place; always three if `fixed`), real grids to half
// spectra (x, y, z) or back (z into a workspace of work_points() complex points,
// y, x).
constexpr int kMaxChains = 2;
enum PassKind { kPassC2C = 0, kPassR2C = 1, kPassC2R = 2 };
struct AxisPasses {
  PassKind kind = kPassC2C;
  int nx = 0, ny = 0, nz = 0, hx = 0, batch = 0;  // hx: complex columns of a row
  long long chunk = 0;  // grids per chunk
  long long sub = 0;    // planes per launch of the x and y passes
  PencilKernel k[3];
  PencilKernel kw;      // kPassC2R: the z pass with weights
  TwoPassKernel two;    // launch not null: two passes instead
  TwoPassArgs two_args;
  BoxKernel box[2];     // func not null: two passes of a box
  BoxArgs box_args;
  RealPassKernel real;  // launch not null: two passes of real grids
  RealPassArgs real_args;
  int chains = 1;       // streams the chunks alternate between
  cudaStream_t side = nullptr;
  cudaEvent_t fork = nullptr, join = nullptr;
  std::mutex* mu = nullptr;
  float2* d_tab = nullptr;
  const float2* tw[3] = {nullptr, nullptr, nullptr};
  const float2* twr = nullptr;
  float scale = 1.0f;
  int do_scale = 0;
  int create(PassKind kind, int nx, int ny, int nz, int batch, int dir, float scale, int do_scale,
             int l2_bytes, bool fixed = false);
  void destroy();
  long long work_points() const;
  // weight (kPassC2R): the input times it, or null
  cudaError_t execute(const void* in, void* out, float2* work, cudaStream_t s,
                      const HartreeWeight* weight = nullptr) const;
  cudaError_t chunk_passes(long long g, const void* in, void* out, float2* work, cudaStream_t s,
                           const HartreeWeight* weight) const;
};

// Defined in the inst_*.cu translation units.
KernelInfo fused_kernel_info(int n, int dir, int variant);   // single-size kernel
KernelInfo mixed_kernel_info(int dir);          // all fused sizes
KernelInfo tc_kernel_info(int n, int dir, int prec, int variant);  // tensor-core kinds
KernelInfo real_kernel_info(int n, int dir);    // real grids (rgrid.cuh); launch null: none
cudaError_t launch_wait_selftest(unsigned* flag, unsigned* status, long long timeout_ns,
                                 cudaStream_t stream);

// Variant choice at plan creation (tune.cu): FFT3D_VARIANT / FFT3D_MIXED_VARIANT
// override; else the FFT3D_TUNE_CACHE entry for this device and problem;
// else, with FFT3D_TUNE=1, tune now (and record); else the built-in default.
int pick_variant(bool mixed, int n, int batch, int precision, int direction, const int* dims,
                 int count,
                 bool* is_default = nullptr);
std::vector<int> variant_candidates(bool mixed, int n, int precision);
int builtin_default_variant(bool mixed, int n, int batch, int precision);

}  // namespace fft3d

// The limits of a plan of `batch` cubic grids, as fft3d_plan_create checks them.
int fft3d_internal_validate(int n, int batch, int precision);
// A plan with a forced variant (plan.cu), for the autotuner.
int fft3d_internal_create_variant(bool mixed, int nx, int batch, int precision, int direction,
                                  const int* dims, int count, int variant, fft3d_plan* out);
