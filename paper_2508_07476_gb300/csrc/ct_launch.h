// Host-side entry points of the kernels (internal to the library).
#pragma once

#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "ct_common.cuh"

namespace ct {

// Set the shared-memory attributes of the kernel instantiations of one radius
// (once per plan and radius, before any launch may be captured into a graph).
cudaError_t prepare_rho_xy_kernels(int rk);
cudaError_t prepare_grad_split_kernels(int rk);

// Where a kernel of the chain goes: the stream, and whether its CTAs may be
// scheduled while the stream's previous kernel drains (`early`; every kernel
// launched through launch_after waits for that kernel first: after_previous()).
// That hides the launch latency of a chain of short kernels (64^3: 50 -> 40 us;
// 173 x 141 x 118: 207 -> 195; a 256^3 chunk: 1118 -> 1099), but an SM that
// never drains keeps its split of L1 and shared memory: the eigen stage after a
// tensor-core pass then runs with little L1 (512^3: 4837 -> 4949 us; a 384^3 chunk,
// 57M voxels: even), and beside other streams the waiting CTAs hold room those could
// use (12 crops on four streams: 6.28 -> 6.41 ms).  So: boxes of at most
// kEarlyMaxVox voxels, outside captured batches.
constexpr int64_t kEarlyMaxVox = (int64_t)1 << 25;
struct Queue {
  cudaStream_t st;
  bool early;
  Queue(cudaStream_t s, bool e = false) : st(s), early(e) {}
};

template <typename... P, typename... A>
cudaError_t launch_after(void (*kernel)(P...), dim3 grid, dim3 block, size_t smem, const Queue& q, A&&... args) {
  cudaLaunchAttribute attr;
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = q.early ? 1 : 0;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = q.st;
  cfg.attrs = &attr;
  cfg.numAttrs = q.early ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, kernel, static_cast<P>(args)...);
}

// How many segments to cut the walk of a streaming kernel into: `ctas` CTAs
// walk n positions each, a segment of L of them costing L + warm (warm: the
// steps before its first output, in steps of the walk), and `slots` CTAs are
// resident at once on `sms` SMs.  The cheapest of up to 64 cuts, whole waves
// of CTAs counted as they run side by side, the last one by the square root of
// the share of an SM's CTAs it still holds (fewer CTAs run faster, but not in
// proportion) and no less than kLoneCta (one waits for its own loads and
// barriers).  seg: a multiple of unit.  64^3, gradient x/y, z and rho z passes:
// 10.8, 8.3, 8.1 us, against 15.4, 16.4, 10.4 with cuts by powers of two above a
// fixed length (grad_z then has 16 CTAs); 173 x 141 x 118, gradient: 25.8 + 18.5 and
// 39.8 + 37.6.  The times are flat in the weights: kLoneCta 0.25 .. 0.8 and
// warm x 0.6 .. 1.5 move none of the measured volumes by more than 1%.
constexpr double kLoneCta = 0.5;
inline int walk_segment(int64_t ctas, int n, int unit, double warm, int slots, int sms) {
  double best = 1e300;
  int best_seg = n;
  for (int s = 1; s <= 64; ++s) {
    const int seg = ((n + s - 1) / s + unit - 1) / unit * unit;
    const int64_t total = ctas * ((n + seg - 1) / seg);
    const int64_t full = total / slots, rest = total - full * slots;
    double waves = (double)full;
    if (rest) {
      const double r = std::sqrt(std::min(1.0, (double)((rest + sms - 1) / sms) * sms / slots));
      waves += std::max(r, kLoneCta);
    }
    const double cost = waves * (seg + warm);
    if (cost < best * 0.99) best = cost, best_seg = seg;  // a finer cut only where it gains
    if (seg <= unit) break;
  }
  return best_seg;
}

// The CTA width (columns) of the kernels that walk along y: of `widths`, the
// first that covers a row of n0 with the least work.
int cta_width(int n0, int halo, double stage, const int* widths, int n);

// CTAs of a kernel resident at once on the current device (its SM count in *sms).
template <typename K>
int resident_ctas(K kernel, int threads, size_t smem, int* sms) {
  int dev = 0, per = 1;
  *sms = 1;
  cudaGetDevice(&dev);
  if (cudaDeviceGetAttribute(sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || *sms < 1) *sms = 1;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem) != cudaSuccess || per < 1) per = 1;
  return per * *sms;
}

// Instantiated radius that serves radius r (zero taps pad the difference), or -1.
int sigma_kernel_radius(int r);
int rho_kernel_radius(int r);

// The gradient and its products: launch_grad_xy writes the x/y-filtered partial
// fields (3 planes over ab = grad_partial_box(ob, vb, R, dims[2])) of vol;
// launch_grad_z takes their z pass and writes J (6 FP32 planes over ob), or
// with gout the gradient g (3 planes over ob: FP16 holding g * 2^-8 in the
// mixed form, FP32 otherwise) for launch_rho_tc_products to form J from.
Box grad_partial_box(const Box& ob, const Box& vb, int rs, int dimz);
// tx / ty / tz: the taps of each axis (anisotropic voxels); scale: the factor of
// each product (1 / (spacing_a spacing_b), xx yy zz xy xz yz).
// zero (nullable): a device counter that the kernel clears (the eigen stage's list).
cudaError_t launch_grad_xy(const uint16_t* vol, const Box& vb, const int dims[3], float* F, const Box& ab,
                           const Taps& tx, const Taps& ty, int rk, int* zero, const Queue& st);
cudaError_t launch_grad_z(const float* F, const Box& ab, void* J, const Box& ob, const Taps& tz,
                          const float scale[6], int rk, bool mixed, bool gout, const Queue& st);

// rho pass along x: out (6 planes over ob) from in (6 planes over ib).
cudaError_t launch_rho_x(const float* in, const Box& ib, const int dims[3], float* out, const Box& ob,
                         const Taps& taps, int rk, const Queue& st);

// rho passes along x and y fused: out (6 planes over ob) from in (6 planes over ib).
cudaError_t launch_rho_xy(const float* in, const Box& ib, const int dims[3], float* out, const Box& ob,
                          const Taps& tx, const Taps& ty, int rk, const Queue& st);

// rho pass along axis 1 (y) or 2 (z), streaming register windows of block_t (8 or 16) outputs.
cudaError_t launch_rho_stream(const float* in, const Box& ib, const int dims[3], float* out, const Box& ob, int axis,
                              const Taps& taps, int rk, int block_t, const Queue& st);

// rho pass along axis 0, 1 or 2 on the tensor cores (banded Toeplitz product,
// TF32 split operands, FP32 accumulation): same contract as launch_rho_x /
// launch_rho_stream.  prepare_rho_tc_kernels sets the shared-memory
// attributes (call before any capture).  Every CTA that gives up a bounded
// wait (ctl.wait_limit polls on another role; copies are waited for up to a
// fixed limit) stops, drains its copies and products, releases its tensor
// memory and adds 1 to *ctl.timeouts (a device word of the caller's plan).
struct TcCtl {
  unsigned int* timeouts;
  uint32_t wait_limit;
  int seg_cap;  // outputs per work unit at most (0: 512); the work is then spread over the SMs
};
cudaError_t prepare_rho_tc_kernels(int rk);
cudaError_t launch_rho_tc(const float* in, const Box& ib, const int dims[3], float* out, const Box& ob, int axis,
                          const Taps& taps, int rk, const TcCtl& ctl, const Queue& st);
// The same pass along axis 1 or 2 reading the gradient instead of the tensor:
// g (3 planes over ib: FP16 holding g * 2^-8 when half, else FP32, as
// launch_grad_z writes them with gout) -> out (6 planes over ob) = the pass of
// the products g_a g_b * scale[k], each formed as launch_grad_z forms it.
cudaError_t launch_rho_tc_products(const void* g, bool half, const Box& ib, const int dims[3], float* out,
                                   const Box& ob, int axis, const Taps& taps, const float scale[6], int rk,
                                   const TcCtl& ctl, const Queue& st);
// Whether a volume nx voxels wide suits launch_rho_tc along axis: 16-byte copies
// of its rows (x extent a multiple of 4).
bool rho_tc_volume_aligned(int nx, int axis);

// ---------------------------------------------------------------- batches
// One persistent launch per stage over a batch of volumes (MultiTable, in
// ct_common.cuh): the item's arguments as the single-item launch takes them;
// *_item fills the item's launch shape (seg: the whole walk, unsplit, since
// the batch's items fill the GPU) and returns its grid; the blocks compute
// every output with the same operations as the single launch, so a batch
// reproduces every item's results bit for bit; launch_*_multi runs the stage
// over a device table of items (grid: the SMs times the blocks each holds, at
// most `blocks`).
struct GxyItem {
  const uint16_t* vol;
  Box vb;
  int dimx, dimy;
  float* F;
  Box ab;
  int seg;
};
struct GzItem {
  const float* F;
  Box ab;
  float* J;
  Box ob;
  int seg;
};
struct RxyItem {
  const float* in;
  Box ib;
  int dimx, dimy;
  float* out;
  Box ob;
  int seg;
};
struct RzItem {
  const float* in;
  Box ib;
  int dim_axis;
  float* out;
  Box ob;
  int seg;
};
uint3 grad_xy_item(int rk, GxyItem& it);
cudaError_t launch_grad_xy_multi(const GxyItem* items, const MultiTable& T, int64_t blocks, const Taps& tx,
                                 const Taps& ty, int rk, cudaStream_t st);
uint3 grad_z_item(int rk, GzItem& it);
cudaError_t launch_grad_z_multi(const GzItem* items, const MultiTable& T, int64_t blocks, const Taps& tz,
                                const float scale[6], int rk, bool mixed, cudaStream_t st);
// the fused x / y stencil at the CTA width `xt`: 128 or 256 (rho_xy_width; the single launch has
// more widths to choose from)
int rho_xy_width(int n0);
uint3 rho_xy_item(int rk, int xt, RxyItem& it);
cudaError_t launch_rho_xy_multi(const RxyItem* items, const MultiTable& T, int64_t blocks, const Taps& tx,
                                const Taps& ty, int rk, int xt, cudaStream_t st);
// the z stencil (axis 2) of k_rho_stream, block_t outputs per thread and block; the
// block shape of an item: rho_stream_block, fixed per batch launch (the single
// launch takes k_rho_z2 over even rows)
uint3 rho_z_item(int rk, int block_t, dim3 block, RzItem& it);
dim3 rho_stream_block(const Box& ob, int axis);
cudaError_t launch_rho_z_multi(const RzItem* items, const MultiTable& T, int64_t blocks, dim3 block,
                               const Taps& taps, int rk, int block_t, cudaStream_t st);

// Persistent grid of a multi-item launch: the SMs times the CTAs each holds.
template <typename K>
int persistent_grid(K kernel, int threads, size_t smem, int64_t blocks) {
  int dev = 0, sms = 1, per = 1;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, kernel, threads, smem) != cudaSuccess || per < 1) per = 1;
  const int64_t g = (int64_t)per * sms;
  return (int)(blocks < g ? (blocks > 0 ? blocks : 1) : g);
}

struct EigOut {
  void* vec;
  void* ha;
  void* ia;
  void* fa;
  int vec_t, ang_t, fa_t;
  Box ab;  // box covered by the output arrays
};

struct Fallback {
  float gap = kDegenerateGap;  // listing threshold of the arithmetic form (degenerate_gap)
  int* count;                 // device counter of listed voxels (reset per launch)
  unsigned long long* total;  // device running total (for statistics)
  int64_t* list;
  int64_t cap;
};

// The near-degeneracy listing threshold of an arithmetic form (FP32 / mixed).
inline float degenerate_gap(bool mixed) { return mixed ? kDegenerateGapMixed : kDegenerateGap; }

// One item of a batched eigen stage (the arguments of launch_eig_angles).
struct EigItem {
  const float* S;
  Box sb, ob;
  const uint8_t* mask;
  Box mb;
  Frame F;
  EigOut o;
  Fallback fb;
};
// Whether an item suits the batched eigen kernels (32-bit indices, rows in the grid).
bool eig_item_ok(const EigItem& it);
uint3 eig_item_grid(bool compact, const EigItem& it);
cudaError_t launch_eig_multi(const EigItem* items, const MultiTable& T, int64_t blocks, bool compact, int vt, int at,
                             int ft, bool plain, float fill, cudaStream_t st);
// The re-solve of every item's listed voxels (at most max_per_item each) in one launch.
cudaError_t launch_eig_fallback_multi(const EigItem* items, int n_items, int64_t max_per_item, float fill, bool mixed,
                                      cudaStream_t st);

// Per-voxel eigen-solve + HA/IA/FA over ob from S (6 planes over sb); mask
// array (nullable) covers mb.  Near-degenerate voxels are appended to fb.
// compact: with a mask, each row segment lists its inside voxels first and
// solves them with full warps (the same arithmetic per voxel).
cudaError_t launch_eig_angles(const float* S, const Box& sb, const Box& ob, const uint8_t* mask, const Box& mb,
                              const Frame& F, float fill, const EigOut& o, bool mixed, const Fallback& fb,
                              bool compact, const Queue& st);
// Re-solve the listed voxels (FP32 Jacobi, or FP64 in the mixed form) and rewrite their outputs.
cudaError_t launch_eig_angles_fallback(const float* S, const Box& sb, const Box& ob, const uint8_t* mask,
                                       const Box& mb, const Frame& F, float fill, const EigOut& o, bool mixed,
                                       const Fallback& fb, int64_t max_items, const Queue& st);

// Stage kernels: eigen only (evals + unoriented evec), and angles only.
cudaError_t launch_eig_only(const float* S, int64_t n, float* evals, float* evec, bool mixed, const Fallback& fb,
                            cudaStream_t st);
cudaError_t launch_eig_only_fallback(const float* S, int64_t n, float* evals, float* evec, bool mixed,
                                     const Fallback& fb, int64_t max_items, const Queue& st);
cudaError_t launch_angles_only(const float* evec, const float* evals, const Box& ob, const uint8_t* mask,
                               const Frame& F, float fill, const EigOut& o, cudaStream_t st);

}  // namespace ct
