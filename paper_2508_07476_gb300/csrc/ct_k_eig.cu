// Eigen-decomposition of the structure tensor and the cardiac descriptors
// (Figure 1b: smallest-eigenvalue eigenvector as the fibre direction;
// Figure 1c: HA, IA, FA in the cylindrical left-ventricle frame; Figure 1a:
// optional myocardial mask).
//
// Every voxel first takes the FP32 closed form (trigonometric roots of the
// characteristic cubic, cross product of two rows of S - l1 I).  Voxels whose
// two smallest eigenvalues nearly coincide, where that form loses half of its
// digits, are appended to a compact list and re-solved by a second kernel:
// FP32 cyclic Jacobi in the FP32 form, FP64 deflation (FP64 Jacobi where even
// that has no gap to work with) in the mixed form.  The list keeps the re-solve off
// the common path, so no warp diverges into it.
#include <algorithm>

#include "ct.h"
#include "ct_common.cuh"
#include "ct_launch.h"

namespace ct {

__device__ __forceinline__ Sym3<float> load_sym(const float* S, int64_t n, int64_t i) {
  Sym3<float> s;
  s.a = __ldca(S + i);
  s.b = __ldca(S + n + i);
  s.c = __ldca(S + 2 * n + i);
  s.d = __ldca(S + 3 * n + i);
  s.e = __ldca(S + 4 * n + i);
  s.f = __ldca(S + 5 * n + i);
  return s;
}

// Robust re-solve of one voxel.
__device__ __forceinline__ void resolve(const Sym3<float>& s, bool mixed, float l[3], float v[3]) {
  if (mixed) {
    if (!eig_deflate(s, l, v)) {
      Sym3<double> sd{(double)s.a, (double)s.b, (double)s.c, (double)s.d, (double)s.e, (double)s.f};
      double ld[3], vd[3];
      eig_jacobi<double>(sd, ld, vd);
      for (int k = 0; k < 3; ++k) {
        l[k] = (float)ld[k];
        v[k] = (float)vd[k];
      }
    }
  } else {
    eig_jacobi<float>(s, l, v);
  }
  float nv = rsqrtf(v[0] * v[0] + v[1] * v[1] + v[2] * v[2]);
  v[0] *= nv; v[1] *= nv; v[2] *= nv;
}

// Outputs of one voxel: oriented vector, HA, IA, FA (or fill outside the mask).
// VT / AT / FT: compile-time encodings of the vector / angle / FA outputs, or
// -1 to take them from `o` at run time.
template <int VT = -1, int AT = -1, int FT = -1, typename IT = int64_t, bool PLAIN = false>
__device__ __forceinline__ void write_voxel(const EigOut& o, IT oi, bool inside, const Frame& F, int x, int y,
                                            int z, const float l[3], float v[3], float fill) {
  const IT n = (IT)box_vox(o.ab);
  if (!inside) {
    store_val<VT, IT>(o.vec, oi, o.vec_t, fill);
    if (o.vec) {
      store_val<VT, IT>(o.vec, n + oi, o.vec_t, fill);
      store_val<VT, IT>(o.vec, 2 * n + oi, o.vec_t, fill);
    }
    store_angle<AT, IT>(o.ha, oi, o.ang_t, fill, false);
    store_angle<AT, IT>(o.ia, oi, o.ang_t, fill, false);
    store_val<FT, IT>(o.fa, oi, o.fa_t, fill);
    return;
  }
  float ha, ia;
  bool framed = ha_ia<PLAIN>(F, x, y, z, v, ha, ia);
  if (!framed) orient_largest(v);
  if (o.vec) {
    store_val<VT, IT>(o.vec, oi, o.vec_t, v[0]);
    store_val<VT, IT>(o.vec, n + oi, o.vec_t, v[1]);
    store_val<VT, IT>(o.vec, 2 * n + oi, o.vec_t, v[2]);
  }
  store_angle<AT, IT>(o.ha, oi, o.ang_t, framed ? ha : fill, framed);
  store_angle<AT, IT>(o.ia, oi, o.ang_t, framed ? ia : fill, framed);
  store_val<FT, IT>(o.fa, oi, o.fa_t, fa_of(l));
}

__device__ __forceinline__ void push_fallback(const Fallback& fb, int64_t i) {
  int slot = atomicAdd(fb.count, 1);
  if (slot < fb.cap) fb.list[slot] = i;
  atomicAdd(fb.total, 1ull);
}

// One thread per voxel on a 3D grid (x from the thread index, y and z from the
// block index, rows beyond 65535 folded into blockIdx.z), so no index division.
// 8 CTAs of 256 threads per SM (32 registers): the kernel streams HBM and
// needs every resident warp to cover its latency.
#ifndef CT_EIG_MINB
#define CT_EIG_MINB 8
#endif
// Whether the re-solve's CTAs may start while the stage still runs (after_previous): not where
// many CTAs of narrow rows would be bound by it.
__device__ __forceinline__ bool starts_next(const Box& ob) {
  return ob.n[0] >= 96 || (int64_t)ob.n[1] * ob.n[2] < 4096;
}
template <int VT, int AT, int FT>
__global__ void __launch_bounds__(256, CT_EIG_MINB)
    k_eig_angles(const float* __restrict__ S, Box sb, Box ob, const uint8_t* __restrict__ mask, Box mb, Frame F,
                 float fill, EigOut o, bool mixed, Fallback fb) {
  after_previous(starts_next(ob));
  const int x = ob.lo[0] + blockIdx.x * blockDim.x + threadIdx.x;
  if (x >= ob.lo[0] + ob.n[0]) return;
  const int row = blockIdx.z * gridDim.y + blockIdx.y;  // y + ny * z within ob
  if (row >= ob.n[1] * ob.n[2]) return;
  const int yr = row % ob.n[1], zr = row / ob.n[1];  // one division per thread, 32-bit
  const int y = ob.lo[1] + yr, z = ob.lo[2] + zr;
  const bool inside = mask == nullptr || __ldg(mask + box_index(mb, x, y, z)) != 0;
  float l[3] = {0.f, 0.f, 0.f}, v[3] = {1.f, 0.f, 0.f};
  if (inside) {
    const Sym3<float> s = load_sym(S, box_vox(sb), box_index(sb, x, y, z));
    if (!eig_closed(s, l, v, fb.gap)) push_fallback(fb, ((int64_t)zr * ob.n[1] + yr) * ob.n[0] + (x - ob.lo[0]));
  }
  write_voxel<VT, AT, FT>(o, box_index(o.ab, x, y, z), inside, F, x, y, z, l, v, fill);
}

// The same for boxes whose planes fit 32-bit indices and whose rows fit the
// grid's y and z: (y, z) from the block index, every index in 32 bits.
__device__ __forceinline__ int box_index32(const Box& b, int x, int y, int z) {
  return ((z - b.lo[2]) * b.n[1] + (y - b.lo[1])) * b.n[0] + (x - b.lo[0]);
}

template <int VT, int AT, int FT, bool PLAIN, typename BLK>
__device__ __forceinline__ void eig32_body(const float* __restrict__ S, Box sb, Box ob,
                                           const uint8_t* __restrict__ mask, Box mb, const Frame& F, float fill,
                                           const EigOut& o, const Fallback& fb, const BLK blk) {
  const int x = ob.lo[0] + blk.x() * blockDim.x + threadIdx.x;
  if (x >= ob.lo[0] + ob.n[0]) return;
  const int y = ob.lo[1] + blk.y(), z = ob.lo[2] + blk.z();
  const bool inside = mask == nullptr || __ldg(mask + box_index32(mb, x, y, z)) != 0;
  float l[3] = {0.f, 0.f, 0.f}, v[3] = {1.f, 0.f, 0.f};
  if (inside) {
    const int ns = sb.n[0] * sb.n[1] * sb.n[2];
    const int si = box_index32(sb, x, y, z);
    Sym3<float> s;
    s.a = __ldca(S + si);
    s.b = __ldca(S + ns + si);
    s.c = __ldca(S + 2 * ns + si);
    s.d = __ldca(S + 3 * ns + si);
    s.e = __ldca(S + 4 * ns + si);
    s.f = __ldca(S + 5 * ns + si);
    if (!eig_closed(s, l, v, fb.gap))
      push_fallback(fb, ((int64_t)blk.z() * ob.n[1] + blk.y()) * ob.n[0] + (x - ob.lo[0]));
  }
  write_voxel<VT, AT, FT, int, PLAIN>(o, box_index32(o.ab, x, y, z), inside, F, x, y, z, l, v, fill);
}

template <int VT, int AT, int FT, bool PLAIN>
__global__ void __launch_bounds__(256, CT_EIG_MINB)
    k_eig_angles32(const float* __restrict__ S, Box sb, Box ob, const uint8_t* __restrict__ mask, Box mb, Frame F,
                   float fill, EigOut o, bool mixed, Fallback fb) {
  (void)mixed;
  after_previous(starts_next(ob));
  eig32_body<VT, AT, FT, PLAIN>(S, sb, ob, mask, mb, F, fill, o, fb, HwBlock{});
}

// The unmasked form: a CTA of kEigRowThreads threads takes up to kEigRowSpan
// consecutive voxels of one row in a loop, so that the row's part of the indices
// and of the frame, and the kernel's set-up, are paid once per CTA and not once
// per voxel.  The solve is bound by its instructions (about 400 per voxel, 87% of
// the issue slots): 173 x 141 x 118 45.0 us with a voxel per thread, 40.8 so; 12 uneven
// crops 6.26 -> 6.17 ms (spans of 4 voxels per thread 6.21, of 2 6.29; 32 or 20 CTAs
// per SM instead of 24, at 32 / 42 registers: 6.24).
constexpr int kEigRowThreads = 64;
constexpr int kEigRowSpan = 8 * kEigRowThreads;
// Whether rows of n voxels without a mask take k_eig_angles_rows.  It walks a row in steps of
// two warps: 1 or 3 warps of voxels leave half a CTA idle in one of one or two steps, and a
// short second span a CTA with little to do; those take a thread per voxel.  12000 / n x n x 300
// voxels, F16 outputs, rows against threads: 24 columns 117 and 84 us, 72 74 and 63, 96 58 and
// 51, 530 54 and 50; but 64 49 and 54, 128 45 and 49, 173 49 and 55, 256 45 and 49, 384 45 and
// 49, 1000 47 and 51.  At 129 to 160 columns rows are up to 4% slower alone and faster beside
// other streams (117 x 192 x 109 and 129 x 69 x 157 in one call 301 and 307 us).
static bool eig_rows(int n) {
  const int warps = (n + 31) / 32, last = n % kEigRowSpan;
  return warps != 1 && warps != 3 && !(n > kEigRowSpan && last > 0 && last <= 128);
}

template <int VT, int AT, int FT, bool PLAIN>
__global__ void __launch_bounds__(kEigRowThreads, 24)
    k_eig_angles_rows(const float* __restrict__ S, Box sb, Box ob, Frame F, float fill, EigOut o, Fallback fb) {
  after_previous(starts_next(ob));
  const int y = ob.lo[1] + blockIdx.y, z = ob.lo[2] + blockIdx.z;
  const int x0 = ob.lo[0] + blockIdx.x * kEigRowSpan;
  const int xend = min(ob.lo[0] + ob.n[0], x0 + kEigRowSpan);
  const int ns = sb.n[0] * sb.n[1] * sb.n[2];
  const float* p = S + box_index32(sb, x0, y, z) + threadIdx.x;
  int oi = box_index32(o.ab, x0, y, z) + threadIdx.x;
#pragma unroll 1
  for (int x = x0 + threadIdx.x; x < xend; x += kEigRowThreads, p += kEigRowThreads, oi += kEigRowThreads) {
    Sym3<float> s;
    s.a = __ldca(p);
    s.b = __ldca(p + ns);
    s.c = __ldca(p + 2 * ns);
    s.d = __ldca(p + 3 * ns);
    s.e = __ldca(p + 4 * ns);
    s.f = __ldca(p + 5 * ns);
    float l[3], v[3];
    if (!eig_closed(s, l, v, fb.gap))
      push_fallback(fb, ((int64_t)blockIdx.z * ob.n[1] + blockIdx.y) * ob.n[0] + (x - ob.lo[0]));
    write_voxel<VT, AT, FT, int, PLAIN>(o, oi, true, F, x, y, z, l, v, fill);
  }
}

// The masked form: a CTA of kEigThreads threads takes kEigSpan consecutive
// voxels of one row (voxel x0 + t + kEigThreads k for thread t, so that the
// mask loads and the fill stores stay coalesced), writes the fill outputs of
// those outside the mask at once and lists the inside ones in shared memory,
// in x order (warp ballots; every warp scans the per-warp counts itself).
// The eigen solve then runs over the list, so that only the last warp of a row
// segment has idle lanes, where a warp per 32 voxels would idle wherever the
// wall boundary cuts it.  Each voxel's arithmetic is that of k_eig_angles32;
// only the thread that does it differs.
// Two-warp CTAs over 512 voxels: 32 CTAs per SM, whose barriers and list
// phases interleave (512^3: 0.97 ms, against 1.09 for 256 threads x 2 voxels,
// 1.01 for 128 x 4, 0.99 for 64 x 4, 1.04 for 64 x 16)
#ifndef CT_EIG_THREADS
#define CT_EIG_THREADS 64
#endif
#ifndef CT_EIG_SPAN_K
#define CT_EIG_SPAN_K 8
#endif
#ifndef CT_EIG_ILP
#define CT_EIG_ILP 1
#endif
constexpr int kEigThreads = CT_EIG_THREADS;        // threads per CTA (tuning choice)
constexpr int kEigSpanK = CT_EIG_SPAN_K;           // voxels per thread per segment (tuning choice)
constexpr int kEigSpan = kEigThreads * kEigSpanK;  // voxels per segment
constexpr int kEigIlp = CT_EIG_ILP;                // list entries per thread whose tensors load together (tuning choice)
constexpr int kEigWarps = kEigThreads / 32;
static_assert(kEigWarps * kEigSpanK <= 32, "one warp scans the per-warp counts");
static_assert(kEigSpan <= 65536, "list entries are 16-bit");

template <int VT, int AT, int FT, bool PLAIN, typename BLK>
__device__ __forceinline__ void eig_compact_body(const float* __restrict__ S, Box sb, Box ob,
                                                 const uint8_t* __restrict__ mask, Box mb, const Frame& F, float fill,
                                                 const EigOut& o, const Fallback& fb, const BLK blk) {
  constexpr int NC = kEigWarps * kEigSpanK;
  __shared__ uint16_t list[kEigSpan];
  __shared__ int cnt[NC];
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int x0 = ob.lo[0] + blk.x() * kEigSpan;
  const int xend = ob.lo[0] + ob.n[0];
  const int y = ob.lo[1] + blk.y(), z = ob.lo[2] + blk.z();
  unsigned in_bits[kEigSpanK];
#pragma unroll
  for (int k = 0; k < kEigSpanK; ++k) {
    const int x = x0 + t + kEigThreads * k;
    const bool valid = x < xend;
    const bool inside = valid && __ldg(mask + box_index32(mb, x, y, z)) != 0;
    if (valid && !inside) {
      float l[3] = {0.f, 0.f, 0.f}, v[3] = {1.f, 0.f, 0.f};
      write_voxel<VT, AT, FT, int, PLAIN>(o, box_index32(o.ab, x, y, z), false, F, x, y, z, l, v, fill);
    }
    in_bits[k] = __ballot_sync(0xffffffffu, inside);
    if (lane == 0) cnt[k * kEigWarps + warp] = __popc(in_bits[k]);
  }
  __syncthreads();
  // every warp scans the counts, in (k, warp) order = x order, itself
  const int c = lane < NC ? cnt[lane] : 0;
  int incl = c;
#pragma unroll
  for (int d = 1; d < NC; d <<= 1) {
    const int u = __shfl_up_sync(0xffffffffu, incl, d);
    if (lane >= d) incl += u;
  }
  const int total = __shfl_sync(0xffffffffu, incl, NC - 1);
  const unsigned below = (1u << lane) - 1u;
#pragma unroll
  for (int k = 0; k < kEigSpanK; ++k) {
    const int base = __shfl_sync(0xffffffffu, incl - c, k * kEigWarps + warp);
    if (in_bits[k] >> lane & 1u) list[base + __popc(in_bits[k] & below)] = (uint16_t)(t + kEigThreads * k);
  }
  __syncthreads();
  const int ns = sb.n[0] * sb.n[1] * sb.n[2];
  for (int i0 = t; i0 < total; i0 += kEigThreads * kEigIlp) {
    int xs[kEigIlp];
    Sym3<float> s[kEigIlp];
#pragma unroll
    for (int u = 0; u < kEigIlp; ++u) {
      const int i = i0 + kEigThreads * u;
      xs[u] = x0 + list[i < total ? i : i0];
      const int si = box_index32(sb, xs[u], y, z);
      s[u].a = __ldca(S + si);
      s[u].b = __ldca(S + ns + si);
      s[u].c = __ldca(S + 2 * ns + si);
      s[u].d = __ldca(S + 3 * ns + si);
      s[u].e = __ldca(S + 4 * ns + si);
      s[u].f = __ldca(S + 5 * ns + si);
    }
#pragma unroll
    for (int u = 0; u < kEigIlp; ++u) {
      if (i0 + kEigThreads * u >= total) break;
      const int x = xs[u];
      float l[3], v[3];
      if (!eig_closed(s[u], l, v, fb.gap))
        push_fallback(fb, ((int64_t)blk.z() * ob.n[1] + blk.y()) * ob.n[0] + (x - ob.lo[0]));
      write_voxel<VT, AT, FT, int, PLAIN>(o, box_index32(o.ab, x, y, z), true, F, x, y, z, l, v, fill);
    }
  }
}

template <int VT, int AT, int FT, bool PLAIN>
__global__ void __launch_bounds__(kEigThreads, CT_EIG_MINB * 256 / kEigThreads)
    k_eig_angles_compact(const float* __restrict__ S, Box sb, Box ob, const uint8_t* __restrict__ mask, Box mb,
                         Frame F, float fill, EigOut o, bool mixed, Fallback fb) {
  (void)mixed;
  after_previous(starts_next(ob));
  eig_compact_body<VT, AT, FT, PLAIN>(S, sb, ob, mask, mb, F, fill, o, fb, HwBlock{});
}

// The eigen stage over a batch of volumes in one persistent launch: masked
// items through the compacted form (kEigThreads per CTA), unmasked ones one
// voxel per thread (kEigMultiThreads per CTA); the encodings and the plain
// frame are the batch's (the plan's).
constexpr int kEigMultiThreads = 256;
template <int VT, int AT, int FT, bool PLAIN, bool COMPACT>
__global__ void __launch_bounds__(COMPACT ? kEigThreads : kEigMultiThreads,
                                  COMPACT ? CT_EIG_MINB * 256 / kEigThreads : CT_EIG_MINB)
    k_eig_multi(const EigItem* __restrict__ items, const MultiTable T, float fill) {
  for_each_vblock<COMPACT ? 4 : 16>(T, [&](int i, const VBlock& v) {
    const EigItem& it = items[i];
    if (COMPACT)
      eig_compact_body<VT, AT, FT, PLAIN>(it.S, it.sb, it.ob, it.mask, it.mb, it.F, fill, it.o, it.fb, v);
    else
      eig32_body<VT, AT, FT, PLAIN>(it.S, it.sb, it.ob, it.mask, it.mb, it.F, fill, it.o, it.fb, v);
  });
}

__global__ void __launch_bounds__(128)
    k_eig_angles_fallback(const float* __restrict__ S, Box sb, Box ob, const uint8_t* __restrict__ mask, Box mb,
                          Frame F, float fill, EigOut o, bool mixed, Fallback fb) {
  after_previous();
  const int64_t cnt = min((int64_t)*fb.count, fb.cap);
  const int64_t ns = box_vox(sb);
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < cnt; j += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = fb.list[j];
    const int x = ob.lo[0] + (int)(i % ob.n[0]);
    const int y = ob.lo[1] + (int)((i / ob.n[0]) % ob.n[1]);
    const int z = ob.lo[2] + (int)(i / ((int64_t)ob.n[0] * ob.n[1]));
    Sym3<float> s = load_sym(S, ns, box_index(sb, x, y, z));
    float l[3], v[3];
    resolve(s, mixed, l, v);
    write_voxel(o, box_index(o.ab, x, y, z), true, F, x, y, z, l, v, fill);
  }
}

// The re-solve of a batch: blockIdx.y = item, each item's listed voxels grid-strided.
__global__ void __launch_bounds__(128)
    k_eig_fallback_multi(const EigItem* __restrict__ items, float fill, bool mixed) {
  const EigItem& it = items[blockIdx.y];
  const int64_t cnt = min((int64_t)*it.fb.count, it.fb.cap);
  const int64_t ns = box_vox(it.sb);
  const Box ob = it.ob;
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < cnt; j += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = it.fb.list[j];
    const int x = ob.lo[0] + (int)(i % ob.n[0]);
    const int y = ob.lo[1] + (int)((i / ob.n[0]) % ob.n[1]);
    const int z = ob.lo[2] + (int)(i / ((int64_t)ob.n[0] * ob.n[1]));
    Sym3<float> s = load_sym(it.S, ns, box_index(it.sb, x, y, z));
    float l[3], v[3];
    resolve(s, mixed, l, v);
    write_voxel(it.o, box_index(it.o.ab, x, y, z), true, it.F, x, y, z, l, v, fill);
  }
}

// The re-solve launches: the listed voxels are few (the list's length is read
// on the device), so a few CTAs per SM stride over it; a grid sized by the box
// would mostly start CTAs that find nothing (batches launch one per item).
static int fallback_grid(int64_t max_items) {
  static const int sms = [] {
    int dev = 0, n = 0;
    cudaGetDevice(&dev);
    return cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev) == cudaSuccess && n > 0 ? n : 152;
  }();
  const int64_t b = (max_items + 127) / 128;
  return (int)std::max<int64_t>(1, std::min<int64_t>(b, 4 * sms));
}

static int grid_for(int64_t n, int threads) {
  int64_t b = (n + threads - 1) / threads;
  const int64_t cap = 152 * 64;  // grid-stride beyond this
  return (int)(b < 1 ? 1 : (b > cap ? cap : b));
}

cudaError_t launch_eig_angles(const float* S, const Box& sb, const Box& ob, const uint8_t* mask, const Box& mb,
                              const Frame& F, float fill, const EigOut& o, bool mixed, const Fallback& fb,
                              bool compact, const Queue& st) {
  int64_t n = box_vox(ob);
  if (n == 0) return cudaSuccess;
  const int rows = ob.n[1] * ob.n[2];
  const int gy = rows < 65535 ? rows : 65535;
  // 128-thread rows where 256 would leave more columns idle (e.g. width 384)
  const int nt = ((ob.n[0] + 127) / 128 * 128 - ob.n[0]) < ((ob.n[0] + 255) / 256 * 256 - ob.n[0]) ? 128 : 256;
  dim3 grid((ob.n[0] + nt - 1) / nt, gy, (rows + gy - 1) / gy);
  // 32-bit indices and a (x, y, z) grid when every plane set fits
  const int64_t lim = ((int64_t)1 << 31) - 1;
  if (ob.n[1] <= 65535 && ob.n[2] <= 65535 && 6 * box_vox(sb) <= lim && 3 * box_vox(o.ab) <= lim &&
      box_vox(mb) <= lim) {
    dim3 g3((ob.n[0] + nt - 1) / nt, ob.n[1], ob.n[2]);
    // unit voxels and a fixed centre take the plain frame
    const bool plain = F.sp[0] == 1.f && F.sp[1] == 1.f && F.sp[2] == 1.f && F.centres == nullptr;
    if (mask != nullptr && compact) {
      dim3 gc((ob.n[0] + kEigSpan - 1) / kEigSpan, ob.n[1], ob.n[2]);
      if (o.vec_t == CT_OUT_F32 && o.ang_t == CT_OUT_F32 && o.fa_t == CT_OUT_F32) {
        if (plain)
          return launch_after(k_eig_angles_compact<0, 0, 0, true>, gc, kEigThreads, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed,
                              fb);
        else
          return launch_after(k_eig_angles_compact<0, 0, 0, false>, gc, kEigThreads, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed,
                              fb);
      } else if (o.vec_t == CT_OUT_F16 && o.ang_t == CT_OUT_F16 && o.fa_t == CT_OUT_F16) {
        if (plain)
          return launch_after(k_eig_angles_compact<1, 1, 1, true>, gc, kEigThreads, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed,
                              fb);
        else
          return launch_after(k_eig_angles_compact<1, 1, 1, false>, gc, kEigThreads, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed,
                              fb);
      } else if (o.vec_t == CT_OUT_F32 && o.ang_t == CT_OUT_U8Q && o.fa_t == CT_OUT_F16 && plain) {
        return launch_after(k_eig_angles_compact<0, 2, 1, true>, gc, kEigThreads, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed,
                            fb);
      } else if (o.ang_t == CT_OUT_U8Q && o.fa_t == CT_OUT_F16) {
        return launch_after(k_eig_angles_compact<-1, 2, 1, false>, gc, kEigThreads, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed,
                            fb);
      } else {
        return launch_after(k_eig_angles_compact<-1, -1, -1, false>, gc, kEigThreads, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed,
                            fb);
      }
    }
    if (mask == nullptr && plain && eig_rows(ob.n[0])) {
      const dim3 gr((ob.n[0] + kEigRowSpan - 1) / kEigRowSpan, ob.n[1], ob.n[2]);
      if (o.vec_t == CT_OUT_F32 && o.ang_t == CT_OUT_F32 && o.fa_t == CT_OUT_F32)
        return launch_after(k_eig_angles_rows<0, 0, 0, true>, gr, kEigRowThreads, 0, st, S, sb, ob, F, fill, o, fb);
      if (o.vec_t == CT_OUT_F16 && o.ang_t == CT_OUT_F16 && o.fa_t == CT_OUT_F16)
        return launch_after(k_eig_angles_rows<1, 1, 1, true>, gr, kEigRowThreads, 0, st, S, sb, ob, F, fill, o, fb);
      if (o.vec_t == CT_OUT_F32 && o.ang_t == CT_OUT_U8Q && o.fa_t == CT_OUT_F16)
        return launch_after(k_eig_angles_rows<0, 2, 1, true>, gr, kEigRowThreads, 0, st, S, sb, ob, F, fill, o, fb);
    }
    if (o.vec_t == CT_OUT_F32 && o.ang_t == CT_OUT_F32 && o.fa_t == CT_OUT_F32) {
      if (plain)
        return launch_after(k_eig_angles32<0, 0, 0, true>, g3, nt, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed, fb);
      else
        return launch_after(k_eig_angles32<0, 0, 0, false>, g3, nt, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed, fb);
    } else if (o.vec_t == CT_OUT_F16 && o.ang_t == CT_OUT_F16 && o.fa_t == CT_OUT_F16) {
      if (plain)
        return launch_after(k_eig_angles32<1, 1, 1, true>, g3, nt, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed, fb);
      else
        return launch_after(k_eig_angles32<1, 1, 1, false>, g3, nt, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed, fb);
    } else if (o.vec_t == CT_OUT_F32 && o.ang_t == CT_OUT_U8Q && o.fa_t == CT_OUT_F16 && plain) {
      return launch_after(k_eig_angles32<0, 2, 1, true>, g3, nt, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed, fb);
    } else if (o.ang_t == CT_OUT_U8Q && o.fa_t == CT_OUT_F16) {
      return launch_after(k_eig_angles32<-1, 2, 1, false>, g3, nt, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed, fb);
    } else {
      return launch_after(k_eig_angles32<-1, -1, -1, false>, g3, nt, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed, fb);
    }
  }
  // the encodings of the common configurations are compiled in; others are read at run time
  if (o.vec_t == CT_OUT_F32 && o.ang_t == CT_OUT_F32 && o.fa_t == CT_OUT_F32)
    return launch_after(k_eig_angles<0, 0, 0>, grid, nt, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed, fb);
  else if (o.vec_t == CT_OUT_F16 && o.ang_t == CT_OUT_F16 && o.fa_t == CT_OUT_F16)
    return launch_after(k_eig_angles<1, 1, 1>, grid, nt, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed, fb);
  else if (o.ang_t == CT_OUT_U8Q && o.fa_t == CT_OUT_F16)
    return launch_after(k_eig_angles<-1, 2, 1>, grid, nt, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed, fb);
  else
    return launch_after(k_eig_angles<-1, -1, -1>, grid, nt, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed, fb);
}

cudaError_t launch_eig_angles_fallback(const float* S, const Box& sb, const Box& ob, const uint8_t* mask,
                                       const Box& mb, const Frame& F, float fill, const EigOut& o, bool mixed,
                                       const Fallback& fb, int64_t max_items, const Queue& st) {
  if (max_items <= 0) return cudaSuccess;
  return launch_after(k_eig_angles_fallback, fallback_grid(max_items), 128, 0, st, S, sb, ob, mask, mb, F, fill, o, mixed,
                      fb);
}

// ------------------------------------------------------------ batches
bool eig_item_ok(const EigItem& it) {
  const int64_t lim = ((int64_t)1 << 31) - 1;
  return it.ob.n[1] <= 65535 && it.ob.n[2] <= 65535 && 6 * box_vox(it.sb) <= lim && 3 * box_vox(it.o.ab) <= lim &&
         box_vox(it.mb) <= lim;
}

uint3 eig_item_grid(bool compact, const EigItem& it) {
  const Box& ob = it.ob;
  return compact ? make_uint3((ob.n[0] + kEigSpan - 1) / kEigSpan, ob.n[1], ob.n[2])
                 : make_uint3((ob.n[0] + kEigMultiThreads - 1) / kEigMultiThreads, ob.n[1], ob.n[2]);
}

template <int VT, int AT, int FT, bool PLAIN, bool COMPACT>
static cudaError_t eig_multi_t(const EigItem* items, const MultiTable& T, int64_t blocks, float fill,
                               cudaStream_t st) {
  constexpr int threads = COMPACT ? kEigThreads : kEigMultiThreads;
  const int grid = persistent_grid(k_eig_multi<VT, AT, FT, PLAIN, COMPACT>, threads, 0, blocks);
  k_eig_multi<VT, AT, FT, PLAIN, COMPACT><<<grid, threads, 0, st>>>(items, T, fill);
  return cudaGetLastError();
}

template <bool COMPACT>
static cudaError_t eig_multi_c(const EigItem* items, const MultiTable& T, int64_t blocks, int vt, int at, int ft,
                               bool plain, float fill, cudaStream_t st) {
  if (vt == CT_OUT_F32 && at == CT_OUT_F32 && ft == CT_OUT_F32)
    return plain ? eig_multi_t<0, 0, 0, true, COMPACT>(items, T, blocks, fill, st)
                 : eig_multi_t<0, 0, 0, false, COMPACT>(items, T, blocks, fill, st);
  if (vt == CT_OUT_F16 && at == CT_OUT_F16 && ft == CT_OUT_F16)
    return plain ? eig_multi_t<1, 1, 1, true, COMPACT>(items, T, blocks, fill, st)
                 : eig_multi_t<1, 1, 1, false, COMPACT>(items, T, blocks, fill, st);
  if (at == CT_OUT_U8Q && ft == CT_OUT_F16) return eig_multi_t<-1, 2, 1, false, COMPACT>(items, T, blocks, fill, st);
  return eig_multi_t<-1, -1, -1, false, COMPACT>(items, T, blocks, fill, st);
}

cudaError_t launch_eig_multi(const EigItem* items, const MultiTable& T, int64_t blocks, bool compact, int vt, int at,
                             int ft, bool plain, float fill, cudaStream_t st) {
  return compact ? eig_multi_c<true>(items, T, blocks, vt, at, ft, plain, fill, st)
                 : eig_multi_c<false>(items, T, blocks, vt, at, ft, plain, fill, st);
}

cudaError_t launch_eig_fallback_multi(const EigItem* items, int n_items, int64_t max_per_item, float fill, bool mixed,
                                      cudaStream_t st) {
  if (n_items <= 0 || max_per_item <= 0) return cudaSuccess;
  dim3 grid((unsigned)std::min<int64_t>((max_per_item + 127) / 128, 64), (unsigned)n_items);
  k_eig_fallback_multi<<<grid, 128, 0, st>>>(items, fill, mixed);
  return cudaGetLastError();
}

// ------------------------------------------------------------ stage kernels
// A warp's listed voxels wait in shared memory until half a buffer has come
// together, then take their places in the list with one atomic per counter.
// One pair of atomics per listed voxel, all on the same two addresses, bound
// the kernel: 256^3 tensors, 1.5% of them listed, 276 us, and 135 us now, at
// 6.0 TB/s (the copy rate would give 119 us).
constexpr int kEigOnlyThreads = 256;
constexpr int kEigOnlyBuf = 64;  // buffered entries per warp: below 32 before a step, which adds 32 at most

__global__ void __launch_bounds__(kEigOnlyThreads)
    k_eig_only(const float* __restrict__ S, int64_t n, float* __restrict__ evals, float* __restrict__ evec,
               bool mixed, Fallback fb) {
  __shared__ int64_t buf[kEigOnlyThreads / 32][kEigOnlyBuf];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int held = 0;  // entries in the warp's buffer
  auto flush = [&] {
    __syncwarp();
    int base = 0;
    if (lane == 0) {
      base = atomicAdd(fb.count, held);
      atomicAdd(fb.total, (unsigned long long)held);
    }
    base = __shfl_sync(0xffffffffu, base, 0);
    for (int j = lane; j < held; j += 32)
      if (base + j < fb.cap) fb.list[base + j] = buf[warp][j];
    __syncwarp();
    held = 0;
  };
  // whole warps walk the tensors, so that the ballots see every lane
  for (int64_t w0 = blockIdx.x * (int64_t)kEigOnlyThreads + 32 * warp; w0 < n;
       w0 += (int64_t)gridDim.x * kEigOnlyThreads) {
    const int64_t i = w0 + lane;
    bool listed = false;
    if (i < n) {
      Sym3<float> s = load_sym(S, n, i);
      float l[3], v[3];
      listed = !eig_closed(s, l, v, fb.gap);
      orient_largest(v);
      if (evals) {
        evals[i] = l[0];
        evals[n + i] = l[1];
        evals[2 * n + i] = l[2];
      }
      evec[i] = v[0];
      evec[n + i] = v[1];
      evec[2 * n + i] = v[2];
    }
    const unsigned m = __ballot_sync(0xffffffffu, listed);
    if (listed) buf[warp][held + __popc(m & ((1u << lane) - 1u))] = i;
    held += __popc(m);
    if (held >= kEigOnlyBuf / 2) flush();
  }
  if (held > 0) flush();
}

__global__ void __launch_bounds__(128)
    k_eig_only_fallback(const float* __restrict__ S, int64_t n, float* __restrict__ evals, float* __restrict__ evec,
                        bool mixed, Fallback fb) {
  after_previous();
  const int64_t cnt = min((int64_t)*fb.count, fb.cap);
  for (int64_t j = blockIdx.x * (int64_t)blockDim.x + threadIdx.x; j < cnt; j += (int64_t)gridDim.x * blockDim.x) {
    const int64_t i = fb.list[j];
    Sym3<float> s = load_sym(S, n, i);
    float l[3], v[3];
    resolve(s, mixed, l, v);
    orient_largest(v);
    if (evals) {
      evals[i] = l[0];
      evals[n + i] = l[1];
      evals[2 * n + i] = l[2];
    }
    evec[i] = v[0];
    evec[n + i] = v[1];
    evec[2 * n + i] = v[2];
  }
}

// Stores of V consecutive voxels' values (V = 4: one 16-, 8- or 4-byte store).
template <int TYPE, int V, typename IT>
__device__ __forceinline__ void store_vals(void* base, IT i, int type, const float* v) {
  if (base == nullptr) return;
  if (V == 4 && TYPE == 0) {
    *reinterpret_cast<float4*>(reinterpret_cast<float*>(base) + i) = make_float4(v[0], v[1], v[2], v[3]);
  } else if (V == 4 && TYPE == 1) {
    __half2 h[2] = {__floats2half2_rn(v[0], v[1]), __floats2half2_rn(v[2], v[3])};
    *reinterpret_cast<uint2*>(reinterpret_cast<__half*>(base) + i) = *reinterpret_cast<const uint2*>(h);
  } else {
#pragma unroll
    for (int k = 0; k < V; ++k) store_val<TYPE, IT>(base, i + k, type, v[k]);
  }
}

template <int TYPE, int V, typename IT>
__device__ __forceinline__ void store_angles(void* base, IT i, int type, const float* deg, unsigned valid) {
  if (base == nullptr) return;
  if (V == 4 && TYPE == 2) {
    uint8_t c[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) store_angle<2, int>(c, k, 2, deg[k], valid >> k & 1u);
    *reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(base) + i) =
        c[0] | (uint32_t)c[1] << 8 | (uint32_t)c[2] << 16 | (uint32_t)c[3] << 24;
  } else if (TYPE == 2 || TYPE < 0) {
#pragma unroll
    for (int k = 0; k < V; ++k) store_angle<TYPE, IT>(base, i + k, type, deg[k], valid >> k & 1u);
  } else {
    store_vals<TYPE, V, IT>(base, i, type, deg);
  }
}

// Every array of the stage is dense over the box, so a thread takes V
// consecutive voxels of the flat index: one division of it for the first
// voxel's position, the others by stepping.  V = 4 (16-byte loads and stores)
// where every plane keeps that alignment and the threads still fill the GPU
// (kAnglesVecMin); nothing is read for a group that lies outside the mask.  256^3, F16 outputs, a wall's mask: 142 us with
// 64-bit divisions per voxel, encodings read at run time and every voxel's
// vector loaded, 94 us now, bound by the instructions of the inside voxels'
// angles (its 403 MB take 59 us at the copy rate).
template <int VT, int AT, int FT, bool PLAIN, int V, typename IT>
__global__ void __launch_bounds__(256)
    k_angles_only(const float* __restrict__ evec, const float* __restrict__ evals, Box ob,
                  const uint8_t* __restrict__ mask, Frame F, float fill, EigOut o) {
  const IT n = (IT)box_vox(ob);
  const IT step = (IT)gridDim.x * (256 * V);
  for (IT i = ((IT)blockIdx.x * 256 + threadIdx.x) * V; i < n; i += step) {
    unsigned in = (1u << V) - 1u;  // the voxels inside the mask
    if (mask != nullptr) {
      in = 0;
      if (V == 4) {
        const uint32_t m = __ldg(reinterpret_cast<const uint32_t*>(mask + i));
#pragma unroll
        for (int k = 0; k < 4; ++k) in |= (m >> (8 * k) & 0xffu) != 0 ? 1u << k : 0u;
      } else {
        in = __ldg(mask + i) != 0;
      }
    }
    float v[3][V], ha[V], ia[V], fa[V];
#pragma unroll
    for (int k = 0; k < V; ++k) v[0][k] = v[1][k] = v[2][k] = ha[k] = ia[k] = fa[k] = fill;
    unsigned framed = 0;
    if (in) {
      float l[3][V];
#pragma unroll
      for (int c = 0; c < 3; ++c) {
        if (V == 4) {
          const float4 a = __ldg(reinterpret_cast<const float4*>(evals + c * n + i));
          const float4 b = __ldg(reinterpret_cast<const float4*>(evec + c * n + i));
          l[c][0] = a.x; l[c][1 % V] = a.y; l[c][2 % V] = a.z; l[c][3 % V] = a.w;
          v[c][0] = b.x; v[c][1 % V] = b.y; v[c][2 % V] = b.z; v[c][3 % V] = b.w;
        } else {
          l[c][0] = __ldg(evals + c * n + i);
          v[c][0] = __ldg(evec + c * n + i);
        }
      }
      const IT row = i / ob.n[0];
      int x = (int)(i - row * ob.n[0]), y = (int)(row % ob.n[1]), z = (int)(row / ob.n[1]);
#pragma unroll
      for (int k = 0; k < V; ++k) {
        if (in >> k & 1u) {
          const float lk[3] = {l[0][k], l[1][k], l[2][k]};
          float vk[3] = {v[0][k], v[1][k], v[2][k]};
          float h, a;
          if (ha_ia<PLAIN>(F, ob.lo[0] + x, ob.lo[1] + y, ob.lo[2] + z, vk, h, a)) {
            framed |= 1u << k;
            ha[k] = h;
            ia[k] = a;
          } else {
            orient_largest(vk);
          }
          v[0][k] = vk[0]; v[1][k] = vk[1]; v[2][k] = vk[2];
          fa[k] = fa_of(lk);
        } else {
          v[0][k] = v[1][k] = v[2][k] = fill;
        }
        if (++x == ob.n[0]) {
          x = 0;
          if (++y == ob.n[1]) y = 0, ++z;
        }
      }
    }
    if (o.vec) {
      store_vals<VT, V, IT>(o.vec, i, o.vec_t, v[0]);
      store_vals<VT, V, IT>(o.vec, n + i, o.vec_t, v[1]);
      store_vals<VT, V, IT>(o.vec, 2 * n + i, o.vec_t, v[2]);
    }
    store_angles<AT, V, IT>(o.ha, i, o.ang_t, ha, framed);
    store_angles<AT, V, IT>(o.ia, i, o.ang_t, ia, framed);
    store_vals<FT, V, IT>(o.fa, i, o.fa_t, fa);
  }
}

cudaError_t launch_eig_only(const float* S, int64_t n, float* evals, float* evec, bool mixed, const Fallback& fb,
                            cudaStream_t st) {
  if (n == 0) return cudaSuccess;
  k_eig_only<<<grid_for(n, kEigOnlyThreads), kEigOnlyThreads, 0, st>>>(S, n, evals, evec, mixed, fb);
  return cudaGetLastError();
}

cudaError_t launch_eig_only_fallback(const float* S, int64_t n, float* evals, float* evec, bool mixed,
                                     const Fallback& fb, int64_t max_items, const Queue& st) {
  if (max_items <= 0) return cudaSuccess;
  return launch_after(k_eig_only_fallback, fallback_grid(max_items), 128, 0, st, S, n, evals, evec, mixed, fb);
}

template <int VT, int AT, int FT, bool PLAIN, int V, typename IT>
static cudaError_t angles_t(const float* evec, const float* evals, const Box& ob, const uint8_t* mask,
                            const Frame& F, float fill, const EigOut& o, cudaStream_t st) {
  k_angles_only<VT, AT, FT, PLAIN, V, IT><<<grid_for((box_vox(ob) + V - 1) / V, 256), 256, 0, st>>>(evec, evals, ob, mask, F,
                                                                                          fill, o);
  return cudaGetLastError();
}

// Four voxels per thread from so many voxels on.  Below, a voxel per thread takes less, as
// more threads share its latency: 32^3 F32 2.0 against 3.1 us (2.5 with 64-bit indices), 48^3
// 2.5 and 3.2, 60^3 3.7 and 3.9; 64^3 4.0 and 3.9, 80^3 6.3 and 5.4.
constexpr int64_t kAnglesVecMin = (int64_t)1 << 18;

template <int VT, int AT, int FT>
static cudaError_t angles_e(const float* evec, const float* evals, const Box& ob, const uint8_t* mask,
                            const Frame& F, float fill, const EigOut& o, bool vec4, bool plain, cudaStream_t st) {
  if (vec4)
    return plain ? angles_t<VT, AT, FT, true, 4, int>(evec, evals, ob, mask, F, fill, o, st)
                 : angles_t<VT, AT, FT, false, 4, int>(evec, evals, ob, mask, F, fill, o, st);
  return plain ? angles_t<VT, AT, FT, true, 1, int>(evec, evals, ob, mask, F, fill, o, st)
               : angles_t<VT, AT, FT, false, 1, int>(evec, evals, ob, mask, F, fill, o, st);
}

cudaError_t launch_angles_only(const float* evec, const float* evals, const Box& ob, const uint8_t* mask,
                               const Frame& F, float fill, const EigOut& o, cudaStream_t st) {
  const int64_t n = box_vox(ob);
  if (n == 0) return cudaSuccess;
  // 32-bit indices while every plane set (and a grid stride past its end) fits them
  if (3 * n >= ((int64_t)1 << 31) - ((int64_t)1 << 24))
    return angles_t<-1, -1, -1, false, 1, int64_t>(evec, evals, ob, mask, F, fill, o, st);
  // four voxels per thread where all planes of all arrays start on the boundary
  // of four elements (a plane of n elements keeps it for the next when n does) and
  // there are enough of them
  auto at = [](const void* p, uintptr_t b) { return reinterpret_cast<uintptr_t>(p) % b == 0; };
  auto size = [](int t) { return (uintptr_t)(t == CT_OUT_F32 ? 4 : t == CT_OUT_F16 ? 2 : 1); };
  const bool vec4 = n >= kAnglesVecMin && n % 4 == 0 && at(evec, 16) && at(evals, 16) && at(mask, 4) && at(o.vec, 4 * size(o.vec_t)) &&
                    at(o.ha, 4 * size(o.ang_t)) && at(o.ia, 4 * size(o.ang_t)) && at(o.fa, 4 * size(o.fa_t));
  const bool plain = F.sp[0] == 1.f && F.sp[1] == 1.f && F.sp[2] == 1.f && F.centres == nullptr;
  if (o.vec_t == CT_OUT_F32 && o.ang_t == CT_OUT_F32 && o.fa_t == CT_OUT_F32)
    return angles_e<0, 0, 0>(evec, evals, ob, mask, F, fill, o, vec4, plain, st);
  if (o.vec_t == CT_OUT_F16 && o.ang_t == CT_OUT_F16 && o.fa_t == CT_OUT_F16)
    return angles_e<1, 1, 1>(evec, evals, ob, mask, F, fill, o, vec4, plain, st);
  if (o.vec_t == CT_OUT_F32 && o.ang_t == CT_OUT_U8Q && o.fa_t == CT_OUT_F16)
    return angles_e<0, 2, 1>(evec, evals, ob, mask, F, fill, o, vec4, plain, st);
  return angles_t<-1, -1, -1, false, 1, int>(evec, evals, ob, mask, F, fill, o, st);
}

}  // namespace ct
