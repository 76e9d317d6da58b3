// Transmural HA profile: histogram of the helical angle against normalised
// wall depth (the paper's analysis module plots this profile from the HA map
// of Figure 1(c)).  A reduction over the pipeline's HA output, privatised per
// CTA in shared memory and flushed once per CTA with 64-bit atomics.
#include <cuda_fp16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>
#include <cmath>

#include "ct.h"

namespace ct {
ct_status set_error(ct_status st, const char* fmt, ...);
}

namespace {

// Measured at 512^3, FP32 HA, masked: 5 CTAs per SM 203 us (4: 217, 6: 203),
// tiles of 16 segments per thread 203 us (8: 217), mask loads in groups of 4
// (one at a time: 210 us).
constexpr int kProfThreads = 256;
constexpr int kProfPerSm = 5;                  // CTAs per SM
constexpr int kProfTile = 16 * kProfThreads;   // segments of a tile at most (16-bit places)
constexpr int kProfGroup = 4;                  // mask loads of a thread in flight
constexpr int kProfMaxBins = 16384;  // 64 KB of shared uint32 counters

struct ProfDev {
  float c[3], a[3];
  float r_in, inv_w;
  int nd, nh;
  float fnd, fnh, h_scale;  // n_depth, n_ha, n_ha / 180
  float depth_scale;        // n_depth / (r_out - r_in)
  float eps_r, eps_0;       // bound on the error of the approximate depth (in bins): eps_r r + eps_0
  int lo[3];
  int n0, n1, n2;
  int segs_row;             // 8-voxel segments per row
  int per_thread;           // mask loads per thread and tile
  uint32_t row_m, n1_m;     // Divisor factors
};

// min(max((int)t, 0), top) for an integral top below 2^22: the clamp first, then
// the truncation by a sum rounded towards zero whose low bits are the integer.
__device__ __forceinline__ int trunc_clamped(float t, float top) {
  return __float_as_int(__fadd_rz(fminf(fmaxf(t, 0.f), top), 8388608.f)) & 0x3fffff;
}

__device__ __forceinline__ float rsqrt_approx(float x) {
  float y;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// A quotient n / d by a multiplication where the host found n d below 2^32
// (m = floor(2^32 / d) + 1), else by the division.
struct Divisor {
  uint32_t d, m;  // m = 0: divide
  __device__ __forceinline__ uint32_t operator()(uint32_t n) const { return m ? __umulhi(n, m) : n / d; }
};

// Bits of the mask bytes of one 8-voxel segment that count (1 per voxel inside).
__device__ __forceinline__ uint32_t nonzero_bytes(uint32_t w) {
  uint32_t b = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) b |= (w >> (8 * k) & 0xffu) != 0 ? 1u << k : 0u;
  return b;
}

template <int TYPE>
__device__ __forceinline__ float load_one(const void* __restrict__ ha, int64_t i, bool& ok) {
  if (TYPE == CT_OUT_F32) {
    const float v = __ldg(reinterpret_cast<const float*>(ha) + i);
    ok = isfinite(v);
    return v;
  } else if (TYPE == CT_OUT_F16) {
    const float v = __half2float(__ldg(reinterpret_cast<const __half*>(ha) + i));
    ok = isfinite(v);
    return v;
  } else {
    const int code = __ldg(reinterpret_cast<const uint8_t*>(ha) + i);
    ok = code != 0;
    return (float)code * (180.f / 256.f) - 90.f;
  }
}

// 8 consecutive HA values from one 8-, 16- or 32-byte load, as they lie.
template <int TYPE>
struct Ha8 {
  static constexpr int W = TYPE == CT_OUT_F32 ? 8 : TYPE == CT_OUT_F16 ? 4 : 2;
  uint32_t w[W];
  __device__ __forceinline__ void load(const void* __restrict__ ha, int64_t i0) {
    if (TYPE == CT_OUT_F32) {
      const uint4* p = reinterpret_cast<const uint4*>(reinterpret_cast<const float*>(ha) + i0);
      const uint4 a = __ldg(p), b = __ldg(p + 1);
      w[0] = a.x; w[1] = a.y; w[2 % W] = a.z; w[3 % W] = a.w;
      w[4 % W] = b.x; w[5 % W] = b.y; w[6 % W] = b.z; w[7 % W] = b.w;
    } else if (TYPE == CT_OUT_F16) {
      const uint4 a = __ldg(reinterpret_cast<const uint4*>(reinterpret_cast<const __half*>(ha) + i0));
      w[0] = a.x; w[1] = a.y; w[2 % W] = a.z; w[3 % W] = a.w;
    } else {
      const uint2 a = __ldg(reinterpret_cast<const uint2*>(reinterpret_cast<const uint8_t*>(ha) + i0));
      w[0] = a.x; w[1] = a.y;
    }
  }
  __device__ __forceinline__ float get(int k, bool& ok) const {
    if (TYPE == CT_OUT_F32) {
      const float v = __uint_as_float(w[k % W]);
      ok = isfinite(v);
      return v;
    } else if (TYPE == CT_OUT_F16) {
      const float v = __half2float(__ushort_as_half((unsigned short)(w[k / 2 % W] >> (16 * (k % 2)))));
      ok = isfinite(v);
      return v;
    } else {
      const int code = w[k / 4 % W] >> (8 * (k % 4)) & 0xff;
      ok = code != 0;
      return (float)code * (180.f / 256.f) - 90.f;
    }
  }
};

// A CTA takes tiles of up to kProfTile 8-voxel segments of the box's rows, a
// grid stride apart.  It first reads the mask of the tile and lists in shared
// memory the segments with a voxel inside (a wall covers a third of its
// volume, but most groups of 32 segments touch it: without the list 42% of the
// lanes had work); then each thread takes listed segments, loads their HA
// (VEC: rows of whole aligned segments, one vector load), finds the 8 bins
// without branches and adds runs of equal bins to the CTA's shared histogram.
// The depth's bin comes from an approximate square root; a depth within its
// error of a bin edge is decided by the definition's arithmetic in a separate
// rare loop, so that every count is the definition's.
// 512^3, FP32 HA, masked, 20 x 180 bins: 203 us, bound by the instructions of the bins
// (without them 89 us; the 402 MB that it reads take 59 us at the copy rate);
// 462 us with a thread's 8 voxels taken where they lie, a square root each and
// 64-bit index divisions.  Small fields gain less, the zeroing and flushing of the
// bins being the same: 64^3 4.7 and 5.9 us, 128^3 9.3 and 12.1, 200^3 18.7 and 29.0.
template <int TYPE, bool VEC>
__global__ void __launch_bounds__(kProfThreads, kProfPerSm) k_transmural(const void* __restrict__ ha,
                                                                         const uint8_t* __restrict__ mask,
                                                                         const __grid_constant__ ProfDev P,
                                                                         unsigned long long* __restrict__ hist) {
  extern __shared__ uint32_t sh[];
  __shared__ uint32_t list[kProfTile];  // segment's place in the tile | voxels that count << 16
  __shared__ uint32_t listed;
  const int t = threadIdx.x, lane = t & 31;
  const int nb = P.nd * P.nh;
  for (int k = t; k < nb; k += kProfThreads) sh[k] = 0u;
  const Divisor by_row{(uint32_t)P.segs_row, P.row_m}, by_n1{(uint32_t)P.n1, P.n1_m};
  const int64_t nseg = (int64_t)P.segs_row * P.n1 * P.n2;
  const int tile = P.per_thread * kProfThreads;
  for (int64_t base = (int64_t)blockIdx.x * tile; base < nseg; base += (int64_t)gridDim.x * tile) {
    // the tile's first segment; the others by small quotients from it
    const int64_t row0 = base / P.segs_row;
    const uint32_t seg0 = (uint32_t)(base - row0 * P.segs_row);
    const int z0 = (int)(row0 / P.n1), y0 = (int)(row0 - (int64_t)z0 * P.n1);
    if (t == 0) listed = 0;
    __syncthreads();
    for (int u0 = 0; u0 < P.per_thread; u0 += kProfGroup) {
      uint32_t in[kProfGroup];  // the loads of a group are in flight together
#pragma unroll
      for (int u = 0; u < kProfGroup; ++u) {
        const uint32_t off = (u0 + u) * kProfThreads + t;
        in[u] = 0;
        if (u0 + u < P.per_thread && base + off < nseg) {
          if (VEC) {
            in[u] = 0xffu;
            if (mask) {
              const uint2 q = __ldg(reinterpret_cast<const uint2*>(mask + 8 * (base + off)));
              in[u] = nonzero_bytes(q.x) | nonzero_bytes(q.y) << 4;
            }
          } else {
            const uint32_t n = seg0 + off, r = by_row(n);
            const int x0 = 8 * (int)(n - r * P.segs_row), nk = min(8, P.n0 - x0);
            in[u] = (1u << nk) - 1u;
            if (mask) {
              const uint8_t* m = mask + (row0 + r) * P.n0 + x0;
#pragma unroll
              for (int k = 0; k < 8; ++k)
                if (k < nk && __ldg(m + k) == 0) in[u] &= ~(1u << k);
            }
          }
        }
      }
      unsigned some[kProfGroup];
      uint32_t sum = 0, at = 0;
#pragma unroll
      for (int u = 0; u < kProfGroup; ++u) {
        some[u] = __ballot_sync(0xffffffffu, in[u] != 0);
        sum += __popc(some[u]);
      }
      if (lane == 0 && sum) at = atomicAdd(&listed, sum);
      at = __shfl_sync(0xffffffffu, at, 0);
#pragma unroll
      for (int u = 0; u < kProfGroup; ++u) {
        if (in[u])
          list[at + __popc(some[u] & ((1u << lane) - 1u))] = (uint32_t)((u0 + u) * kProfThreads + t) | in[u] << 16;
        at += __popc(some[u]);
      }
    }
    __syncthreads();
    const int total = listed;
    for (int j = t; j < total; j += kProfThreads) {
      const uint32_t e = list[j], in = e >> 16;
      const uint32_t n = seg0 + (e & 0xffffu), r = by_row(n);
      const int64_t row = row0 + r;
      const int x0 = 8 * (int)(n - r * P.segs_row);
      const uint32_t yy = y0 + r, dzz = by_n1(yy);
      const int y = (int)(yy - dzz * P.n1), z = z0 + (int)dzz;
      const int64_t i0 = row * P.n0 + x0;
      Ha8<TYPE> h8;
      if (VEC) h8.load(ha, i0);
      const float fx = (float)(P.lo[0] + x0);  // exact: positions are below 2^24
      const float dy = (float)(P.lo[1] + y) - P.c[1], dz = (float)(P.lo[2] + z) - P.c[2];
      auto radius2 = [&](int k) {
        const float dx = (fx + (float)k) - P.c[0];
        const float t = dx * P.a[0] + dy * P.a[1] + dz * P.a[2];
        const float rx = dx - t * P.a[0], ry = dy - t * P.a[1], rz = dz - t * P.a[2];
        return rx * rx + ry * ry + rz * rz;
      };
      auto ha_bin = [&](float h) { return trunc_clamped((h + 90.f) * P.h_scale, P.fnh - 1.f); };
      int bin[8];
      unsigned edge = 0;  // voxels whose depth lies within rounding of a bin's edge
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        bool ok = false;
        float h = 0.f;
        if (VEC)
          h = h8.get(k, ok);
        else if (in >> k & 1u)
          h = load_one<TYPE>(ha, i0 + k, ok);
        ok = ok && (in >> k & 1u);
        const float rr = radius2(k);
        const float rad = rr * rsqrt_approx(rr);  // (NaN at 0, which takes the definition's arithmetic)
        const float d = (rad - P.r_in) * P.depth_scale;
        const bool near = !(fabsf(d - rintf(d)) > fmaf(rad, P.eps_r, P.eps_0));
        if (ok && near) edge |= 1u << k;
        ok = ok && !near && d >= 0.f && d < P.fnd;
        bin[k] = ok ? trunc_clamped(d, P.fnd - 1.f) * P.nh + ha_bin(h) : -1;
      }
      int start = 0;
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        const bool end = k == 7 || bin[k + 1 < 8 ? k + 1 : 7] != bin[k];
        if (end && bin[k] >= 0) atomicAdd(&sh[bin[k]], (uint32_t)(k + 1 - start));
        if (end) start = k + 1;
      }
      while (edge) {
        const int k = __ffs(edge) - 1;
        edge &= edge - 1;
        bool ok;
        const float h = load_one<TYPE>(ha, i0 + k, ok);
        const float d = (sqrtf(radius2(k)) - P.r_in) * P.inv_w;
        if (d >= 0.f && d < 1.f) atomicAdd(&sh[trunc_clamped(d * P.fnd, P.fnd - 1.f) * P.nh + ha_bin(h)], 1u);
      }
    }
    __syncthreads();  // the list is free for the next tile
  }
  __syncthreads();
  for (int k = t; k < nb; k += kProfThreads)
    if (sh[k]) atomicAdd(hist + k, (unsigned long long)sh[k]);
}

template <int TYPE>
cudaError_t launch_profile(const void* ha, const uint8_t* mask, const ProfDev& P, unsigned long long* hist, int grid,
                           size_t smem, bool vec, cudaStream_t st) {
  cudaError_t e;
  if (vec) {
    e = cudaFuncSetAttribute(k_transmural<TYPE, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) k_transmural<TYPE, true><<<grid, kProfThreads, smem, st>>>(ha, mask, P, hist);
  } else {
    e = cudaFuncSetAttribute(k_transmural<TYPE, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
    if (e == cudaSuccess) k_transmural<TYPE, false><<<grid, kProfThreads, smem, st>>>(ha, mask, P, hist);
  }
  return e == cudaSuccess ? cudaGetLastError() : e;
}

}  // namespace

extern "C" ct_status ct_transmural_profile(const ct_profile_spec* spec, const int64_t vol_dims[3],
                                           const int64_t lo[3], const int64_t n[3], const void* d_ha,
                                           const uint8_t* d_mask, uint64_t* d_hist, void* stream) {
  if (!spec || !vol_dims || !lo || !n || !d_ha || !d_hist) return ct::set_error(CT_ERR_INVALID, "NULL argument");
  for (int k = 0; k < 3; ++k)
    if (vol_dims[k] < 1 || n[k] < 1 || lo[k] < 0 || lo[k] + n[k] > vol_dims[k] || vol_dims[k] > (1 << 24))
      return ct::set_error(CT_ERR_INVALID, "box outside the volume");
  if (n[0] > (1 << 30) || n[1] * n[2] > ((int64_t)1 << 40)) return ct::set_error(CT_ERR_INVALID, "box too large");
  if (spec->n_depth < 1 || spec->n_ha < 1 || (int64_t)spec->n_depth * spec->n_ha > kProfMaxBins)
    return ct::set_error(CT_ERR_INVALID, "n_depth * n_ha must be in [1, %d]", kProfMaxBins);
  if (!(spec->r_out > spec->r_in) || !std::isfinite(spec->r_in) || !std::isfinite(spec->r_out))
    return ct::set_error(CT_ERR_INVALID, "r_out must exceed r_in");
  if (spec->ha_type != CT_OUT_F32 && spec->ha_type != CT_OUT_F16 && spec->ha_type != CT_OUT_U8Q)
    return ct::set_error(CT_ERR_INVALID, "unknown HA encoding %d", spec->ha_type);
  if (spec->reserved != 0) return ct::set_error(CT_ERR_INVALID, "reserved must be 0");
  const double an = std::sqrt(spec->lv_axis[0] * spec->lv_axis[0] + spec->lv_axis[1] * spec->lv_axis[1] +
                              spec->lv_axis[2] * spec->lv_axis[2]);
  if (!(an > 0.0) || !std::isfinite(an)) return ct::set_error(CT_ERR_INVALID, "axis must be finite and non-zero");
  ProfDev P;
  for (int k = 0; k < 3; ++k) {
    P.c[k] = (float)spec->lv_center[k];
    P.a[k] = (float)(spec->lv_axis[k] / an);
    P.lo[k] = (int)lo[k];
  }
  P.r_in = (float)spec->r_in;
  P.inv_w = (float)(1.0 / (spec->r_out - spec->r_in));
  P.nd = spec->n_depth;
  P.nh = spec->n_ha;
  P.fnd = (float)P.nd;
  P.fnh = (float)P.nh;
  P.h_scale = (float)P.nh / 180.f;
  P.depth_scale = P.inv_w * P.fnd;
  // the approximate radius is within 2^-21 of the exact one, and each of the few
  // roundings on either way within 2^-23 of its operands
  P.eps_r = 1e-6f * P.depth_scale;
  P.eps_0 = 1e-6f * (std::fabs(P.r_in) * P.depth_scale + P.fnd);
  P.n0 = (int)n[0];
  P.n1 = (int)n[1];
  P.n2 = (int)n[2];
  P.segs_row = (P.n0 + 7) / 8;
  const int64_t segs = (int64_t)P.segs_row * n[1] * n[2];
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess || sms < 1) sms = 1;
  const int64_t want = (int64_t)sms * kProfPerSm;
  // tiles as large as still gives every CTA one
  P.per_thread = (int)std::min<int64_t>(kProfTile / kProfThreads, std::max<int64_t>(1, segs / (want * kProfThreads)));
  const int64_t tile = (int64_t)P.per_thread * kProfThreads;
  int grid = (int)std::max<int64_t>(1, std::min<int64_t>(want, (segs + tile - 1) / tile));
  // A CTA's tiles lie `grid` tiles apart, and the work of a tile depends on its
  // place in the plane (none above and below the wall): a stride of whole planes
  // would give a CTA the same place again and again (608 CTAs at 512^3: 282 us),
  // so of the grids within 8% of the largest the one is taken whose stride is
  // nearest to the golden section of a plane, which spreads any number of tiles
  // evenly over it.
  if (grid == want) {
    const double tiles_per_plane = (double)P.segs_row * P.n1 / (double)tile;
    double best = 2.0;
    for (int g = (int)want; g > want - want / 12; --g) {
      const double f = g / tiles_per_plane, off = std::fabs(f - std::floor(f) - 0.6180339887);
      if (off < best - 1e-9) best = off, grid = g;
    }
  }
  // a quotient's numerator is below its divisor + the tile
  auto factor = [](uint64_t d) {
    return d >= 2 && (d + kProfTile + 1) * d < ((uint64_t)1 << 32) ? (uint32_t)(((uint64_t)1 << 32) / d + 1) : 0u;
  };
  P.row_m = factor(P.segs_row);
  P.n1_m = factor(P.n1);
  const size_t smem = sizeof(uint32_t) * (size_t)P.nd * P.nh;
  // vector loads: rows of whole 8-voxel segments on 16-byte aligned arrays
  const bool vec = n[0] % 8 == 0 && (uintptr_t)d_ha % 16 == 0 && (d_mask == nullptr || (uintptr_t)d_mask % 8 == 0);
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = cudaSuccess;
  unsigned long long* h = reinterpret_cast<unsigned long long*>(d_hist);
  switch (spec->ha_type) {
    case CT_OUT_F32: e = launch_profile<CT_OUT_F32>(d_ha, d_mask, P, h, grid, smem, vec, st); break;
    case CT_OUT_F16: e = launch_profile<CT_OUT_F16>(d_ha, d_mask, P, h, grid, smem, vec, st); break;
    default: e = launch_profile<CT_OUT_U8Q>(d_ha, d_mask, P, h, grid, smem, vec, st); break;
  }
  if (e == cudaSuccess) e = cudaGetLastError();
  if (e != cudaSuccess) return ct::set_error(CT_ERR_CUDA, "profile launch failed: %s", cudaGetErrorString(e));
  return CT_OK;
}
