// gpf_build_index on a multi-level hashed grid.
//
// Level L has cubic cells of edge c0 * 2^L. Each Gaussian lives on the finest
// level on which its k-sigma bounds span at most S cells per axis, and is
// listed in the (level, cell) bucket of every cell of that box that holds a
// hit point. Lists of all levels share one array of 2^hash_bits buckets,
// radix-sorted by bucket (stable, so a list's order is deterministic).
// Hit points are sorted by their cell on the query level K (dense linear
// keys), which orders the forward's tiles and gives the backward the hit
// points of any query-level cell. Gaussians are also sorted by the
// query-level cell of their mean, the order the backward walks them in.
//
// Kernels, in stream order:
//   query_keys (hit point keys, occupancy bits of every level)
//   preprocess (records, level boxes, entry counts, order keys, level mask)
//   emit (bucket, Gaussian) entries
//   sorts, a pass of all three per launch: hit points by cell, Gaussians into
//   the backward's order, entries by bucket
//   ranges (per-cell starts of the hit points, bucket ranges of the entries)
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>

#include "gpf_internal.h"

namespace gpf {

namespace {

constexpr int kThreads = 256;
constexpr int kBlockWarps = kThreads / kWarp;

// The sum over a block of up to four per-thread counts,
// each in [0, 2^32); thread 0 gets the sums. The header counters take one
// atomic per block: atomics to one address are serialised, so per-warp
// updates from 10^6 threads cost tens of microseconds.
__device__ __forceinline__ void block_counts(uint32_t (&v)[4], uint32_t (*s)[4]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
#pragma unroll
  for (int k = 0; k < 4; ++k) v[k] = __reduce_add_sync(kFullMask, v[k]);
  if (lane == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) s[warp][k] = v[k];
  }
  __syncthreads();
  if (threadIdx.x == 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      uint32_t t = 0;
      for (int w = 0; w < (int)blockDim.x / kWarp; ++w) t += s[w][k];
      v[k] = t;
    }
  }
}
// Boxes with more cells than this on their level are refused (overflow flag).
constexpr int64_t kMaxBoxCells = int64_t(1) << 16;
// Boxes of up to this many cells keep a bit mask of the occupied ones; emit
// tests the cells of the others again.
constexpr int64_t kMaskCells = 64;

// Groups of Gaussians whose entry counts add up to one word of gpart, which
// then holds one word per kSuper groups: the entry offset of a group is the
// sum of at most kSuper groups and n / (kSuper * group) super-groups.
constexpr int kSuper = 64;
__host__ __device__ __forceinline__ int64_t group_count(int64_t n, int group) {
  return (n + group - 1) / group;
}

// Adds the digits of this lane's sort key (if ok) to the block's digit counts
// cnt[pass * kSortBins + digit]: one atomic per run of lanes with equal digits
// (hit points of neighbouring pixels share the high digits of their cell keys,
// and atomics to one address are serialised). All lanes of the warp call it.
__device__ __forceinline__ void count_digits(uint32_t key, bool ok, int passes, uint32_t* cnt) {
  const int lane = threadIdx.x & 31;
  const uint32_t left = __shfl_up_sync(kFullMask, key, 1);
  const uint32_t valid = __ballot_sync(kFullMask, ok);     // a prefix of the lanes
  for (int p = 0; p < passes; ++p) {
    const uint32_t d = (key >> (8 * p)) & 255u;
    const bool head = ok && (lane == 0 || d != ((left >> (8 * p)) & 255u));
    const uint32_t heads = __ballot_sync(kFullMask, head);
    if (head) {
      const uint32_t later = heads & ~((2u << lane) - 1u);
      const int end = later ? __ffs(later) - 1 : __popc(valid);
      atomicAdd(&cnt[p * kSortBins + d], (uint32_t)(end - lane));
    }
  }
}
__device__ __forceinline__ void flush_digits(const uint32_t* cnt, int passes,
                                             uint32_t* __restrict__ out) {
  for (int i = threadIdx.x; i < passes * kSortBins; i += blockDim.x)
    if (cnt[i]) atomicAdd(&out[i], cnt[i]);
}

__device__ __forceinline__ bool occupied(const uint32_t* occ, uint32_t b) {
  return (occ[b >> 5] >> (b & 31u)) & 1u;
}

// GPF_BF16 / GPF_BF16_MEAN32 field -> float32 [(10 + C), n] rows: mean, quat, logscale,
// spectrum (the decoding stated at gpf_field).
__global__ void decode_bf16_kernel(gpf_field f, float* __restrict__ dec) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n = f.n;
  if (g >= n) return;
  const float* anc = f.anchor + 4 * (g / GPF_BF16_GROUP);
  const uint16_t* quat = static_cast<const uint16_t*>(f.quat);
  const uint16_t* lsc = static_cast<const uint16_t*>(f.logscale);
  const uint16_t* spec = static_cast<const uint16_t*>(f.spectrum);
  const float4 a = *reinterpret_cast<const float4*>(anc);
  if (f.storage == GPF_BF16) {
    const uint16_t* mean = static_cast<const uint16_t*>(f.mean);
    dec[g] = __fadd_rn(a.x, bf16_to_f32(mean[g]));
    dec[n + g] = __fadd_rn(a.y, bf16_to_f32(mean[n + g]));
    dec[2 * n + g] = __fadd_rn(a.z, bf16_to_f32(mean[2 * n + g]));
  } else {
    const float* mean = static_cast<const float*>(f.mean);
#pragma unroll
    for (int k = 0; k < 3; ++k) dec[k * n + g] = mean[k * n + g];
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) dec[(3 + k) * n + g] = bf16_to_f32(quat[k * n + g]);
#pragma unroll
  for (int k = 0; k < 3; ++k) dec[(7 + k) * n + g] = __fadd_rn(a.w, bf16_to_f32(lsc[k * n + g]));
  for (int c = 0; c < f.channels; ++c) dec[(10 + c) * n + g] = bf16_to_f32(spec[c * n + g]);
}

// gpf_field_quantize: one half-warp per group of 16 Gaussians, one lane per
// Gaussian; min / max over the group by xor shuffles within the half-warp.
__global__ void quantize_bf16_kernel(gpf_field src, gpf_field dst) {
  const int64_t g = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t n = src.n;
  const bool live = g < n;
  const float* mean = static_cast<const float*>(src.mean);
  const float* quat = static_cast<const float*>(src.quat);
  const float* lsc = static_cast<const float*>(src.logscale);
  const float* spec = static_cast<const float*>(src.spectrum);
  float mu[3], l[3];
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    mu[k] = live ? mean[k * n + g] : 0.0f;
    l[k] = live ? lsc[k * n + g] : 0.0f;
  }
  float lo[4], hi[4];
#pragma unroll
  for (int k = 0; k < 3; ++k) lo[k] = hi[k] = mu[k];
  lo[3] = fminf(l[0], fminf(l[1], l[2]));
  hi[3] = fmaxf(l[0], fmaxf(l[1], l[2]));
  if (!live) {
#pragma unroll
    for (int k = 0; k < 4; ++k) { lo[k] = INFINITY; hi[k] = -INFINITY; }
  }
#pragma unroll
  for (int o = GPF_BF16_GROUP / 2; o > 0; o >>= 1) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      lo[k] = fminf(lo[k], __shfl_xor_sync(kFullMask, lo[k], o, GPF_BF16_GROUP));
      hi[k] = fmaxf(hi[k], __shfl_xor_sync(kFullMask, hi[k], o, GPF_BF16_GROUP));
    }
  }
  float ref[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) ref[k] = __fmul_rn(__fadd_rn(lo[k], hi[k]), 0.5f);
  if (!live) return;
  if (g % GPF_BF16_GROUP == 0)
    *reinterpret_cast<float4*>(const_cast<float*>(dst.anchor) + 4 * (g / GPF_BF16_GROUP)) =
        make_float4(ref[0], ref[1], ref[2], ref[3]);
  const bool mean32 = dst.storage == GPF_BF16_MEAN32;
  uint16_t* dquat = static_cast<uint16_t*>(const_cast<void*>(dst.quat));
  uint16_t* dlsc = static_cast<uint16_t*>(const_cast<void*>(dst.logscale));
  uint16_t* dspec = static_cast<uint16_t*>(const_cast<void*>(dst.spectrum));
#pragma unroll
  for (int k = 0; k < 3; ++k) {
    if (mean32)
      static_cast<float*>(const_cast<void*>(dst.mean))[k * n + g] = mu[k];
    else
      static_cast<uint16_t*>(const_cast<void*>(dst.mean))[k * n + g] =
          f32_to_bf16(__fsub_rn(mu[k], ref[k]));
    dlsc[k * n + g] = f32_to_bf16(__fsub_rn(l[k], ref[3]));
  }
#pragma unroll
  for (int k = 0; k < 4; ++k) dquat[k * n + g] = f32_to_bf16(quat[k * n + g]);
  for (int c = 0; c < src.channels; ++c) dspec[c * n + g] = f32_to_bf16(spec[c * n + g]);
}

// The bits of a box's occupancy mask per row and per slice: 3 and 9 for boxes of
// up to 3 cells an axis, 4 and 16 for up to 4 (constants for the code that sets
// them), else the box's own.
__device__ __forceinline__ uint2 mask_strides(uint32_t nx, uint32_t ny, uint32_t nz) {
  const uint32_t most = max(nx, max(ny, nz));
  return most <= 3 ? make_uint2(3u, 9u) : most <= 4 ? make_uint2(4u, 16u)
                                                    : make_uint2(nx, nx * ny);
}

// The occupancy mask of a box of at most N cells an axis: the N x N reads of a z
// slice go out together, without a branch per cell.
template <int N>
__device__ __forceinline__ unsigned long long small_box_mask(
    const Grid& grid, const uint32_t* __restrict__ occ, int L, uint32_t lx, uint32_t ly,
    uint32_t lz, uint32_t sx, uint32_t sy, uint32_t sz) {
  unsigned long long mask = 0;
  uint64_t cell = cell_word(L, lx, ly, lz);
  for (uint32_t dz = 0; dz <= sz; ++dz, cell += uint64_t(1) << 40) {
    uint32_t bkt[N * N], word[N * N];
#pragma unroll
    for (int j = 0; j < N * N; ++j) {
      bkt[j] = bucket_of_word(grid, cell + (uint64_t)(j % N) + ((uint64_t)(j / N) << 20));
      word[j] = (uint32_t)(j % N) <= sx && (uint32_t)(j / N) <= sy ? __ldg(occ + (bkt[j] >> 5)) : 0u;
    }
    uint32_t bits = 0;
#pragma unroll
    for (int j = 0; j < N * N; ++j) bits |= ((word[j] >> (bkt[j] & 31u)) & 1u) << j;
    mask |= (unsigned long long)bits << (N * N * dz);
  }
  return mask;
}

// Per Gaussian: record, level box, the number of cells of that box holding a
// hit point (its list entries) and its key in the backward's order.
__global__ void __launch_bounds__(kThreads, 4)
preprocess_kernel(gpf_field f, Grid grid, float cutoff, int brute,
                                  float* __restrict__ rec, int rs, VetRec* __restrict__ vet,
                                  const uint32_t* __restrict__ occ,
                                  uint32_t* __restrict__ gcount, uint8_t* __restrict__ glive,
                                  unsigned long long* __restrict__ gmask,
                                  uint2* __restrict__ qbox,
                                  uint32_t* __restrict__ okey, uint32_t* __restrict__ oval,
                                  int passes, uint32_t* __restrict__ digit_counts,
                                  uint32_t* __restrict__ gpart, DeviceHeader* header) {
  __shared__ uint32_t s_digits[kSortMaxPasses * kSortBins];   // of the order keys
  for (int i = threadIdx.x; i < passes * kSortBins; i += blockDim.x) s_digits[i] = 0;
  __syncthreads();
  const int64_t n = f.n;
  const int64_t n_groups = group_count(n, (int)blockDim.x);
  uint32_t level_bits = 0;
  uint32_t v[4] = {0u, 0u, 0u, 0u};    // live, small, huge, bad of this thread
  for (int64_t group = blockIdx.x; group < n_groups; group += gridDim.x) {
  const int64_t g = group * blockDim.x + threadIdx.x;
  bool live = false, small = false, huge = false, bad = false;
  uint32_t order_key = 0, entries = 0;
  if (g < n) {
    const float* mean = static_cast<const float*>(f.mean);
    const float* spec = static_cast<const float*>(f.spectrum);
    const float mu[3] = {mean[g], mean[n + g], mean[2 * n + g]};
    const Frame fr = gaussian_frame(static_cast<const float*>(f.quat),
                                    static_cast<const float*>(f.logscale), n, g);
    // the record's first 16 floats in registers, stored as four float4 once
    // the level is known (rs is a multiple of 4, the record 16-byte aligned)
    float rv[16];
    const float smax = fmaxf(fr.s[0], fmaxf(fr.s[1], fr.s[2]));
    // non-finite parameters: an infinite log-scale shows in max s; the rest
    // in the record (checked where it is stored)
    uint32_t nf = ~__float_as_uint(smax) & 0x7f800000u ? 0u : 1u;
    rv[0] = mu[0]; rv[1] = mu[1]; rv[2] = mu[2];
    // bounding sphere of the k-sigma ellipsoid, widened by 1e-4 for rounding
    rv[3] = isinf(cutoff) ? INFINITY : cutoff * smax * 1.0001f;
#pragma unroll
    for (int j = 0; j < 3; ++j) {
      const float inv = 1.0f / fr.s[j];
#pragma unroll
      for (int k = 0; k < 3; ++k) rv[4 + 3 * j + k] = fr.R[k][j] * inv;
    }
#pragma unroll
    for (int c = 0; c < 3; ++c) rv[13 + c] = c < f.channels ? spec[(int64_t)c * n + g] : 0.0f;
    // the order the backward walks Gaussians in: class (0 = bounds within
    // 2 x 2 x 2 query-level cells, 1 = larger, 2 = no hit point in reach);
    // the large ones largest first (log4 of their bounds' volume in query
    // cells), so that none of them starts last; then the cell of the mean on
    // a coarse level
    const int K = grid.qlevel, os = grid.oshift;
    const uint32_t mkey =
        ((coord0(mu[2], grid.oz, grid.inv_cell0, grid.max0z) >> os) * grid.ody +
         (coord0(mu[1], grid.oy, grid.inv_cell0, grid.max0y) >> os)) * grid.odx +
        (coord0(mu[0], grid.ox, grid.inv_cell0, grid.max0x) >> os);
    const int cls_shift = grid.obits - 2;
    const int size_shift = cls_shift - kOrderSizeBits;
    uint32_t cls = 1, size_rank = 0;
    oval[g] = (uint32_t)g;
    if (!brute) {
      uint32_t lo[3], hi[3];
      gaussian_cells0(grid, fr, mu, cutoff, lo, hi);
      qbox[g] = pack_qbox(lo, hi, grid.qlevel);    // the backward's cell range
      if ((hi[0] >> K) - (lo[0] >> K) <= 1 && (hi[1] >> K) - (lo[1] >> K) <= 1 &&
          (hi[2] >> K) - (lo[2] >> K) <= 1) {
        // (those of as many cells together: a warp of the backward takes 32 of
        // them side by side, at the pace of the longest)
        cls = 0;
        size_rank = 3u - (((hi[0] >> K) != (lo[0] >> K)) + ((hi[1] >> K) != (lo[1] >> K)) +
                          ((hi[2] >> K) != (lo[2] >> K)));
      } else {
        const uint64_t vq = (uint64_t)((hi[0] >> K) - (lo[0] >> K) + 1) *
                            ((hi[1] >> K) - (lo[1] >> K) + 1) * ((hi[2] >> K) - (lo[2] >> K) + 1);
        const uint32_t lg = 63u - (uint32_t)__clzll((long long)vq);
        const uint32_t top = (1u << kOrderSizeBits) - 1u;
        size_rank = top - min(lg >> 1, top);
      }
      int L = 0;
      for (; L < grid.levels - 1; ++L) {
        const uint32_t sx = (hi[0] >> L) - (lo[0] >> L), sy = (hi[1] >> L) - (lo[1] >> L),
                       sz = (hi[2] >> L) - (lo[2] >> L);
        if (max(sx, max(sy, sz)) < (uint32_t)grid.max_span) break;
      }
      const uint32_t lx = lo[0] >> L, ly = lo[1] >> L, lz = lo[2] >> L;
      const uint32_t sx = (hi[0] >> L) - lx, sy = (hi[1] >> L) - ly, sz = (hi[2] >> L) - lz;
      const int64_t vol = (int64_t)(sx + 1) * (sy + 1) * (sz + 1);
      uint32_t cnt = 0;
      if (sx > 255 || sy > 255 || sz > 255 || vol > kMaxBoxCells) {
        vet[g] = VetRec{mu[0], mu[1], mu[2], rv[3], 0ull, 0ull};
        atomicExch(&header->overflow, 1u);
      } else {
        rv[3] = rec_radius_with_level(rv[3], (uint32_t)L);
        vet[g] = VetRec{mu[0], mu[1], mu[2], rv[3], kCellGuard - pack_cell(lx, ly, lz),
                        kCellGuard + pack_cell(lx + sx, ly + sy, lz + sz)};
        level_bits |= 1u << L;
        // bit c of the mask: the c-th cell of the box (x fastest, rows and
        // slices mask_strides apart) holds a hit point; emit walks the set bits
        unsigned long long mask = 0;
        if (sx <= 2 && sy <= 2 && sz <= 2) {
          mask = small_box_mask<3>(grid, occ, L, lx, ly, lz, sx, sy, sz);
          cnt = (uint32_t)__popcll(mask);
        } else if (sx <= 3 && sy <= 3 && sz <= 3) {
          mask = small_box_mask<4>(grid, occ, L, lx, ly, lz, sx, sy, sz);
          cnt = (uint32_t)__popcll(mask);
        } else {
          uint32_t c = 0;
          for (uint32_t iz = lz; iz <= lz + sz; ++iz)
            for (uint32_t iy = ly; iy <= ly + sy; ++iy)
              for (uint32_t ix = lx; ix <= lx + sx; ++ix, ++c)
                if (occupied(occ, bucket_of(grid, L, ix, iy, iz))) {
                  ++cnt;
                  if (c < 64) mask |= 1ull << c;
                }
        }
        gmask[g] = mask;
      }
      live = cnt > 0;
      if (grid.blevel >= 0) ++cnt;      // the centre entry (kept for every Gaussian)
      gcount[g] = cnt;
      entries = cnt;
      if (!live) cls = 2;
      small = live && cls == 0;
      huge = live && cls == 1 && size_rank <= 1;
    }
    order_key = mkey | (size_rank << size_shift) | (cls << cls_shift);
    okey[g] = order_key;
    glive[g] = (brute || live) ? 1 : 0;
    float4* r4 = reinterpret_cast<float4*>(rec + g * rs);
#pragma unroll
    for (int v = 0; v < 4; ++v)
      r4[v] = make_float4(rv[4 * v], rv[4 * v + 1], rv[4 * v + 2], rv[4 * v + 3]);
    // every parameter finite: a NaN or infinite mean, quaternion or
    // log-scale leaves a non-finite value in the record's mean or M = S^-1 R^T
    // (an infinite log-scale in max s), and a spectrum value is stored as is
#pragma unroll
    for (int v = 0; v < 16; ++v)
      if (v != 3) nf |= ~__float_as_uint(rv[v]) & 0x7f800000u ? 0u : 1u;
    for (int c = 16; c < rs; ++c) {
      const float sv = c - 13 < f.channels ? spec[(int64_t)(c - 13) * n + g] : 0.0f;
      nf |= ~__float_as_uint(sv) & 0x7f800000u ? 0u : 1u;
      rec[g * rs + c] = sv;
    }
    bad = nf != 0u;
  }
  count_digits(order_key, g < n, passes, s_digits);
  v[0] += live;
  v[1] += small;
  v[2] += huge;
  v[3] |= bad;
  if (gpart) {
    const uint32_t ent = __reduce_add_sync(kFullMask, entries);
    if ((threadIdx.x & 31) == 0 && ent) {
      atomicAdd(&gpart[group], ent);
      atomicAdd(&gpart[n_groups + group / kSuper], ent);
    }
  }
  }  // groups
  __shared__ uint32_t s_cnt[kBlockWarps][4];
  __shared__ uint32_t s_mask;
  if (threadIdx.x == 0) s_mask = 0;
  __syncthreads();
  const uint32_t m = __reduce_or_sync(kFullMask, level_bits);
  if ((threadIdx.x & 31) == 0 && m) atomicOr(&s_mask, m);
  block_counts(v, s_cnt);      // its __syncthreads also orders s_mask
  if (threadIdx.x == 0) {
    // the level bits: only when this block adds one (the mask fills up early)
    if (s_mask & ~*(volatile uint32_t*)&header->level_mask) atomicOr(&header->level_mask, s_mask);
    if (v[0]) atomicAdd(&header->n_live, v[0]);
    if (v[1]) atomicAdd(&header->n_small, v[1]);
    if (v[2]) atomicAdd(&header->n_huge, v[2]);
    if (v[3]) atomicExch(&header->nonfinite, 1u);
  }
  flush_digits(s_digits, passes, digit_counts);
}

__global__ void query_keys_kernel(Grid grid, const float* __restrict__ x,
                                  const float* __restrict__ nrm, const float* __restrict__ wo,
                                  const uint8_t* __restrict__ valid, int64_t m,
                                  uint32_t* __restrict__ key, uint32_t* __restrict__ val,
                                  uint32_t* __restrict__ occ, int mark,
                                  uint32_t* __restrict__ qbits, int passes,
                                  uint32_t* __restrict__ digit_counts, DeviceHeader* header) {
  __shared__ uint32_t s_digits[kSortMaxPasses * kSortBins];   // of the sort keys
  for (int d = threadIdx.x; d < passes * kSortBins; d += blockDim.x) s_digits[d] = 0;
  __syncthreads();
  uint32_t v[4] = {0u, 0u, 0u, 0u};            // active, bad hit points of this thread
  const int64_t chunks = (m + kThreads - 1) / kThreads;
  for (int64_t chunk = blockIdx.x; chunk < chunks; chunk += gridDim.x) {
  const int64_t i = chunk * kThreads + threadIdx.x;
  bool active = false, bad = false;
  uint32_t k = grid.key_inactive;  // sort key
  uint32_t c0[3] = {0u, 0u, 0u};   // level-0 cell of an active hit point
  if (i < m) {
    // hemisphere gate n . w_o > 0: the float32 sum when it is far enough
    // from zero for its sign to be exact (its error is below 3 u sum|a_i b_i|,
    // u = 2^-24), else the float64 sum (the three products of float32 values
    // are exact in float64, so its sign is exact)
    const float a0 = nrm[i], a1 = nrm[m + i], a2 = nrm[2 * m + i];
    const float b0 = wo[i], b1 = wo[m + i], b2 = wo[2 * m + i];
    const float d32 = fmaf(a0, b0, fmaf(a1, b1, a2 * b2));
    const float mag = fabsf(a0 * b0) + fabsf(a1 * b1) + fabsf(a2 * b2);
    bool facing;
    if (fabsf(d32) > 1e-6f * mag && mag > 1e-30f) {
      facing = d32 > 0.0f;
    } else {
      const double d = __dadd_rn(__dadd_rn(__dmul_rn((double)a0, (double)b0),
                                           __dmul_rn((double)a1, (double)b1)),
                                 __dmul_rn((double)a2, (double)b2));
      facing = d > 0.0;
    }
    active = facing && (valid == nullptr || valid[i] != 0);
    if (active) {
      bad = !(isfinite(x[i]) && isfinite(x[m + i]) && isfinite(x[2 * m + i]));
      const uint32_t cx = coord0(x[i], grid.ox, grid.inv_cell0, grid.max0x);
      const uint32_t cy = coord0(x[m + i], grid.oy, grid.inv_cell0, grid.max0y);
      const uint32_t cz = coord0(x[2 * m + i], grid.oz, grid.inv_cell0, grid.max0z);
      const int K = grid.qlevel;
      k = qkey_of(grid, cx >> K, cy >> K, cz >> K);
      if (grid.qsub > 0) {
        // then the Morton code of the sub-cell on level K - qsub (x in the
        // lowest bit of each triple), so that a run of 32 hit points covers
        // a compact part of its cell
        const int s = K - grid.qsub;
        uint32_t mort = 0u;
        for (int b = grid.qsub - 1; b >= 0; --b)
          mort = (mort << 3) | (((cz >> (s + b)) & 1u) << 2) | (((cy >> (s + b)) & 1u) << 1) |
                 ((cx >> (s + b)) & 1u);
        k = (k << (3 * grid.qsub)) | mort;
      }
      c0[0] = cx; c0[1] = cy; c0[2] = cz;
    }
    key[i] = k;
    val[i] = (uint32_t)i;
  }
  if (mark) {
    // occupancy bits of every level, by the first lane of every run of lanes
    // in the same cell (differ: the bits in which a lane's cell differs from
    // its left neighbour's, so level L differs when differ >> L is not zero).
    // The levels from the query level up are marked once per query-level cell:
    // by the lane that finds the cell's own bit unset.
    const bool lactive = __shfl_up_sync(kFullMask, active ? 1 : 0, 1) != 0;
    uint32_t differ = 0;
#pragma unroll
    for (int a = 0; a < 3; ++a) differ |= c0[a] ^ __shfl_up_sync(kFullMask, c0[a], 1);
    if ((threadIdx.x & 31) == 0 || !lactive) differ = 0xffffffffu;
    if (!active) differ = 0;
    const int K = grid.qlevel;
    bool first = false;
    if ((differ >> K) != 0 && K < grid.levels) {
      const uint32_t kc = qkey_of(grid, c0[0] >> K, c0[1] >> K, c0[2] >> K);
      const uint32_t bit = 1u << (kc & 31u);
      first = !(qbits[kc >> 5] & bit) && !(atomicOr(&qbits[kc >> 5], bit) & bit);
    }
    // all the levels' words are read before the first bit is set
    uint32_t bkt[kMaxLevels], word[kMaxLevels];
#pragma unroll
    for (int L = 0; L < kMaxLevels; ++L) {
      word[L] = 0xffffffffu;
      if (L < grid.levels && (L < K ? (differ >> L) != 0 : first)) {
        bkt[L] = bucket_of(grid, L, c0[0] >> L, c0[1] >> L, c0[2] >> L);
        word[L] = occ[bkt[L] >> 5];
      }
    }
#pragma unroll
    for (int L = 0; L < kMaxLevels; ++L)
      if (word[L] != 0xffffffffu) {
        const uint32_t bit = 1u << (bkt[L] & 31u);
        if (!(word[L] & bit)) atomicOr(&occ[bkt[L] >> 5], bit);
      }
  }
  count_digits(k, i < m, passes, s_digits);
  v[0] += active;
  v[1] |= bad;
  }  // chunks
  __shared__ uint32_t s_cnt[kBlockWarps][4];
  block_counts(v, s_cnt);     // its __syncthreads also orders s_digits
  flush_digits(s_digits, passes, digit_counts);
  if (threadIdx.x == 0 && v[0]) atomicAdd(&header->n_active, v[0]);
  if (threadIdx.x == 0 && v[1]) atomicExch(&header->nonfinite, 1u);
}

// One (bucket, Gaussian) entry per occupied cell of every Gaussian's level
// box, in the box's cell order, at the Gaussian's offset (the entries of the
// Gaussians before it). A Gaussian whose cells share a bucket appears there on
// consecutive entries; the pair loops take only the first. A block takes the
// groups of preprocess in strides and adds up the counts before each; a warp lays the
// entries of its 32 Gaussians end to end and writes 32 at a time, so that the
// stores are coalesced and no lane waits for the Gaussian with the most cells
// (a thread per Gaussian: 53 us and scattered 4-byte stores at 3.8 M entries).
__global__ void __launch_bounds__(kThreads)
emit_kernel(Grid grid, int64_t n, int64_t p_max, const VetRec* __restrict__ vet,
            const uint32_t* __restrict__ occ,
            const unsigned long long* __restrict__ gmask, const uint32_t* __restrict__ gcount,
            const uint32_t* __restrict__ gpart, uint32_t* __restrict__ gkey,
            uint32_t* __restrict__ gval, int passes, uint32_t* __restrict__ digit_counts,
            uint32_t* __restrict__ cocc, uint32_t* __restrict__ focc, DeviceHeader* header) {
  // the digit counts of the entry sort, added here as the keys are written
  __shared__ uint32_t cnt[kSortMaxPasses * kSortBins];
  __shared__ uint32_t s_warp[2][kBlockWarps], s_before[2][kBlockWarps];
  for (int i = threadIdx.x; i < passes * kSortBins; i += blockDim.x) cnt[i] = 0;
  __syncthreads();
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t n_groups = group_count(n, (int)blockDim.x);
  int odd = 0;           // the shared sums alternate: one barrier per group
  for (int64_t group = blockIdx.x; group < n_groups; group += gridDim.x, odd ^= 1) {
  const int64_t g = group * blockDim.x + threadIdx.x;
  // the entries of the groups before this one
  {
    const uint32_t sup = (uint32_t)(group / kSuper);
    uint32_t before = 0;
    for (uint32_t i = threadIdx.x; i < sup; i += blockDim.x) before += gpart[n_groups + i];
    for (uint32_t i = sup * kSuper + threadIdx.x; i < (uint32_t)group; i += blockDim.x)
      before += gpart[i];
    before = __reduce_add_sync(kFullMask, before);
    if (lane == 0) s_before[odd][warp] = before;
  }
  const uint32_t c = g < n ? gcount[g] : 0u;
  uint32_t incl = c;
#pragma unroll
  for (int o = 1; o < kWarp; o <<= 1) {
    const uint32_t t = __shfl_up_sync(kFullMask, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == kWarp - 1) s_warp[odd][warp] = incl;
  __syncthreads();
  uint32_t warp_base = 0, total_here = 0;
  for (int w = 0; w < (int)blockDim.x / kWarp; ++w) {
    total_here += s_before[odd][w] + s_warp[odd][w];
    warp_base += s_before[odd][w] + (w < warp ? s_warp[odd][w] : 0u);
  }
  const uint32_t off = warp_base + incl - c;             // this Gaussian's offset
  if (group == n_groups - 1 && threadIdx.x == 0) {
    const uint32_t total = total_here;
    header->n_pairs = total;
    if ((int64_t)total > p_max) atomicExch(&header->overflow, 1u);
  }
  auto put = [&](int64_t pos, const CellHash& h, uint32_t id) {
    if (pos >= p_max) return;
    gkey[pos] = h.bucket;
    gval[pos] = id | h.tag;
    for (int p = 0; p < passes; ++p)
      atomicAdd(&cnt[p * kSortBins + ((h.bucket >> (8 * p)) & 255u)], 1u);
  };
  uint32_t bx = 0, by = 0, bz = 0;        // lowest cell of the box, the level above bx
  uint32_t nx = 0, ny = 0, nz = 0;        // cells per axis (0: no box)
  unsigned long long mask = 0;
  uint32_t centre = 0;
  if (g < n) {
    const VetRec r = load_vet(vet + g);
    if (r.nlo != 0ull) {
      const unsigned long long lo = kCellGuard - r.nlo, hi = r.hig - kCellGuard;
      bx = (uint32_t)lo & kCoordMax;
      by = (uint32_t)(lo >> 21) & kCoordMax;
      bz = (uint32_t)(lo >> 42) & kCoordMax;
      nx = ((uint32_t)hi & kCoordMax) - bx + 1;
      ny = ((uint32_t)(hi >> 21) & kCoordMax) - by + 1;
      nz = ((uint32_t)(hi >> 42) & kCoordMax) - bz + 1;
      bx |= rec_level(r.radius) << kCoordBits;
    }
    if (grid.blevel >= 0) {
      // the centre entry: the cell of the mean on the centre level
      const int Lb = grid.blevel;
      const uint32_t cx = coord0(r.x, grid.ox, grid.inv_cell0, grid.max0x) >> Lb;
      const uint32_t cy = coord0(r.y, grid.oy, grid.inv_cell0, grid.max0y) >> Lb;
      const uint32_t cz = coord0(r.z, grid.oz, grid.inv_cell0, grid.max0z) >> Lb;
      put(off, cell_hash(grid, Lb, cx, cy, cz, kCentreSalt), (uint32_t)g);
      const uint32_t bit = cocc_bit(grid, cx, cy, cz);
      atomicOr(cocc + (bit >> 5), 1u << (bit & 31u));
      if (grid.fwords) atomicOr(focc + focc_word(grid, cx, cy, cz), 1u << (cx & 31u));
      centre = 1;
    }
  }
  const bool masked = nx * ny * nz <= (uint32_t)kMaskCells;
  if (masked && nx) mask = gmask[g];
  const uint2 strides = mask_strides(nx, ny, nz);
  const uint32_t size = strides.x | (strides.y << 8);    // masked boxes: at most 64 each
  // the masked boxes of the warp, their set cells end to end: item f belongs
  // to the first lane whose inclusive count exceeds f; bit i of a box's mask is
  // cell (i mod row, (i mod slice) / row, i / slice); i < 64, so the quotients
  // computed as floor((i + 0.5) / d) in float32 are exact
  const uint32_t my = masked && nx ? c - centre : 0u;
  uint32_t mi = my;
#pragma unroll
  for (int o = 1; o < kWarp; o <<= 1) {
    const uint32_t t = __shfl_up_sync(kFullMask, mi, o);
    if (lane >= o) mi += t;
  }
  const uint32_t total = __shfl_sync(kFullMask, mi, kWarp - 1);
  for (uint32_t f0 = 0; f0 < total; f0 += kWarp) {
    const uint32_t f = f0 + lane;
    int o = 0;
#pragma unroll
    for (int st = 16; st > 0; st >>= 1)
      if (__shfl_sync(kFullMask, mi, o + st - 1) <= f) o += st;
    const uint32_t j = f - __shfl_sync(kFullMask, mi - my, o);
    const unsigned long long om = __shfl_sync(kFullMask, mask, o);
    const uint32_t x = __shfl_sync(kFullMask, bx, o), y = __shfl_sync(kFullMask, by, o),
                   z = __shfl_sync(kFullMask, bz, o), w = __shfl_sync(kFullMask, size, o);
    const uint32_t pos = __shfl_sync(kFullMask, off + centre, o) + j;
    if (f < total) {
      const uint32_t i = nth_bit(om, j);
      const uint32_t onx = w & 0xffu, onxy = w >> 8;
      const uint32_t dz = (uint32_t)(((float)i + 0.5f) * (1.0f / (float)onxy));
      const uint32_t r = i - dz * onxy;
      const uint32_t dy = (uint32_t)(((float)r + 0.5f) * (1.0f / (float)onx));
      put(pos, cell_hash(grid, (int)(x >> kCoordBits), (x & kCoordMax) + r - dy * onx, y + dy,
                         z + dz),
          (uint32_t)(g - lane) + (uint32_t)o);
    }
  }
  // the larger boxes one at a time, 32 cells at a time
  for (uint32_t todo = __ballot_sync(kFullMask, !masked); todo; todo &= todo - 1u) {
    const int o = __ffs(todo) - 1;
    const uint32_t x = __shfl_sync(kFullMask, bx, o), y = __shfl_sync(kFullMask, by, o),
                   z = __shfl_sync(kFullMask, bz, o);
    const uint32_t ox = __shfl_sync(kFullMask, nx, o), oy = __shfl_sync(kFullMask, ny, o),
                   oz = __shfl_sync(kFullMask, nz, o);
    const uint32_t cells = ox * oy * oz;                 // at most kMaxBoxCells
    uint32_t pos = __shfl_sync(kFullMask, off + centre, o);
    for (uint32_t i0 = 0; i0 < cells; i0 += kWarp) {
      const uint32_t i = i0 + lane;
      CellHash h{};
      bool set = false;
      if (i < cells) {
        h = cell_hash(grid, (int)(x >> kCoordBits), (x & kCoordMax) + i % ox, y + i / ox % oy,
                      z + i / (ox * oy));
        set = occupied(occ, h.bucket);
      }
      const uint32_t sm = __ballot_sync(kFullMask, set);
      if (set)
        put((int64_t)pos + __popc(sm & lanemask_lt()), h, (uint32_t)(g - lane) + (uint32_t)o);
      pos += (uint32_t)__popc(sm);
    }
  }
  }  // groups
  __syncthreads();
  flush_digits(cnt, passes, digit_counts);
}

// qstart[c] for every query-level cell c < n_out: the number of active hit
// points in cells before c, found in their sorted keys. A warp takes
// kStartCells consecutive cells: it finds the first point of its first cell
// and of the cell after its last by a 32-way search (4-5 probes of 10^6
// points), fills them with one value when no point lies between - nearly every
// run: hit points lie on surfaces, 10^5 of the 2 * 10^7 cells of a 1M-Gaussian
// scene hold one - and else searches that interval once per cell, 16 cells per
// lane at a time. Bound by the 4 B per cell it writes. Counting the points per
// cell with atomics and scanning the counts read and wrote every cell three
// times and cleared it once (22 M cells: 160 us and a 89 MB memset).
constexpr uint32_t kStartCells = 512;
__device__ __forceinline__ void cell_starts(uint32_t block, const uint32_t* __restrict__ skey,
                                            int shift, const DeviceHeader* header,
                                            uint32_t n_out, uint32_t* __restrict__ qstart) {
  constexpr int kPer = kStartCells / kWarp;
  const int lane = threadIdx.x & 31;
  const uint32_t w = (block * (uint32_t)kThreads + threadIdx.x) / kWarp;
  if (w > (n_out - 1) / kStartCells) return;
  const uint32_t c0 = w * kStartCells;
  const uint32_t n = header->n_active;
  // first positions of cells c0 and c0 + kStartCells (both searches at once)
  const uint32_t target[2] = {c0, c0 + kStartCells};
  uint32_t a[2] = {0u, 0u}, b[2] = {n, n};       // the answer lies in [a, b]
  while (a[0] < b[0] || a[1] < b[1]) {
    bool below[2];
    uint32_t step[2];
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      step[k] = (b[k] - a[k] + kWarp - 1) / kWarp;
      const uint32_t p = a[k] + (lane + 1) * step[k] - 1;
      below[k] = a[k] < b[k] && p < b[k] && (__ldg(skey + p) >> shift) < target[k];
    }
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const uint32_t cnt = (uint32_t)__popc(__ballot_sync(kFullMask, below[k]));
      if (a[k] < b[k]) {
        const uint32_t na = min(a[k] + cnt * step[k], b[k]);
        b[k] = min(b[k], a[k] + (cnt + 1) * step[k] - 1);
        a[k] = na;
      }
    }
  }
  uint32_t at[kPer];
#pragma unroll
  for (int j = 0; j < kPer; ++j) at[j] = a[0];
  // (keys of a sort that gave up may be out of order: every read stays below n)
  if (a[1] > a[0]) {
    uint32_t len = a[1] - a[0];
    while (len > 0) {
      const uint32_t half = (len + 1) >> 1;
#pragma unroll
      for (int j = 0; j < kPer; ++j) {
        const uint32_t c = c0 + (uint32_t)(j / 4) * (4 * kWarp) + 4 * lane + (j & 3);
        if ((__ldg(skey + at[j] + half - 1) >> shift) < c) at[j] += half;
      }
      len -= half;
    }
  }
#pragma unroll
  for (int j = 0; j < kPer; j += 4) {
    const uint32_t c = c0 + (uint32_t)(j / 4) * (4 * kWarp) + 4 * lane;
    if (c + 3 < n_out) {
      *reinterpret_cast<uint4*>(qstart + c) = make_uint4(at[j], at[j + 1], at[j + 2], at[j + 3]);
    } else {
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (c + i < n_out) qstart[c + i] = at[j + i];
    }
  }
}

// [start, end) of every non-empty bucket from the boundaries of the sorted
// keys, and its bit in listed: a lookup reads the table only where the bit is
// set, so the table (134 MB at 2^24 buckets) is never cleared and the many
// empty lookups stay in the 2 MB of bits.
__device__ __forceinline__ void bucket_ranges(uint32_t block, const uint32_t* __restrict__ keys,
                                              const DeviceHeader* header, int64_t n_cap,
                                              uint2* __restrict__ range,
                                              uint32_t* __restrict__ listed) {
  const int64_t i = (int64_t)block * kThreads + threadIdx.x;
  if (header->stalled) return;
  int64_t n = header->n_pairs;
  if (n > n_cap) n = n_cap;
  if (i >= n) return;
  const uint32_t k = keys[i];
  if (i == 0 || keys[i - 1] != k) {
    range[k].x = (uint32_t)i;
    atomicOr(&listed[k >> 5], 1u << (k & 31u));
  }
  if (i == n - 1 || keys[i + 1] != k) range[k].y = (uint32_t)(i + 1);
}

// The active hit points' positions and ids in sorted order: the pair loops, the
// tile costs and the backward's packing read them in turn instead of gathering
// three floats per point by id each time.
__device__ __forceinline__ void sorted_positions(uint32_t block, const float* __restrict__ x,
                                                 const uint32_t* __restrict__ qval, int64_t m,
                                                 const DeviceHeader* header,
                                                 float4* __restrict__ qpos) {
  const int64_t k = (int64_t)block * kThreads + threadIdx.x;
  if (k >= (int64_t)header->n_active || header->stalled) return;
  const uint32_t q = qval[k];
  qpos[k] = make_float4(x[q], x[m + q], x[2 * m + q], __uint_as_float(q));
}

// After the sorts, in one launch: the query-level cells' starts (the first
// start_blocks blocks), the hit points' positions (the next pos_blocks) and the
// buckets' ranges (the others).
__global__ void __launch_bounds__(kThreads)
ranges_kernel(uint32_t start_blocks, const uint32_t* __restrict__ skey, int shift,
              uint32_t n_out, uint32_t* __restrict__ qstart, uint32_t pos_blocks,
              const float* __restrict__ x, const uint32_t* __restrict__ qval, int64_t m,
              float4* __restrict__ qpos, const uint32_t* __restrict__ keys, int64_t n_cap,
              uint2* __restrict__ range, uint32_t* __restrict__ listed,
              const DeviceHeader* header) {
  const uint32_t b = blockIdx.x;
  if (b < start_blocks) cell_starts(b, skey, shift, header, n_out, qstart);
  else if (b < start_blocks + pos_blocks)
    sorted_positions(b - start_blocks, x, qval, m, header, qpos);
  else bucket_ranges(b - start_blocks - pos_blocks, keys, header, n_cap, range, listed);
}

__global__ void index_flags_kernel(const DeviceHeader* header, uint32_t* flags) {
  *flags = index_flags(header);
}

// Blocks of the kernels that add digit counts: at the end each block adds up to
// 256 counts per sort pass to the same words, which serialise, so a few blocks
// per SM take several groups each rather than every group its own block (2, 8
// and unlimited blocks per SM: density estimate of 1M photons 864, 812 and 829
// us a pass, eight views over 1M Gaussians 4.64, 4.50 and 4.59 ms).
inline unsigned shared_blocks(unsigned groups) { return std::min(groups, 152u * 8u); }
inline unsigned blocks_for(int64_t n, int t = kThreads) {
  return (unsigned)((n + t - 1) / t);
}

}  // namespace

gpf_field float32_view(const IndexDims& d, const IndexBuffers& b, const gpf_field& f) {
  if (f.storage == GPF_F32) return f;
  // rows of the field's own length n, packed at the start of the buffer
  const int64_t n = f.n;
  gpf_field v = f;
  v.storage = GPF_F32;
  v.mean = b.dec;
  v.quat = b.dec + 3 * n;
  v.logscale = b.dec + 7 * n;
  v.spectrum = b.dec + 10 * n;
  v.anchor = nullptr;
  return v;
}

size_t gpart_words(int64_t n) {
  const int64_t groups = group_count(n, kThreads) + 1;
  return (size_t)(groups + groups / kSuper + 1);
}

cudaError_t launch_build(const IndexDims& d, const IndexBuffers& b, const gpf_field& f_in,
                         const gpf_queries& q, cudaStream_t stream) {
  const Grid& grid = d.grid;
  // everything that starts from zero lies in one range: the header, the
  // occupancy bits, the sorts' counts and status words, the entry sums
  cudaError_t e = cudaMemsetAsync(b.header, 0, b.clear_bytes, stream);
  if (e != cudaSuccess) return e;
  // 0. 16-bit storage: decode every parameter to float32 once
  if (f_in.storage != GPF_F32 && f_in.n > 0) {
    decode_bf16_kernel<<<blocks_for(f_in.n), kThreads, 0, stream>>>(f_in, b.dec);
    note_launches(1);
  }
  const gpf_field f = float32_view(d, b, f_in);
  const SortTask sort_q{b.qkey[0], b.qval[0], b.qkey[1], b.qval[1], q.m, nullptr, grid.key_bits,
                        b.qsort_ws};
  const SortTask sort_o{b.okey[0], b.oval[0], b.okey[1], b.oval[1], f.n, nullptr, grid.obits,
                        b.osort_ws};
  const SortTask sort_g{b.gkey[0], b.gval[0], b.gkey[1], b.gval[1], d.p_max, &b.header->n_pairs,
                        grid.hash_bits, b.gsort_ws};
  const bool lists = !d.brute && f.n > 0;
  // 1. hit point keys and occupancy bits of every level
  if (q.m > 0) {
    query_keys_kernel<<<shared_blocks(blocks_for(q.m)), kThreads, 0, stream>>>(
        grid, q.x, q.normal, q.wo, q.valid, q.m, b.qkey[0], b.qval[0], b.occ, d.brute ? 0 : 1,
        b.qbits, radix_sort_passes(grid.key_bits), radix_sort_counts(b.qsort_ws), b.header);
    note_launches(1);
  }
  // 2. Gaussian records, level boxes, entry counts, order keys, level mask;
  // 3. (bucket, Gaussian) entries
  if (f.n > 0) {
    const unsigned blocks = shared_blocks(blocks_for(f.n));
    preprocess_kernel<<<blocks, kThreads, 0, stream>>>(
        f, grid, d.cutoff, d.brute ? 1 : 0, b.rec, rec_stride(d.channels), b.vet, b.occ,
        b.gcount, b.glive, b.gmask, b.qbox, b.okey[0], b.oval[0], radix_sort_passes(grid.obits),
        radix_sort_counts(b.osort_ws), lists ? b.gpart : nullptr, b.header);
    note_launches(1);
    if (lists) {
      emit_kernel<<<blocks, kThreads, 0, stream>>>(
          grid, f.n, d.p_max, b.vet, b.occ, b.gmask, b.gcount,
          b.gpart, b.gkey[0], b.gval[0], radix_sort_passes(grid.hash_bits),
          radix_sort_counts(b.gsort_ws), b.cocc, b.focc, b.header);
      note_launches(1);
    }
  }
  // 4. side by side: hit points by query-level cell (inactive ones last),
  // Gaussians in the backward's order, entries by bucket
  const SortTask sorts[3] = {sort_q, sort_o, sort_g};
  e = radix_sort_counted(sorts, lists ? 3 : 2, &b.header->stalled, stream);
  if (e != cudaSuccess) return e;
  // 5. the cells' starts, the hit points' positions and the bucket ranges
  {
    const uint32_t n_out = grid.n_keys + 2;
    const unsigned starts =
        blocks_for(((int64_t)n_out + kStartCells - 1) / kStartCells * kWarp);
    const unsigned ranges = lists ? blocks_for(d.p_max) : 0u;
    const unsigned pos = blocks_for(q.m);
    ranges_kernel<<<starts + pos + ranges, kThreads, 0, stream>>>(
        starts, b.qkey[b.qsorted], 3 * grid.qsub, n_out, b.qstart, pos, q.x, b.qval[b.qsorted],
        q.m, b.qpos, b.gkey[b.gsorted], d.p_max, b.brange, b.listed, b.header);
    note_launches(1);
  }
  if (lists && d.split_items > 0 && q.m > 0) {
    e = launch_tile_split(d, b, q, stream);
    if (e != cudaSuccess) return e;
  }
  return cudaGetLastError();
}

cudaError_t launch_index_flags(const DeviceHeader* header, uint32_t* flags, cudaStream_t stream) {
  index_flags_kernel<<<1, 1, 0, stream>>>(header, flags);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_quantize(const gpf_field& src, const gpf_field& dst, cudaStream_t stream) {
  if (src.n == 0) return cudaSuccess;
  // whole groups per block: kThreads is a multiple of GPF_BF16_GROUP
  quantize_bf16_kernel<<<blocks_for(src.n), kThreads, 0, stream>>>(src, dst);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace gpf
