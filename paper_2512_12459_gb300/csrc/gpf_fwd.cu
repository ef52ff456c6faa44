// gpf_radiance_fwd: radiance at hit points (Sec. 4.2, aggregation equation;
// the soft falloff and soft normalisation of the query listing of Algorithm S3).
//
// A tile is 32 consecutive hit points in cell-sorted order; a warp takes it, or
// a team of warps where there are few tiles. The lanes look up their cell's
// list on every grid level that holds Gaussians and group equal cells:
//   * levels with few distinct cells (the Gaussians there are large next to the
//     tile) are walked together. The lists of all their cells are laid end to
//     end and vetted 32 entries at a time, an entry per lane: the entry belongs
//     to this level and cell, it was not already taken from an earlier cell of
//     the tile, and its bounding sphere reaches the tile's box. The ids that
//     pass are queued and their records loaded 32 at a time, tested against a
//     lower bound of their Mahalanobis distance to the box, staged in shared
//     memory, and every lane evaluates all of them at its own hit point.
//   * levels with many distinct cells (the Gaussians are small next to the
//     spacing of the hit points) are pooled: the lanes' own lists are laid end to
//     end, a level after the other, and taken 32 (hit point, entry) items at a
//     time, one per lane; a segmented sum over the lanes returns each hit
//     point's share to its lane.
// Every lane applies the exact predicate Q <= k^2, so the result equals the
// brute-force sum over {i : Q_i <= k^2}. With no cell lists (k = +INF or
// brute force) the candidates are all Gaussians, in index order.
#include <cuda_runtime.h>
#include <math.h>

#include <cmath>
#include <stdint.h>

#include "gpf_internal.h"

namespace gpf {

namespace {

constexpr int kFwdWarps = 4;
constexpr int kFwdThreads = kFwdWarps * kWarp;
// Units of a tile's estimated work (tile_cost_kernel).
constexpr uint32_t kCostPerEntry = 8, kCostPerTile = 8 * 32 * 10;
constexpr uint32_t kTileUnits = 0x80000000u;   // of a tile's parts: taken by several units
constexpr int kQueue = 128;   // vetted ids of a warp that wait for their records

struct FwdArgs {
  Grid grid;
  const uint32_t* qval;    // sorted hit point ids
  const float4* qpos;      // sorted positions and ids of the active ones
  DeviceHeader* header;
  const float* albedo;     // [C,M] or null
  int64_t m;
  const float* rec;
  const VetRec* vet;
  const uint2* brange;     // [n_buckets] [start, end) of each bucket's list
  const uint32_t* listed;  // [n_buckets / 32] set: the bucket has a list
  const uint32_t* gval;    // sorted entries (Gaussian ids)
  int64_t n;               // Gaussians (brute force)
  int mode;
  float r, r2, inv_rr;     // falloff radius, its square, 1/max(r, 1e-6)
  float eps;
  float kde_scale;         // disk kernel: 1 / (pi r^2)
  float cut, cut2;         // k, k^2
  float tscale;            // sqrt(3 log2 e) / max(r, 1e-6): the falloff root in base 2
  float* out;              // [C,M]
  float* z;                // [M] or null
  unsigned long long* counts;  // count mode: [candidates, included]
  const uint32_t* tparts;  // split forward: parts of each tile, kTileUnits (null: no splitting)
  const uint4* xunit;      // split forward: (tile, unit of units and parts, first slot) of each unit
  uint32_t* xheavy;        // disk kernel: tiles deferred to the second launch
  int late;                // 1: the second launch, over the deferred tiles
  float* xsum;             // split forward: [slot][C + 1][32] partial sums
};

__device__ __forceinline__ float warp_min(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fminf(v, __shfl_xor_sync(kFullMask, v, o));
  return v;
}
__device__ __forceinline__ float warp_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(kFullMask, v, o));
  return v;
}

// Pair kernels: the Gaussian weight alone, with the soft falloff psi, or the
// disk of the photon density estimate.
constexpr int kKernGauss = 0, kKernFalloff = 1, kKernDisk = 2;
constexpr float kNegHalfLog2e = -0.72134752044448170368f;   // -log2(e) / 2

// |d| from d2 = |d|^2: one reciprocal square root and one Newton step on the
// square root (residual d2 - s^2 by a fused multiply-add), which leaves about
// 1 ulp of relative error, as a correctly rounded square root would within an
// ulp, without its special-case branch.
__device__ __forceinline__ float dist_of(float d2) {
  const float y = rsqrt_approx(d2);
  const float s = d2 * y;
  return fmaf(0.5f * y, fmaf(-s, s, d2), s);
}

// w = exp(-Q/2) psi(|d|) of an included pair as 2^-(Q log2(e)/2 + t'^2), with
// t' = sqrt(3 log2 e) (|d| - r)/r beyond the falloff radius r (zero within).
template <int KERN>
__device__ __forceinline__ float pair_exp2(float Q, float dx, float dy, float dz,
                                           const FwdArgs& a) {
  float e = Q * kNegHalfLog2e;
  if (KERN == kKernFalloff) {
    const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    const float t = fmaxf(dist_of(d2) - a.r, 0.0f) * a.tscale;   // as eval_staged: same w
    e = fmaf(-t, t, e);
  }
  return ex2_approx(e);
}

// Weight of one pair: w = exp(-Q/2) psi(|d|) when Q <= k^2 (hit = true); for
// the disk kernel w = 1 when |d| <= r (Eq. kde; 1/(pi r^2) is applied once
// per hit point). In count mode only evaluated and included pairs are counted.
template <int KERN, bool COUNT>
__device__ __forceinline__ float pair_weight(const float* __restrict__ r, float px, float py,
                                             float pz, const FwdArgs& a, bool& hit,
                                             uint32_t& n_eval, uint32_t& n_inc) {
  const float dx = px - r[0], dy = py - r[1], dz = pz - r[2];
  if (KERN == kKernDisk) {
    const float d2 = fmaf(dx, dx, fmaf(dy, dy, dz * dz));
    hit = d2 <= a.r2;
    if (COUNT) {
      ++n_eval;
      n_inc += hit ? 1u : 0u;
      hit = false;
    }
    return hit ? 1.0f : 0.0f;
  }
  const float u0 = fmaf(r[4], dx, fmaf(r[5], dy, r[6] * dz));
  const float u1 = fmaf(r[7], dx, fmaf(r[8], dy, r[9] * dz));
  const float u2 = fmaf(r[10], dx, fmaf(r[11], dy, r[12] * dz));
  const float Q = fmaf(u0, u0, fmaf(u1, u1, u2 * u2));
  if (COUNT) {
    ++n_eval;
    n_inc += Q <= a.cut2 ? 1u : 0u;
    hit = false;
    return 0.0f;
  }
  hit = Q <= a.cut2;
  if (!hit) return 0.0f;
  return pair_exp2<KERN>(Q, dx, dy, dz, a);
}

// Accumulate one Gaussian record r into this lane's sums (or count it).
template <int C, int KERN, bool COUNT>
__device__ __forceinline__ void eval_pair(const float* __restrict__ r, float px, float py, float pz,
                                          const FwdArgs& a, float (&L)[C], float& Z,
                                          uint32_t& n_eval, uint32_t& n_inc) {
  bool hit;
  const float w = pair_weight<KERN, COUNT>(r, px, py, pz, a, hit, n_eval, n_inc);
  if (hit) {
#pragma unroll
    for (int c = 0; c < C; ++c) L[c] = fmaf(w, r[13 + c], L[c]);
    Z += w;
  }
}

// Staged records, a field after the other so that one 16-byte load gives a
// field of four records as two packed pairs: -mu (3), M (9), Phi (C).
__host__ __device__ constexpr int stage_fields(int C) { return 12 + C; }

// Every staged record of the walked levels at this lane's hit point, four at a
// time as straight-line code, two records to an instruction: the evaluation is
// bound by the instructions it issues, about 25 per record packed and 40 not.
// Every value is rounded as in pair_weight. nk is a multiple of 4: the slots
// past the last record hold a NaN mean, which fails Q <= k^2, and finite Phi,
// so their weight is 0. The sums take the records in turn, a scalar operation
// each: sums of the even and the odd records apart would save 2 of 25
// instructions a record and change the order.
template <int C, int KERN>
__device__ __forceinline__ void eval_staged(const float* __restrict__ st, int nk, float px,
                                            float py, float pz, const FwdArgs& a,
                                            float (&L)[C], float& Z) {
  const f32x2 px2 = pack2(px, px), py2 = pack2(py, py), pz2 = pack2(pz, pz);
  const f32x2 c_e = pack2(-kNegHalfLog2e, -kNegHalfLog2e);
  const f32x2 c_neg = pack2(-1.0f, -1.0f), c_half = pack2(0.5f, 0.5f);
  const f32x2 c_r = pack2(-a.r, -a.r), c_t = pack2(a.tscale, a.tscale);
  for (int s = 0; s < nk; s += 4) {
    auto field = [&](int f) {
      return *reinterpret_cast<const ulonglong2*>(st + f * kWarp + s);
    };
    f32x2 w[2];
    {
      const ulonglong2 nx = field(0), ny = field(1), nz = field(2);
      const f32x2 dx[2] = {add2(px2, nx.x), add2(px2, nx.y)};
      const f32x2 dy[2] = {add2(py2, ny.x), add2(py2, ny.y)};
      const f32x2 dz[2] = {add2(pz2, nz.x), add2(pz2, nz.y)};
      f32x2 d2[2];
      if (KERN != kKernGauss) {
#pragma unroll
        for (int h = 0; h < 2; ++h)
          d2[h] = fma2(dx[h], dx[h], fma2(dy[h], dy[h], mul2(dz[h], dz[h])));
      }
      if (KERN == kKernDisk) {
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          float d0, d1;
          unpack2(d2[h], d0, d1);
          w[h] = pack2(d0 <= a.r2 ? 1.0f : 0.0f, d1 <= a.r2 ? 1.0f : 0.0f);
        }
      } else {
        f32x2 u[3][2];
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const ulonglong2 m0 = field(3 + 3 * j), m1 = field(4 + 3 * j), m2 = field(5 + 3 * j);
          u[j][0] = fma2(m0.x, dx[0], fma2(m1.x, dy[0], mul2(m2.x, dz[0])));
          u[j][1] = fma2(m0.y, dx[1], fma2(m1.y, dy[1], mul2(m2.y, dz[1])));
        }
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const f32x2 Q = fma2(u[0][h], u[0][h], fma2(u[1][h], u[1][h], mul2(u[2][h], u[2][h])));
          f32x2 e = mul2(Q, c_e);          // minus the exponent
          if (KERN == kKernFalloff) {
            float d0, d1;
            unpack2(d2[h], d0, d1);
            const f32x2 y = pack2(rsqrt_approx(d0), rsqrt_approx(d1));
            const f32x2 sq = mul2(d2[h], y);
            const f32x2 res = fma2(mul2(sq, c_neg), sq, d2[h]);
            const f32x2 dist = fma2(mul2(y, c_half), res, sq);
            float t0, t1;
            unpack2(add2(dist, c_r), t0, t1);
            const f32x2 t = mul2(pack2(fmaxf(t0, 0.0f), fmaxf(t1, 0.0f)), c_t);
            e = fma2(t, t, e);
          }
          float q0, q1, e0, e1;
          unpack2(Q, q0, q1);
          unpack2(e, e0, e1);
          w[h] = pack2(ex2_approx(-(q0 <= a.cut2 ? e0 : INFINITY)),     // 2^-inf = +0
                       ex2_approx(-(q1 <= a.cut2 ? e1 : INFINITY)));
        }
      }
    }
    float v[4];
    unpack2(w[0], v[0], v[1]);
    unpack2(w[1], v[2], v[3]);
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const float4 phi = *reinterpret_cast<const float4*>(st + (12 + c) * kWarp + s);
      L[c] = fmaf(v[3], phi.w, fmaf(v[2], phi.z, fmaf(v[1], phi.y, fmaf(v[0], phi.x, L[c]))));
    }
    Z = ((Z + v[0]) + v[1]) + v[2] + v[3];
  }
}

// The pairs that eval_staged would evaluate and include (count mode).
template <int C>
__device__ __forceinline__ void count_staged(const float* __restrict__ st, int nk, float px,
                                             float py, float pz, const FwdArgs& a,
                                             uint32_t& n_eval, uint32_t& n_inc) {
  for (int s = 0; s < nk; ++s) {
    auto f = [&](int k) { return st[k * kWarp + s]; };
    const float dx = px + f(0), dy = py + f(1), dz = pz + f(2);
    const float u0 = fmaf(f(3), dx, fmaf(f(4), dy, f(5) * dz));
    const float u1 = fmaf(f(6), dx, fmaf(f(7), dy, f(8) * dz));
    const float u2 = fmaf(f(9), dx, fmaf(f(10), dy, f(11) * dz));
    ++n_eval;
    n_inc += fmaf(u0, u0, fmaf(u1, u1, u2 * u2)) <= a.cut2 ? 1u : 0u;
  }
}

// Hands the per-lane partial sums pc of the lanes with f set to their owner
// key (owner lane) in acc[c][key]. The flushing lanes of one key are
// contiguous, so a segmented inclusive sum over the lanes leaves each key's
// total in its last lane, which adds it to acc. Lanes that flush restart
// from zero.
template <int C>
__device__ __forceinline__ void pooled_flush(float (*acc)[kWarp], int lane, int key_in, bool f,
                                             float (&pc)[C + 1]) {
  const int key = f ? key_in : 2 * kWarp + lane;
  float t[C + 1];
#pragma unroll
  for (int c = 0; c <= C; ++c) t[c] = f ? pc[c] : 0.0f;
#pragma unroll
  for (int d = 1; d < kWarp; d <<= 1) {
    const int kd = __shfl_up_sync(kFullMask, key, d);
    float u[C + 1];
#pragma unroll
    for (int c = 0; c <= C; ++c) u[c] = __shfl_up_sync(kFullMask, t[c], d);
    if (lane >= d && kd == key) {
#pragma unroll
      for (int c = 0; c <= C; ++c) t[c] += u[c];
    }
  }
  const int kn = __shfl_down_sync(kFullMask, key, 1);
  if (f && (lane == kWarp - 1 || kn != key)) {
#pragma unroll
    for (int c = 0; c <= C; ++c) acc[c][key] += t[c];
  }
  if (f) {
#pragma unroll
    for (int c = 0; c <= C; ++c) pc[c] = 0.0f;
  }
  __syncwarp();
}

// A record, in 32-byte loads where its stride allows them: a gather is bound
// by the lines its instructions touch, one per lane whatever the width.
template <int RS>
__device__ __forceinline__ void load_rec(const float* __restrict__ rec, uint32_t g, float (&r)[RS]) {
  const float* src = rec + (int64_t)g * RS;
  if constexpr (RS % 8 == 0) {
#pragma unroll
    for (int v = 0; v < RS; v += 8) ld_global_v8(src + v, r + v);
  } else {
#pragma unroll
    for (int v = 0; v < RS / 4; ++v) {
      const float4 t = __ldg(reinterpret_cast<const float4*>(src) + v);
      r[4 * v] = t.x; r[4 * v + 1] = t.y; r[4 * v + 2] = t.z; r[4 * v + 3] = t.w;
    }
  }
}

// Its first eight values (mean, radius, the first of M), and the others.
template <int RS>
__device__ __forceinline__ void load_rec_head(const float* __restrict__ rec, uint32_t g,
                                              float (&r)[RS]) {
  const float* src = rec + (int64_t)g * RS;
  if constexpr (RS % 8 == 0) {
    ld_global_v8(src, r);
  } else {
#pragma unroll
    for (int v = 0; v < 2; ++v) {
      const float4 t = __ldg(reinterpret_cast<const float4*>(src) + v);
      r[4 * v] = t.x; r[4 * v + 1] = t.y; r[4 * v + 2] = t.z; r[4 * v + 3] = t.w;
    }
  }
}
template <int RS>
__device__ __forceinline__ void load_rec_tail(const float* __restrict__ rec, uint32_t g,
                                              float (&r)[RS]) {
  const float* src = rec + (int64_t)g * RS;
  if constexpr (RS % 8 == 0) {
#pragma unroll
    for (int v = 8; v < RS; v += 8) ld_global_v8(src + v, r + v);
  } else {
#pragma unroll
    for (int v = 2; v < RS / 4; ++v) {
      const float4 t = __ldg(reinterpret_cast<const float4*>(src) + v);
      r[4 * v] = t.x; r[4 * v + 1] = t.y; r[4 * v + 2] = t.z; r[4 * v + 3] = t.w;
    }
  }
}

// The shared memory of a warp. Sizes follow the index: levels * coop segments
// at most, levels ranges per lane.
struct WarpShared {
  float* stage;            // [max(rec stride, stage fields)][32]
  float (*acc)[kWarp];     // [C + 1][32] pooled-mode sums per hit point
  float4* box;             // [3] the tile's box: (lo, hi.x), (hi.yz, centre.xy),
                           // (centre.z, half extents)
  uint2* range;            // [levels][32]
  unsigned long long* cell;  // [segments + 3] pack_cell
  uint4* seg;              // [segments + 1] where it begins in the stream, first entry of its
                           // list - that, tag, level | first segment of that level << 8 |
                           // entries of its last chunk - 1 << 16
  uint32_t* queue;         // [kQueue]
};
__host__ __device__ constexpr int stage_words(int C) {
  return kWarp * (rec_stride(C) > stage_fields(C) ? rec_stride(C) : stage_fields(C));
}
__host__ __device__ constexpr int warp_shared_words(int C, int levels, int coop) {
  // (the cells' count rounded up to even, for 16-byte pieces)
  return stage_words(C) + (C + 1) * kWarp + 12 + 2 * levels * kWarp +
         (levels * coop + 4) / 2 * 2 * 2 + (levels * coop + 1) * 4 + kQueue;
}
template <int C>
__device__ __forceinline__ WarpShared warp_shared(float* base, int wib, int levels, int coop) {
  float* p = base + wib * warp_shared_words(C, levels, coop);
  WarpShared w;
  w.stage = p;
  p += stage_words(C);
  w.acc = reinterpret_cast<float(*)[kWarp]>(p);
  p += (C + 1) * kWarp;
  w.box = reinterpret_cast<float4*>(p);
  p += 12;
  w.range = reinterpret_cast<uint2*>(p);
  p += 2 * levels * kWarp;
  w.cell = reinterpret_cast<unsigned long long*>(p);
  p += (levels * coop + 4) / 2 * 2 * 2;
  w.seg = reinterpret_cast<uint4*>(p);
  p += (levels * coop + 1) * 4;
  w.queue = reinterpret_cast<uint32_t*>(p);
  return w;
}

// What bounds it: issue and the latency of dependent gathers together (1M
// Gaussians, one 1024 x 1024 view, ncu: 2.1 instructions a cycle and SM, 20
// resident warps, long and short scoreboard the largest stalls, DRAM 5 %). So
// the lists of a tile are walked as one stream of full chunks, whatever level
// and cell they belong to, an entry is rejected on one 32-byte load, and only
// survivors load their record. 5 blocks of 4 warps per SM: at 6 (80 registers)
// the spills cost 5 % more than the warps bring.
//
// The order of the sums is part of the result (a training step's last bits
// decide which pairs the next one includes), so what is free is only who takes
// a sum, not how it is made up (1M Gaussians, a view of 1024 x 1024, query cells
// of 0.02: a chunk loop per cell and level 693 us, this loop 602, and 548 when it
// summed in an order of its own): a tile's walked sums take the entries level by
// level, cell by cell, in list order; its pooled sums take each level's items
// 32 at a time, a lane each; and a tile of P parts (Grid: split_items) adds P
// such sums, each over every P-th chunk of 32 of every list. One warp takes all
// the parts, one after the other, on one look-up of the lists; only a tile that
// would keep a warp too long is given to several, some parts each
// (tile_parts_kernel). Two cases choose their own order: calls of few tiles,
// whose lists a team of warps shares, and the disk kernel, which nothing
// differentiates: there a tile that turns out longer than its estimate (eight
// sampled points may miss the one in a dense cell) is deferred, before its lists
// are walked, to a second launch, which splits it kHeavyParts ways: one such tile
// begun late kept its warp for 290 us after all the others of a 215 us density
// estimate had ended. Longer means an eighth of what every warp has to do;
// nothing is deferred below kHeavyChunks chunks (16, 48, 144: the estimate 799,
// 812, 883 us a pass). If they were too many for the list of units, the second
// launch takes them whole (all of them, so that the sums do not depend on which
// warp came first).
constexpr uint32_t kHeavyParts = 8, kHeavyChunks = 48;
__device__ __forceinline__ uint32_t heavy_chunks(const DeviceHeader* h) {
  const unsigned long long share =
      h->split_cost / ((unsigned long long)kCostPerEntry * kWarp * 152u * 20u);
  return max(kHeavyChunks, (uint32_t)min(share / 8, 1ull << 20));
}
__device__ __forceinline__ bool heavy_fits(const DeviceHeader* h) {
  return h->n_xslots + kHeavyParts * h->n_heavy <= (unsigned long long)GPF_MAX_SPLIT_UNITS;
}

// COUNT: count the evaluated and included pairs instead of summing radiance.
// TEAM: warps of a block that share a tile, each taking every TEAM-th chunk of
// its lists; their sums are added in order.
template <int C, bool BRUTE, int KERN, bool COUNT, int TEAM>
__global__ void __launch_bounds__(TEAM > 4 ? TEAM * kWarp : kFwdThreads,
                                  TEAM > 4 ? 1 : C <= 4 ? 5 : 4)
fwd_kernel(const __grid_constant__ FwdArgs a) {
  constexpr int RS = rec_stride(C);
  constexpr bool kOrdered = TEAM == 1 && KERN != kKernDisk;   // sums in the order stated above
  constexpr bool kDefer = KERN == kKernDisk && !BRUTE && !COUNT;
  extern __shared__ __align__(16) float s_mem[];
  __shared__ unsigned long long s_unit;
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5;
  if (index_unusable(a.header)) return;
  const Grid& G = a.grid;
  const WarpShared ws = warp_shared<C>(s_mem, wib, G.levels, G.coop);
  // the staged slots start finite: eval_staged reads whole groups of four
  for (int i = lane; i < stage_words(C); i += kWarp) ws.stage[i] = 0.0f;
  const int64_t n_act = a.header->n_active;
  const int64_t n_tiles = (a.m + kWarp - 1) / kWarp;
  // the units of the tiles that several warps take come first, then every tile
  // as one unit (those tiles' are skipped)
  const int64_t n_x = a.tparts ? (int64_t)a.header->n_xunits : 0;
  const bool late = kDefer && a.late;
  const bool late_split = late && heavy_fits(a.header);
  const int64_t n_units =
      late ? (int64_t)a.header->n_heavy * (late_split ? (int64_t)kHeavyParts : 1) : n_x + n_tiles;
  const uint32_t limit = kDefer && !late && a.tparts ? heavy_chunks(a.header) : 0xffffffffu;
  unsigned long long* const next_unit = late ? &a.header->next_heavy : &a.header->next_tile;
  const uint32_t lmask = a.header->level_mask;
  uint32_t n_eval = 0, n_inc = 0;
  // persistent: every warp (team) takes the next unit until none is left, so a
  // warp that drew a light tile goes on with another one
  for (;;) {
  int64_t unit;
  if (TEAM > 1) {
    __syncthreads();
    if (threadIdx.x == 0) s_unit = atomicAdd(next_unit, 1ull);
    __syncthreads();
    unit = (int64_t)s_unit;
  } else {
    __syncwarp();
    unsigned long long unit_u = 0;
    if (lane == 0) unit_u = atomicAdd(next_unit, 1ull);
    unit = (int64_t)__shfl_sync(kFullMask, unit_u, 0);
  }
  if (unit >= n_units) break;
  // this unit's tile, its parts [p0, p1) of `parts`, and, where other units have
  // the tile's other parts, the slot of part 0
  int64_t tile;
  uint32_t p0 = 0, p1 = 1, parts = 1, slot = 0;
  bool split = false;
  if (late) {
    split = late_split;
    tile = a.xheavy[split ? unit / kHeavyParts : unit];
    if (split) {
      parts = kHeavyParts;
      p0 = (uint32_t)(unit % kHeavyParts);
      p1 = p0 + 1;
      slot = a.header->n_xslots + (uint32_t)unit - p0;
    }
  } else if (unit < n_x) {
    const uint4 xu = a.xunit[unit];
    const uint32_t i = xu.y & 0xffu, of = (xu.y >> 8) & 0xffu;
    tile = xu.x;
    slot = xu.z;
    split = true;
    parts = kOrdered ? xu.y >> 16 : of;
    p0 = kOrdered ? i * parts / of : i;
    p1 = kOrdered ? (i + 1) * parts / of : i + 1;
  } else {
    tile = unit - n_x;
    if (a.tparts) {
      const uint32_t tp = a.tparts[tile];
      if (tp & kTileUnits) continue;          // taken by its units
      if (kOrdered) p1 = parts = tp;
    }
  }
  const int64_t base = tile * kWarp;
  const int64_t k = base + lane;
  const bool in_range = k < a.m;
  const bool active = k < n_act;
  if (!COUNT && !split && in_range && !active && (TEAM == 1 || wib == 0)) {
    const uint32_t q = a.qval[k];
#pragma unroll
    for (int c = 0; c < C; ++c) a.out[(int64_t)c * a.m + q] = 0.0f;
    if (a.z) a.z[q] = 0.0f;
  }
  if (base >= n_act) continue;  // the whole warp or team (never a split tile)

  float px = 0.f, py = 0.f, pz = 0.f;
  uint32_t q = 0;
  if (active) {
    const float4 p = __ldg(a.qpos + k);
    px = p.x;
    py = p.y;
    pz = p.z;
    q = __float_as_uint(p.w);
  }

  // ---- walked levels: their distinct cells' lists as segments, end to end;
  // pooled levels: each lane's lists of a level end to end, a level after the
  // other (range[p] of the p-th pooled level: first entry - items before, items
  // up to and with this lane's). The pooled levels are the finest ones: a
  // coarser level has no more distinct cells.
  int n_seg = 0, n_pool = 0;
  uint32_t total = 0;                     // entries of the segments
  uint32_t pool_chunks = 0;               // chunks of the pooled levels
  unsigned long long pool_levels = 0;     // 4 bits per pooled level
  // parts take whole chunks of each list, so their segments begin with a chunk
  const bool pad = kOrdered && parts > 1;
  if (!BRUTE) {
    const uint32_t c0x = coord0(px, G.ox, G.inv_cell0, G.max0x);
    const uint32_t c0y = coord0(py, G.oy, G.inv_cell0, G.max0y);
    const uint32_t c0z = coord0(pz, G.oz, G.inv_cell0, G.max0z);
    // the lane's list on every used level: first the bits of all levels, then
    // the ranges of those that have one
    {
      uint32_t bkt[kMaxLevels], word[kMaxLevels];
#pragma unroll
      for (int lev = 0; lev < kMaxLevels; ++lev) {
        word[lev] = 0;
        if (lev < G.levels && ((lmask >> lev) & 1u) && active) {
          bkt[lev] = bucket_of(G, lev, c0x >> lev, c0y >> lev, c0z >> lev);
          word[lev] = __ldg(a.listed + (bkt[lev] >> 5));
        }
      }
#pragma unroll
      for (int lev = 0; lev < kMaxLevels; ++lev) {
        if (lev < G.levels && ((lmask >> lev) & 1u)) {
          uint2 rg = make_uint2(0u, 0u);
          if (active && ((word[lev] >> (bkt[lev] & 31u)) & 1u)) rg = __ldg(a.brange + bkt[lev]);
          ws.range[lev * kWarp + lane] = rg;
        }
      }
    }
    // tile box of the active hit points
    const float bx0 = warp_min(active ? px : INFINITY), bx1 = warp_max(active ? px : -INFINITY);
    const float by0 = warp_min(active ? py : INFINITY), by1 = warp_max(active ? py : -INFINITY);
    const float bz0 = warp_min(active ? pz : INFINITY), bz1 = warp_max(active ? pz : -INFINITY);
    if (lane == 0) {         // in shared memory: the evaluation needs the registers
      ws.box[0] = make_float4(bx0, by0, bz0, bx1);
      ws.box[1] = make_float4(by1, bz1, 0.5f * (bx0 + bx1), 0.5f * (by0 + by1));
      ws.box[2] = make_float4(0.5f * (bz0 + bz1), 0.5f * (bx1 - bx0), 0.5f * (by1 - by0),
                              0.5f * (bz1 - bz0));
    }
    __syncwarp();
    for (int lev = 0; lev < G.levels; ++lev) {
      if (!((lmask >> lev) & 1u)) continue;
      const uint32_t lx = c0x >> lev, ly = c0y >> lev, lz = c0z >> lev;
      const unsigned long long packed = active ? pack_cell(lx, ly, lz) : ~0ull;
      const uint32_t peers = __match_any_sync(kFullMask, packed);
      const bool leader = active && (peers & lanemask_lt()) == 0;
      const uint32_t uniq = __ballot_sync(kFullMask, leader);
      const int nu = __popc(uniq);
      const uint2 rg = ws.range[lev * kWarp + lane];    // (0, 0) for inactive lanes
      const bool walked = nu <= G.coop;
      // (a cell without a list holds no Gaussian that another cell repeats)
      const uint32_t len = walked && !leader ? 0u : rg.y - rg.x;
      const uint32_t room = walked && pad ? (len + kWarp - 1) / kWarp * kWarp : len;
      uint32_t incl = room;
#pragma unroll
      for (int o = 1; o < kWarp; o <<= 1) {
        const uint32_t t = __shfl_up_sync(kFullMask, incl, o);
        if (lane >= o) incl += t;
      }
      const uint32_t all = __shfl_sync(kFullMask, incl, kWarp - 1);
      if (walked) {
        const uint32_t hm = __ballot_sync(kFullMask, len > 0u);
        if (len > 0u) {
          const int s = n_seg + __popc(hm & lanemask_lt());
          const uint32_t before = total + incl - room;
          ws.cell[s] = packed;
          ws.seg[s] = make_uint4(before, rg.x - before, cell_hash(G, lev, lx, ly, lz).tag,
                                 (uint32_t)lev | ((uint32_t)n_seg << 8) |
                                     (((len - 1u) & 31u) << 16));
        }
        n_seg += __popc(hm);
        total += all;
      } else {
        // (slot n_pool <= lev: the ranges of this and later levels are read first)
        ws.range[n_pool * kWarp + lane] = make_uint2(rg.x - (incl - len), incl);
        pool_chunks += (all + kWarp - 1) / kWarp;
        pool_levels |= (unsigned long long)lev << (4 * n_pool);
        ++n_pool;
      }
    }
    if (lane == 0) ws.seg[n_seg].x = total;
    __syncwarp();
  }
  const uint32_t n_chunks = (total + kWarp - 1) / kWarp;
  if (kDefer && !split && n_chunks + pool_chunks > limit) {
    if ((TEAM == 1 || wib == 0) && lane == 0)
      a.xheavy[atomicAdd(&a.header->n_heavy, 1ull)] = (uint32_t)tile;
    continue;
  }

  float L[C], Z = 0.0f;                   // this hit point's sums over the unit's parts
#pragma unroll
  for (int c = 0; c < C; ++c) L[c] = 0.0f;
  for (uint32_t pt = p0; pt < p1; ++pt) {
  // chunk c of the unit's lists, the pooled levels' first, is taken for
  // c mod of == part
  const uint32_t part = TEAM > 1 ? pt * TEAM + wib : pt;
  const uint32_t of = TEAM > 1 ? parts * TEAM : parts;
  float W[C], V = 0.0f;                   // the walked sums of this part
#pragma unroll
  for (int c = 0; c < C; ++c) W[c] = 0.0f;
#pragma unroll
  for (int c = 0; c <= C; ++c) ws.acc[c][lane] = 0.0f;
  __syncwarp();

  if (BRUTE) {
    float* my_rec = ws.stage;
    for (int64_t g0 = (int64_t)part * kWarp; g0 < a.n; g0 += (int64_t)of * kWarp) {
      const int64_t g = g0 + lane;
      const int cnt = (int)min((int64_t)kWarp, a.n - g0);
      if (g < a.n) {
        const float4* src = reinterpret_cast<const float4*>(a.rec + g * RS);
        float4* dst = reinterpret_cast<float4*>(my_rec + lane * RS);
#pragma unroll
        for (int v = 0; v < RS / 4; ++v) dst[v] = src[v];
      }
      __syncwarp();
      if (active)
        for (int s = 0; s < cnt; ++s)
          eval_pair<C, KERN, COUNT>(my_rec + s * RS, px, py, pz, a, W, V, n_eval, n_inc);
      __syncwarp();
    }
  } else {
    uint32_t chunk = (part + of - pool_chunks % of) % of;
    if (chunk < n_chunks) {
      const float cut_keep = a.cut * 1.0001f;
      int top = 1;                          // the segment search's first step
      while (2 * top < n_seg) top *= 2;
      // up to 32 segments (none is empty): lane l keeps where the l-th begins, and
      // a chunk's segments follow from the beginnings inside it, without a search
      const bool few = n_seg <= kWarp;
      const uint32_t seg_at =
          few && lane < n_seg ? ws.seg[lane].x : 0xffffffffu;
      const uint32_t le = lanemask_lt() | (1u << lane);
      // entry e of the stream: its segment (the last that begins at or before e)
      // and entry word (all ones, which no cell has: none), with the previous
      // word of its list
      auto fetch = [&](uint32_t chunk, int& seg, uint32_t& v, uint32_t& vprev, bool& first) {
        const uint32_t e = chunk * kWarp + lane;
        seg = 0;
        v = 0xffffffffu;
        vprev = 0u;
        first = true;
        if (few) {
          const uint32_t c0 = chunk * kWarp;
          const uint32_t inside = __reduce_or_sync(
              kFullMask, seg_at > c0 && seg_at - c0 < kWarp ? 1u << (seg_at - c0) : 0u);
          seg = __popc(__ballot_sync(kFullMask, seg_at <= c0)) - 1 + __popc(inside & le);
        }
        if (e < total) {
          if (!few)
            for (int st = top; st > 0; st >>= 1)
              if (seg + st <= n_seg - 1 && ws.seg[seg + st].x <= e) seg += st;
          // (a padded list's last chunk)
          if (pad && ws.seg[seg + 1].x == (chunk + 1) * kWarp &&
              (uint32_t)lane > (ws.seg[seg].w >> 16))
            return;
          const uint2 sg = *reinterpret_cast<const uint2*>(ws.seg + seg);
          const uint32_t* p = a.gval + (sg.y + e);         // modulo 2^32
          v = __ldg(p);
          first = e == sg.x;                 // of its list
          if (!first && lane == 0) vprev = __ldg(p - 1);   // (else the lane to the left has it)
        }
      };
      int qn = 0;                            // queued ids
      for (;;) {
        // vet entries until the queue may overflow; the entry words of the
        // next chunk are fetched while one is vetted
        int seg_n;
        uint32_t v_n, vp_n;
        bool first_n;
        fetch(chunk, seg_n, v_n, vp_n, first_n);
        while (chunk < n_chunks && qn <= kQueue - kWarp) {
          const int seg = seg_n;
          const uint32_t v = v_n;
          const uint32_t left = __shfl_up_sync(kFullMask, v, 1);
          // a Gaussian listed twice in a bucket sits on consecutive entries
          const bool again = !first_n && v == (lane == 0 ? vp_n : left);
          const uint2 sl = reinterpret_cast<const uint2*>(ws.seg + seg)[1];   // tag, level
          bool keep = (v & ~G.id_mask) == sl.x && !again;
          const uint32_t g = v & G.id_mask;
          VetRec r;
          if (keep) r = load_vet(a.vet + g);
          chunk += of;
          fetch(chunk, seg_n, v_n, vp_n, first_n);
          if (keep) {
            // sphere test: distance from mu to the tile box vs k * max s
            const float4 b0 = ws.box[0], b1 = ws.box[1];
            const float ex = fmaxf(fmaxf(b0.x - r.x, r.x - b0.w), 0.0f);
            const float ey = fmaxf(fmaxf(b0.y - r.y, r.y - b1.x), 0.0f);
            const float ez = fmaxf(fmaxf(b0.z - r.z, r.z - b1.y), 0.0f);
            // it must live on this level and cover this cell, and must not
            // have been taken from an earlier cell of this tile
            keep = fmaf(ex, ex, fmaf(ey, ey, ez * ez)) <= r.radius * r.radius &&
                   rec_level(r.radius) == (sl.y & 0xffu) && cell_in(r, ws.cell[seg]);
            for (int j = (int)((sl.y >> 8) & 0xffu); j < seg && keep; j += 2)   // two loads at a time
              keep = !(cell_in(r, ws.cell[j]) || (j + 1 < seg && cell_in(r, ws.cell[j + 1])));
          }
          const uint32_t kb = __ballot_sync(kFullMask, keep);
          if (keep) ws.queue[qn + __popc(kb & lanemask_lt())] = g;
          qn += __popc(kb);
        }
        __syncwarp();
        const bool done = chunk >= n_chunks;
        const int take = done ? qn : qn & ~(kWarp - 1);
        for (int i = 0; i < take; i += kWarp) {
          bool keep = i + lane < take;
          float rr[RS];
          if (keep) {
            load_rec<RS>(a.rec, ws.queue[i + lane], rr);
            if (KERN != kKernDisk) {
              const float4 b1 = ws.box[1], b2 = ws.box[2];
              keep = box_distance(rr + 4, b1.z - rr[0], b1.w - rr[1], b2.x - rr[2], b2.y, b2.z,
                                  b2.w) <= cut_keep;
            }
          }
          const uint32_t kb = __ballot_sync(kFullMask, keep);
          const int nk = __popc(kb);
          if (keep) {
            float* d = ws.stage + __popc(kb & lanemask_lt());
#pragma unroll
            for (int f = 0; f < 3; ++f) d[f * kWarp] = -rr[f];
#pragma unroll
            for (int f = 0; f < 9 + C; ++f) d[(3 + f) * kWarp] = rr[4 + f];
          } else if (nk + __popc(~kb & lanemask_lt()) < ((nk + 3) & ~3)) {
            ws.stage[nk + __popc(~kb & lanemask_lt())] = NAN;    // fills the last group of four
          }
          __syncwarp();
          if (COUNT) {
            if (active) count_staged<C>(ws.stage, nk, px, py, pz, a, n_eval, n_inc);
          } else {
            eval_staged<C, KERN>(ws.stage, nk, px, py, pz, a, W, V);
          }
          __syncwarp();
        }
        if (done) break;
        // the rest of the queue moves to its front
        const uint32_t rest = take + lane < qn ? ws.queue[take + lane] : 0u;
        __syncwarp();
        qn -= take;
        if (lane < qn) ws.queue[lane] = rest;
        __syncwarp();
      }
    }

    // ---- pooled levels: 32 (hit point, entry) items at a time, one per lane.
    // A lane sums what it evaluates for one owner at a time and hands the
    // sum over (pooled_flush) when the owner of its item slot, or the level,
    // changes, so no lane waits for the longest list and every sum has a fixed
    // order. The cell-box test is not needed here: an entry that reached this
    // bucket from another cell on the same level has a box that misses
    // this hit point, so Q > k^2 rejects it; the level test and the
    // duplicate test keep any Gaussian from being counted twice.
    if (part < pool_chunks) {
      // the level that is fetched: its chunks [lbeg, lend) of the pooled ones, its
      // items, where this lane's begin, and the lanes that have items, in order:
      // (lane, first item, tag, first entry - first item)
      int pl = -1, lev_f = 0;
      uint32_t lbeg = 0, lend = 0, items = 0, own_at = 0xffffffffu;
      uint4* owners = reinterpret_cast<uint4*>(ws.queue);
      static_assert(sizeof(uint4) * kWarp <= sizeof(uint32_t) * kQueue, "room for every lane");
      const uint32_t le = lanemask_lt() | (1u << lane);
      // item of this lane in chunk c: its owner (kWarp: none), the owner's tag,
      // level, entry word and the previous word of its list
      auto fetch = [&](uint32_t c, int& own, int& lev, uint32_t& tag, uint32_t& v,
                       uint32_t& vprev, bool& first) {
        own = kWarp;
        lev = lev_f;
        tag = v = vprev = 0u;
        first = true;
        if (c >= pool_chunks) return;
        if (c >= lend) {
          do {
            ++pl;
            items = ws.range[pl * kWarp + kWarp - 1].y;
            lbeg = lend;
            lend += (items + kWarp - 1) / kWarp;
          } while (c >= lend);
          lev = lev_f = (int)((pool_levels >> (4 * pl)) & 15u);
          const uint2 rg = ws.range[pl * kWarp + lane];
          uint32_t excl = __shfl_up_sync(kFullMask, rg.y, 1);
          if (lane == 0) excl = 0;
          const bool any = rg.y > excl;
          own_at = any ? excl : 0xffffffffu;
          const uint32_t has = __ballot_sync(kFullMask, any);
          if (any)
            owners[__popc(has & lanemask_lt())] =
                make_uint4((uint32_t)lane, excl,
                           cell_hash(G, lev_f, coord0(px, G.ox, G.inv_cell0, G.max0x) >> lev_f,
                                     coord0(py, G.oy, G.inv_cell0, G.max0y) >> lev_f,
                                     coord0(pz, G.oz, G.inv_cell0, G.max0z) >> lev_f).tag,
                           rg.x);
          __syncwarp();
        }
        const uint32_t i0 = (c - lbeg) * kWarp, i = i0 + lane;
        const uint32_t inside = __reduce_or_sync(
            kFullMask, own_at > i0 && own_at - i0 < kWarp ? 1u << (own_at - i0) : 0u);
        const uint32_t begun = __ballot_sync(kFullMask, own_at <= i0);
        if (i < items) {
          const uint4 ow = owners[__popc(begun) - 1 + __popc(inside & le)];
          own = (int)ow.x;
          tag = ow.z;
          const uint32_t at = ow.w + i;                // modulo 2^32
          v = __ldg(a.gval + at);
          first = i == ow.y;
          if (!first && lane == 0) vprev = __ldg(a.gval + (at - 1u));
        }
        __syncwarp();                                  // (before the next level's owners)
      };
      int cur = -1, cur_lev = -1;  // owner of this lane's item slot in the previous chunk
      float pc[C + 1];
#pragma unroll
      for (int c = 0; c <= C; ++c) pc[c] = 0.0f;
      float qx = 0.0f, qy = 0.0f, qz = 0.0f;
      int own_n, lev_n;
      uint32_t tag_n, v_n, vp_n;
      bool first_n;
      fetch(part, own_n, lev_n, tag_n, v_n, vp_n, first_n);
      for (uint32_t b = part; b < pool_chunks; b += of) {
        const int own = own_n, lev = lev_n;
        const uint32_t v = v_n;
        const uint32_t left = __shfl_up_sync(kFullMask, v, 1);
        const bool again = !first_n && v == (lane == 0 ? vp_n : left);
        const bool take = own < kWarp && (v & ~G.id_mask) == tag_n && !again;
        float rr[RS];
        if (take) load_rec_head<RS>(a.rec, v & G.id_mask, rr);
        fetch(b + of, own_n, lev_n, tag_n, v_n, vp_n, first_n);
        const bool chg = own != cur || lev != cur_lev;
        if (__any_sync(kFullMask, chg)) {
          pooled_flush<C>(ws.acc, lane, cur, chg && cur >= 0 && cur < kWarp, pc);
          const int src = own & (kWarp - 1);
          qx = __shfl_sync(kFullMask, px, src);
          qy = __shfl_sync(kFullMask, py, src);
          qz = __shfl_sync(kFullMask, pz, src);
          cur = own;
          cur_lev = lev;
        }
        // the rest of the record only where its bounding sphere holds the point
        bool near = take && rec_level(rr[3]) == (uint32_t)lev;
        if (near) {
          const float dx = qx - rr[0], dy = qy - rr[1], dz = qz - rr[2];
          near = fmaf(dx, dx, fmaf(dy, dy, dz * dz)) <= rr[3] * rr[3];
        }
        if (near) {
          load_rec_tail<RS>(a.rec, v & G.id_mask, rr);
          bool hit;
          const float w = pair_weight<KERN, COUNT>(rr, qx, qy, qz, a, hit, n_eval, n_inc);
          if (hit) {
#pragma unroll
            for (int c = 0; c < C; ++c) pc[c] = fmaf(w, rr[13 + c], pc[c]);
            pc[C] += w;
          }
        }
      }
      pooled_flush<C>(ws.acc, lane, cur, cur >= 0 && cur < kWarp, pc);
    }
  }

  if (!COUNT) {
    // the walked and the pooled sums of this lane's hit point
    __syncwarp();
#pragma unroll
    for (int c = 0; c < C; ++c) W[c] += ws.acc[c][lane];
    V += ws.acc[C][lane];
    if (TEAM > 1) {
      // the team's sums, added in warp order by warp 0
#pragma unroll
      for (int c = 0; c < C; ++c) ws.acc[c][lane] = W[c];
      ws.acc[C][lane] = V;
      __syncthreads();
      if (wib > 0) continue;      // (a team's unit has one part)
      for (int w = 1; w < TEAM; ++w) {
        const WarpShared o = warp_shared<C>(s_mem, w, G.levels, G.coop);
#pragma unroll
        for (int c = 0; c < C; ++c) W[c] += o.acc[c][lane];
        V += o.acc[C][lane];
      }
    }
    if (split) {
      // this part's sums; fwd_split_combine_kernel adds the parts in order
      float* xs = a.xsum + (size_t)(slot + pt) * (C + 1) * kWarp;
#pragma unroll
      for (int c = 0; c < C; ++c) xs[c * kWarp + lane] = W[c];
      xs[C * kWarp + lane] = V;
    } else {
#pragma unroll
      for (int c = 0; c < C; ++c) L[c] += W[c];
      Z += V;
    }
  }
  }  // parts

  if (!COUNT && !split && active && (TEAM == 1 || wib == 0)) {
    float scale = 1.0f;
    if (a.mode == GPF_NORMALIZED) scale = 1.0f / fmaxf(Z, a.eps);
    else if (a.mode == GPF_DISK_KDE) scale = a.kde_scale;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const float rho = a.albedo ? a.albedo[(int64_t)c * a.m + q] : 1.0f;
      a.out[(int64_t)c * a.m + q] = rho * (L[c] * scale);
    }
    if (a.z) a.z[q] = Z;
  }
  }  // tile loop

  if (COUNT) {
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      n_eval += __shfl_xor_sync(kFullMask, n_eval, o);
      n_inc += __shfl_xor_sync(kFullMask, n_inc, o);
    }
    if (lane == 0) {
      atomicAdd(&a.counts[0], (unsigned long long)n_eval);
      atomicAdd(&a.counts[1], (unsigned long long)n_inc);
    }
  }
}

// The split tiles' outputs: one warp per tile that several units took, adding
// its parts in part order, then the epilogue of fwd_kernel. ordered: the units
// wrote the tile's own parts (else a part each).
template <int C>
__global__ void fwd_split_combine_kernel(FwdArgs a, bool ordered, bool deferred) {
  const int lane = threadIdx.x & 31;
  const int64_t u = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (index_unusable(a.header)) return;
  const int64_t n_x = a.header->n_xunits;
  uint32_t tile, slot, parts;
  if (u < n_x) {
    const uint4 xu = a.xunit[u];
    if ((xu.y & 0xffu) != 0u) return;
    tile = xu.x;
    slot = xu.z;
    parts = ordered ? xu.y >> 16 : (xu.y >> 8) & 0xffu;
  } else {
    if (!deferred || !heavy_fits(a.header) || u - n_x >= (int64_t)a.header->n_heavy) return;
    tile = a.xheavy[u - n_x];
    slot = a.header->n_xslots + kHeavyParts * (uint32_t)(u - n_x);
    parts = kHeavyParts;
  }
  const int64_t k = (int64_t)tile * kWarp + lane;
  float L[C], Z = 0.0f;
#pragma unroll
  for (int c = 0; c < C; ++c) L[c] = 0.0f;
#pragma unroll 4
  for (uint32_t p = 0; p < parts; ++p) {
    const float* xs = a.xsum + (size_t)(slot + p) * (C + 1) * kWarp;
#pragma unroll
    for (int c = 0; c < C; ++c) L[c] += xs[c * kWarp + lane];
    Z += xs[C * kWarp + lane];
  }
  if (k >= a.m) return;
  const uint32_t q = a.qval[k];
  const bool active = k < (int64_t)a.header->n_active;
  float scale = 1.0f;
  if (a.mode == GPF_NORMALIZED) scale = 1.0f / fmaxf(Z, a.eps);
  else if (a.mode == GPF_DISK_KDE) scale = a.kde_scale;
#pragma unroll
  for (int c = 0; c < C; ++c) {
    const float rho = a.albedo ? a.albedo[(int64_t)c * a.m + q] : 1.0f;
    a.out[(int64_t)c * a.m + q] = active ? rho * (L[c] * scale) : 0.0f;
  }
  if (a.z) a.z[q] = active ? Z : 0.0f;
}

// Two estimates for every tile of 32 hit points, from a sample of eight of its
// points (every fourth: neighbouring points of the cell order see similar
// lists), over every used level: where the sample falls in at most Grid::coop
// cells, from the distinct cells' lists, walked by the whole warp; else from the
// points' own lists, times four for the points not sampled.
//  * The parts of its sums (parts, and by group of tiles in xpart): a walked
//    entry counts 8 and a pooled one 1, and a tile of more than split_items has
//    one part per split_items. They fix the order of the sums, so this count is
//    not an estimate to be improved.
//  * The work of a warp (cost, and the sum over all tiles): 32 entries of either
//    kind cost it about the same (a least-squares fit over the units of a
//    1M-Gaussian view: 1.5 us per 32 walked, 1.6 us per 32 pooled entries, and
//    17 us a unit).
// Four tiles per warp, eight lanes each.
__global__ void tile_cost_kernel(Grid grid, const DeviceHeader* header,
                                 const float4* __restrict__ qpos, int64_t m,
                                 const uint2* __restrict__ brange,
                                 const uint32_t* __restrict__ listed, uint32_t split_items,
                                 uint32_t* __restrict__ tparts, uint32_t* __restrict__ xpart,
                                 uint32_t* __restrict__ tcost, unsigned long long* total) {
  const int lane = threadIdx.x & 31;
  const int64_t gt = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  const int64_t tile = gt >> 3;
  const int64_t n_tiles = (m + kWarp - 1) / kWarp;
  const int64_t n_act = header->n_active;
  const int64_t k = tile * kWarp + (lane & 7) * 4;
  const bool active = tile < n_tiles && k < n_act && !index_unusable(header);
  const uint32_t group = 0xffu << (lane & ~7);      // the 8 lanes of this tile
  uint32_t c0x = 0, c0y = 0, c0z = 0;
  uint2 rg[kMaxLevels];
  const uint32_t lmask = header->level_mask;
  if (active) {
    const float4 p = __ldg(qpos + k);
    c0x = coord0(p.x, grid.ox, grid.inv_cell0, grid.max0x);
    c0y = coord0(p.y, grid.oy, grid.inv_cell0, grid.max0y);
    c0z = coord0(p.z, grid.oz, grid.inv_cell0, grid.max0z);
  }
#pragma unroll
  for (int lev = 0; lev < kMaxLevels; ++lev) {
    rg[lev] = make_uint2(0u, 0u);
    if (active && lev < grid.levels && ((lmask >> lev) & 1u))
      rg[lev] = bucket_list(listed, brange, bucket_of(grid, lev, c0x >> lev, c0y >> lev, c0z >> lev));
  }
  uint32_t walked = 0, pooled = 0;       // entries, of this sampled point
#pragma unroll
  for (int lev = 0; lev < kMaxLevels; ++lev) {
    if (lev >= grid.levels || !((lmask >> lev) & 1u)) continue;
    const unsigned long long packed =
        active ? ((unsigned long long)(c0x >> lev) | ((unsigned long long)(c0y >> lev) << 20) |
                  ((unsigned long long)(c0z >> lev) << 40))
               : ~0ull;
    const uint32_t peers = __match_any_sync(kFullMask, packed) & group;
    const bool leader = active && (peers & lanemask_lt()) == 0;
    const int nu = __popc(__ballot_sync(kFullMask, leader) & group);
    const uint32_t len = rg[lev].y - rg[lev].x;
    // (eight samples see at most 8 cells: all 8 distinct reads as more than 8)
    if (nu > min(grid.coop, 7)) pooled += len;
    else if (leader) walked += len;
  }
  // the eight lanes of a tile are consecutive: sum them
#pragma unroll
  for (int o = 1; o < 8; o <<= 1) {
    walked += __shfl_xor_sync(kFullMask, walked, o);
    pooled += __shfl_xor_sync(kFullMask, pooled, o);
  }
  const uint32_t items = 8u * walked + 4u * pooled;
  uint32_t cost = kCostPerEntry * (walked + 4u * pooled);
  if (tile < n_tiles && tile * kWarp < n_act) cost += kCostPerTile;
  if ((lane & 7) == 0 && tile < n_tiles) {
    const uint32_t parts = items <= split_items
                               ? 1u
                               : min((items + split_items - 1) / split_items,
                                     (uint32_t)GPF_MAX_TILE_PARTS);
    tparts[tile] = parts;
    tcost[tile] = cost;
    if (parts > 1) atomicAdd(&xpart[tile / kTileGroup], parts);
  }
  __shared__ uint32_t s_sum;
  if (threadIdx.x == 0) s_sum = 0;
  __syncthreads();
  const uint32_t sum = __reduce_add_sync(kFullMask, (lane & 7) == 0 ? min(cost, 1u << 26) : 0u);
  if (lane == 0 && sum) atomicAdd(&s_sum, sum);
  __syncthreads();
  if (threadIdx.x == 0 && s_sum) atomicAdd(total, (unsigned long long)s_sum);
}

// The parts' slots and the units. Each part of a split tile has a slot, after
// those of the split tiles before it (a block adds up the groups before its
// own: there is one word per 256 tiles, and most of them are zero); a tile
// whose slots would not all fit under GPF_MAX_SPLIT_UNITS has one part. A tile
// is given to several units, some of its parts each, when its work exceeds 1 /
// kSplitShare of all tiles' (a quarter of what a resident warp has to do
// anyway): a unit of its own for every part repeats the tile's look-ups, 17 us
// each (22 K tiles of a 1M field were 35 K units). Which place in the list a
// tile's units get depends on the order of the blocks; its sums do not.
constexpr uint32_t kSplitShare = 152 * 20 * 4;
__global__ void __launch_bounds__(kTileGroup)
tile_parts_kernel(int64_t n_tiles, uint32_t split_items, uint32_t* __restrict__ tparts,
                  const uint32_t* __restrict__ xpart, const uint32_t* __restrict__ tcost,
                  const unsigned long long* total, uint4* __restrict__ xunit,
                  uint32_t* n_units, uint32_t* n_slots) {
  __shared__ uint32_t s_before[kTileGroup / kWarp], s_parts[kTileGroup / kWarp],
      s_units[kTileGroup / kWarp], s_first;
  const bool last = blockIdx.x == gridDim.x - 1;
  if (xpart[blockIdx.x] == 0u && !last) return;      // one part each, as written
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t t = (int64_t)blockIdx.x * kTileGroup + threadIdx.x;
  uint32_t before = 0;
  for (uint32_t i = threadIdx.x; i < blockIdx.x; i += kTileGroup) before += xpart[i];
  before = __reduce_add_sync(kFullMask, before);
  uint32_t parts = t < n_tiles ? tparts[t] : 1u;
  auto scan = [&](uint32_t v) {                      // inclusive, over the warp
#pragma unroll
    for (int o = 1; o < kWarp; o <<= 1) {
      const uint32_t u = __shfl_up_sync(kFullMask, v, o);
      if (lane >= o) v += u;
    }
    return v;
  };
  const uint32_t mine = parts > 1 ? parts : 0u, incl = scan(mine);
  if (lane == 0) s_before[warp] = before;
  if (lane == kWarp - 1) s_parts[warp] = incl;
  __syncthreads();
  uint32_t slot = incl - mine, slots = 0;
  for (int w = 0; w < kTileGroup / kWarp; ++w) {
    slot += s_before[w] + (w < warp ? s_parts[w] : 0u);
    slots += s_before[w] + s_parts[w];
  }
  if (last && threadIdx.x == 0) *n_slots = min(slots, (uint32_t)GPF_MAX_SPLIT_UNITS);
  uint32_t units = 1;
  if (parts > 1) {
    if ((uint64_t)slot + parts > (uint64_t)GPF_MAX_SPLIT_UNITS) {
      parts = 1;
    } else {
      const unsigned long long share =
          max((unsigned long long)split_items, *total / kSplitShare + 1ull);
      units = (uint32_t)min((tcost[t] + share - 1) / share, (unsigned long long)parts);
    }
    tparts[t] = parts | (units > 1 ? kTileUnits : 0u);
  }
  const uint32_t my_units = units > 1 ? units : 0u, uincl = scan(my_units);
  if (lane == kWarp - 1) s_units[warp] = uincl;
  __syncthreads();
  if (threadIdx.x == 0) {
    uint32_t sum = 0;
    for (int w = 0; w < kTileGroup / kWarp; ++w) sum += s_units[w];
    s_first = sum ? atomicAdd(n_units, sum) : 0u;
  }
  __syncthreads();
  if (units <= 1) return;
  uint32_t o = s_first + uincl - units;              // no more units than slots: they fit
  for (int w = 0; w < warp; ++w) o += s_units[w];
  for (uint32_t i = 0; i < units; ++i)
    xunit[o + i] = make_uint4((uint32_t)t, i | (units << 8) | (parts << 16), slot, 0u);
}

// The hybrid forward's split units: a split tile's parts follow those of the split tiles before
// it (a block adds up the groups before its own: there is one word per 256
// tiles, and most of them are zero); a tile whose units would not all fit
// under GPF_MAX_SPLIT_UNITS runs unsplit, and its slots below the limit are
// marked empty.
__global__ void __launch_bounds__(kTileGroup)
tile_units_kernel(int64_t n_tiles, uint32_t* __restrict__ tparts,
                  const uint32_t* __restrict__ xpart, uint4* __restrict__ xunit,
                  uint32_t* n_units) {
  __shared__ uint32_t s_sum[kTileGroup / kWarp], s_warp[kTileGroup / kWarp];
  const bool last = blockIdx.x == gridDim.x - 1;
  if (xpart[blockIdx.x] == 0u && !last) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int64_t t = (int64_t)blockIdx.x * kTileGroup + threadIdx.x;
  uint32_t before = 0;
  for (uint32_t i = threadIdx.x; i < blockIdx.x; i += kTileGroup) before += xpart[i];
  before = __reduce_add_sync(kFullMask, before);
  const uint32_t parts = t < n_tiles ? tparts[t] : 1u;
  uint32_t incl = parts > 1 ? parts : 0u;
#pragma unroll
  for (int o = 1; o < kWarp; o <<= 1) {
    const uint32_t v = __shfl_up_sync(kFullMask, incl, o);
    if (lane >= o) incl += v;
  }
  if (lane == 0) s_sum[warp] = before;
  if (lane == kWarp - 1) s_warp[warp] = incl;
  __syncthreads();
  uint32_t o = incl - (parts > 1 ? parts : 0u), total = 0;
  for (int w = 0; w < kTileGroup / kWarp; ++w) {
    o += s_sum[w] + (w < warp ? s_warp[w] : 0u);
    total += s_sum[w] + s_warp[w];
  }
  if (last && threadIdx.x == 0) *n_units = min(total, (uint32_t)GPF_MAX_SPLIT_UNITS);
  if (parts <= 1) return;
  const bool fits = (uint64_t)o + parts <= (uint64_t)GPF_MAX_SPLIT_UNITS;
  if (!fits) tparts[t] = 1;
  for (uint32_t p = 0; p < parts && o + p < (uint32_t)GPF_MAX_SPLIT_UNITS; ++p)
    xunit[o + p] = make_uint4((uint32_t)t, p, parts, fits ? 1u : 0u);
}

}  // namespace

cudaError_t launch_split_units(int64_t n_tiles, uint32_t* tparts, const uint32_t* xpart,
                               uint4* xunit, uint32_t* n_units, cudaStream_t stream) {
  tile_units_kernel<<<(unsigned)tile_groups(n_tiles), kTileGroup, 0, stream>>>(
      n_tiles, tparts, xpart, xunit, n_units);
  note_launches(1);
  return cudaGetLastError();
}

cudaError_t launch_tile_split(const IndexDims& d, const IndexBuffers& b, const gpf_queries& q,
                              cudaStream_t stream) {
  const int64_t n_tiles = (q.m + kWarp - 1) / kWarp;
  tile_cost_kernel<<<(unsigned)((n_tiles * 8 + 255) / 256), 256, 0, stream>>>(
      d.grid, b.header, b.qpos, q.m, b.brange, b.listed, (uint32_t)d.split_items, b.tparts,
      b.xpart, b.tcost, &b.header->split_cost);
  tile_parts_kernel<<<(unsigned)tile_groups(n_tiles), kTileGroup, 0, stream>>>(
      n_tiles, (uint32_t)d.split_items, b.tparts, b.xpart, b.tcost, &b.header->split_cost,
      b.xunit, &b.header->n_xunits, &b.header->n_xslots);
  note_launches(2);
  return cudaGetLastError();
}

// Warps per tile: the chip holds 152 SMs x 20 warps of the forward at once, so
// fewer tiles than that leave it waiting for the longest list of one warp (the
// 512 tiles of a 4,096-Gaussian cube: 377 us with a warp each, 62 with 16; with
// both lines four times as high, 15,000 tiles take 422 us a pass instead of 419).
static int forward_team(int64_t n_tiles) {
  return n_tiles <= 152 * 8 ? 16 : n_tiles <= 152 * 32 ? 4 : 1;
}

cudaError_t launch_forward(const IndexDims& d, const IndexBuffers& b, const gpf_queries& q,
                           const gpf_query_params& p, int64_t n, float* out, float* z,
                           unsigned long long* counts, const KernelEvents& ev,
                           cudaStream_t stream) {
  if (counts) {
    cudaError_t e = cudaMemsetAsync(counts, 0, 2 * sizeof(unsigned long long), stream);
    if (e != cudaSuccess) return e;
  }
  if (q.m == 0) return cudaSuccess;
  FwdArgs a;
  a.grid = d.grid;
  a.qval = b.qval[b.qsorted];
  a.qpos = b.qpos;
  a.header = b.header;
  a.albedo = q.albedo;
  a.m = q.m;
  a.rec = b.rec;
  a.vet = b.vet;
  a.brange = b.brange;
  a.listed = b.listed;
  a.gval = b.gval[b.gsorted];
  a.n = n;
  a.mode = p.mode;
  const bool psi = isfinite(p.r_max);
  a.r = psi ? p.r_max : 0.0f;
  a.r2 = psi ? p.r_max * p.r_max : 0.0f;
  a.inv_rr = psi ? 1.0f / fmaxf(p.r_max, 1e-6f) : 0.0f;
  a.eps = p.eps;
  a.kde_scale = psi ? (float)(1.0 / (M_PI * (double)p.r_max * (double)p.r_max)) : 0.0f;
  a.cut = d.cutoff;
  a.cut2 = isinf(d.cutoff) ? INFINITY : d.cutoff * d.cutoff;
  a.tscale = (float)((double)a.inv_rr * std::sqrt(3.0 * M_LOG2E));
  a.out = out;
  a.z = z;
  a.counts = counts;
  a.late = 0;
  const bool split = d.split_items > 0 && !d.brute && n > 0;
  a.tparts = split ? b.tparts : nullptr;
  a.xunit = split ? b.xunit : nullptr;
  a.xheavy = split ? b.xheavy : nullptr;
  a.xsum = split ? b.xsum : nullptr;
  {
    const cudaError_t e =
        cudaMemsetAsync(&b.header->next_heavy, 0, 3 * sizeof(unsigned long long), stream);
    if (e != cudaSuccess) return e;
  }
  const int64_t n_tiles = (q.m + kWarp - 1) / kWarp;
  const int64_t units = n_tiles + (split ? GPF_MAX_SPLIT_UNITS : 0);
  const int team = forward_team(n_tiles);
  const int64_t want = team > 1 ? units : (units + kFwdWarps - 1) / kFwdWarps;
#define GPF_FWD_LAUNCH(CC, BR, PS, CN, TM)                                                   \
  do {                                                                                       \
    constexpr int warps = TM > 4 ? TM : kFwdWarps;                                           \
    const int smem =                                                                         \
        (int)sizeof(float) * warps * warp_shared_words(CC, d.grid.levels, d.grid.coop);      \
    const auto kernel = fwd_kernel<CC, BR, PS, CN, TM>;                                      \
    /* the limit belongs to the kernel, which other indexes launch from other threads: */    \
    /* always the same value, the most any index needs */                                    \
    constexpr int most =                                                                     \
        (int)sizeof(float) * warps * warp_shared_words(CC, GPF_MAX_LEVELS, GPF_MAX_COOP_CELLS); \
    static_assert(most <= 227 * 1024, "a block's shared memory");                            \
    if (most > 48 * 1024) {                                                                  \
      const cudaError_t e =                                                                  \
          cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, most);   \
      if (e != cudaSuccess) return e;                                                        \
    }                                                                                        \
    const unsigned blocks = (unsigned)persistent_blocks(                                     \
        reinterpret_cast<const void*>(kernel), warps * kWarp, want, smem);                   \
    kernel<<<blocks, warps * kWarp, smem, stream>>>(a);                                      \
    if (split && !CN && PS == kKernDisk) {                                                   \
      FwdArgs late = a;                                                                      \
      late.late = 1;                                                                         \
      kernel<<<blocks, warps * kWarp, smem, stream>>>(late);                                 \
      note_launches(1);                                                                      \
    }                                                                                        \
  } while (0)
#define GPF_FWD_TEAMS(CC, PS)                                          \
  do {                                                                 \
    if (team == 16) GPF_FWD_LAUNCH(CC, false, PS, false, 16);          \
    else if (team == 4) GPF_FWD_LAUNCH(CC, false, PS, false, 4);       \
    else GPF_FWD_LAUNCH(CC, false, PS, false, 1);                      \
  } while (0)
#define GPF_FWD_CASE(CC)                                                              \
  case CC:                                                                            \
    if (d.brute) {                                                                    \
      if (counts) GPF_FWD_LAUNCH(CC, true, kKernGauss, true, 1);                      \
      else if (kern == kKernDisk) GPF_FWD_LAUNCH(CC, true, kKernDisk, false, 1);      \
      else if (kern == kKernFalloff) GPF_FWD_LAUNCH(CC, true, kKernFalloff, false, 1); \
      else GPF_FWD_LAUNCH(CC, true, kKernGauss, false, 1);                            \
    } else {                                                                          \
      if (counts) GPF_FWD_LAUNCH(CC, false, kKernGauss, true, 1);                     \
      else if (kern == kKernDisk) GPF_FWD_TEAMS(CC, kKernDisk);                       \
      else if (kern == kKernFalloff) GPF_FWD_TEAMS(CC, kKernFalloff);                 \
      else GPF_FWD_TEAMS(CC, kKernGauss);                                             \
    }                                                                                 \
    note_launches(1);                                                                 \
    if (split && !counts) {                                                           \
      fwd_split_combine_kernel<CC><<<GPF_MAX_SPLIT_UNITS / 4, 128, 0, stream>>>(      \
          a, team == 1 && kern != kKernDisk, kern == kKernDisk);                      \
      note_launches(1);                                                               \
    }                                                                                 \
    break;
  const int kern = p.mode == GPF_DISK_KDE ? kKernDisk : psi ? kKernFalloff : kKernGauss;
  if (ev.start) {
    const cudaError_t e = cudaEventRecord(ev.start, stream);
    if (e != cudaSuccess) return e;
  }
  switch (d.channels) {
    GPF_FWD_CASE(1)
    GPF_FWD_CASE(2)
    GPF_FWD_CASE(3)
    GPF_FWD_CASE(4)
    GPF_FWD_CASE(5)
    GPF_FWD_CASE(6)
    GPF_FWD_CASE(7)
    GPF_FWD_CASE(8)
    default:
      return cudaErrorInvalidValue;
  }
#undef GPF_FWD_CASE
#undef GPF_FWD_TEAMS
#undef GPF_FWD_LAUNCH
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return ev.stop ? cudaEventRecord(ev.stop, stream) : cudaSuccess;
}

}  // namespace gpf
