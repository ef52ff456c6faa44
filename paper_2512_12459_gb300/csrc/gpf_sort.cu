// Device-wide exclusive scan of uint32 values and a stable LSD radix sort of
// (uint32 key, uint32 value) pairs, 8 bits per pass.
//
// Sort (single pass per digit, decoupled look-back; Merrill and Garland,
// "Single-pass Parallel Prefix Scan with Decoupled Look-back", 2016, and
// Adinets and Merrill, "Onesweep", 2022):
//   0. one kernel counts the digits of every pass over all keys (the global
//      digit counts do not depend on the order the earlier passes leave);
//   1. per pass, one kernel for up to three sorts side by side (a sort that
//      has no such pass takes no blocks): a block claims the next tile of its
//      sort, 3072 keys (small sorts 1024), from an atomic counter, so every
//      earlier tile is held by a block that is already running; keys and
//      values are read into registers, and each warp ranks its own, 32 at a
//      time (groups of equal digits from bit ballots, per-warp digit counters
//      in shared memory);
//      the block publishes its digit counts, orders its keys by digit in
//      shared memory, adds up the counts the earlier tiles published for each
//      digit, walking back until a tile whose inclusive prefix is known,
//      publishes its own inclusive prefix and writes its keys out in digit
//      order (runs of equal digits land on consecutive addresses).
//   Every wait in the walk is bounded: after kSpinLimit polls the block sets
//   the caller's stall flag, stops waiting and writes only in-bounds
//   addresses; the sorted output is then invalid and the flag says so.
//   Counts are below kMaxSortN = 2^30 (30-bit status values).
// The element count may live on the device (it is produced by an earlier
// kernel); grids are sized for the capacity and blocks past the count return
// early, so a whole build can be captured in a CUDA graph.
#include <cuda_runtime.h>
#include <stdint.h>

#include <algorithm>

#include "gpf_internal.h"

namespace gpf {

namespace {

constexpr int kScanThreads = 256;
constexpr int kScanPerThread = 8;
constexpr int kScanTile = kScanThreads * kScanPerThread;  // 2048

constexpr int kSortThreads = 256;
constexpr int kSortWarps = kSortThreads / kWarp;
constexpr int kSortPerThread = 12;
constexpr int kSortTile = kSortThreads * kSortPerThread;  // 3072
constexpr int kSortSmallPer = 4;
constexpr int kSortSmall = kSortThreads * kSortSmallPer;  // 1024
// Sorts of at most this many elements take tiles of kSortSmall keys: up to here
// the large ones are fewer than fit on the chip at once (512 K keys: 171 of 608).
// The line at 2^17 left a pass over a 4,096-Gaussian cube at 145 us instead of
// 135 and one over 100K Gaussians at 419 instead of 416; without small tiles a
// small training step took 284 instead of 266.
constexpr int64_t kSmallMax = int64_t(1) << 19;
constexpr int kLookBack = 8;     // status words read per step of the look-back
constexpr int kBins = 256;

// Exclusive scan across a block of kScanThreads threads; returns the prefix
// of this thread and writes the block total to *total.
__device__ __forceinline__ uint32_t block_exclusive_scan(uint32_t v, uint32_t* total) {
  __shared__ uint32_t warp_sums[kScanThreads / kWarp];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  uint32_t incl = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    uint32_t t = __shfl_up_sync(kFullMask, incl, o);
    if (lane >= o) incl += t;
  }
  if (lane == 31) warp_sums[warp] = incl;
  __syncthreads();
  if (warp == 0) {
    uint32_t s = lane < kScanThreads / kWarp ? warp_sums[lane] : 0u;
    uint32_t si = s;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      uint32_t t = __shfl_up_sync(kFullMask, si, o);
      if (lane >= o) si += t;
    }
    if (lane < kScanThreads / kWarp) warp_sums[lane] = si - s;
    if (lane == kScanThreads / kWarp - 1) *total = si;
  }
  __syncthreads();
  uint32_t r = warp_sums[warp] + incl - v;
  __syncthreads();
  return r;
}

__global__ void scan_reduce_kernel(const uint32_t* __restrict__ in, int64_t n,
                                   uint32_t* __restrict__ partial) {
  const int64_t base = (int64_t)blockIdx.x * kScanTile;
  uint32_t s = 0;
#pragma unroll
  for (int r = 0; r < kScanPerThread; ++r) {
    int64_t i = base + (int64_t)r * kScanThreads + threadIdx.x;
    if (i < n) s += in[i];
  }
  __shared__ uint32_t total;
  block_exclusive_scan(s, &total);
  if (threadIdx.x == 0) partial[blockIdx.x] = total;
}

// One block scans all partials (exclusive, in place) and stores the total.
__global__ void scan_partials_kernel(uint32_t* __restrict__ partial, int64_t nb,
                                     uint32_t* __restrict__ total_out) {
  __shared__ uint32_t total;
  uint32_t carry = 0;
  for (int64_t base = 0; base < nb; base += kScanThreads) {
    int64_t i = base + threadIdx.x;
    uint32_t v = i < nb ? partial[i] : 0u;
    uint32_t ex = block_exclusive_scan(v, &total);
    if (i < nb) partial[i] = carry + ex;
    carry += total;
    __syncthreads();
  }
  if (threadIdx.x == 0 && total_out) *total_out = carry;
}

// in and out may be the same array (each thread reads its elements before
// writing them).
__global__ void scan_down_kernel(const uint32_t* in, int64_t n,
                                 const uint32_t* __restrict__ partial, uint32_t* out) {
  const int64_t base = (int64_t)blockIdx.x * kScanTile + (int64_t)threadIdx.x * kScanPerThread;
  uint32_t v[kScanPerThread];
  uint32_t s = 0;
#pragma unroll
  for (int r = 0; r < kScanPerThread; ++r) {
    int64_t i = base + r;
    v[r] = i < n ? in[i] : 0u;
    s += v[r];
  }
  __shared__ uint32_t total;
  uint32_t run = block_exclusive_scan(s, &total) + partial[blockIdx.x];
#pragma unroll
  for (int r = 0; r < kScanPerThread; ++r) {
    int64_t i = base + r;
    if (i < n) out[i] = run;
    run += v[r];
  }
}

__device__ __forceinline__ uint32_t load_count(const uint32_t* d_n, int64_t n_max) {
  if (d_n == nullptr) return (uint32_t)n_max;
  uint32_t n = *d_n;
  return (int64_t)n > n_max ? (uint32_t)n_max : n;
}

// ---- single-pass (decoupled look-back) sort

constexpr int kMaxPasses = kSortMaxPasses;     // 32-bit keys
static_assert(kSortBins == kBins, "8-bit digits");
constexpr uint32_t kFlagAgg = 1u << 30;        // the tile's own count is published
constexpr uint32_t kFlagPre = 2u << 30;        // the inclusive prefix is published
constexpr uint32_t kValMask = kFlagAgg - 1u;
constexpr uint32_t kSpinLimit = 1u << 22;      // polls of one status word before giving up

__device__ __forceinline__ uint32_t ld_status(const uint32_t* p) {
  uint32_t v;
  asm volatile("ld.relaxed.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
__device__ __forceinline__ void st_status(uint32_t* p, uint32_t v) {
  asm volatile("st.relaxed.gpu.global.u32 [%0], %1;" ::"l"(p), "r"(v) : "memory");
}

// Digit counts of every pass over all keys: ghist[pass * 256 + digit].
__global__ void onesweep_hist_kernel(const uint32_t* __restrict__ keys, const uint32_t* d_n,
                                     int64_t n_max, int passes, uint32_t* __restrict__ ghist) {
  __shared__ uint32_t cnt[kMaxPasses * kBins];
  for (int i = threadIdx.x; i < kMaxPasses * kBins; i += blockDim.x) cnt[i] = 0;
  __syncthreads();
  const uint32_t n = load_count(d_n, n_max);
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  // plain shared-memory atomics: cheaper here than grouping equal digits first
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < (int64_t)n; i += stride) {
    const uint32_t k = keys[i];
    for (int p = 0; p < passes; ++p) atomicAdd(&cnt[p * kBins + ((k >> (8 * p)) & (kBins - 1))], 1u);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < passes * kBins; i += blockDim.x)
    if (cnt[i]) atomicAdd(&ghist[i], cnt[i]);
}

// One pass of one sort: the job's blocks claim its tiles from its own counter.
struct PassJob {
  const uint32_t* keys_in;
  const uint32_t* vals_in;
  uint32_t* keys_out;
  uint32_t* vals_out;
  const uint32_t* d_n;      // element count on the device, or null (n_max)
  int64_t n_max;
  const uint32_t* ghist;    // [kBins] digit counts of this pass
  uint32_t* status;         // [tiles][kBins]
  uint32_t* counter;        // tiles claimed so far
  uint32_t blocks;          // blocks of the launch that work on this job
  int shift;
  int small;                // tiles of kSortSmall keys instead of kSortTile
};
struct PassArgs {
  PassJob job[kSortMaxJobs];
  uint32_t tile_base;
  uint32_t spin_limit;
  uint32_t* stalled;
};

struct PassShared {
  uint32_t keys[kSortTile];
  uint32_t vals[kSortTile];
  uint32_t wcnt[kSortWarps][kBins];   // digit counts of each warp, then its bases
  uint32_t tile_start[kBins];
  uint32_t out_base[kBins];
  uint32_t total;
  uint32_t tile;
};

template <int PER>
__device__ __forceinline__ void onesweep_tile(const PassJob& a, PassShared& s, uint32_t tile_base,
                                              uint32_t spin_limit, uint32_t* stalled) {
  constexpr int kTile = kSortThreads * PER;
  constexpr int kWarpKeys = PER * kWarp;   // each warp ranks its own keys
  const int t = threadIdx.x;        // kSortThreads == kBins: thread t owns digit t
  const int lane = t & 31, warp = t >> 5;
  if (t == 0) s.tile = tile_base + atomicAdd(a.counter, 1u);
#pragma unroll
  for (int w = 0; w < kSortWarps; ++w) s.wcnt[w][t] = 0;
  const uint32_t n = load_count(a.d_n, a.n_max);
  const uint32_t my_ghist = a.ghist[t];
  __syncthreads();
  const uint32_t tile = s.tile;
  const int64_t base = (int64_t)tile * kTile;
  if (base >= (int64_t)n) return;                    // the whole block
  const int tile_n = (int)min((int64_t)kTile, (int64_t)n - base);
  const int shift = a.shift;

  // 1. ranks inside the warp's keys (taken 32 at a time in order); the keys stay
  //    in registers, all loaded before the first is ranked
  uint32_t rd[PER], key[PER];
#pragma unroll
  for (int it = 0; it < PER; ++it) {
    const int li = warp * kWarpKeys + it * kWarp + lane;
    key[it] = li < tile_n ? __ldg(a.keys_in + base + li) : 0u;
  }
#pragma unroll
  for (int it = 0; it < PER; ++it) {
    const int li = warp * kWarpKeys + it * kWarp + lane;
    const bool ok = li < tile_n;
    const uint32_t d = (key[it] >> shift) & (kBins - 1);
    // the lanes with the same digit: nine ballots (validity, then each digit
    // bit), cheaper here than __match_any_sync
    uint32_t peers = __ballot_sync(kFullMask, ok);
    if (!ok) peers = ~peers;
#pragma unroll
    for (int b = 0; b < 8; ++b) {
      const uint32_t m = __ballot_sync(kFullMask, (d >> b) & 1u);
      peers &= ((d >> b) & 1u) ? m : ~m;
    }
    uint32_t r0 = 0;
    if (ok) r0 = s.wcnt[warp][d];
    __syncwarp();
    if (ok && (peers & lanemask_lt()) == 0) s.wcnt[warp][d] = r0 + (uint32_t)__popc(peers);
    __syncwarp();
    rd[it] = r0 + (uint32_t)__popc(peers & lanemask_lt());
  }
  __syncthreads();
  // 2. digit t: the warps' bases and the tile's count; publish the count
  //    (tile 0: its inclusive prefix). The values are fetched meanwhile.
  uint32_t val[PER];
#pragma unroll
  for (int it = 0; it < PER; ++it) {
    const int li = warp * kWarpKeys + it * kWarp + lane;
    val[it] = li < tile_n ? __ldg(a.vals_in + base + li) : 0u;
  }
  uint32_t c = 0;
#pragma unroll
  for (int w = 0; w < kSortWarps; ++w) {
    const uint32_t x = s.wcnt[w][t];
    s.wcnt[w][t] = c;
    c += x;
  }
  st_status(a.status + (int64_t)tile * kBins + t, (tile == 0 ? kFlagPre : kFlagAgg) | c);
  s.tile_start[t] = block_exclusive_scan(c, &s.total);
  const uint32_t digit_start = block_exclusive_scan(my_ghist, &s.total);
  // 3. keys in digit order in shared memory
#pragma unroll
  for (int it = 0; it < PER; ++it) {
    const int li = warp * kWarpKeys + it * kWarp + lane;
    if (li < tile_n) {
      const uint32_t d = (key[it] >> shift) & (kBins - 1);
      const uint32_t pos = s.tile_start[d] + s.wcnt[warp][d] + rd[it];
      s.keys[pos] = key[it];
      s.vals[pos] = val[it];
    }
  }
  // 4. digit t in the earlier tiles: walk back to the nearest inclusive
  //    prefix, kLookBack tiles a step (their status words are read together:
  //    one after the other, the chain of L2 latencies was most of a pass)
  uint32_t excl = 0;
  if (tile > 0) {
    int64_t j = (int64_t)tile - 1;
    uint32_t spins = 0;
    bool found = false;
    while (j >= 0 && !found) {
      uint32_t sv[kLookBack];
#pragma unroll
      for (int i = 0; i < kLookBack; ++i)
        sv[i] = j - i >= 0 ? ld_status(a.status + (j - i) * kBins + t) : kFlagPre;
      // not there yet: poll this one word (eight at a time from every waiting
      // block kept the tiles that are being ranked from the L2)
      while ((sv[0] & ~kValMask) == 0u && ++spins < spin_limit) {
        __nanosleep(64);
        sv[0] = ld_status(a.status + j * kBins + t);
      }
      if ((sv[0] & ~kValMask) == 0u) {
        atomicExch(stalled, 1u);
        break;
      }
      int used = 0;
#pragma unroll
      for (int i = 0; i < kLookBack; ++i) {
        const uint32_t flag = sv[i] & ~kValMask;
        if (!found && used == i && flag != 0u) {
          excl += sv[i] & kValMask;
          used = i + 1;
          found = flag == kFlagPre;
        }
      }
      j -= used;
    }
    st_status(a.status + (int64_t)tile * kBins + t, kFlagPre | ((excl + c) & kValMask));
  }
  s.out_base[t] = digit_start + excl - s.tile_start[t];
  __syncthreads();
  // 5. out in digit order: runs of one digit go to consecutive addresses
  for (int p = t; p < tile_n; p += kSortThreads) {
    const uint32_t k = s.keys[p];
    const uint32_t dst = s.out_base[(k >> shift) & (kBins - 1)] + (uint32_t)p;
    if (dst < n) {
      a.keys_out[dst] = k;
      a.vals_out[dst] = s.vals[p];
    }
  }
}

// One pass of up to kSortMaxJobs independent sorts: the blocks are shared out
// over the jobs in order. A pass of one sort leaves most of the chip waiting
// on its look-back and its tail; the index build's three sorts in one launch
// fill it, and launch once per pass instead of three times.
__global__ void __launch_bounds__(kSortThreads, 4)
onesweep_pass_kernel(const __grid_constant__ PassArgs a) {
  __shared__ PassShared s;
  uint32_t blk = blockIdx.x;
  int j = 0;
#pragma unroll
  for (int k = 0; k < kSortMaxJobs - 1; ++k)
    if (j == k && blk >= a.job[k].blocks) {
      blk -= a.job[k].blocks;
      j = k + 1;
    }
  const PassJob& job = a.job[j];
  if (job.small) onesweep_tile<kSortSmallPer>(job, s, a.tile_base, a.spin_limit, a.stalled);
  else onesweep_tile<kSortPerThread>(job, s, a.tile_base, a.spin_limit, a.stalled);
}

}  // namespace

int64_t scan_partials_count(int64_t n) { return (n + kScanTile - 1) / kScanTile; }

size_t scan_workspace_bytes(int64_t n_max) {
  return align_up((size_t)(scan_partials_count(n_max) + 1) * sizeof(uint32_t));
}

cudaError_t exclusive_scan_u32(const uint32_t* in, uint32_t* out, int64_t n,
                               uint32_t* total_out, void* ws, cudaStream_t stream) {
  if (n <= 0) {
    if (total_out) return cudaMemsetAsync(total_out, 0, sizeof(uint32_t), stream);
    return cudaSuccess;
  }
  const int64_t nb = scan_partials_count(n);
  uint32_t* partial = static_cast<uint32_t*>(ws);
  scan_reduce_kernel<<<(unsigned)nb, kScanThreads, 0, stream>>>(in, n, partial);
  scan_partials_kernel<<<1, kScanThreads, 0, stream>>>(partial, nb, total_out);
  scan_down_kernel<<<(unsigned)nb, kScanThreads, 0, stream>>>(in, n, partial, out);
  note_launches(3);
  return cudaGetLastError();
}

bool radix_small(int64_t n_max) { return n_max <= kSmallMax; }

int64_t radix_tiles(int64_t n_max) {
  const int64_t tile = radix_small(n_max) ? kSortSmall : kSortTile;
  return (n_max + tile - 1) / tile;
}

namespace {
constexpr size_t kCountBytes = sizeof(uint32_t) * (kMaxPasses * kBins + kMaxPasses);
}

// The digit counts and tile counters of every pass, then the per-pass tile
// status words: all of it is zero before a sort.
size_t radix_sort_workspace_bytes(int64_t n_max, int bits) {
  // (for every count up to n_max: the most small tiles may exceed n_max's own)
  const int64_t tiles = std::max(radix_tiles(n_max), radix_tiles(std::min(n_max, kSmallMax)));
  return align_up(kCountBytes) +
         align_up((size_t)radix_sort_passes(bits) * tiles * kBins * sizeof(uint32_t));
}

int radix_sort_passes(int bits) { return bits <= 0 ? 0 : (bits + 7) / 8; }

// Two tiles of keys and values in and out, the digit counts and tile
// counter of one pass, two tiles of status words.
size_t sort_wait_probe_bytes() {
  return sizeof(uint32_t) * (8 * (size_t)kSortTile + kBins + 1 + 2 * kBins);
}

cudaError_t launch_sort_wait_probe(void* buf, uint32_t spin_limit, uint32_t* stalled,
                                   cudaStream_t stream) {
  cudaError_t e = cudaMemsetAsync(buf, 0, sort_wait_probe_bytes(), stream);
  if (e != cudaSuccess) return e;
  uint32_t* w = static_cast<uint32_t*>(buf);
  uint32_t* ghist = w + 8 * kSortTile;
  PassArgs a{};
  a.job[0] = PassJob{w, w + 2 * kSortTile, w + 4 * kSortTile, w + 6 * kSortTile, nullptr,
                     2 * kSortTile, ghist, ghist + kBins + 1, ghist + kBins, 1u, 0, 0};
  // one block, claiming tile 1 (tile_base 1): tile 0 is never processed, so
  // its status words stay 0 and the walk back from tile 1 waits on them
  a.tile_base = 1u;
  a.spin_limit = spin_limit;
  a.stalled = stalled;
  onesweep_pass_kernel<<<1, kSortThreads, 0, stream>>>(a);
  note_launches(1);
  return cudaGetLastError();
}

uint32_t* radix_sort_counts(void* ws) { return static_cast<uint32_t*>(ws); }

cudaError_t radix_sort_counted(const SortTask* tasks, int count, uint32_t* stalled,
                               cudaStream_t stream) {
  if (count > kSortMaxJobs) return cudaErrorInvalidValue;
  int passes = 0;
  for (int k = 0; k < count; ++k) {
    if (tasks[k].n_max >= kMaxSortN) return cudaErrorInvalidValue;
    if (tasks[k].n_max > 0) passes = std::max(passes, radix_sort_passes(tasks[k].bits));
  }
  for (int pass = 0; pass < passes; ++pass) {
    PassArgs a{};
    a.spin_limit = kSpinLimit;
    a.stalled = stalled;
    unsigned blocks = 0;
    for (int k = 0; k < count; ++k) {
      const SortTask& t = tasks[k];
      if (t.n_max <= 0 || pass >= radix_sort_passes(t.bits)) continue;
      const int64_t tiles = radix_tiles(t.n_max);
      uint32_t* counts = static_cast<uint32_t*>(t.ws);       // [kMaxPasses][kBins], counters
      uint32_t* status = reinterpret_cast<uint32_t*>(static_cast<char*>(t.ws) +
                                                     align_up(kCountBytes));
      const bool odd = pass & 1;
      a.job[k] = PassJob{odd ? t.k1 : t.k0, odd ? t.v1 : t.v0, odd ? t.k0 : t.k1,
                         odd ? t.v0 : t.v1, t.d_n, t.n_max, counts + pass * kBins,
                         status + (size_t)pass * tiles * kBins, counts + kMaxPasses * kBins + pass,
                         (uint32_t)tiles, pass * 8, radix_small(t.n_max) ? 1 : 0};
      blocks += (unsigned)tiles;
    }
    onesweep_pass_kernel<<<blocks, kSortThreads, 0, stream>>>(a);
    note_launches(1);
  }
  return cudaGetLastError();
}

cudaError_t radix_sort_pairs(const SortTask& t, uint32_t* stalled, cudaStream_t stream) {
  if (t.n_max <= 0) return cudaSuccess;
  if (t.n_max >= kMaxSortN) return cudaErrorInvalidValue;
  const int passes = radix_sort_passes(t.bits);
  if (passes == 0) return cudaSuccess;
  const cudaError_t e =
      cudaMemsetAsync(t.ws, 0, radix_sort_workspace_bytes(t.n_max, t.bits), stream);
  if (e != cudaSuccess) return e;
  const unsigned hblocks = (unsigned)std::min<int64_t>(radix_tiles(t.n_max), 1024);
  onesweep_hist_kernel<<<hblocks, kSortThreads, 0, stream>>>(t.k0, t.d_n, t.n_max, passes,
                                                             radix_sort_counts(t.ws));
  note_launches(1);
  return radix_sort_counted(&t, 1, stalled, stream);
}

}  // namespace gpf
