// Device helpers shared by the kernel translation units.
#pragma once

#include <cuda_runtime.h>

#include <atomic>

#include "tpc_internal.h"

namespace tpc {
namespace TPC_NS {
namespace {

constexpr int kBlock = 256;

__device__ __forceinline__ unsigned f2o(float f) {
  const unsigned u = __float_as_uint(f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}
__device__ __forceinline__ float o2f(unsigned u) {
  return __uint_as_float((u & 0x80000000u) ? (u & 0x7fffffffu) : ~u);
}
__device__ __forceinline__ int clampi(int v, int lo, int hi) { return v < lo ? lo : (v > hi ? hi : v); }

__device__ __forceinline__ int bin_of(float v, float v0, float inv, int n) {
  return clampi((int)floorf((v - v0) * inv), 0, n - 1);
}

// Visit sorted clusters of a row grid whose bins cover [ylo,yhi] x [zlo,zhi]
// (a superset of the clusters inside the box: bin index is monotone in the
// coordinate).
template <typename Fn>
__device__ __forceinline__ void for_window(const int* __restrict__ bin_first, const RowGrid& g,
                                           float ylo, float yhi, float zlo, float zhi, Fn&& fn) {
  if (g.ncl == 0 || !(ylo <= yhi) || !(zlo <= zhi)) return;
  const int iy0 = bin_of(ylo, g.y0, g.invDy, g.nY), iy1 = bin_of(yhi, g.y0, g.invDy, g.nY);
  const int iz0 = bin_of(zlo, g.z0, g.invDz, g.nZ), iz1 = bin_of(zhi, g.z0, g.invDz, g.nZ);
  for (int iz = iz0; iz <= iz1; ++iz) {
    const int b = g.bin0 + iz * g.nY;
    const int lo = bin_first[b + iy0], hi = bin_first[b + iy1 + 1];
    for (int k = lo; k < hi; ++k) fn(k);
  }
}

// The clusters of up to kStrips z strips of a search window as one run of
// candidates.  A window of a few cm covers one or two strips holding about one
// cluster each (bins of some 5 cm with half a cluster), so what a search waits
// for is its chain of dependent loads, and what it diverges over is the nesting
// of strips and clusters: the strips' ranges are requested together, and the
// lanes of a warp run one loop over their candidates, not one per strip.
constexpr int kStrips = 3;

struct StripRun {
  int l0, l1, l2;  // the strips' first clusters
  int n0, n1, n;   // candidates of the first, the first two, all strips
  __device__ __forceinline__ int at(int c) const {
    return c < n0 ? l0 + c : c < n1 ? l1 + (c - n0) : l2 + (c - n1);
  }
};

// Strips iz .. min(iz + kStrips - 1, iz1), y bins iy0 .. iy1.
__device__ __forceinline__ StripRun strip_run(const int* __restrict__ bin_first, const RowGrid& g,
                                              int iy0, int iy1, int iz, int iz1) {
  const int* b = bin_first + g.bin0 + iz * g.nY;
  int h1 = 0, h2 = 0;
  StripRun r;
  r.l1 = r.l2 = 0;
  r.l0 = b[iy0];
  const int h0 = b[iy1 + 1];
  if (iz + 1 <= iz1) {
    r.l1 = b[g.nY + iy0];
    h1 = b[g.nY + iy1 + 1];
  }
  if (iz + 2 <= iz1) {
    r.l2 = b[2 * g.nY + iy0];
    h2 = b[2 * g.nY + iy1 + 1];
  }
  r.n0 = h0 - r.l0;
  r.n1 = r.n0 + (h1 - r.l1);
  r.n = r.n1 + (h2 - r.l2);
  return r;
}

__device__ __forceinline__ int block_exscan(int v, int* sh_warp, int* total) {
  const int lane = threadIdx.x & 31, wid = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xffffffffu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) sh_warp[wid] = x;
  __syncthreads();
  if (wid == 0) {
    const int nw = blockDim.x >> 5;
    int w = lane < nw ? sh_warp[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xffffffffu, w, o);
      if (lane >= o) w += y;
    }
    if (lane < nw) sh_warp[lane] = w;
  }
  __syncthreads();
  const int base = wid ? sh_warp[wid - 1] : 0;
  if (total) *total = sh_warp[(blockDim.x >> 5) - 1];
  __syncthreads();
  return base + x - v;
}

// Exclusive scan of the block counts in one block; writes the total.
__global__ void k_scan_partials(int* part, int nparts, int* total) {
  __shared__ int sh[32];
  __shared__ int carry;
  if (threadIdx.x == 0) carry = 0;
  __syncthreads();
  for (int base = 0; base < nparts; base += blockDim.x) {
    const int i = base + threadIdx.x;
    const int v = i < nparts ? part[i] : 0;
    int tot;
    const int ex = block_exscan(v, sh, &tot);
    if (i < nparts) part[i] = carry + ex;
    __syncthreads();
    if (threadIdx.x == 0) carry += tot;
    __syncthreads();
  }
  if (threadIdx.x == 0) *total = carry;
}

// Items per warp of the kernels whose warps take up to 32 items, their headers
// loaded by the lanes side by side, one after the other: fewer where 32 would
// leave warps without work (the items of a warp are a serial chain).
__device__ __forceinline__ int warp_share(int n, int warps) {
  return max(1, min(32, (n + warps - 1) / warps));
}

// Device-side work queue: each call hands the calling lanes the next item
// indices of the queue (one atomic per warp), so uneven items (tracklets of
// 3..150 rows, sectors of 10x different occupancy) balance dynamically across
// a persistent grid.
__device__ __forceinline__ int queue_next(int* q) {
  const unsigned mask = __activemask();
  const int lane = threadIdx.x & 31;
  const int leader = __ffs(mask) - 1;
  int base = 0;
  if (lane == leader) base = atomicAdd(q, __popc(mask));
  base = __shfl_sync(mask, base, leader);
  return base + __popc(mask & ((1u << lane) - 1u));
}

// Next item of a lane: the first is the lane's own number in the grid, for the
// `stat` lanes of the blocks that start together; every other one comes from
// the queue, whose count starts there.  Blocks start one per SM before any SM
// gets its second, so the first items, the longest ones, are spread evenly over
// the SMs.  (All from the queue, the blocks that asked first took them: with the
// 17,000 tracks of an event, too few for every lane, some schedulers had four
// warps of filter steps and others none.)
__device__ __forceinline__ int next_item(int* q, bool& first, int stat) {
  if (first) {
    first = false;
    const int g = blockIdx.x * blockDim.x + threadIdx.x;
    if (g < stat) return g;
  }
  return stat + queue_next(q);
}

// Refill of the per-lane state machines (all lanes of the warp call it once per
// loop iteration): lanes without an item wait until kRefill of them do, or until
// no lane has one, and fetch together.  Loading an item costs as much as a step
// or two, and run for one or two lanes at a time it would cost that in every
// iteration.  (Two full frames, k_tl_chain / k_tl_refit / k_fit1: 0.82 / 1.07 /
// 1.34 ms at 1, 0.51 / 0.81 / 1.05 at 8, 0.58 / 0.96 / 0.99 at 24.)
constexpr int kRefill = 8;
__device__ __forceinline__ bool refill(bool busy, bool done, bool& all_done) {
  const unsigned b = __ballot_sync(0xffffffffu, busy);
  const unsigned w = __ballot_sync(0xffffffffu, !busy && !done);
  all_done = (b | w) == 0u;
  return !busy && !done && (b == 0u || __popc(w) >= kRefill);
}

// Order of kOrdChunk consecutive items by length, longest first: order[base +
// rank] = item for the chunk's items item(0..n-1), with len(i) < kOrdBuckets
// (the longest in bucket 0; -1: nothing to do, last).  The lanes of a warp then
// run items of one length side by side, start and end together, and still take
// them from one stretch of the list, which keeps their cluster accesses close.
// (By length over the whole list the lanes fill as well, but two full frames'
// k_tl_chain and k_fit1 took 0.73 and 1.64 ms instead of 0.51 and 1.05.)
constexpr int kOrdChunk = 4096;
template <typename Item, typename Len>
__device__ __forceinline__ void order_chunk(int n, Item&& item, Len&& len, int* order) {
  constexpr int kPer = kOrdChunk / kBlock;
  __shared__ int cnt[kOrdBuckets], sh[32];
  static_assert(kOrdBuckets <= kBlock && kOrdChunk % kBlock == 0, "chunk shape");
  if (threadIdx.x < kOrdBuckets) cnt[threadIdx.x] = 0;
  __syncthreads();
  int it[kPer], b[kPer], slot[kPer];
#pragma unroll
  for (int j = 0; j < kPer; ++j) {
    const int q = j * kBlock + threadIdx.x;
    b[j] = -1;
    if (q < n) {
      it[j] = item(q);
      b[j] = kOrdBuckets - 1 - min(kOrdBuckets - 1, len(it[j]) + 1);
    }
  }
#pragma unroll
  for (int j = 0; j < kPer; ++j)
    if (b[j] >= 0) slot[j] = atomicAdd(&cnt[b[j]], 1);
  __syncthreads();
  const int ex = block_exscan(threadIdx.x < kOrdBuckets ? cnt[threadIdx.x] : 0, sh, nullptr);
  if (threadIdx.x < kOrdBuckets) cnt[threadIdx.x] = ex;
  __syncthreads();
#pragma unroll
  for (int j = 0; j < kPer; ++j)
    if (b[j] >= 0) order[cnt[b[j]] + slot[j]] = it[j];
  __syncthreads();
}

// Scheduling order from per-item buckets: order[start of bucket b + slot] = i
// for the first min(*n, cap) items.  Every block scans the kOrdBuckets counts
// in shared memory.  The order only decides which item a thread takes next;
// no result depends on it (slots within a bucket follow atomic arrival).
__global__ void k_order_scatter(const int* __restrict__ bucket, const int* __restrict__ slot,
                                const int* __restrict__ cnt, const int* n, long cap,
                                const int* err, int* __restrict__ order) {
  __shared__ int base[kOrdBuckets];
  if (threadIdx.x == 0) {
    int acc = 0;
    for (int b = 0; b < kOrdBuckets; ++b) {
      base[b] = acc;
      acc += cnt[b];
    }
  }
  __syncthreads();
  if (*err) return;
  const int m = (int)min((long)*n, cap);
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < m; i += gridDim.x * blockDim.x)
    order[base[bucket[i]] + slot[i]] = i;
}

}  // namespace

inline unsigned blocks_for(long n, int b) { return (unsigned)((n + b - 1) / b); }

// Lanes of the blocks of kernel K (block size `block`, shared memory `smem`, a
// function of the block size) that start together in a grid of `grid` blocks.
template <auto K>
inline int resident_lanes(int block, size_t smem, unsigned grid, int sms) {
  static std::atomic<int> per_sm[kBlock / 32 + 1];  // by warps of the block; 0: not asked yet
  std::atomic<int>& c = per_sm[min(block, kBlock) / 32];
  int nb = c.load(std::memory_order_relaxed);
  if (nb == 0) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, K, block, smem) != cudaSuccess || nb < 1)
      nb = 1;
    c.store(nb, std::memory_order_relaxed);
  }
  return (int)min((long)grid, (long)nb * sms) * block;
}

// Persistent grid of a heavy kernel for launch slot `slot`.
inline unsigned persistent_grid(const LaunchCfg& lc, int slot, int sms) {
  return (unsigned)(sms * lc.per_sm[slot]);
}

}  // namespace TPC_NS
}  // namespace tpc
