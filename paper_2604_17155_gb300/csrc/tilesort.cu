// tilesort.cu -- depth order inside every screen tile (the "depth ordered list" of Eq. 2).
//
// After binning, each tile owns a contiguous slot range of 64-bit keys (float32 depth bits << 32 |
// Gaussian index); the keys are unique, so sorting them ascending gives depth order with ties in
// index order, and every list of a pass is sorted before the walks read it. A list is bucket sorted
// (bucket.cuh) in shared memory by a team sized to it: lists of up to kWarpSortCap keys by one warp
// each of a persistent kernel (k_sort_tiles, no CTA barrier), which queues the others; up to kMidCap
// keys by a CTA of four warps (k_sort_mid); longer ones, in runs of kSortCap keys that are merged,
// by a CTA of eight (k_sort_queued). A list in which many depths are equal, which the warp's or the CTA's sort
// refuses, is split by its whole keys in the queue's kernels, and one that still crowds takes the stable LSD radix
// sort of radix.cuh there.
//
// Latency of shared-memory atomics and loads bounds these kernels, so passes over the keys and warps
// in flight count: with three or four radix passes a list, the sort of 1.1e9 keys in 1.3 million lists
// (200 views of 1600 x 1060) took 16.5 ms, with one bucket pass 9.6 (its keys read and written once at
// the copy rate: 2.6); 5.4e7 keys in 250,000 lists 0.88 -> 0.51 ms. Teams: lists of 1025..2048 keys
// by two warps with 32 keys a thread (159 registers, 12 warps an SM) gave 10.5 ms.
#include <cuda_runtime.h>

#include <algorithm>

#include "bucket.cuh"
#include "icgs_internal.h"
#include "radix.cuh"

namespace icgs {

namespace {

constexpr int kSortThreads = radix::kThreads;  // CTA of the queued sort
constexpr int kWarpSortCap = 1024;             // longest list a warp sorts alone
constexpr int kWarpSortWarps = 4;              // warps per CTA of k_sort_tiles
constexpr int kWarpSortChunk = 4;              // most tiles a warp claims per work-counter increment
constexpr int kMidCap = 2 * kWarpSortCap;       // queued lists up to this length: k_sort_mid
constexpr int kMidThreads = 128;               // its CTA

constexpr int kWarpBins = 2048;                 // bins of a warp's bucket sort: two a key of its longest list

struct WarpSortSmem {
  unsigned long long keys[kWarpSortCap];
  bucket::Bins<1, kWarpBins> bins;
};

__device__ __forceinline__ void tile_range(const uint32_t* tile_off, int t, uint32_t capacity,
                                           uint32_t& b, uint32_t& e) {
  b = min(tile_off[t], capacity);
  e = min(tile_off[t + 1], capacity);
  if (e < b) e = b;
}

// Number of elements of A among the first d outputs of merging A and B (keys are unique).
__device__ __forceinline__ int merge_path(const unsigned long long* A, int na, const unsigned long long* B,
                                          int nb, int d);

// Every tile list of the pass, by warps that claim chunk tiles at a time from the work counter: lists of up
// to kWarpSortCap keys are bucket sorted in place by the claiming warp, longer and crowded ones queued. 16
// warps an SM, by shared memory (12 KB each) and registers (32 keys a lane): CTAs of three warps fit 18,
// but at 96 registers that spill (large scene 10.7 ms against 10.5).
__global__ void __launch_bounds__(32 * kWarpSortWarps, 4) k_sort_tiles(const uint32_t* __restrict__ tile_off,
                                                                    unsigned long long* __restrict__ entries,
                                                                    uint32_t capacity, int ntiles, int chunk,
                                                                    uint32_t* __restrict__ queue, DevStatus* status) {
  extern __shared__ __align__(16) unsigned long long s_dyn[];  // kWarpSortWarps x WarpSortSmem
  WarpSortSmem& m = reinterpret_cast<WarpSortSmem*>(s_dyn)[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  while (true) {
    uint32_t t0 = 0;
    if (lane == 0) t0 = atomicAdd(&status->sort_next, (uint32_t)chunk);
    t0 = __shfl_sync(0xFFFFFFFFu, t0, 0);
    if (t0 >= (uint32_t)ntiles) break;
    const int t1 = min(ntiles, (int)t0 + chunk);
    {  // start the chunk's keys towards L2 while the first list is sorted
      uint32_t cb, ce, cx;
      tile_range(tile_off, (int)t0, capacity, cb, cx);
      tile_range(tile_off, t1 - 1, capacity, cx, ce);
      const char* p0 = reinterpret_cast<const char*>(entries + cb);
      const size_t bytes = (size_t)(ce - cb) * sizeof(unsigned long long);
      for (size_t o = (size_t)lane * 128; o < bytes; o += 32 * 128)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(p0 + o));
    }
    for (int t = (int)t0; t < t1; ++t) {
      uint32_t b, e;
      tile_range(tile_off, t, capacity, b, e);
      const int n = (int)(e - b);
      if (n <= 1) continue;
      bool done = false;
      if (n <= kWarpSortCap) done = bucket::sort_list<1, kWarpSortCap / 32>(entries + b, n, m.keys, m.bins);
      if (!done) {  // queued: up to kMidCap keys from the front, longer lists from the back
        if (lane == 0) {
          if (n <= kMidCap) queue[atomicAdd(&status->big_tiles, 1u)] = (uint32_t)t;
          else queue[ntiles - 1 - (int)atomicAdd(&status->long_tiles, 1u)] = (uint32_t)t;
        }
      }
    }
  }
}

// Number of elements of A among the first d outputs of merging A and B (keys are unique).
__device__ __forceinline__ int merge_path(const unsigned long long* A, int na, const unsigned long long* B,
                                          int nb, int d) {
  int lo = max(0, d - nb), hi = min(d, na);
  while (lo < hi) {
    const int i = (lo + hi) >> 1;
    if (A[i] < B[d - 1 - i]) lo = i + 1;
    else hi = i;
  }
  return lo;
}

// Merges the sorted runs A[0, na) and B[0, nb) into out[0, na + nb) with the CTA's NT threads,
// each producing an equal share of the outputs (merge path).
template <int NT>
__device__ __forceinline__ void merge_runs(const unsigned long long* A, int na, const unsigned long long* B, int nb,
                                           unsigned long long* out, int t) {
  const int n = na + nb;
  const int per = (n + NT - 1) / NT;
  const int d0 = min(n, t * per), d1 = min(n, d0 + per);
  if (d0 >= d1) return;
  int ia = merge_path(A, na, B, nb, d0);
  int ib = d0 - ia;
  for (int d = d0; d < d1; ++d) {
    const bool takeA = ib >= nb || (ia < na && A[ia] < B[ib]);
    out[d] = takeA ? A[ia++] : B[ib++];
  }
}

// Sorts the queued lists of up to kMidCap keys (queue[0, big_tiles)), a grid-stride loop with a CTA per list:
// those of more than kWarpSortCap keys by a bucket sort of the CTA; the crowded ones, and the shorter lists
// that a warp's bucket sort refused, by splitting them. What remains by two warps: warp w sorts one half (at most
// kWarpSortCap keys) with the warp radix sort in its part of two shared pools, the halves are gathered into the first
// pool, and a merge-path merge (every thread an equal share of the outputs) writes the list back to its slot range.
__global__ void __launch_bounds__(kMidThreads, 6) k_sort_mid(const uint32_t* __restrict__ tile_off,
                                                             unsigned long long* __restrict__ entries, uint32_t capacity,
                                                             const uint32_t* __restrict__ queue,
                                                             const DevStatus* status) {
  extern __shared__ __align__(16) unsigned long long s_dyn[];  // pools P0, P1 of 2 x kWarpSortCap keys, scratch
  unsigned long long* P0 = s_dyn;
  unsigned long long* P1 = s_dyn + 2 * kWarpSortCap;
  __shared__ int s_len[2];
  using MidBins = bucket::Bins<kMidThreads / 32, 2 * kMidCap / (kMidThreads / 32)>;
  MidBins& bins = *reinterpret_cast<MidBins*>(P1);
  static_assert(sizeof(MidBins) <= 2 * kWarpSortCap * sizeof(unsigned long long), "bins in P1");
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  radix::WarpScratch& sc = reinterpret_cast<radix::WarpScratch*>(P1 + 2 * kWarpSortCap)[w & 1];
  if (w < 2)
    for (int i = lane; i < radix::kBins; i += 32) sc.match[i] = 0u;
  const uint32_t count = status->big_tiles;
  for (uint32_t q = blockIdx.x; q < count; q += gridDim.x) {
    uint32_t b, e;
    tile_range(tile_off, queue[q], capacity, b, e);
    const int n = (int)(e - b);
    if (n > kWarpSortCap && bucket::sort_list<kMidThreads / 32, kMidCap / kMidThreads>(entries + b, n, P0, bins)) continue;  // uniform
    if (bucket::split_list<kMidThreads / 32, kMidCap / kMidThreads>(entries + b, n, P0, bins)) continue;  // uniform
    if (w < 2) {
      __syncwarp();
      const int h = (n + 1) / 2;
      const int lo = min(n, w * h), len = min(h, n - lo);
      unsigned long long* a = P0 + w * kWarpSortCap;
      unsigned long long* bb = P1 + w * kWarpSortCap;
      if (len > 1) {
        const unsigned long long* run = radix::warp_sort_keys(entries + b + lo, len, a, bb, sc);
        if (run != a) {  // gather the half into the first pool
          for (int pos = lane; pos < len; pos += 32) a[pos] = run[pos];
          __syncwarp();
        }
      } else if (len == 1 && lane == 0) {
        a[0] = entries[b + lo];
      }
      if (lane == 0) s_len[w] = max(0, len);
    }
    __syncthreads();
    merge_runs<kMidThreads>(P0, s_len[0], P0 + kWarpSortCap, s_len[1], entries + b, threadIdx.x);
    __syncthreads();
  }
}

// Sorts the m (1 < m <= kSortCap) keys at g in place with the block radix sort sized to m.
__device__ __forceinline__ void block_sort_list(unsigned long long* g, int m, unsigned long long* a,
                                                unsigned long long* b, radix::BlockScratch& sc) {
  if (m <= 1024) radix::block_sort<4>(g, m, a, b, sc);
  else if (m <= 2048) radix::block_sort<8>(g, m, a, b, sc);
  else if (m <= 3072) radix::block_sort<12>(g, m, a, b, sc);
  else radix::block_sort<16>(g, m, a, b, sc);
}

// Sorts the queued lists of more than kMidCap keys (the last long_tiles entries of the queue) in
// place, a grid-stride loop with a CTA per list: in runs of up to kSortCap keys, each by a bucket sort or, when
// crowded, by splitting it or by the block radix sort; a longer list then by pairwise merge-path merges ping-ponging between its
// slot range and the same range of the scratch array. (A bucket sort of 2 kSortCap keys in both buffers at
// once spilled its 32 keys a thread and was slower, 1.06 ms a pass against 0.65.)
__global__ void __launch_bounds__(kSortThreads, 2) k_sort_queued(const uint32_t* __restrict__ tile_off,
                                                                 unsigned long long* __restrict__ entries,
                                                                 unsigned long long* __restrict__ scratch,
                                                                 uint32_t capacity, const uint32_t* __restrict__ queue,
                                                                 int ntiles, const DevStatus* status) {
  constexpr int CAP = kSortCap, kWarps = kSortThreads / 32;
  using QueueBins = bucket::Bins<kWarps, 2 * CAP / kWarps>;
  static_assert(sizeof(QueueBins) <= CAP * sizeof(unsigned long long), "bins in the second buffer");
  extern __shared__ __align__(16) unsigned long long s_dyn[];  // 2 x CAP keys
  __shared__ radix::BlockScratch sc;
  QueueBins& bins = *reinterpret_cast<QueueBins*>(s_dyn + CAP);
  for (int i = threadIdx.x; i < radix::kWarps * radix::kBins; i += kSortThreads) sc.match[i] = 0u;
  __syncthreads();
  const uint32_t count = status->long_tiles;
  for (uint32_t q = blockIdx.x; q < count; q += gridDim.x) {
    uint32_t b, e;
    tile_range(tile_off, queue[ntiles - 1 - (int)q], capacity, b, e);
    const int n = (int)(e - b);
    for (int r0 = 0; r0 < n; r0 += CAP) {  // sorted runs (the whole list when it fits)
      const int m = min(CAP, n - r0);
      if (m > 1 && !bucket::sort_list<kWarps, CAP / kSortThreads>(entries + b + r0, m, s_dyn, bins) &&
          !bucket::split_list<kWarps, CAP / kSortThreads>(entries + b + r0, m, s_dyn, bins))
        block_sort_list(entries + b + r0, m, s_dyn, s_dyn + CAP, sc);
    }
    if (n <= CAP) continue;  // uniform
    unsigned long long* src = entries + b;
    unsigned long long* dst = scratch + b;
    for (int width = CAP; width < n; width <<= 1) {
      for (int lo = 0; lo < n; lo += 2 * width) {
        const int na = min(width, n - lo);
        const int nb = max(0, min(width, n - lo - width));
        const unsigned long long* A = src + lo;
        const unsigned long long* Bp = src + lo + na;
        const int tot = na + nb;
        const int per = (tot + kSortThreads - 1) / kSortThreads;
        const int d0 = min(tot, (int)threadIdx.x * per), d1 = min(tot, d0 + per);
        if (d0 < d1) {
          int ia = merge_path(A, na, Bp, nb, d0);
          int ib = d0 - ia;
          for (int d = d0; d < d1; ++d) {
            const bool takeA = ib >= nb || (ia < na && A[ia] < Bp[ib]);
            dst[lo + d] = takeA ? A[ia++] : Bp[ib++];
          }
        }
      }
      __syncthreads();
      unsigned long long* tmp = src;
      src = dst;
      dst = tmp;
    }
    if (src != entries + b)
      for (int k = threadIdx.x; k < n; k += kSortThreads) entries[b + k] = src[k];
    __syncthreads();
  }
}

}  // namespace

int sm_count() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms > 0 ? sms : 1;
}

// Orders every tile list of the pass: the warp-per-list kernel, then the queued lists. The queue
// counters of the status block are zero (the scan of the pass's counts empties them).
void launch_tile_sort(const Problem& p, int cb, const Workspace& ws, cudaStream_t s) {
  const int ntiles = cb * p.tiles;
  const int sms = sm_count();
  const int smem = kWarpSortWarps * (int)sizeof(WarpSortSmem);
  cudaFuncSetAttribute(k_sort_tiles, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  int per_sm = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm, k_sort_tiles, 32 * kWarpSortWarps, smem);
  const int grid = sms * (per_sm > 0 ? per_sm : 1);
  // Claims of several tiles save counter atomics, but a pass with few tiles a warp needs every warp at once:
  // one view of 2,500 tiles in claims of four kept 625 of 1,824 warps busy (89 us, against 47 in claims of one).
  const int chunk = std::max(1, std::min(kWarpSortChunk, ntiles / (8 * grid * kWarpSortWarps)));
  k_sort_tiles<<<grid, 32 * kWarpSortWarps, smem, s>>>(ws.tile_off, reinterpret_cast<unsigned long long*>(ws.entries),
                                                       p.capacity, ntiles, chunk, ws.big_list, ws.status);
  unsigned long long* entries = reinterpret_cast<unsigned long long*>(ws.entries);
  unsigned long long* scratch = reinterpret_cast<unsigned long long*>(ws.entries_tmp);
  const int psmem = 2 * (2 * kWarpSortCap * (int)sizeof(unsigned long long) + (int)sizeof(radix::WarpScratch));
  cudaFuncSetAttribute(k_sort_mid, cudaFuncAttributeMaxDynamicSharedMemorySize, psmem);
  int per_sm2 = 0;
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per_sm2, k_sort_mid, kMidThreads, psmem);
  k_sort_mid<<<sms * (per_sm2 > 0 ? per_sm2 : 1), kMidThreads, psmem, s>>>(ws.tile_off, entries, p.capacity, ws.big_list,
                                                                    ws.status);
  const int qsmem = 2 * kSortCap * (int)sizeof(unsigned long long);
  cudaFuncSetAttribute(k_sort_queued, cudaFuncAttributeMaxDynamicSharedMemorySize, qsmem);
  k_sort_queued<<<sms * 2, kSortThreads, qsmem, s>>>(ws.tile_off, entries, scratch, p.capacity, ws.big_list, ntiles,
                                                     ws.status);
  note_launches(3);
}

}  // namespace icgs
