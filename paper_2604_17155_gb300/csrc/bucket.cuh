// bucket.cuh -- depth order of one tile list in one pass (the "depth ordered list" of Eq. 2): a bucket
// sort by depth whose buckets hold about half a key on average, finished by counting inside each bucket.
//
// A key is (float32 depth bits << 32) | Gaussian index; keys are unique. The list's range of depth words
// is mapped linearly (a multiply-high) onto the bins, two or more a key, so bins follow depth order. Each
// key takes its rank in its bin from the counter's atomic (any order within a bin will do), the counters
// are scanned into offsets, the keys are placed, and a key's final slot is its bin's offset plus the number
// of smaller keys in the bin, by the whole 64-bit key: the unique (depth, index) order, ties included.
// That is two shared-memory passes over the keys, whatever the depth range; the radix sort of radix.cuh takes
// one per 8 bits of it (three or four, with a ranking by lane masks each).
//
// Counting inside bins costs the sum of the squared bin lengths. The ranks give that sum before anything is
// moved. A list whose depths crowd into few bins (above kCrowd pairs of keys in a bin, per key) is binned
// again by its own distribution: each bin is split linearly into two bins a key that it holds, at twice its
// offset, so that a band of depths a few bins wide spreads over all of them. A list that still crowds
// (many equal depths) is refused, untouched, and goes to the radix sort.
//
// 4e7 keys in lists of 700: uniform depths 0.76 ms by radix passes, 0.33 so; nine in ten keys in 1/512 of
// the range 0.99, by splitting 0.53; 97 in a hundred in 1024 words with ties 1.06, 0.80.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace icgs {
namespace bucket {

constexpr unsigned kAll = 0xFFFFFFFFu;
// Most pairs of keys that share a bin, per key: counting among 2 kCrowd keys costs about what the second
// binning does, counting among 2 kCrowdSplit about what the radix sort does.
constexpr uint32_t kCrowd = 8, kCrowdSplit = 32;

// Shared memory of a team of NW warps with BW bins a warp: 16-bit counters and one more (the end).
template <int NW, int BW>
struct Bins {
  uint4 word[NW * BW / 8 + 1];
  uint32_t base[NW + 1];  // keys in the bins of the warps before (NW > 1)
  uint32_t lo[NW], hi[NW], pairs[NW];
};

template <int NW>
__device__ __forceinline__ void team_sync() {
  if (NW == 1) __syncwarp();
  else __syncthreads();
}

// Sorts the n (1 < n <= 32 NW R) keys at g in place; false, with g untouched, for a crowded list. By one
// warp (NW = 1) or by a CTA of NW warps, all of whose threads call it; s_keys holds n keys.
template <int NW, int R, int BW>
__device__ __forceinline__ bool sort_list(unsigned long long* g, int n, unsigned long long* s_keys, Bins<NW, BW>& sb) {
  static_assert(BW % 256 == 0 && 64 * NW * R <= NW * BW && NW * BW <= 65535, "chunks of 256 bins, two bins a key, 16 bits");
  constexpr int T = 32 * NW;
  const int tid = NW == 1 ? threadIdx.x & 31 : threadIdx.x;
  const int lane = threadIdx.x & 31, w = NW == 1 ? 0 : threadIdx.x >> 5;
  // a warp alone: two to four bins a key for short lists, whose scan would cost more than their keys
  int nb = NW * BW;
  if (NW == 1) nb = min(nb, max(256, 2 << (32 - __clz(n - 1))));
  unsigned long long k[R];
  uint32_t hmin = kAll, hmax = 0u;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (r * T >= n) break;
    const int pos = r * T + tid;
    k[r] = pos < n ? g[pos] : 0ull;
  }
  for (int i = tid; i < nb / 8; i += T) sb.word[i] = make_uint4(0u, 0u, 0u, 0u);
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (r * T >= n) break;
    if (r * T + tid < n) {
      const uint32_t h = (uint32_t)(k[r] >> 32);
      hmin = min(hmin, h);
      hmax = max(hmax, h);
    }
  }
  hmin = __reduce_min_sync(kAll, hmin);
  hmax = __reduce_max_sync(kAll, hmax);
  if (NW > 1) {
    if (lane == 0) {
      sb.lo[w] = hmin;
      sb.hi[w] = hmax;
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < NW; ++v) {
      hmin = min(hmin, sb.lo[v]);
      hmax = max(hmax, sb.hi[v]);
    }
  } else {
    __syncwarp();
  }
  // bin = (word - hmin) scale / 2^32 with scale a little below nb 2^32 / (range + 1), so that it stays below nb
  // (three roundings of 2^-24 against a margin of 2^-20); a range of fewer words than bins is taken as it is
  const uint32_t range = hmax - hmin;
  const bool narrow = range < (uint32_t)nb;
  const uint32_t scale =
      narrow ? 0u : (uint32_t)((float)nb * 4294967296.0f / ((float)range + 1.0f) * (1.0f - 0x1p-20f));
  auto bin_of = [&](unsigned long long key) -> uint32_t {
    const uint32_t x = (uint32_t)(key >> 32) - hmin;
    return narrow ? x : __umulhi(x, scale);
  };
  uint32_t* const cnt = reinterpret_cast<uint32_t*>(sb.word);
  const unsigned short* const off = reinterpret_cast<const unsigned short*>(sb.word);
  uint32_t rank2[(R + 1) / 2];  // ranks in the bins, two to a register
  auto rank = [&](int r) -> uint32_t { return r & 1 ? rank2[r / 2] >> 16 : rank2[r / 2] & 0xFFFFu; };
  // Takes a key's rank in bin d; the number of keys that were there.
  auto count = [&](int r, uint32_t d) -> uint32_t {
    const uint32_t sh = (d & 1u) * 16u;
    const uint32_t old = (atomicAdd(&cnt[d >> 1], 1u << sh) >> sh) & 0xFFFFu;
    rank2[r / 2] = r & 1 ? rank2[r / 2] | (old << 16) : old;
    return old;
  };
  // After the counts: whether the pairs of keys that share a bin are too many (uniform over the team).
  auto crowded = [&](uint32_t pairs, uint32_t limit) -> bool {
    pairs = __reduce_add_sync(kAll, pairs);
    if (NW > 1 && lane == 0) sb.pairs[w] = pairs;
    team_sync<NW>();
    if (NW > 1) {
      pairs = 0u;
#pragma unroll
      for (int v = 0; v < NW; ++v) pairs += sb.pairs[v];
    }
    return pairs > limit * (uint32_t)n;
  };
  // Counts to offsets: each warp scans its bins, 256 at a time (8 a lane), then the warps' totals are added.
  auto scan = [&]() {
    uint32_t run = 0u;
    uint4* const mine = sb.word + w * (BW / 8);
    const int chunks = (NW == 1 ? nb : BW) / 256;
    for (int c = 0; c < chunks; ++c) {
      uint4 v = mine[c * 32 + lane];
      const uint32_t t = v.x + v.y + v.z + v.w, s = (t & 0xFFFFu) + (t >> 16);
      uint32_t incl = s;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t y = __shfl_up_sync(kAll, incl, o);
        if (lane >= o) incl += y;
      }
      uint32_t e = run + incl - s;
      uint32_t* q = &v.x;
#pragma unroll
      for (int h = 0; h < 4; ++h) {
        const uint32_t lo = q[h] & 0xFFFFu, hi = q[h] >> 16;
        q[h] = e | ((e + lo) << 16);
        e += lo + hi;
      }
      mine[c * 32 + lane] = v;
      run += __shfl_sync(kAll, incl, 31);
    }
    if (NW == 1) {
      if (lane == 0) cnt[nb / 2] = (uint32_t)n;
      __syncwarp();
      return;
    }
    if (lane == 0) sb.lo[w] = run;
    if (tid == 0) cnt[nb / 2] = 0u;
    __syncthreads();
    if (tid <= NW) {
      uint32_t b = 0u;
#pragma unroll
      for (int v = 0; v < NW; ++v) b += v < tid ? sb.lo[v] : 0u;
      sb.base[tid] = b;
    }
    __syncthreads();
  };
  auto offset = [&](uint32_t d) -> uint32_t { return NW == 1 ? off[d] : off[d] + sb.base[d / BW]; };
  // The slot of a key of the bin at [s0, s1): s0 and the smaller keys of the bin.
  auto slot_of = [&](unsigned long long key, uint32_t s0, uint32_t s1) -> uint32_t {
    uint32_t slot = s0;
    if (s1 - s0 > 1u)
      for (uint32_t j = s0; j < s1; ++j) slot += s_keys[j] < key ? 1u : 0u;
    return slot;
  };

  uint32_t pairs = 0u;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (r * T >= n) break;
    if (r * T + tid < n) pairs += count(r, bin_of(k[r]));
  }
  if (!crowded(pairs, kCrowd)) {
    scan();
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (r * T >= n) break;
      if (r * T + tid < n) s_keys[offset(bin_of(k[r])) + rank(r)] = k[r];
    }
    team_sync<NW>();
    for (int pos = tid; pos < n; pos += T) {
      const unsigned long long key = s_keys[pos];
      const uint32_t d = bin_of(key);
      g[slot_of(key, offset(d), offset(d + 1))] = key;
    }
    team_sync<NW>();
    return true;
  }
  if (narrow) {  // a bin is one depth
    team_sync<NW>();
    return false;
  }
  // Each bin split in two bins a key: the product's low word is the key's place within its bin. 2 n <= nb.
  scan();
  uint32_t bin2[(R + 1) / 2];
  auto bin = [&](int r) -> uint32_t { return r & 1 ? bin2[r / 2] >> 16 : bin2[r / 2] & 0xFFFFu; };
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (r * T >= n) break;
    if (r * T + tid < n) {
      const uint32_t x = (uint32_t)(k[r] >> 32) - hmin, d = __umulhi(x, scale);
      const uint32_t s0 = offset(d), s1 = offset(d + 1);
      const uint32_t e = 2u * s0 + __umulhi(x * scale, 2u * (s1 - s0));
      bin2[r / 2] = r & 1 ? bin2[r / 2] | (e << 16) : e;
    }
  }
  team_sync<NW>();
  for (int i = tid; i < nb / 8; i += T) sb.word[i] = make_uint4(0u, 0u, 0u, 0u);
  team_sync<NW>();
  pairs = 0u;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (r * T >= n) break;
    if (r * T + tid < n) pairs += count(r, bin(r));
  }
  if (crowded(pairs, kCrowdSplit)) {
    team_sync<NW>();
    return false;
  }
  scan();
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (r * T >= n) break;
    if (r * T + tid < n) s_keys[offset(bin(r)) + rank(r)] = k[r];
  }
  team_sync<NW>();
  // The new bins are not to be had from a key alone: the slots are found by each key's owner (over the ranks),
  // then the keys move within shared memory, so that they leave in order.
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (r * T >= n) break;
    if (r * T + tid < n) {
      const uint32_t slot = slot_of(k[r], offset(bin(r)), offset(bin(r) + 1));
      rank2[r / 2] = r & 1 ? (rank2[r / 2] & 0xFFFFu) | (slot << 16) : (rank2[r / 2] & 0xFFFF0000u) | slot;
    }
  }
  team_sync<NW>();
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (r * T >= n) break;
    if (r * T + tid < n) s_keys[rank(r)] = k[r];
  }
  team_sync<NW>();
  for (int pos = tid; pos < n; pos += T) g[pos] = s_keys[pos];
  team_sync<NW>();
  return true;
}

}  // namespace bucket
}  // namespace icgs
