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
// moved. A list of one depth is binned again by its indices. A list whose depths crowd into few bins (above kCrowd pairs
// of keys in a bin, per key) is binned again by its own distribution: each bin is split linearly into two bins
// a key that it holds, at twice its offset, so that a band of depths a few bins wide spreads over all of them.
// Short lists, and those whose bins hold one depth each, are counted out as far as that is cheaper. A list that
// still crowds (many equal depths) is refused, untouched, and goes to split_list, and what that refuses to the
// radix sort.
//
// 2e7 keys in lists of 700 / 4,000 (a warp's / a CTA's; ms, the fixed 0.07 of a call included), all by radix passes
// and so: uniform depths 0.29 / 0.33 and 0.20 / 0.26; one depth 0.36 / 0.30 and 0.23 / 0.30; two depths 1.35 / 1.09
// and 0.65 / 0.70; sixteen 1.29 / 1.09 and 0.71 / 0.58; nine in ten of one depth 1.33 / 1.03 and 0.78 / 0.93;
// 95 in a hundred in 400 words 0.51 / 0.92 and 0.44 / 0.52.
#pragma once

#include <cstdint>

#include <cuda_runtime.h>

namespace icgs {
namespace bucket {

constexpr unsigned kAll = 0xFFFFFFFFu;
// Most pairs of keys that share a bin, per key: counting among 2 kCrowd keys costs about what the second
// binning does, counting among 2 kCrowdSplit about what the radix sort does. Lists of up to kShort keys are
// counted out rather than split (64 keys of two depths 0.50 ms so, 0.39 by counting), and those of up to
// kCountOut rather than refused: they cannot have as many pairs (128 keys, nine in ten of one depth 2.04 against
// 0.70, 1.46 by radix passes).
constexpr uint32_t kCrowd = 8, kCrowdSplit = 32;
constexpr int kShort = 64, kCountOut = 128;

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

// Smallest and largest word over the team.
template <int NW, int BW>
__device__ __forceinline__ uint2 team_range(Bins<NW, BW>& sb, uint32_t lo, uint32_t hi) {
  lo = __reduce_min_sync(kAll, lo);
  hi = __reduce_max_sync(kAll, hi);
  if (NW > 1) {
    if ((threadIdx.x & 31) == 0) {
      sb.lo[threadIdx.x >> 5] = lo;
      sb.hi[threadIdx.x >> 5] = hi;
    }
    __syncthreads();
#pragma unroll
    for (int v = 0; v < NW; ++v) {
      lo = min(lo, sb.lo[v]);
      hi = max(hi, sb.hi[v]);
    }
  } else {
    __syncwarp();
  }
  return make_uint2(lo, hi);
}
// After the counts, the team's pairs of keys that share a bin.
template <int NW, int BW>
__device__ __forceinline__ uint32_t team_pairs(Bins<NW, BW>& sb, uint32_t pairs) {
  pairs = __reduce_add_sync(kAll, pairs);
  if (NW > 1 && (threadIdx.x & 31) == 0) sb.pairs[threadIdx.x >> 5] = pairs;
  team_sync<NW>();
  if (NW > 1) {
    pairs = 0u;
#pragma unroll
    for (int v = 0; v < NW; ++v) pairs += sb.pairs[v];
  }
  return pairs;
}
// Counts to offsets: each warp scans its bins, 256 at a time (8 a lane), then the warps' totals are added.
template <int NW, int BW>
__device__ __forceinline__ void scan_bins(Bins<NW, BW>& sb, int n, int nb) {
  const int tid = NW == 1 ? threadIdx.x & 31 : threadIdx.x;
  const int lane = threadIdx.x & 31, w = NW == 1 ? 0 : threadIdx.x >> 5;
  uint32_t* const cnt = reinterpret_cast<uint32_t*>(sb.word);
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
}
template <int NW, int BW>
__device__ __forceinline__ uint32_t offset_of(const Bins<NW, BW>& sb, uint32_t d) {
  const unsigned short* const off = reinterpret_cast<const unsigned short*>(sb.word);
  return NW == 1 ? off[d] : off[d] + sb.base[d / BW];
}
// The slot of a key of the bin at [s0, s1): s0 and the smaller keys of the bin.
__device__ __forceinline__ uint32_t slot_of(const unsigned long long* s_keys, unsigned long long key, uint32_t s0, uint32_t s1) {
  uint32_t slot = s0;
  if (s1 - s0 > 1u)
    for (uint32_t j = s0; j < s1; ++j) slot += s_keys[j] < key ? 1u : 0u;
  return slot;
}
__device__ __forceinline__ unsigned long long swapped(unsigned long long key) { return key << 32 | key >> 32; }
// A key in global memory, read here and not kept from an earlier read.
__device__ __forceinline__ unsigned long long key_at(const unsigned long long* at) {
  unsigned long long v;
  asm volatile("ld.global.b64 %0, [%1];" : "=l"(v) : "l"(at));
  return v;
}

// Sorts the n (1 < n <= 32 NW R) keys at g in place; false, with g untouched, for a crowded list. By one
// warp (NW = 1) or by a CTA of NW warps, all of whose threads call it; s_keys holds n keys.
template <int NW, int R, int BW>
__device__ __forceinline__ bool sort_list(unsigned long long* g, int n, unsigned long long* s_keys, Bins<NW, BW>& sb) {
  static_assert(BW % 256 == 0 && 64 * NW * R <= NW * BW && NW * BW <= 65535, "chunks of 256 bins, two bins a key, 16 bits");
  constexpr int T = 32 * NW;
  const int tid = NW == 1 ? threadIdx.x & 31 : threadIdx.x;
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
  const uint2 ends = team_range(sb, hmin, hmax);
  hmin = ends.x;
  // bin = (word - hmin) scale / 2^32 with scale a little below nb 2^32 / (range + 1), so that it stays below nb
  // (three roundings of 2^-24 against a margin of 2^-20); a range of fewer words than bins is taken as it is
  uint32_t range = ends.y - hmin;
  bool narrow = range < (uint32_t)nb;
  auto scale_of = [&]() -> uint32_t {
    return narrow ? 0u : (uint32_t)((float)nb * 4294967296.0f / ((float)range + 1.0f) * (1.0f - 0x1p-20f));
  };
  uint32_t scale = scale_of();
  auto bin_of = [&](unsigned long long key) -> uint32_t {
    const uint32_t x = (uint32_t)(key >> 32) - hmin;
    return narrow ? x : __umulhi(x, scale);
  };
  uint32_t* const cnt = reinterpret_cast<uint32_t*>(sb.word);
  uint32_t rank2[(R + 1) / 2];  // ranks in the bins, two to a register
  auto rank = [&](int r) -> uint32_t { return r & 1 ? rank2[r / 2] >> 16 : rank2[r / 2] & 0xFFFFu; };
  // Takes a key's rank in bin d; the number of keys that were there.
  auto count = [&](int r, uint32_t d) -> uint32_t {
    const uint32_t sh = (d & 1u) * 16u;
    const uint32_t old = (atomicAdd(&cnt[d >> 1], 1u << sh) >> sh) & 0xFFFFu;
    rank2[r / 2] = r & 1 ? rank2[r / 2] | (old << 16) : old;
    return old;
  };
  auto offset = [&](uint32_t d) -> uint32_t { return offset_of(sb, d); };
  const uint32_t most = n <= kCountOut ? kCountOut / 2 : kCrowdSplit;
  uint32_t pairs;
  bool done, flat = false;
  while (true) {
    pairs = 0u;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (r * T >= n) break;
      if (r * T + tid < n) pairs += count(r, bin_of(k[r]));
    }
    done = team_pairs(sb, pairs) <= (n <= kShort || (narrow && range > 0u) ? most : kCrowd) * (uint32_t)n;
    if (done || range > 0u || flat) break;
    // One depth: again by the indices, the halves of the keys swapped until they are written back. (Asked before the
    // counts, this cost the other lists 2%.)
    flat = true;
    uint32_t lo = kAll, hi = 0u;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (r * T >= n) break;
      if (r * T + tid < n) {
        k[r] = swapped(k[r]);
        lo = min(lo, (uint32_t)(k[r] >> 32));
        hi = max(hi, (uint32_t)(k[r] >> 32));
      }
    }
    const uint2 e = team_range(sb, lo, hi);
    hmin = e.x;
    range = e.y - e.x;
    narrow = range < (uint32_t)nb;
    scale = scale_of();
    for (int i = tid; i < nb / 8; i += T) sb.word[i] = make_uint4(0u, 0u, 0u, 0u);
    team_sync<NW>();
  }
  if (done) {
    scan_bins(sb, n, nb);
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (r * T >= n) break;
      if (r * T + tid < n) s_keys[offset(bin_of(k[r])) + rank(r)] = k[r];
    }
    team_sync<NW>();
    for (int pos = tid; pos < n; pos += T) {
      const unsigned long long key = s_keys[pos];
      const uint32_t d = bin_of(key);
      g[slot_of(s_keys, key, offset(d), offset(d + 1))] = flat ? swapped(key) : key;
    }
    team_sync<NW>();
    return true;
  }
  if (narrow) {  // a bin is one word
    team_sync<NW>();
    return false;
  }
  // Each bin split in two bins a key: the product's low word is the key's place within its bin. 2 n <= nb.
  scan_bins(sb, n, nb);
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
  if (team_pairs(sb, pairs) > most * (uint32_t)n) {
    team_sync<NW>();
    return false;
  }
  scan_bins(sb, n, nb);
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
      const uint32_t slot = slot_of(s_keys, k[r], offset(bin(r)), offset(bin(r) + 1));
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
  for (int pos = tid; pos < n; pos += T) g[pos] = flat ? swapped(s_keys[pos]) : s_keys[pos];
  team_sync<NW>();
  return true;
}

// Sorts a list that sort_list refused: the same binning and splitting by the whole key, a bin between its smallest
// and largest key; false, with g untouched, for one that crowds after kSplits splits. By a CTA of NW warps. The keys
// are read from memory at each pass, kAhead at a time: held in registers beside their bins and ranks they spill, and
// made sort_list spill too (lists of 1,000 uniform depths 0.20 -> 0.32 ms).
constexpr int kSplits = 3;
template <int NW, int R, int BW>
__device__ __forceinline__ bool split_list(unsigned long long* g, int n, unsigned long long* s_keys, Bins<NW, BW>& sb) {
  static_assert(NW > 1, "a CTA");
  constexpr int T = 32 * NW, nb = NW * BW, kAhead = 8;
  static_assert(R % kAhead == 0, "whole groups of keys");
  const int tid = threadIdx.x;
  uint32_t* const cnt = reinterpret_cast<uint32_t*>(sb.word);
  auto each = [&](auto f) {  // f(r, key) for the thread's keys
#pragma unroll
    for (int r0 = 0; r0 < R; r0 += kAhead) {
      if (r0 * T >= n) break;
      unsigned long long key[kAhead];
#pragma unroll
      for (int h = 0; h < kAhead; ++h) {
        const int pos = (r0 + h) * T + tid;
        key[h] = pos < n ? key_at(g + pos) : 0ull;
      }
#pragma unroll
      for (int h = 0; h < kAhead; ++h)
        if ((r0 + h) * T + tid < n) f(r0 + h, key[h]);
    }
  };
  auto clear = [&]() {
    __syncthreads();
    for (int i = tid; i < nb / 8; i += T) sb.word[i] = make_uint4(0u, 0u, 0u, 0u);
    __syncthreads();
  };
  uint32_t hmin = kAll, hmax = 0u, imin = kAll, imax = 0u;
  each([&](int, unsigned long long key) {
    hmin = min(hmin, (uint32_t)(key >> 32));
    hmax = max(hmax, (uint32_t)(key >> 32));
    imin = min(imin, (uint32_t)key);
    imax = max(imax, (uint32_t)key);
  });
  const uint2 h = team_range(sb, hmin, hmax);
  __syncthreads();
  const uint2 i = team_range(sb, imin, imax);
  // z: the key as one number without gaps, and its upper 32 bits x: keys of equal depths differ in it by their indices
  const unsigned long long irange = (unsigned long long)(i.y - i.x) + 1ull;
  const unsigned long long z_max = (h.y - h.x) * irange + (irange - 1ull);  // below 2^64
  const int shift = max(0, 32 - __clzll(z_max));
  auto whole = [&](unsigned long long key) -> unsigned long long {
    return ((uint32_t)(key >> 32) - h.x) * irange + ((uint32_t)key - i.x);
  };
  uint32_t bin2[R / 2] = {}, rank2[R / 2] = {};  // two to a register
  auto get = [](const uint32_t (&v)[R / 2], int r) -> uint32_t { return r & 1 ? v[r / 2] >> 16 : v[r / 2] & 0xFFFFu; };
  auto put = [](uint32_t (&v)[R / 2], int r, uint32_t x) {
    v[r / 2] = r & 1 ? (v[r / 2] & 0xFFFFu) | (x << 16) : (v[r / 2] & 0xFFFF0000u) | x;
  };
  clear();
  {  // the first bins, as sort_list's
    const uint32_t top = (uint32_t)(z_max >> shift);
    const uint32_t scale =
        top < (uint32_t)nb ? 0u : (uint32_t)((float)nb * 4294967296.0f / ((float)top + 1.0f) * (1.0f - 0x1p-20f));
    each([&](int r, unsigned long long key) {
      const uint32_t x = (uint32_t)(whole(key) >> shift), d = scale == 0u ? x : __umulhi(x, scale);
      put(bin2, r, d);
      atomicAdd(&cnt[d >> 1], 1u << ((d & 1u) * 16u));
    });
  }
  __syncthreads();
  uint2* const span_of = reinterpret_cast<uint2*>(s_keys);  // a bin's smallest and largest x, at its offset
  for (int split = 1;; ++split) {
    scan_bins(sb, n, nb);
    for (int pos = tid; pos < n; pos += T) span_of[pos] = make_uint2(kAll, 0u);
    __syncthreads();
    each([&](int r, unsigned long long key) {
      const uint32_t s0 = offset_of(sb, get(bin2, r));
      if (offset_of(sb, get(bin2, r) + 1) - s0 > 1u) {
        const uint32_t x = (uint32_t)(whole(key) >> shift);
        atomicMin(&span_of[s0].x, x);
        atomicMax(&span_of[s0].y, x);
      }
    });
    __syncthreads();
    each([&](int r, unsigned long long key) {
      const uint32_t s0 = offset_of(sb, get(bin2, r)), c2 = 2u * (offset_of(sb, get(bin2, r) + 1) - s0);
      uint32_t e = 2u * s0;  // 2 n <= nb
      if (c2 > 2u) {
        const unsigned long long z = whole(key);
        const uint2 m = span_of[s0];
        if (m.x < m.y)  // monotone in x, whatever the roundings
          e += min(c2 - 1u, (uint32_t)((float)((uint32_t)(z >> shift) - m.x) * __fdividef((float)c2, (float)(m.y - m.x) + 1.0f)));
        else if (shift > 0)  // by the bits below x
          e += __umulhi((uint32_t)((z << (64 - shift)) >> 32), c2);
      }
      put(bin2, r, e);
    });
    clear();
    uint32_t pairs = 0u;
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (r * T >= n) break;
      if (r * T + tid < n) {
        const uint32_t d = get(bin2, r), sh = (d & 1u) * 16u;
        const uint32_t old = (atomicAdd(&cnt[d >> 1], 1u << sh) >> sh) & 0xFFFFu;
        put(rank2, r, old);
        pairs += old;
      }
    }
    if (team_pairs(sb, pairs) <= kCrowdSplit * (uint32_t)n) break;
    if (split == kSplits) {
      __syncthreads();
      return false;
    }
  }
  scan_bins(sb, n, nb);
  each([&](int r, unsigned long long key) { s_keys[offset_of(sb, get(bin2, r)) + get(rank2, r)] = key; });
  __syncthreads();
  each([&](int r, unsigned long long key) {
    put(rank2, r, slot_of(s_keys, key, offset_of(sb, get(bin2, r)), offset_of(sb, get(bin2, r) + 1)));
  });
  __syncthreads();
  each([&](int r, unsigned long long key) { s_keys[get(rank2, r)] = key; });
  __syncthreads();
  for (int pos = tid; pos < n; pos += T) g[pos] = s_keys[pos];
  __syncthreads();
  return true;
}

}  // namespace bucket
}  // namespace icgs
