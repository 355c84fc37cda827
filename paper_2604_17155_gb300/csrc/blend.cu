// blend.cu -- the per-tile front-to-back walks (Eq. 2, Eq. 4-6), one CTA per 16x16 screen tile.
//
//   k_blend_accumulate  colorize: for every (pixel, Gaussian) blend weight w = alpha T (Eq. 4)
//   (2: <= 7 channels)  accumulate V = sum w (Eq. 5) and S_k = sum w t_k (Eq. 6 numerator), reduced
//                       over the tile's pixels; then ONE global atomic group per (Gaussian, tile)
//                       lands in the per-(camera, Gaussian) accumulator.
//   k_blend_render      render: img_k = sum w C_k (Eq. 1-3) with C from the payload.
//   (2: <= 4 channels)
//   k_blend_adjoint     gradient: dL/dt_k = sum w a_k and, per Gaussian, dL/do = sum over pixels of
//   (2: <= 4 channels)  (g T - sum_{n>m} g_n w_n / (1-alpha)) * alpha/o with g = beta + a . t.
//   k_blend_refine2     refinement: render and accumulation of the residuals in one kernel (<= 3 channels).
//
// The kernels named ...2 walk by 8-lane groups (groupwalk.cuh): 64 threads with four pixels each, every
// group its own hit list over its 8x4 or 4x8 pixel block, pixel pairs in packed FP32. They issue in 72%
// (accumulation) to 78% of the cycles, with the ALU and FMA pipes at 45-60%; what is left is the list's own waste (a warp's
// four groups run to the longest of their lists, 1.08 of their mean). Against one list a warp and two
// pixels a thread, at 800 x 800: accumulating 100 views 9.3 -> 6.0 ms, rendering them 9.0 -> 4.2, the
// adjoint of 40 views 6.5 -> 3.7.
//
// The others (more channels, whose per-pixel values and sums fill the registers) have 256 threads with one
// pixel each: warp w covers the 8x4 block ((w&1)*8, (w>>1)*4), skips a Gaussian whose padded support box
// misses its block (a ballot; the accumulate walk then also tests the ellipse), and skips a whole batch
// once all its pixels stopped. Sums go over a warp by a halving butterfly that leaves value v's sum in
// lane v * 32/NP, and over warps with shared-memory atomics.
#include <cuda_runtime.h>

#include "icgs_device.cuh"
#include "groupwalk.cuh"
#include "icgs_internal.h"
#include "walk.cuh"

namespace icgs {

namespace {

using namespace walk;

template <int N>
struct Log2 {
  static constexpr int value = 1 + Log2<N / 2>::value;
};
template <>
struct Log2<1> {
  static constexpr int value = 0;
};

template <int N>
struct NextPow2 {
  static constexpr int value = N <= 1 ? 1 : N <= 2 ? 2 : N <= 4 ? 4 : N <= 8 ? 8 : N <= 16 ? 16 : 32;
};

// Warp sums of NP values (NP a power of two <= 32) with NP - 1 + 5 - log2(NP) shuffles and no
// selects, for values held in lane-permuted slots: slot i of lane l holds value index i ^ m(l),
// m(l) = (l >> (5 - log2 NP)) & (NP - 1). At each level a lane keeps its lower half of slots and
// adds its partner's upper half, which holds the same value indices (the partner's m differs in
// exactly that level's bit). Lane l returns the warp sum of value m(l). The caller permutes its
// per-pixel factors once (they do not change during the walk).
template <int NP>
__device__ __forceinline__ float warp_permuted_reduce(float (&v)[NP]) {
  constexpr int P = Log2<NP>::value;
#pragma unroll
  for (int lvl = 0; lvl < P; ++lvl) {
    const int off = 16 >> lvl;
    const int half = NP >> (lvl + 1);
#pragma unroll
    for (int i = 0; i < half; ++i) v[i] += __shfl_xor_sync(kFull, v[i + half], off);
  }
  float r = v[0];
#pragma unroll
  for (int off = 16 >> P; off > 0; off >>= 1) r += __shfl_xor_sync(kFull, r, off);
  return r;
}
// ------------------------------------------------------------------------------------------
// colorize: V and S per (camera, Gaussian)
// ------------------------------------------------------------------------------------------
template <int KC>
__global__ void __launch_bounds__(kThreads, KC <= 8 ? 5 : 4) k_blend_accumulate(
    const uint32_t* __restrict__ tile_off, const uint64_t* __restrict__ entries, uint32_t capacity,
    const ProjRec* __restrict__ rec, int64_t n, int width, int height, int tiles_x, int tiles,
    const void* __restrict__ targets, int dtype, int K, int k0, int cam0, const float* __restrict__ sub_img,
    float* __restrict__ acc, int RS, int64_t acc_cam_stride, DevStatus* status) {
  static_assert(KC >= 8, "up to 7 channels take the group walk");
  constexpr int NV = KC + 1;                      // V and S_0..S_{KC-1}
  // 16 channels reduce V on its own, so that the sums fill a 16-value reduction instead of a
  // 32-value one padded with 15 zeros; otherwise V is value 0 of the reduction.
  constexpr bool kSplitV = KC == 16;
  constexpr int NS = kSplitV ? KC : NV;           // values in the warp reduction
  constexpr int NP = NextPow2<NS>::value;
  constexpr int SHIFT = 5 - Log2<NP>::value;      // lane l returns the sum of value l >> SHIFT
  __shared__ float4 s_geo[kBatch], s_aux[kBatch];
  __shared__ float2 s_half[kBatch];
  __shared__ uint32_t s_id[kBatch];
  __shared__ float s_acc[kBatch][NV];
  const TileCtx c = tile_ctx(tile_off, capacity, tiles, tiles_x, width, height);
  const unsigned long long* list = tile_list(entries, c.b);
  const int lane = threadIdx.x & 31;
  float tv[KC];
#pragma unroll
  for (int k = 0; k < KC; ++k) tv[k] = 0.0f;
  if (c.inside) {
    const int64_t base = (((int64_t)(cam0 + c.j) * height + c.py) * width + c.px) * K + k0;
#pragma unroll
    for (int k = 0; k < KC; ++k)
      if (k0 + k < K) tv[k] = load_target(targets, base + k, dtype);
    check_finite(tv, status);
    if (sub_img) {  // refinement: residual targets t - img, img of this pass's cameras
      const int64_t ib = (((int64_t)c.j * height + c.py) * width + c.px) * K + k0;
#pragma unroll
      for (int k = 0; k < KC; ++k)
        if (k0 + k < K) tv[k] -= sub_img[ib + k];
    }
  }
  for (int k = threadIdx.x; k < kBatch * NV; k += kThreads) (&s_acc[0][0])[k] = 0.0f;
  const ProjRec* rec_cam = rec + (int64_t)c.j * n;
  float* acc_cam = acc + (int64_t)c.j * acc_cam_stride;
  const int my_value = lane >> SHIFT;
  const bool reducer = (lane & ((1 << SHIFT) - 1)) == 0 && my_value < NS;
  const int my_col = (kSplitV ? 1 : 0) + my_value;  // the s_acc column of this lane's sum
  // Value q of a hit is w u[q], u = (1, t_0, .., t_{KC-1}, 0, ..), or the channels alone when V is
  // reduced on its own. This lane keeps value q in slot q ^ my_value (warp_permuted_reduce), so u
  // is permuted here once, by one conditional swap per bit of my_value.
  float u[NP];
#pragma unroll
  for (int q = 0; q < NP; ++q) {
    const int k = q - (kSplitV ? 0 : 1);
    u[q] = k < 0 ? 1.0f : (k < KC ? tv[k >= 0 && k < KC ? k : 0] : 0.0f);
  }
#pragma unroll
  for (int bit = 1; bit < NP; bit <<= 1) {
    const bool sw = (my_value & bit) != 0;
#pragma unroll
    for (int q = 0; q < NP; ++q) {
      if (q & bit) continue;
      const float x = u[q], y = u[q | bit];
      u[q] = sw ? y : x;
      u[q | bit] = sw ? x : y;
    }
  }
  float T = 1.0f;
  bool done = !c.inside;
  uint32_t npairs = 0;
  for (uint32_t start = 0; start < c.len; start += kBatch) {
    const int nb = (int)min((uint32_t)kBatch, c.len - start);
    __syncthreads();
    load_batch(list, start, nb, rec_cam, n, c.ox, c.oy, s_geo, s_aux, s_half, s_id);
    __syncthreads();
    if (!__all_sync(kFull, done)) {
#pragma unroll
      for (int half = 0; half < kBatch / 32; ++half) {
        uint32_t bits = warp_hit_bits<true>(s_geo, s_aux, s_half, half * 32, nb, c);
        while (bits) {  // only the Gaussians whose box touches this warp's block, in depth order
          const int g = half * 32 + __ffs(bits) - 1;
          bits &= bits - 1;
          const float w = blend_weight(s_geo[g], s_aux[g], c.pxf, c.pyf, T, done, npairs);
          if (__any_sync(kFull, w > 0.0f)) {
            float v[NP];
#pragma unroll
            for (int q = 0; q < NP; ++q) v[q] = __fmul_rn(w, u[q]);
            const float r = warp_permuted_reduce<NP>(v);
            if (reducer) atomicAdd(&s_acc[g][my_col], r);
            if constexpr (kSplitV) {
              float ws = w;
#pragma unroll
              for (int off = 16; off > 0; off >>= 1) ws += __shfl_xor_sync(kFull, ws, off);
              if (lane == 1) atomicAdd(&s_acc[g][0], ws);
            }
          }
        }
      }
    }
    __syncthreads();
    if ((int)threadIdx.x < nb) {
      const int g = threadIdx.x;
      if (s_acc[g][0] > 0.0f) {
        float* dst = acc_cam + (int64_t)s_id[g] * RS;
        if (k0 == 0) atomicAdd(dst, s_acc[g][0]);
#pragma unroll
        for (int k = 0; k < KC; ++k)
          if (k0 + k < K) atomicAdd(dst + 1 + k0 + k, s_acc[g][k + 1]);
#pragma unroll
        for (int k = 0; k < NV; ++k) s_acc[g][k] = 0.0f;
      }
    }
    if (__syncthreads_and(done)) break;
  }
  if (k0 == 0) add_pair_count(npairs, status);
}

// The same accumulation for up to 7 channels by 8-lane groups (groupwalk.cuh): 64 threads, two pixel
// pairs each, a hit list per 8x4 block. A group reduces each of its hits over its 8 lanes (a halving
// butterfly of 4 shuffles for up to 3 channels, 7 for up to 7) and stores the sums (no atomics: a group
// takes a Gaussian once per batch) in its row of s_part; after the batch one thread per Gaussian
// adds the rows of the groups that list it, and one atomic group per (Gaussian, tile) lands in the
// accumulator.
constexpr int kPP = 2;  // pixel pairs a lane of the walks below
constexpr int kGThreads = GroupCfg<kPP>::kThreads;
constexpr int kGroups = GroupCfg<kPP>::kGroups;

// V decides, through the pivots of the solve, which Gaussians are solved in FP64, so its sum over a pixel
// block keeps one order, that of a halving over the block's rows and then its columns (rows 4 apart, 2, 1,
// columns 4 apart, 2, 1): over 8x8 blocks up to three channels, over 8x4 blocks with more. The groups have
// the shape with which the levels fall inside a lane, inside a group and, last, between two groups:
// TALL 4x8 blocks keep V as the sums of their four columns, which two groups' columns 4 apart then join. (With V
// a sum of each group like the others the accumulation of 100 views took 5.8 ms, but a handful of three
// million Gaussians at the limit changed between the FP32 and the FP64 solve.) The rows of a block's sums
// are what fills the shared memory: 10 CTAs an SM.
// Refinement, whose V decides nothing, sums it like S (not ORDERED): 8x4 blocks, rows of half the size.
template <int KC, bool ORDERED = true>
struct GroupAcc {
  static_assert(KC >= 1 && KC <= 7, "1..7 channels");
  static constexpr bool kTall = ORDERED && KC <= 3;
  // values of a reduction: kTall S alone, else V and S
  static constexpr int NP = kTall ? (KC == 3 ? 4 : 2) : NextPow2<KC + 1>::value;
  static constexpr int SHIFT = 3 - Log2<NP>::value;         // lane l of a group returns value l >> SHIFT
  static constexpr int kRow = kTall ? 8 : NP;               // floats of a row: kTall V by columns, then S
  float part[kGroups][kBatch + 1][kRow];                    // slot kBatch: where the list padding goes
  GroupIds<kPP> ids;
};

// Group sums of NT values held in lane-permuted slots (warp_permuted_reduce over 8 lanes).
template <int NT>
__device__ __forceinline__ float group_permuted_reduce(float (&v)[NT]) {
  constexpr int P = Log2<NT>::value;
#pragma unroll
  for (int lvl = 0; lvl < P; ++lvl) {
    const int half = NT >> (lvl + 1);
#pragma unroll
    for (int i = 0; i < half; ++i) v[i] += __shfl_xor_sync(kFull, v[i + half], 4 >> lvl);
  }
  float r = v[0];
#pragma unroll
  for (int off = 4 >> P; off > 0; off >>= 1) r += __shfl_xor_sync(kFull, r, off);
  return r;
}

// The walk of one tile for target values tv of the lane's pixels ([2 u + x]: pair u, pixel x). UNCHECKED: they
// may be infinite or NaN without the call failing (residuals of more than three channels).
template <int KC, bool ORDERED, bool UNCHECKED>
__device__ __forceinline__ void group_accumulate(GroupBatch<kPP>& s, GroupAcc<KC, ORDERED>& sa,
                                                 const GroupCtx<kPP, GroupAcc<KC, ORDERED>::kTall>& c,
                                                 const unsigned long long* list, const ProjRec* __restrict__ rec_cam,
                                                 int64_t n, const float (&tv)[2 * kPP][KC], float* __restrict__ acc_cam,
                                                 int RS, int K, int k0, DevStatus* status) {
  using S = GroupAcc<KC, ORDERED>;
  constexpr bool kTall = S::kTall;
  constexpr int NP = S::NP, k1 = kTall ? 0 : 1;  // S_0 is value k1
  const int lane = threadIdx.x & 31;
  // Value k of a hit is its weights times u[k], u = (t_0, .., t_{KC-1}, 0, ..) with, not kTall, a 1 for V
  // first, summed over the pixels.
  // This lane keeps it in slot k ^ m (warp_permuted_reduce): u is permuted here once.
  const int m = (lane & 7) >> S::SHIFT;
  f2 U[2 * kPP][NP / 2];
#pragma unroll
  for (int x = 0; x < 2 * kPP; ++x) {
    float u[NP];
#pragma unroll
    for (int k = 0; k < NP; ++k)
      u[k] = k < k1 ? 1.0f : (k < k1 + KC ? tv[x][k >= k1 && k < k1 + KC ? k - k1 : 0] : 0.0f);
#pragma unroll
    for (int bit = 1; bit < NP; bit <<= 1) {
      const bool sw = (m & bit) != 0;
#pragma unroll
      for (int k = 0; k < NP; ++k) {
        if (k & bit) continue;
        const float a = u[k], b = u[k | bit];
        u[k] = sw ? b : a;
        u[k | bit] = sw ? a : b;
      }
    }
#pragma unroll
    for (int k = 0; k < NP / 2; ++k) U[x][k] = pack2(u[2 * k], u[2 * k + 1]);
  }
  // The lane's place in a row: kTall, lanes 1, 2, 6, 7 the columns of V that they end up with (2, 0, 1, 3) and
  // lanes 0, 3, 4 sums of the value that they return; else the value they return, ORDERED V in place of value 0.
  const int l = lane & 7;
  const bool has_v = kTall ? l == 1 || l == 2 || l == 6 || l == 7 : ORDERED && l == 0;
  const bool writer = kTall ? has_v || (l == 0 || l == 4 || (l == 3 && KC == 3))
                            : (l & ((1 << S::SHIFT) - 1)) == 0 && m < 1 + KC;
  const int my_col = !kTall ? m : (has_v ? 2 * (l & 1) + (l >> 2) : 4 + m);
  char* const my_part = reinterpret_cast<char*>(&sa.part[c.group][0][my_col]);
  const uint16_t* const my_list = s.lists.row[c.group];
  GroupT<kPP> T(c);
  uint32_t npairs = 0;
  int buf = 0;
  const uint32_t list_end = c.b + c.len;
  const uint32_t id0 = group_id<kPP>(list, c.b, list_end, n, threadIdx.x);
  uint32_t id_next = group_id<kPP>(list, c.b + kBatch, list_end, n, threadIdx.x);
  GroupFetch fetch = group_fetch(id0, rec_cam);
  group_put<kPP, kTall>(fetch, (int)min((uint32_t)kBatch, c.len), c.ox, c.oy, s.geo, s.lim, threadIdx.x);
  sa.ids.id[buf][threadIdx.x] = id0;
  __syncthreads();
  // two barriers a batch: the next batch is staged between them, when the walk of this one has ended
  for (uint32_t start = 0; start < c.len; start += kBatch, buf ^= 1) {
    const int nb = (int)min((uint32_t)kBatch, c.len - start);
    const uint32_t next = start + kBatch, id_fetched = id_next;
    if (next < c.len) {  // in flight during the walk
      fetch = group_fetch(id_fetched, rec_cam);
      id_next = group_id<kPP>(list, c.b + next + kBatch, list_end, n, threadIdx.x);
    }
    const int steps = group_lists(s.geo, s.lim, s.lists, c, nb, group_alive(T.alive()), threadIdx.x, sa.ids.hits);
    auto reduce = [&](uint32_t o, const GroupW<kPP>& w) {
      float v[NP];
#pragma unroll
      for (int k = 0; k < NP / 2; ++k) {
        f2 x = 0ull;
#pragma unroll
        for (int u = 0; u < kPP; ++u) {
          const f2 w0 = pack2(w.v[u].x, w.v[u].x), w1 = pack2(w.v[u].y, w.v[u].y);
          x = u == 0 ? mul2(w0, U[0][k]) : fma2(w0, U[2 * u][k], x);
          x = fma2(w1, U[2 * u + 1][k], x);
        }
        const float2 y = unpack2(x);
        v[2 * k] = y.x;
        v[2 * k + 1] = y.y;
      }
      const float r = group_permuted_reduce<NP>(v);  // the group's sum of value m
      float V = r;
      if constexpr (ORDERED) {  // the lane's rows, then the rows of the lanes, each keeping one of its columns
        const float2 t = unpack2(add2(pack2(w.v[0].x, w.v[0].y), pack2(w.v[1].x, w.v[1].y)));
        const bool odd = (lane & 4) != 0;
        V = (odd ? t.y : t.x) + __shfl_xor_sync(kFull, odd ? t.x : t.y, 4);
        V += __shfl_xor_sync(kFull, V, 2);
        if (!kTall) {  // the columns: 4 apart (above), 2, 1
          V += __shfl_xor_sync(kFull, V, 1);
          V += __shfl_xor_sync(kFull, V, 4);
        }
      }
      if (writer) *reinterpret_cast<float*>(my_part + o * S::kRow / 4) = has_v ? V : r;
    };
    for (int i = 0; i < steps; i += 2) {
      const uint2 o = s.lists.pair(my_list, i);
      const GroupAlpha<kPP> a1 = group_alpha(s.geo, o.x, c), a2 = group_alpha(s.geo, o.y, c);  // independent of T
      reduce(o.x, group_take(a1, T, npairs));
      reduce(o.y, group_take(a2, T, npairs));
    }
    __syncthreads();
    {
      const int g = threadIdx.x;
      float sum[8];  // V, S_0, ..
#pragma unroll
      for (int k = 0; k < 8; ++k) sum[k] = 0.0f;
      if (g < nb) {
        const uint32_t hits = *reinterpret_cast<const uint16_t*>(&sa.ids.hits[g][0]);
        if constexpr (kTall) {
#pragma unroll
          for (int q = 0; q < kGroups; q += 2) {  // an 8x8 block
            const uint32_t both = (hits >> (q < 4 ? q : q + 4)) & 3u;
            if (both == 0u) continue;
            float4 a = make_float4(0.0f, 0.0f, 0.0f, 0.0f), b = a;
            if (both & 1u) {
              a = *reinterpret_cast<const float4*>(sa.part[q][g]);
#pragma unroll
              for (int k = 0; k < KC; ++k) sum[1 + k] += sa.part[q][g][4 + k];
            }
            if (both & 2u) {
              b = *reinterpret_cast<const float4*>(sa.part[q + 1][g]);
#pragma unroll
              for (int k = 0; k < KC; ++k) sum[1 + k] += sa.part[q + 1][g][4 + k];
            }
            sum[0] += ((a.x + b.x) + (a.z + b.z)) + ((a.y + b.y) + (a.w + b.w));
          }
        } else {
#pragma unroll
          for (int q = 0; q < kGroups; ++q) {
            if (hits & (1u << (q < 4 ? q : q + 4))) {
              const float* row = sa.part[q][g];
              if constexpr (NP == 2) {
                const float2 x = *reinterpret_cast<const float2*>(row);
                sum[0] += x.x;
                sum[1] += x.y;
              } else {
                // an infinite residual makes 0 t NaN: it stays with the Gaussians that have weight in its block
                if (UNCHECKED && !(row[0] > 0.0f)) continue;
#pragma unroll
                for (int k = 0; k < NP; k += 4) {
                  const float4 x = *reinterpret_cast<const float4*>(row + k);
                  sum[k] += x.x;
                  sum[k + 1] += x.y;
                  sum[k + 2] += x.z;
                  sum[k + 3] += x.w;
                }
              }
            }
          }
        }
        if (sum[0] > 0.0f) {
          float* dst = acc_cam + (int64_t)sa.ids.id[buf][g] * RS;
          if (KC == 3 && K == 3) {
            atomicAdd(reinterpret_cast<float4*>(dst), make_float4(sum[0], sum[1], sum[2], sum[3]));
          } else {
            if (k0 == 0) atomicAdd(dst, sum[0]);
#pragma unroll
            for (int k = 0; k < KC; ++k)
              if (k0 + k < K) atomicAdd(dst + 1 + k0 + k, sum[k + 1]);
          }
        }
      }
    }
    if (next < c.len) {
      group_put<kPP, kTall>(fetch, (int)min((uint32_t)kBatch, c.len - next), c.ox, c.oy, s.geo, s.lim, threadIdx.x);
      sa.ids.id[buf ^ 1][threadIdx.x] = id_fetched;
    }
    if (!__syncthreads_or(T.alive())) break;
  }
  if (k0 == 0) add_pair_count(npairs, status);
}

// Calls f(x, offset) for each of the lane's pixels inside the image: x = 2 u + side, offset in pixels
// from the lane's first pixel.
template <bool TALL, typename F>
__device__ __forceinline__ void for_pixels(const GroupCtx<kPP, TALL>& c, int width, F f) {
#pragma unroll
  for (int u = 0; u < kPP; ++u) {
    const int64_t row = (int64_t)(GroupShape<kPP, TALL>::kRowStep * u) * width;
    if (c.in0[u]) f(2 * u, row);
    if (c.in1[u]) f(2 * u + 1, row + 1);
  }
}

// Flags a value that is not finite among the lane's pixels, all of whose loads it waits for at once.
template <int KC>
__device__ __forceinline__ void check_finite(const float (&tv)[2 * kPP][KC], DevStatus* status) {
  bool bad = false;
#pragma unroll
  for (int x = 0; x < 2 * kPP; ++x)
#pragma unroll
    for (int k = 0; k < KC; ++k) bad |= !isfinite(tv[x][k]);
  if (bad) atomicOr(&status->flags, kFlagNonfinite);
}

// The CTA's tile: camera of the images, first pixel.
struct TilePlace {
  int cam, x0, y0;
};
__device__ __forceinline__ TilePlace tile_place(int cam0, int tiles_x, int tiles) {
  const int j = (int)blockIdx.x / tiles, t = (int)blockIdx.x - j * tiles;
  return {cam0 + j, t % tiles_x * kTile, t / tiles_x * kTile};
}
// Visits the kc values from channel k0 of the tile's pixels, along the rows of the image: f(address, y < rows) for
// eight rows at a time.
template <typename T, typename F>
__device__ __forceinline__ void for_tile_values(const TilePlace& p, T* images, int width, int height, int K, int k0, int kc,
                                                F f) {
  const int y0 = p.y0 + (int)(threadIdx.x >> 5) * 8;
  const int cols = min(kTile, width - p.x0), rows = min(8, height - y0), lane = threadIdx.x & 31;
  T* const first = images + (((int64_t)p.cam * height + y0) * width + p.x0) * K + k0;
  for (int e = lane; e < cols * kc; e += 32) {
    T* const at = first + (kc == K ? e : (e / kc) * K + e % kc);
#pragma unroll
    for (int y = 0; y < 8; ++y) f(at + (int64_t)y * width * K, y < rows);
  }
}
// A tile without Gaussians: zeros in its pixels, or its targets only checked. By rows, since the lanes' own
// pixels, 4 bytes of 24 an instruction, touch each sector several times (rendering 100 empty views of 1600 x 1060:
// 0.82 ms by pixels, 0.47 by rows).
__device__ __forceinline__ void zero_tile(const TilePlace& p, float* __restrict__ images, int width, int height, int K,
                                          int k0, int kc) {
  for_tile_values(p, images, width, height, K, k0, kc, [](float* at, bool in) {
    if (in) *at = 0.0f;
  });
}
__device__ __forceinline__ void check_tile(const TilePlace& p, const void* targets, int dtype, int width, int height,
                                           int K, DevStatus* status) {
  uint32_t top = 0u;  // the largest magnitude: infinity and NaN lie above every other value
  if (dtype == 0) {
    for_tile_values(p, static_cast<const uint32_t*>(targets), width, height, K, 0, K,
                    [&](const uint32_t* at, bool in) { top = max(top, in ? __ldg(at) & 0x7FFFFFFFu : 0u); });
  } else {
    for_tile_values(p, static_cast<const uint16_t*>(targets), width, height, K, 0, K,
                    [&](const uint16_t* at, bool in) { top = max(top, in ? __ldg(at) & 0x7FFFu : 0u); });
  }
  if (top >= (dtype == 0 ? 0x7F800000u : dtype == 1 ? 0x7F80u : 0x7C00u)) atomicOr(&status->flags, kFlagNonfinite);
}
__device__ __forceinline__ bool tile_empty(const uint32_t* __restrict__ tile_off, uint32_t capacity) {
  return min(tile_off[blockIdx.x + 1], capacity) <= min(tile_off[blockIdx.x], capacity);
}

template <int KC, bool RESIDUAL>
__global__ void __launch_bounds__(kGThreads, KC <= 3 ? 10 : 8) k_blend_accumulate2(
    const uint32_t* __restrict__ tile_off, const uint64_t* __restrict__ entries, uint32_t capacity,
    const ProjRec* __restrict__ rec, int64_t n, int width, int height, int tiles_x, int tiles,
    const void* __restrict__ targets, int dtype, int K, int k0, int cam0, const float* __restrict__ sub_img,
    float* __restrict__ acc, int RS, int64_t acc_cam_stride, DevStatus* status) {
  __shared__ GroupBatch<kPP> s;
  __shared__ __align__(16) GroupAcc<KC> sa;
  const auto c = group_ctx<kPP, GroupAcc<KC>::kTall>(tile_off, capacity, tiles, tiles_x, width, height, threadIdx.x);
  if (threadIdx.x == 0) group_pad(s.geo);
  float tv[2 * kPP][KC];
#pragma unroll
  for (int x = 0; x < 2 * kPP; ++x)
#pragma unroll
    for (int k = 0; k < KC; ++k) tv[x][k] = 0.0f;
  const int64_t base = (((int64_t)(cam0 + c.j) * height + c.py) * width + c.px) * K + k0;
  const int64_t ib = (((int64_t)c.j * height + c.py) * width + c.px) * K + k0;
  for_pixels(c, width, [&](int x, int64_t off) {
#pragma unroll
    for (int k = 0; k < KC; ++k)
      if (k0 + k < K) tv[x][k] = load_target(targets, base + off * K + k, dtype);
  });
  if (KC > 3) check_finite(tv, status);
  if constexpr (RESIDUAL) {  // refinement: residual targets t - img, img of this pass's cameras
    for_pixels(c, width, [&](int x, int64_t off) {
#pragma unroll
      for (int k = 0; k < KC; ++k)
        if (k0 + k < K) tv[x][k] -= sub_img[ib + off * K + k];
    });
  }
  if (KC <= 3) check_finite(tv, status);
  if (c.len == 0) return;  // uniform
  group_accumulate<KC, true, RESIDUAL && (KC > 3)>(s, sa, c, reinterpret_cast<const unsigned long long*>(entries),
                                                   rec + (int64_t)c.j * n, n, tv, acc + (int64_t)c.j * acc_cam_stride, RS, K, k0, status);
}

// ------------------------------------------------------------------------------------------
// render: img = sum w C
// ------------------------------------------------------------------------------------------
template <int KC>
__global__ void __launch_bounds__(kThreads) k_blend_render(
    const uint32_t* __restrict__ tile_off, const uint64_t* __restrict__ entries, uint32_t capacity,
    const ProjRec* __restrict__ rec, int64_t n, int width, int height, int tiles_x, int tiles,
    const float* __restrict__ payload, int K, int k0, int cam0, float* __restrict__ images) {
  __shared__ float4 s_geo[kBatch], s_aux[kBatch];
  __shared__ float2 s_half[kBatch];
  __shared__ uint32_t s_id[kBatch];
  __shared__ float s_col[kBatch][KC];
  const TileCtx c = tile_ctx(tile_off, capacity, tiles, tiles_x, width, height);
  const unsigned long long* list = tile_list(entries, c.b);
  const ProjRec* rec_cam = rec + (int64_t)c.j * n;
  const float* pay_cam = payload + (int64_t)c.j * n * K;
  float img[KC];
#pragma unroll
  for (int k = 0; k < KC; ++k) img[k] = 0.0f;
  float T = 1.0f;
  bool done = !c.inside;
  for (uint32_t start = 0; start < c.len; start += kBatch) {
    const int nb = (int)min((uint32_t)kBatch, c.len - start);
    __syncthreads();
    load_batch(list, start, nb, rec_cam, n, c.ox, c.oy, s_geo, s_aux, s_half, s_id);
    __syncthreads();
    for (int idx = threadIdx.x; idx < nb * KC; idx += kThreads) {
      const int g = idx / KC, k = idx - g * KC;
      s_col[g][k] = k0 + k < K ? pay_cam[(int64_t)s_id[g] * K + k0 + k] : 0.0f;
    }
    __syncthreads();
    if (!__all_sync(kFull, done)) {
#pragma unroll
      for (int half = 0; half < kBatch / 32; ++half) {
        uint32_t bits = warp_hit_bits(s_geo, s_aux, s_half, half * 32, nb, c);
        while (bits && !done) {
          const int g = half * 32 + __ffs(bits) - 1;
          bits &= bits - 1;
          float al, ex;
          bool cap;
          const float w = blend_step(s_geo[g], s_aux[g], c.pxf, c.pyf, T, done, al, ex, cap);
          if (w > 0.0f) {
#pragma unroll
            for (int k = 0; k < KC; ++k) img[k] = fmaf(w, s_col[g][k], img[k]);
          }
        }
      }
    }
    if (__syncthreads_and(done)) break;
  }
  if (c.inside) {
    float* dst = images + (((int64_t)(cam0 + c.j) * height + c.py) * width + c.px) * K + k0;
#pragma unroll
    for (int k = 0; k < KC; ++k)
      if (k0 + k < K) dst[k] = img[k];
  }
}

// The render by 8-lane groups (groupwalk.cuh) for up to 4 channels: two pixel pairs a lane, a hit list per
// 8x4 block. The colours are staged twice each, so that a channel of a pixel pair is one packed FMA.
// A skipped step adds 0 c, which is exact for a finite c; once a staged colour is not finite (weird)
// the tile's steps test the weight instead.
struct GroupColours {
  float4 c01[kBatch + 1], c23[kBatch + 1];  // (c0, c0, c1, c1), (c2, c2, c3, c3); slot kBatch: zeros
};

// The channels of the thread's staged Gaussian.
template <int KC>
__device__ __forceinline__ void stage_colours(const float* __restrict__ pay_cam, uint32_t id, int nb, int K, int k0,
                                              GroupColours& col, int* weird) {
  const int g = threadIdx.x;
  if (g >= nb) return;
  const float* src = pay_cam + (int64_t)id * K + k0;
  float v[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
  for (int k = 0; k < KC; ++k)
    if (k0 + k < K) v[k] = src[k];
  bool bad = false;
#pragma unroll
  for (int k = 0; k < KC; ++k) bad |= !isfinite(v[k]);
  col.c01[g] = make_float4(v[0], v[0], v[1], v[1]);
  if (KC > 2) col.c23[g] = make_float4(v[2], v[2], v[3], v[3]);
  if (bad) *weird = 1;
}

// x with each half replaced by old's where that pixel's weight is 0 (only when guard is set)
__device__ __forceinline__ f2 guarded(bool guard, const float2 w, f2 x, f2 old) {
  if (!guard) return x;
  const float2 a = unpack2(x), b = unpack2(old);
  return pack2(w.x > 0.0f ? a.x : b.x, w.y > 0.0f ? a.y : b.y);
}

template <int KC, bool TALL>
__device__ __forceinline__ void group_render(GroupBatch<kPP>& s, GroupColours& col, int* weird, const GroupCtx<kPP, TALL>& c,
                                             const unsigned long long* list, const ProjRec* __restrict__ rec_cam,
                                             int64_t n, const float* __restrict__ pay_cam, int K, int k0,
                                             f2 (&img)[kPP][KC]) {
  if (threadIdx.x == 0) {
    *weird = 0;
    col.c01[kBatch] = col.c23[kBatch] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  }
#pragma unroll
  for (int u = 0; u < kPP; ++u)
#pragma unroll
    for (int k = 0; k < KC; ++k) img[u][k] = pack2(0.0f, 0.0f);
  const uint16_t* const my_list = s.lists.row[c.group];
  GroupT<kPP> T(c);
  uint32_t unused = 0;
  __syncthreads();
  const uint32_t list_end = c.b + c.len;
  uint32_t id_next = group_id<kPP>(list, c.b, list_end, n, threadIdx.x);
  auto stage = [&](uint32_t first) {  // the batch at slot first of the list, whose indices id_next holds
    const int nb = (int)min((uint32_t)kBatch, list_end - first);
    group_put<kPP, TALL>(group_fetch(id_next, rec_cam), nb, c.ox, c.oy, s.geo, s.lim, threadIdx.x);
    stage_colours<KC>(pay_cam, id_next, nb, K, k0, col, weird);
  };
  stage(c.b);
  __syncthreads();
  for (uint32_t start = 0; start < c.len; start += kBatch) {
    const int nb = (int)min((uint32_t)kBatch, c.len - start);
    id_next = group_id<kPP>(list, c.b + start + kBatch, list_end, n, threadIdx.x);
    const int steps = group_lists(s.geo, s.lim, s.lists, c, nb, group_alive(T.alive()), threadIdx.x, nullptr);
    auto blend = [&](uint32_t o, const GroupW<kPP>& w, bool guard) {
      const ulonglong2 c01 = *reinterpret_cast<const ulonglong2*>(reinterpret_cast<const char*>(col.c01) + o);
      ulonglong2 c23 = make_ulonglong2(0ull, 0ull);
      if constexpr (KC > 2) c23 = *reinterpret_cast<const ulonglong2*>(reinterpret_cast<const char*>(col.c23) + o);
      const f2 ck[4] = {c01.x, c01.y, c23.x, c23.y};
#pragma unroll
      for (int u = 0; u < kPP; ++u) {
        const f2 w2 = pack2(w.v[u].x, w.v[u].y);
#pragma unroll
        for (int k = 0; k < KC; ++k) img[u][k] = guarded(guard, w.v[u], fma2(w2, ck[k], img[u][k]), img[u][k]);
      }
    };
    auto walk = [&](bool guard) {
      for (int i = 0; i < steps; i += 2) {
        const uint2 o = s.lists.pair(my_list, i);
        const GroupAlpha<kPP> a1 = group_alpha(s.geo, o.x, c), a2 = group_alpha(s.geo, o.y, c);
        blend(o.x, group_take<false>(a1, T, unused), guard);
        blend(o.y, group_take<false>(a2, T, unused), guard);
      }
    };
    if (*weird) walk(true);
    else walk(false);
    if (!__syncthreads_or(T.alive())) break;
    if (start + kBatch < c.len) stage(c.b + start + kBatch);
    __syncthreads();
  }
}

template <int KC>
__global__ void __launch_bounds__(kGThreads, 13) k_blend_render2(
    const uint32_t* __restrict__ tile_off, const uint64_t* __restrict__ entries, uint32_t capacity,
    const ProjRec* __restrict__ rec, int64_t n, int width, int height, int tiles_x, int tiles,
    const float* __restrict__ payload, int K, int k0, int cam0, float* __restrict__ images) {
  static_assert(KC <= 4, "up to 4 channels");
  __shared__ GroupBatch<kPP> s;
  __shared__ GroupColours col;
  __shared__ int weird;
  if (tile_empty(tile_off, capacity)) {  // uniform
    zero_tile(tile_place(cam0, tiles_x, tiles), images, width, height, K, k0, min(KC, K - k0));
    return;
  }
  const GroupCtx<kPP> c = group_ctx<kPP>(tile_off, capacity, tiles, tiles_x, width, height, threadIdx.x);
  if (threadIdx.x == 0) group_pad(s.geo);
  f2 img[kPP][KC];
  group_render<KC>(s, col, &weird, c, reinterpret_cast<const unsigned long long*>(entries), rec + (int64_t)c.j * n, n,
                   payload + (int64_t)c.j * n * K, K, k0, img);
  float* dst = images + (((int64_t)(cam0 + c.j) * height + c.py) * width + c.px) * K + k0;
  for_pixels(c, width, [&](int x, int64_t off) {
#pragma unroll
    for (int k = 0; k < KC; ++k)
      if (k0 + k < K) {
        const float2 v = unpack2(img[x >> 1][k]);
        dst[off * K + k] = (x & 1) ? v.y : v.x;
      }
  });
}

// ------------------------------------------------------------------------------------------
// adjoint: dL/dt and dL/do. Payload per (camera, Gaussian) = (a_0..a_{K-1}, beta).
// ------------------------------------------------------------------------------------------
template <int KC>
__device__ __forceinline__ void load_payload(const float* __restrict__ pay_cam, int nb, int K, const uint32_t* s_id,
                                             float (*s_pay)[KC + 1]) {
  for (int idx = threadIdx.x; idx < nb * (KC + 1); idx += kThreads) {
    const int g = idx / (KC + 1), k = idx - g * (KC + 1);
    float v = 0.0f;
    if (k < KC) {
      if (k < K) v = pay_cam[(int64_t)s_id[g] * (K + 1) + k];
    } else {
      v = pay_cam[(int64_t)s_id[g] * (K + 1) + K];
    }
    s_pay[g][k] = v;
  }
}

template <int KC>
__global__ void __launch_bounds__(kThreads, KC <= 16 ? 4 : (KC <= 32 ? 2 : 1)) k_blend_adjoint(
    const uint32_t* __restrict__ tile_off, const uint64_t* __restrict__ entries, uint32_t capacity,
    const ProjRec* __restrict__ rec, int64_t n, int width, int height, int tiles_x, int tiles,
    const void* __restrict__ targets, int dtype, const float* __restrict__ payload, int K, int cam0,
    float* __restrict__ grad_t, float* __restrict__ grad_o) {
  __shared__ float4 s_geo[kBatch], s_aux[kBatch];
  __shared__ float2 s_half[kBatch];
  __shared__ uint32_t s_id[kBatch];
  __shared__ float s_pay[kBatch][KC + 1];
  __shared__ float s_go[kBatch];
  const TileCtx c = tile_ctx(tile_off, capacity, tiles, tiles_x, width, height);
  const unsigned long long* list = tile_list(entries, c.b);
  const int lane = threadIdx.x & 31;
  const ProjRec* rec_cam = rec + (int64_t)c.j * n;
  const float* pay_cam = payload + (int64_t)c.j * n * (K + 1);
  float tv[KC], gt[KC];
#pragma unroll
  for (int k = 0; k < KC; ++k) { tv[k] = 0.0f; gt[k] = 0.0f; }
  const int64_t pix = ((int64_t)(cam0 + c.j) * height + c.py) * width + c.px;
  if (c.inside) {
#pragma unroll
    for (int k = 0; k < KC; ++k)
      if (k < K) tv[k] = load_target(targets, pix * K + k, dtype);
  }
  // pass 1: F = sum_n g_n w_n and dL/dt = sum_n w_n a_n
  float F = 0.0f;
  {
    float T = 1.0f;
    bool done = !c.inside;
    for (uint32_t start = 0; start < c.len; start += kBatch) {
      const int nb = (int)min((uint32_t)kBatch, c.len - start);
      __syncthreads();
      load_batch(list, start, nb, rec_cam, n, c.ox, c.oy, s_geo, s_aux, s_half, s_id);
      __syncthreads();
      load_payload<KC>(pay_cam, nb, K, s_id, s_pay);
      __syncthreads();
      if (!__all_sync(kFull, done)) {
#pragma unroll
        for (int half = 0; half < kBatch / 32; ++half) {
          uint32_t bits = warp_hit_bits(s_geo, s_aux, s_half, half * 32, nb, c);
          while (bits && !done) {
            const int g = half * 32 + __ffs(bits) - 1;
            bits &= bits - 1;
            float al, ex;
            bool cap;
            const float w = blend_step(s_geo[g], s_aux[g], c.pxf, c.pyf, T, done, al, ex, cap);
            if (w > 0.0f) {
              float gg = s_pay[g][KC];
#pragma unroll
              for (int k = 0; k < KC; ++k) {
                gg = fmaf(s_pay[g][k], tv[k], gg);
                gt[k] = fmaf(w, s_pay[g][k], gt[k]);
              }
              F = fmaf(gg, w, F);
            }
          }
        }
      }
      if (__syncthreads_and(done)) break;
    }
  }
  if (grad_t && c.inside) {
#pragma unroll
    for (int k = 0; k < KC; ++k)
      if (k < K) grad_t[pix * K + k] = gt[k];
  }
  if (!grad_o) return;
  // pass 2: dL/dalpha_m = g_m T_m - (F - P_m) / (1 - alpha_m), P_m = sum_{n<=m} g_n w_n
  for (int k = threadIdx.x; k < kBatch; k += kThreads) s_go[k] = 0.0f;
  float T = 1.0f, P = 0.0f;
  bool done = !c.inside;
  for (uint32_t start = 0; start < c.len; start += kBatch) {
    const int nb = (int)min((uint32_t)kBatch, c.len - start);
    __syncthreads();
    load_batch(list, start, nb, rec_cam, n, c.ox, c.oy, s_geo, s_aux, s_half, s_id);
    __syncthreads();
    load_payload<KC>(pay_cam, nb, K, s_id, s_pay);
    __syncthreads();
    if (!__all_sync(kFull, done)) {
#pragma unroll
      for (int half = 0; half < kBatch / 32; ++half) {
       uint32_t bits = warp_hit_bits(s_geo, s_aux, s_half, half * 32, nb, c);
       // dL/dalpha_m of one hit for this pixel (0 when skipped or capped); updates T and P
       auto d_opacity = [&](int g) -> float {
         if (done) return 0.0f;
         const float Tm = T;
         float al = 0.0f, ex = 0.0f;
         bool cap = false;
         const float w = blend_step(s_geo[g], s_aux[g], c.pxf, c.pyf, T, done, al, ex, cap);
         if (!(w > 0.0f)) return 0.0f;
         float gg = s_pay[g][KC];
#pragma unroll
         for (int k = 0; k < KC; ++k) gg = fmaf(s_pay[g][k], tv[k], gg);
         P = fmaf(gg, w, P);
         const float dalpha = gg * Tm - __fdividef(F - P, 1.0f - al);
         return cap ? 0.0f : dalpha * ex;
       };
       // two consecutive hits (in depth order) share one warp reduction of their two values
       while (bits) {
        const int g1 = half * 32 + __ffs(bits) - 1;
        bits &= bits - 1;
        const int g2 = bits ? half * 32 + __ffs(bits) - 1 : -1;
        bits &= bits - 1;
        const float d1 = d_opacity(g1);
        const float d2 = g2 >= 0 ? d_opacity(g2) : 0.0f;
        if (__any_sync(kFull, d1 != 0.0f || d2 != 0.0f)) {
          // lanes < 16 end with the sum of d1, lanes >= 16 with the sum of d2
          const bool upper = (lane & 16) != 0;
          float r = (upper ? d2 : d1) + __shfl_xor_sync(kFull, upper ? d1 : d2, 16);
#pragma unroll
          for (int o = 8; o > 0; o >>= 1) r += __shfl_xor_sync(kFull, r, o);
          if (lane == 0) atomicAdd(&s_go[g1], r);
          if (lane == 16 && g2 >= 0) atomicAdd(&s_go[g2], r);
        }
       }
      }
    }
    __syncthreads();
    if ((int)threadIdx.x < nb) {
      const float v = s_go[threadIdx.x];
      if (v != 0.0f) {
        atomicAdd(grad_o + s_id[threadIdx.x], v);
        s_go[threadIdx.x] = 0.0f;
      }
    }
    if (__syncthreads_and(done)) break;
  }
}

// The adjoint walk by 8-lane groups (groupwalk.cuh) for up to 4 channels: two pixel pairs a lane, a hit
// list per 8x4 block, the payload staged twice each for packed arithmetic. Pass 2 adds a lane's four
// pixels, reduces two hits at a time over the group's 8 lanes (3 shuffles) and stores the sums in the
// group's row; after the batch one thread per Gaussian adds the rows and one atomic lands in grad_o.
// A skipped step adds 0 a to dL/dt and 0 g to F and P, g = a . t + beta: exact while a and g are finite.
// Once a staged payload could make g overflow at some pixel of the tile, or is not finite, or a target is not
// (weird), the tile's steps test the weight instead.
template <int KC>
struct GroupPayload {
  static constexpr int NQ = (KC + 2) / 2;      // float4 rows of two doubled values: a_0.., beta
  float4 q[NQ][kBatch + 1];
};

// t_max: the largest magnitude of the tile's targets. |g| and every partial sum of it stay below
// |beta| + t_max sum |a_k| (1 + 2^-21), so a bound below 2^126 rules an overflow out; a NaN, or an infinite
// a or beta, fails the comparison too (t_max = 0 makes it NaN).
template <int KC>
__device__ __forceinline__ void stage_payload(const float* __restrict__ pay_cam, uint32_t id, int nb, int K, float t_max,
                                              GroupPayload<KC>& pay, int* weird) {
  const int g = threadIdx.x;
  if (g >= nb) return;
  const float* src = pay_cam + (int64_t)id * (K + 1);  // K == KC
  float sum_a = 0.0f, beta = 0.0f;
#pragma unroll
  for (int r = 0; r < GroupPayload<KC>::NQ; ++r) {
    const float x = src[2 * r], y = 2 * r + 1 <= KC ? src[2 * r + 1 <= KC ? 2 * r + 1 : 0] : 0.0f;
    pay.q[r][g] = make_float4(x, x, y, y);
    if (2 * r < KC) sum_a += fabsf(x);
    else beta = x;
    if (2 * r + 1 < KC) sum_a += fabsf(y);
    else if (2 * r + 1 == KC) beta = y;
  }
  if (!(fmaf(t_max, sum_a, fabsf(beta)) < 0x1p126f)) *weird = 1;
}

// The staged payload of the Gaussian at byte offset o: a[0..KC-1], beta in a[KC].
template <int KC>
__device__ __forceinline__ void load_group_payload(const GroupPayload<KC>& pay, uint32_t o, f2 (&a)[KC + 1]) {
#pragma unroll
  for (int r = 0; r < GroupPayload<KC>::NQ; ++r) {
    const ulonglong2 v = *reinterpret_cast<const ulonglong2*>(reinterpret_cast<const char*>(pay.q[r]) + o);
    a[2 * r] = v.x;
    if (2 * r + 1 <= KC) a[2 * r + 1 <= KC ? 2 * r + 1 : 0] = v.y;
  }
}

template <int KC>
__global__ void __launch_bounds__(kGThreads, KC <= 3 ? 10 : 8) k_blend_adjoint2(
    const uint32_t* __restrict__ tile_off, const uint64_t* __restrict__ entries, uint32_t capacity,
    const ProjRec* __restrict__ rec, int64_t n, int width, int height, int tiles_x, int tiles,
    const void* __restrict__ targets, int dtype, const float* __restrict__ payload, int K, int cam0,
    float* __restrict__ grad_t, float* __restrict__ grad_o) {
  static_assert(KC <= 4, "up to 4 channels");
  __shared__ GroupBatch<kPP> s;
  __shared__ GroupPayload<KC> pay;
  __shared__ GroupIds<kPP> ids;
  __shared__ float s_go[kGroups][kBatch + 1];
  __shared__ float s_tmax[kGThreads / 32];
  __shared__ int weird;
  const GroupCtx<kPP> c = group_ctx<kPP>(tile_off, capacity, tiles, tiles_x, width, height, threadIdx.x);
  const unsigned long long* list = reinterpret_cast<const unsigned long long*>(entries);
  const int lane = threadIdx.x & 31;
  const ProjRec* rec_cam = rec + (int64_t)c.j * n;
  const float* pay_cam = payload + (int64_t)c.j * n * (K + 1);
  if (threadIdx.x == 0) {
    weird = 0;
#pragma unroll
    for (int r = 0; r < GroupPayload<KC>::NQ; ++r) pay.q[r][kBatch] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  }
  if (threadIdx.x == 0) group_pad(s.geo);
  const int64_t pix0 = ((int64_t)(cam0 + c.j) * height + c.py) * width + c.px;
  if (c.len == 0) {  // uniform
    if (grad_t) zero_tile(TilePlace{cam0 + c.j, (int)c.ox, (int)c.oy}, grad_t, width, height, KC, 0, KC);
    return;
  }
  f2 tv[kPP][KC];
  float t_max;
  {
    float t[2 * kPP][KC];
#pragma unroll
    for (int x = 0; x < 2 * kPP; ++x)
#pragma unroll
      for (int k = 0; k < KC; ++k) t[x][k] = 0.0f;
    uint32_t m = 0u;  // non-negative floats order like their bit patterns, with infinity and NaN above
    for_pixels(c, width, [&](int x, int64_t off) {
#pragma unroll
      for (int k = 0; k < KC; ++k) {
        t[x][k] = load_target(targets, (pix0 + off) * K + k, dtype);
        m = max(m, __float_as_uint(fabsf(t[x][k])));
      }
    });
    m = __reduce_max_sync(kFull, m);
    if (lane == 0) s_tmax[threadIdx.x >> 5] = __uint_as_float(m);
    __syncthreads();
    t_max = __uint_as_float(max(__float_as_uint(s_tmax[0]), __float_as_uint(s_tmax[1])));
    static_assert(kGThreads == 64, "two warps");
    if (!(t_max < INFINITY)) weird = 1;
#pragma unroll
    for (int u = 0; u < kPP; ++u)
#pragma unroll
      for (int k = 0; k < KC; ++k) tv[u][k] = pack2(t[2 * u][k], t[2 * u + 1][k]);
  }
  const uint32_t list_end = c.b + c.len;
  uint32_t id_next = 0;
  auto stage = [&](uint32_t first, int to) {  // the batch at slot first of the list, whose indices id_next holds
    const int nb = (int)min((uint32_t)kBatch, list_end - first);
    group_put<kPP>(group_fetch(id_next, rec_cam), nb, c.ox, c.oy, s.geo, s.lim, threadIdx.x);
    ids.id[to][threadIdx.x] = id_next;
    stage_payload<KC>(pay_cam, id_next, nb, K, t_max, pay, &weird);
  };
  // g = a . t + beta of pixel pair u
  auto gain = [&](const f2 (&a)[KC + 1], int u) -> f2 {
    f2 g = a[KC];
#pragma unroll
    for (int k = 0; k < KC; ++k) g = fma2(a[k], tv[u][k], g);
    return g;
  };
  const uint16_t* const my_list = s.lists.row[c.group];
  uint32_t unused = 0;
  // pass 1: F = sum_n g_n w_n and dL/dt = sum_n w_n a_n, per pixel
  f2 F[kPP];
  {
    f2 gt[kPP][KC];
#pragma unroll
    for (int u = 0; u < kPP; ++u) {
      F[u] = pack2(0.0f, 0.0f);
#pragma unroll
      for (int k = 0; k < KC; ++k) gt[u][k] = pack2(0.0f, 0.0f);
    }
    GroupT<kPP> T(c);
    id_next = group_id<kPP>(list, c.b, list_end, n, threadIdx.x);
    stage(c.b, 0);
    __syncthreads();
    for (uint32_t start = 0; start < c.len; start += kBatch) {
      const int nb = (int)min((uint32_t)kBatch, c.len - start);
      id_next = group_id<kPP>(list, c.b + start + kBatch, list_end, n, threadIdx.x);
      const int steps = group_lists(s.geo, s.lim, s.lists, c, nb, group_alive(T.alive()), threadIdx.x, nullptr);
      auto gather = [&](uint32_t o, const GroupW<kPP>& w, bool guard) {
        f2 a[KC + 1];
        load_group_payload<KC>(pay, o, a);
#pragma unroll
        for (int u = 0; u < kPP; ++u) {
          const f2 w2 = pack2(w.v[u].x, w.v[u].y);
#pragma unroll
          for (int k = 0; k < KC; ++k) gt[u][k] = guarded(guard, w.v[u], fma2(w2, a[k], gt[u][k]), gt[u][k]);
          F[u] = guarded(guard, w.v[u], fma2(gain(a, u), w2, F[u]), F[u]);
        }
      };
      auto walk = [&](bool guard) {
        for (int i = 0; i < steps; i += 2) {
          const uint2 o = s.lists.pair(my_list, i);
          const GroupAlpha<kPP> a1 = group_alpha(s.geo, o.x, c), a2 = group_alpha(s.geo, o.y, c);
          gather(o.x, group_take<false>(a1, T, unused), guard);
          gather(o.y, group_take<false>(a2, T, unused), guard);
        }
      };
      if (weird) walk(true);
      else walk(false);
      if (!__syncthreads_or(T.alive())) break;
      if (start + kBatch < c.len) stage(c.b + start + kBatch, 0);
      __syncthreads();
    }
    if (grad_t) {
      for_pixels(c, width, [&](int x, int64_t off) {
#pragma unroll
        for (int k = 0; k < KC; ++k) {
          const float2 v = unpack2(gt[x >> 1][k]);
          grad_t[(pix0 + off) * K + k] = (x & 1) ? v.y : v.x;
        }
      });
    }
  }
  if (!grad_o) return;
  // pass 2: dL/dalpha_m = g_m T_m - (F - P_m) / (1 - alpha_m), P_m = sum_{n<=m} g_n w_n; times
  // dalpha/do = exp(-q/2), 0 where skipped or where alpha was capped
  __syncthreads();
  GroupT<kPP> T(c);
  f2 P[kPP];
#pragma unroll
  for (int u = 0; u < kPP; ++u) P[u] = pack2(0.0f, 0.0f);
  const bool second = (lane & 4) != 0;  // this lane's half of the group returns the second hit's sum
  float* const my_go = s_go[c.group];
  int buf = 0;
  id_next = group_id<kPP>(list, c.b, list_end, n, threadIdx.x);
  stage(c.b, buf);
  __syncthreads();
  for (uint32_t start = 0; start < c.len; start += kBatch, buf ^= 1) {
    const int nb = (int)min((uint32_t)kBatch, c.len - start);
    id_next = group_id<kPP>(list, c.b + start + kBatch, list_end, n, threadIdx.x);
    const int steps = group_lists(s.geo, s.lim, s.lists, c, nb, group_alive(T.alive()), threadIdx.x, ids.hits);
    auto step = [&](uint32_t o, const GroupAlpha<kPP>& al, bool guard) -> float {
      GroupT<kPP> Tm = T;
      const GroupW<kPP> w = group_take<false>(al, T, unused);
      f2 a[KC + 1];
      load_group_payload<KC>(pay, o, a);
      float sum = 0.0f;
#pragma unroll
      for (int u = 0; u < kPP; ++u) {
        const f2 g = gain(a, u);
        P[u] = guarded(guard, w.v[u], fma2(g, pack2(w.v[u].x, w.v[u].y), P[u]), P[u]);
        const float2 rest = unpack2(sub2(F[u], P[u]));
        const float2 om = unpack2(sub2(T.ones, pack2(al.alpha[u].x, al.alpha[u].y)));
        const f2 da = fma2(g, pack2(Tm.v[u].x, Tm.v[u].y), pack2(-__fdividef(rest.x, om.x), -__fdividef(rest.y, om.y)));
        const float2 d = unpack2(mul2(da, pack2(al.e[u].x, al.e[u].y)));
        const float d0 = w.v[u].x > 0.0f && al.oe[u].x < kAlphaMax ? d.x : 0.0f;
        const float d1 = w.v[u].y > 0.0f && al.oe[u].y < kAlphaMax ? d.y : 0.0f;
        sum = u == 0 ? d0 + d1 : sum + (d0 + d1);
      }
      return sum;
    };
    auto walk = [&](bool guard) {
      for (int i = 0; i < steps; i += 2) {
        const uint2 o = s.lists.pair(my_list, i);
        const GroupAlpha<kPP> a1 = group_alpha(s.geo, o.x, c), a2 = group_alpha(s.geo, o.y, c);
        const float d1 = step(o.x, a1, guard), d2 = step(o.y, a2, guard);
        float v[2] = {second ? d2 : d1, second ? d1 : d2};
        const float r = group_permuted_reduce<2>(v);
        const uint32_t mine = second ? o.y : o.x;
        if ((lane & 3) == 0) my_go[mine / 16] = r;
      }
    };
    if (weird) walk(true);
    else walk(false);
    __syncthreads();
    {
      const int g = threadIdx.x;
      if (g < nb) {
        float sum = 0.0f;
        const uint32_t hits = *reinterpret_cast<const uint16_t*>(&ids.hits[g][0]);
#pragma unroll
        for (int q = 0; q < kGroups; ++q)
          if (hits & (1u << (q < 4 ? q : q + 4))) sum += s_go[q][g];
        if (sum != 0.0f) atomicAdd(grad_o + ids.id[buf][g], sum);
      }
    }
    if (start + kBatch < c.len) stage(c.b + start + kBatch, buf ^ 1);
    if (!__syncthreads_or(T.alive())) break;
  }
}

// One refinement walk (Alg. 1 lines 8-9) for up to 3 channels by 8-lane groups: pass 1 renders the
// current colours of the lane's pixels (as k_blend_render2), pass 2 accumulates the residual targets
// t - img (as k_blend_accumulate2 with a rendered image subtracted), over the tile list sorted once.
// Same arithmetic as the two separate walks, without the image round trip. The colours of pass 1 share
// the shared memory of pass 2's partial sums.
template <int KC>
__global__ void __launch_bounds__(kGThreads, 13) k_blend_refine2(
    const uint32_t* __restrict__ tile_off, const uint64_t* __restrict__ entries, uint32_t capacity,
    const ProjRec* __restrict__ rec, int64_t n, int width, int height, int tiles_x, int tiles,
    const void* __restrict__ targets, int dtype, int K, int cam0, const float* __restrict__ payload,
    float* __restrict__ acc, int RS, int64_t acc_cam_stride, DevStatus* status) {
  static_assert(KC <= 3, "up to 3 channels");
  static_assert(sizeof(GroupColours) <= sizeof(GroupAcc<KC, false>), "the colours fit where the sums go");
  __shared__ GroupBatch<kPP> s;
  __shared__ __align__(16) GroupAcc<KC, false> sa;
  __shared__ int weird;
  if (tile_empty(tile_off, capacity)) {  // uniform
    check_tile(tile_place(cam0, tiles_x, tiles), targets, dtype, width, height, K, status);
    return;
  }
  const auto c = group_ctx<kPP, GroupAcc<KC, false>::kTall>(tile_off, capacity, tiles, tiles_x, width, height, threadIdx.x);
  if (threadIdx.x == 0) group_pad(s.geo);
  const unsigned long long* list = reinterpret_cast<const unsigned long long*>(entries);
  const ProjRec* rec_cam = rec + (int64_t)c.j * n;
  f2 img[kPP][KC];
  group_render<KC>(s, reinterpret_cast<GroupColours&>(sa), &weird, c, list, rec_cam, n,
                   payload + (int64_t)c.j * n * K, K, 0, img);
  float tv[2 * kPP][KC];
#pragma unroll
  for (int x = 0; x < 2 * kPP; ++x)
#pragma unroll
    for (int k = 0; k < KC; ++k) tv[x][k] = 0.0f;
  const int64_t base = (((int64_t)(cam0 + c.j) * height + c.py) * width + c.px) * K;
  for_pixels(c, width, [&](int x, int64_t off) {
#pragma unroll
    for (int k = 0; k < KC; ++k) {
      const float2 v = unpack2(img[x >> 1][k]);
      tv[x][k] = load_target(targets, base + off * K + k, dtype) - ((x & 1) ? v.y : v.x);
    }
    walk::check_finite(tv[x], status);
  });
  __syncthreads();
  group_accumulate<KC, false, false>(s, sa, c, list, rec_cam, n, tv, acc + (int64_t)c.j * acc_cam_stride, RS, K, 0, status);
}

template <int KC>
void accumulate_chunk(const Problem& p, int cb, int cam0, const void* targets, int dtype, int k0,
                      const float* sub_img, const Workspace& ws, cudaStream_t s) {
  const int64_t stride = p.L == 0 ? 0 : p.n * (int64_t)p.acc_stride;
  if constexpr (KC <= 7) {
    const auto kern = sub_img ? k_blend_accumulate2<KC, true> : k_blend_accumulate2<KC, false>;
    kern<<<cb * p.tiles, kGThreads, 0, s>>>(ws.tile_off, ws.entries, p.capacity, ws.rec, p.n, p.width, p.height,
                                            p.tiles_x, p.tiles, targets, dtype, p.K, k0, cam0, sub_img, ws.acc,
                                            p.acc_stride, stride, ws.status);
  } else {
    k_blend_accumulate<KC><<<cb * p.tiles, kThreads, 0, s>>>(ws.tile_off, ws.entries, p.capacity, ws.rec, p.n,
                                                              p.width, p.height, p.tiles_x, p.tiles, targets, dtype,
                                                              p.K, k0, cam0, sub_img, ws.acc, p.acc_stride, stride,
                                                              ws.status);
  }
  note_launches(1);
}

template <int KC>
void render_chunk(const Problem& p, int cb, int cam0, int k0, const Workspace& ws, float* images,
                  cudaStream_t s) {
  if constexpr (KC <= 4) {
    k_blend_render2<KC><<<cb * p.tiles, kGThreads, 0, s>>>(ws.tile_off, ws.entries, p.capacity, ws.rec, p.n,
                                                           p.width, p.height, p.tiles_x, p.tiles, ws.payload, p.K,
                                                           k0, cam0, images);
  } else {
    k_blend_render<KC><<<cb * p.tiles, kThreads, 0, s>>>(ws.tile_off, ws.entries, p.capacity, ws.rec, p.n,
                                                          p.width, p.height, p.tiles_x, p.tiles, ws.payload, p.K,
                                                          k0, cam0, images);
  }
  note_launches(1);
}

}  // namespace

// Channels are processed in chunks of at most 16 per walk; the chunk width is the smallest
// instantiated width that covers the remaining channels (1+KC values are reduced per Gaussian,
// padded to a power of two: 2, 4 and 8 in the group walk, 16 and, V apart, 16 in the other). The group
// walk holds four pixels' values and the sums of a thread in registers, up to 7 channels.
void launch_blend_accumulate(const Problem& p, int cb, int cam0, const void* targets, int dtype,
                             const float* sub_img, const Workspace& ws, cudaStream_t s) {
  if (!sub_img && tc_accumulate_applies(p, dtype)) {
    launch_blend_accumulate_tc(p, cb, cam0, targets, dtype, ws, s);
    return;
  }
  for (int k0 = 0; k0 < p.K; k0 += 16) {
    const int kc = p.K - k0;
    if (kc == 1) accumulate_chunk<1>(p, cb, cam0, targets, dtype, k0, sub_img, ws, s);
    else if (kc == 2) accumulate_chunk<2>(p, cb, cam0, targets, dtype, k0, sub_img, ws, s);
    else if (kc == 3) accumulate_chunk<3>(p, cb, cam0, targets, dtype, k0, sub_img, ws, s);
    else if (kc <= 7) accumulate_chunk<7>(p, cb, cam0, targets, dtype, k0, sub_img, ws, s);
    else if (kc <= 15) accumulate_chunk<15>(p, cb, cam0, targets, dtype, k0, sub_img, ws, s);
    else accumulate_chunk<16>(p, cb, cam0, targets, dtype, k0, sub_img, ws, s);
  }
}

void launch_blend_render(const Problem& p, int cb, int cam0, const Workspace& ws, float* images,
                         cudaStream_t s) {
  for (int k0 = 0; k0 < p.K; k0 += 16) {
    const int kc = p.K - k0;
    if (kc == 1) render_chunk<1>(p, cb, cam0, k0, ws, images, s);
    else if (kc == 2) render_chunk<2>(p, cb, cam0, k0, ws, images, s);
    else if (kc == 3) render_chunk<3>(p, cb, cam0, k0, ws, images, s);
    else if (kc == 4) render_chunk<4>(p, cb, cam0, k0, ws, images, s);
    else if (kc <= 8) render_chunk<8>(p, cb, cam0, k0, ws, images, s);
    else render_chunk<16>(p, cb, cam0, k0, ws, images, s);
  }
}

// The refinement walk (render of the current colours, then accumulation of the residual targets)
// in one kernel for up to 3 channels; returns false when the channel count needs the two walks.
bool launch_blend_refine(const Problem& p, int cb, int cam0, const void* targets, int dtype, const Workspace& ws,
                         cudaStream_t s) {
  if (p.K > 3) return false;
  const int64_t stride = p.L == 0 ? 0 : p.n * (int64_t)p.acc_stride;
#define ICGS_REF(KC)                                                                                         \
  k_blend_refine2<KC><<<cb * p.tiles, kGThreads, 0, s>>>(ws.tile_off, ws.entries, p.capacity, ws.rec, p.n,     \
                                                          p.width, p.height, p.tiles_x, p.tiles, targets, dtype, \
                                                          p.K, cam0, ws.payload, ws.acc, p.acc_stride, stride,   \
                                                          ws.status)
  if (p.K == 1) ICGS_REF(1);
  else if (p.K == 2) ICGS_REF(2);
  else ICGS_REF(3);
#undef ICGS_REF
  note_launches(1);
  return true;
}

void launch_blend_adjoint(const Problem& p, int cb, int cam0, const void* targets, int dtype,
                          const Workspace& ws, float* grad_targets, bool want_grad_o, cudaStream_t s) {
  float* go = want_grad_o ? ws.grad_o_acc : nullptr;
#define ICGS_ADJ(KC)                                                                                       \
  k_blend_adjoint<KC><<<cb * p.tiles, kThreads, 0, s>>>(ws.tile_off, ws.entries, p.capacity, ws.rec, p.n,  \
                                                         p.width, p.height, p.tiles_x, p.tiles, targets,     \
                                                         dtype, ws.payload, p.K, cam0, grad_targets, go)
#define ICGS_ADJ2(KC)                                                                                        \
  k_blend_adjoint2<KC><<<cb * p.tiles, kGThreads, 0, s>>>(ws.tile_off, ws.entries, p.capacity, ws.rec, p.n,  \
                                                           p.width, p.height, p.tiles_x, p.tiles, targets,     \
                                                           dtype, ws.payload, p.K, cam0, grad_targets, go)
  if (p.K == 1) ICGS_ADJ2(1);
  else if (p.K == 2) ICGS_ADJ2(2);
  else if (p.K == 3) ICGS_ADJ2(3);
  else if (p.K == 4) ICGS_ADJ2(4);
  else if (p.K <= 8) ICGS_ADJ(8);
  else if (p.K <= 16) ICGS_ADJ(16);
  else if (p.K <= 32) ICGS_ADJ(32);
  else ICGS_ADJ(64);
#undef ICGS_ADJ
#undef ICGS_ADJ2
  note_launches(1);
}

}  // namespace icgs
