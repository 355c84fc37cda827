// groupwalk.cuh -- the tile walk by 8-lane groups, shared by the CUDA-core kernels of blend.cu for few
// channels and the tensor-core walk of contract_tc.cu: a depth-ordered hit list of its own for every
// small pixel block, and packed two-pixel arithmetic.
//
// What bounds these walks is instruction issue (70-80% of the cycles issued) with shared-memory reads
// or the FP32 pipes close behind, so the layout is chosen for instructions per contributing (pixel, Gaussian) pair:
//   - The 8 lanes of a group own one block: 8x4 or 4x8 pixels with PP = 2 pixel pairs a lane (64 threads a
//     tile), 4x4 with PP = 1 (128 threads). A warp's four groups step through their own lists
//     side by side, so a warp takes as many steps as its longest list has entries. Measured on the relight
//     scene, per (Gaussian, tile) instance: 1.69 steps of 64 pixels with one list per 8x8 warp block, 1.25
//     with 4x4 groups, 0.81 steps of 128 pixels with 8x4 groups. PP = 2 halves what a step costs besides
//     the pixels (list, geometry, reduction, list building); PP = 1 keeps more warps where shared memory
//     limits the CTAs.
//   - The arithmetic of a pixel pair is packed (add/mul/fma.rn.f32x2: two IEEE operations per issue). To
//     need no moves, a batch can be staged with every scalar twice in a row.
//   - Lists are padded with a Gaussian of opacity 0 and so need no end test.
//   - Each batch's indices and records are loaded one and two batches ahead.
// The decisions and the weights are those of walk.cuh's blend_step, bit for bit: the same rounded
// operations in the same order (min.NaN keeps a NaN product NaN, so that it fails alpha >= 1/255, as
// it failed the fast reject).
#pragma once

#include <cuda_runtime.h>

#include "icgs_device.cuh"
#include "icgs_internal.h"
#include "packed.cuh"
#include "walk.cuh"

namespace icgs {
namespace walk {

// A pair of ones that the compiler keeps in registers instead of rebuilding it at every use.
__device__ __forceinline__ f2 opaque_ones() {
  f2 d;
  asm volatile("mov.b64 %0, {%1, %1};" : "=l"(d) : "f"(1.0f));
  return d;
}
__device__ __forceinline__ float min_nan(float a, float b) {
  float d;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}

constexpr uint32_t kGPad = kBatch * 16;  // byte offset of the padding Gaussian

template <int PP>
struct GroupCfg {
  static_assert(PP == 1 || PP == 2, "one or two pixel pairs a lane");
  static constexpr int kThreads = 128 / PP, kWarps = 4 / PP, kGroups = 16 / PP;
};

// A group's block of pixels: 4x4 with PP = 1, 8x4 with PP = 2 or, TALL, 4x8. A lane's pixels: (px, py),
// (px + 1, py) and, with PP = 2, the same kRowStep rows below.
template <int PP, bool TALL>
struct GroupShape {
  static_assert(PP == 2 || !TALL, "4x8 blocks have two pixel pairs a lane");
  static constexpr float kHalfX = PP == 2 && !TALL ? 3.5f : 1.5f;  // pixel centres off the block's centre
  static constexpr float kHalfY = TALL ? 3.5f : 1.5f;
  static constexpr int kRowStep = TALL ? 4 : 2;
};

// The walk's threads are numbered tid = 0 .. GroupCfg::kThreads - 1, which a kernel with other warps beside
// them passes on.
template <int PP, bool TALL = false>
struct GroupCtx {
  using Shape = GroupShape<PP, TALL>;
  int j, t, px, py;         // camera, tile, first pixel
  bool in0[PP], in1[PP];    // the pixels inside the image
  float ox, oy;             // tile origin in image pixels
  f2 x2, y2[PP];            // pixel centres, tile-relative
  float bx, by;             // origin of the warp's block, tile-relative
  int group;                // this lane's group in the tile
  uint32_t b, len;
};

template <int PP, bool TALL = false>
__device__ __forceinline__ GroupCtx<PP, TALL> group_ctx(const uint32_t* __restrict__ tile_off, uint32_t capacity, int tiles,
                                                  int tiles_x, int width, int height, int tid) {
  GroupCtx<PP, TALL> c;
  constexpr int kStep = GroupShape<PP, TALL>::kRowStep;
  const int bid = blockIdx.x;
  c.j = bid / tiles;
  c.t = bid - c.j * tiles;
  const int tyi = c.t / tiles_x, txi = c.t - tyi * tiles_x;
  const int warp = tid >> 5, lane = tid & 31;
  const int gq = lane >> 3, l = lane & 7;
  const int bx = PP == 2 ? 0 : (warp & 1) * 8, by = PP == 2 ? warp * 8 : (warp >> 1) * 8;
  const int lx = TALL ? bx + gq * 4 + (l & 1) * 2 : bx + (gq & 1) * 4 * PP + (PP == 2 ? l & 3 : l & 1) * 2;
  const int ly = TALL ? by + (l >> 1) : by + (gq >> 1) * 4 + (PP == 2 ? l >> 2 : l >> 1);
  c.group = warp * 4 + gq;
  c.px = txi * kTile + lx;
  c.py = tyi * kTile + ly;
  c.ox = (float)(txi * kTile);
  c.oy = (float)(tyi * kTile);
  c.x2 = pack2((float)lx + 0.5f, (float)lx + 1.5f);
#pragma unroll
  for (int u = 0; u < PP; ++u) {
    c.in0[u] = c.px < width && c.py + kStep * u < height;
    c.in1[u] = c.px + 1 < width && c.py + kStep * u < height;
    c.y2[u] = pack2((float)(ly + kStep * u) + 0.5f, (float)(ly + kStep * u) + 0.5f);
  }
  c.bx = (float)bx;
  c.by = (float)by;
  const uint32_t b = min(tile_off[bid], capacity);
  uint32_t e = min(tile_off[bid + 1], capacity);
  if (e < b) e = b;
  c.b = b;
  c.len = e - b;
  return c;
}

// The transmittances of a lane's pixels: a pixel that has stopped, or lies outside the image, has T = 0.
template <int PP>
struct GroupT {
  float2 v[PP];
  f2 ones;
  template <bool TALL>
  __device__ __forceinline__ GroupT(const GroupCtx<PP, TALL>& c, float one = 1.0f) : ones(opaque_ones()) {
#pragma unroll
    for (int u = 0; u < PP; ++u) v[u] = make_float2(c.in0[u] ? one : 0.0f, c.in1[u] ? one : 0.0f);
  }
  __device__ __forceinline__ bool alive() const {
    bool a = false;
#pragma unroll
    for (int u = 0; u < PP; ++u) a = a || v[u].x > 0.0f || v[u].y > 0.0f;
    return a;
  }
};

// The geometry of a batch of kBatch Gaussians as the groups read it (slot kBatch: the padding). The means
// are negated, so that the offset pixel - mean is one packed addition. With DUP every value is stored
// twice, so that a packed operand is read and not assembled (three 16-byte loads a step); without, a
// step takes a 16-byte and an 8-byte load and six moves, for half the shared memory. What only the list
// test reads is apart: lim = (E_lim, packed half-sizes of the support box) per Gaussian.
struct GroupOperands {
  f2 nx, ny, A, Bc, C, o;
};
template <bool DUP>
struct GroupGeo;
template <>
struct GroupGeo<true> {
  float4 xy[kBatch + 1], ab[kBatch + 1], co[kBatch + 1];  // (-mx, -mx, -my, -my), (A, A, Bc, Bc), (C, C, o, o)
  __device__ __forceinline__ void put_mean(int g, float nx, float ny, float A, float Bc) {
    xy[g] = make_float4(nx, nx, ny, ny);
    ab[g] = make_float4(A, A, Bc, Bc);
  }
  __device__ __forceinline__ void put_rest(int g, float C, float o) { co[g] = make_float4(C, C, o, o); }
  __device__ __forceinline__ GroupOperands at(uint32_t off) const {
    const ulonglong2 m = *reinterpret_cast<const ulonglong2*>(reinterpret_cast<const char*>(xy) + off);
    const ulonglong2 q = *reinterpret_cast<const ulonglong2*>(reinterpret_cast<const char*>(ab) + off);
    const ulonglong2 r = *reinterpret_cast<const ulonglong2*>(reinterpret_cast<const char*>(co) + off);
    return {m.x, m.y, q.x, q.y, r.x, r.y};
  }
};
template <>
struct GroupGeo<false> {
  float4 xyab[kBatch + 1];  // (-mx, -my, A, Bc)
  float2 co[kBatch + 1];    // (C, o)
  __device__ __forceinline__ void put_mean(int g, float nx, float ny, float A, float Bc) { xyab[g] = make_float4(nx, ny, A, Bc); }
  __device__ __forceinline__ void put_rest(int g, float C, float o) { co[g] = make_float2(C, o); }
  __device__ __forceinline__ GroupOperands at(uint32_t off) const {
    const float4 m = *reinterpret_cast<const float4*>(reinterpret_cast<const char*>(xyab) + off);
    const float2 r = *reinterpret_cast<const float2*>(reinterpret_cast<const char*>(co) + (off >> 1));
    return {pack2(m.x, m.x), pack2(m.y, m.y), pack2(m.z, m.z), pack2(m.w, m.w), pack2(r.x, r.x), pack2(r.y, r.y)};
  }
};

// The groups' hit lists of a batch: byte offsets (16 per Gaussian) into the geometry, or with BYTES the
// slots themselves, which saves a KB where shared memory decides the CTAs per SM. A row stride of 144
// bytes puts four groups' rows in distinct banks.
template <int PP, bool BYTES = false>
struct GroupLists {
  static constexpr int kStride = BYTES ? 64 : 72;  // entries of a row
  uint16_t row[GroupCfg<PP>::kGroups][kStride / (BYTES ? 2 : 1)];

  // the byte offsets of entries i, i + 1 (i even) of a group's row
  __device__ __forceinline__ static uint2 pair(const uint16_t* row, int i) {
    if constexpr (BYTES) {
      const uint32_t v = row[i >> 1];
      return make_uint2((v & 0xFFu) << 4, (v >> 8) << 4);
    } else {
      const uint32_t v = *reinterpret_cast<const uint32_t*>(row + i);
      return make_uint2(v & 0xFFFFu, v >> 16);
    }
  }
};

// Geometry and lists of a walk that holds one batch at a time.
template <int PP>
struct GroupBatch {
  GroupGeo<true> geo;
  float2 lim[kBatch];
  GroupLists<PP> lists;
};

// The Gaussians' indices, of this batch and of the one before, and per Gaussian and warp the groups
// that list it (bit q: group q of the warp).
template <int PP>
struct GroupIds {
  uint32_t id[2][kBatch];
  uint8_t hits[kBatch][GroupCfg<PP>::kWarps];
};

// The padding slot (one thread).
template <bool DUP>
__device__ __forceinline__ void group_pad(GroupGeo<DUP>& geo) {
  geo.put_mean(kBatch, 0.0f, 0.0f, 0.0f, 0.0f);
  geo.put_rest(kBatch, 0.0f, 0.0f);
}

__device__ __forceinline__ float lg2_approx(float x) {
  float y;
  asm("lg2.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}
__device__ __forceinline__ float sqrt_approx(float x) {
  float y;
  asm("sqrt.approx.ftz.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// Staging of a batch, one thread a Gaussian (PP = 2) or two (PP = 1: the even one the mean and (A, Bc),
// the odd one (C, opacity) and what the list test reads). In three parts, so that the two dependent
// loads are off the path: a batch's indices are loaded two batches ahead, its records one batch ahead.
template <int PP>
__device__ __forceinline__ int group_slot(int tid) {
  return PP == 2 ? tid : tid >> 1;
}
struct GroupFetch {
  float4 box, par;
};
// The index of the thread's Gaussian of the batch that starts at slot first; 0 past the list's end.
template <int PP>
__device__ __forceinline__ uint32_t group_id(const unsigned long long* list, uint32_t first, uint32_t end, int64_t n,
                                             int tid) {
  const uint32_t at = first + (uint32_t)group_slot<PP>(tid);
  return at < end ? min((uint32_t)list[at], (uint32_t)(n - 1)) : 0u;
}
__device__ __forceinline__ GroupFetch group_fetch(uint32_t id, const ProjRec* __restrict__ rec_cam) {
  GroupFetch f;
  f.par = rec_cam[id].par;
  f.box = rec_cam[id].box;
  return f;
}
// E_lim is explained at group_lists. -E_thr = log2(255 o) (o >= 1/255 in every list), widened by 1e-4
// of itself and 7.2e-5; the approximate logarithm and roots are within 2^-20, and the square is
// widened by 1e-5.
template <int PP, bool TALL = false, bool DUP>
__device__ __forceinline__ void group_put(const GroupFetch& f, int nb, float ox, float oy, GroupGeo<DUP>& geo,
                                          float2* lim, int tid) {
  const int g = group_slot<PP>(tid);
  if (g >= nb) return;
  const float A = -kHalfLog2e * f.par.x, Bc = -2.0f * kHalfLog2e * f.par.y, C = -kHalfLog2e * f.par.z;
  if (PP == 2 || (tid & 1) == 0) {
    const float2 lo = unpack_half2(f.box.z);
    const float mx = __fadd_rn(__fsub_rn(f.box.x, ox), __fmul_rn(lo.x, kMeanLoScaleInv));
    const float my = __fadd_rn(__fsub_rn(f.box.y, oy), __fmul_rn(lo.y, kMeanLoScaleInv));
    geo.put_mean(g, -mx, -my, A, Bc);
  }
  if (PP == 2 || (tid & 1) == 1) {
    constexpr float hx = GroupShape<PP, TALL>::kHalfX, hy = GroupShape<PP, TALL>::kHalfY;
    const float thr = fmaf(fmaxf(lg2_approx(255.0f * f.par.w), 0.0f), 1.0001f, 7.2e-5f);
    const float corner = fmaf(hx * hx, fabsf(A), fmaf(hy * hy, fabsf(C), hx * hy * fabsf(Bc)));
    const float reach = sqrt_approx(thr) + sqrt_approx(corner);
    geo.put_rest(g, C, f.par.w);
    lim[g] = make_float2(-1.00001f * reach * reach, f.box.w);
  }
}

// Builds the warp's four hit lists of the batch and returns the longest one's length (warp-uniform).
// One Gaussian per lane is tested against the four blocks: can it pass alpha >= 1/255 at one of the
// block's pixel centres? Those lie within (hx, hy) of the block's centre. The Gaussian is listed when the
// centre is within (hx, hy) of its support box and when E = A dx^2 + Bc dx dy + C dy^2 there is at least
// E_lim = -(sqrt(-E_thr) + sqrt(-E_corner))^2: sqrt(-E) is a norm of the offset from the mean, so a pixel
// at the threshold E_thr is at most sqrt(-E_corner) closer than the centre, E_corner the lowest E of the
// offsets (+-hx, +-hy). Against the exact ellipse-rectangle test this lists 3-4% more for a third of
// the instructions. The margin for rounding is 2e-5 of |A dx^2| + |C dy^2|, which bounds half the sum of
// the three terms' magnitudes (the conic is positive definite); E itself is a few 2^-24 of those off.
// alive: bit q set while group q has a pixel that has not stopped. hits: the per-Gaussian masks, when
// wanted. any: the Gaussians that some group of the warp lists (two words, ORed into), counts: the
// tile's list lengths by group, when wanted.
template <int PP, bool TALL, bool DUP, bool BYTES>
__device__ __forceinline__ int group_lists(const GroupGeo<DUP>& geo, const float2* lim_of, GroupLists<PP, BYTES>& lists,
                                           const GroupCtx<PP, TALL>& c, int nb, uint32_t alive, int tid,
                                           uint8_t (*hits)[GroupCfg<PP>::kWarps], uint32_t* any = nullptr,
                                           uint32_t* counts = nullptr) {
  const int warp = tid >> 5, lane = tid & 31;
  constexpr int kStride = GroupLists<PP, BYTES>::kStride;
  constexpr float wx = TALL ? 4.0f : 4.0f * PP;  // block width
  uint16_t* const rows = lists.row[warp * 4];
  // pad every entry first, by 16-byte stores
  constexpr uint32_t kPad = BYTES ? (uint32_t)kBatch * 0x01010101u : kGPad | (kGPad << 16);
  constexpr int kRowStores = 4 * kStride * (BYTES ? 1 : 2) / 16;
#pragma unroll
  for (int i = 0; i < kRowStores; i += 32)
    if (i + lane < kRowStores) reinterpret_cast<uint4*>(rows)[i + lane] = make_uint4(kPad, kPad, kPad, kPad);
  __syncwarp();
  // Lane (q, j) writes the entries of group q whose Gaussians lie in the j-th four of each 32.
  const int gq = lane >> 3, j4 = (lane & 7) * 4;
  uint16_t* const my_row = reinterpret_cast<uint16_t*>(reinterpret_cast<char*>(rows) + gq * kStride * (BYTES ? 1 : 2));
  int cnt = 0;
#pragma unroll
  for (int half = 0; half < kBatch / 32; ++half) {
    if (half * 32 >= nb) break;  // uniform
    const int g = half * 32 + lane;
    bool h[4] = {false, false, false, false};
    if (g < nb) {
      const GroupOperands op = geo.at((uint32_t)g * 16u);
      const float2 lim = lim_of[g], half2 = unpack_half2(lim.y);
      const float hx = half2.x + GroupShape<PP, TALL>::kHalfX, hy = half2.y + GroupShape<PP, TALL>::kHalfY;
      // two blocks at a time, side by side: (0, 1) and (2, 3), below them or, TALL, to their right
#pragma unroll
      for (int v = 0; v < 2; ++v) {
        const float cx = TALL ? c.bx + 8.0f * (float)v : c.bx, cy = TALL ? c.by + 4.0f : c.by + (4.0f * (float)v + 2.0f);
        const f2 dx = add2(pack2(cx + 0.5f * wx, cx + 1.5f * wx), op.nx);
        const f2 ax = mul2(mul2(op.A, dx), dx), bx = mul2(op.Bc, dx);
        const float2 dxs = unpack2(dx);
        const f2 dy = add2(pack2(cy, cy), op.ny);
        const f2 sq = fma2(mul2(op.C, dy), dy, ax);
        const float2 e = unpack2(fma2(pack2(-2e-5f, -2e-5f), sq, fma2(bx, dy, sq)));
        const bool in_y = fabsf(unpack2(dy).x) <= hy;
        h[2 * v] = e.x >= lim.x && fabsf(dxs.x) <= hx && in_y;
        h[2 * v + 1] = e.y >= lim.x && fabsf(dxs.y) <= hx && in_y;
      }
    }
    uint32_t m[4];
#pragma unroll
    for (int q = 0; q < 4; ++q) m[q] = __ballot_sync(kFull, h[q] && ((alive >> q) & 1u));
    if (hits && g < nb) {
      uint32_t byte = 0u;
#pragma unroll
      for (int q = 0; q < 4; ++q) byte |= ((m[q] >> lane) & 1u) << q;
      hits[g][warp] = (uint8_t)byte;
    }
    if (any) any[half] |= (m[0] | m[1]) | (m[2] | m[3]);
    const uint32_t mine = gq < 2 ? (gq == 0 ? m[0] : m[1]) : (gq == 2 ? m[2] : m[3]);
    int at = cnt + __popc(mine & ((1u << j4) - 1u));
    const uint32_t four = mine >> j4;
#pragma unroll
    for (int b = 0; b < 4; ++b) {
      const bool in = (four >> b) & 1u;
      if constexpr (BYTES) {
        if (in) reinterpret_cast<uint8_t*>(my_row)[at] = (uint8_t)(half * 32 + j4 + b);
      } else {
        if (in) my_row[at] = (uint16_t)((half * 32 + j4 + b) * 16);
      }
      at += in ? 1 : 0;
    }
    cnt += __popc(mine);
  }
  if (counts && (lane & 7) == 0) counts[warp * 4 + gq] = (uint32_t)cnt;
  __syncwarp();
  return __reduce_max_sync(kFull, cnt);
}

// Which of the warp's groups still have a pixel that has not stopped (bit q for group q).
__device__ __forceinline__ uint32_t group_alive(bool alive) {
  const uint32_t m = __ballot_sync(kFull, alive);
  return ((m & 0xFFu) ? 1u : 0u) | ((m & 0xFF00u) ? 2u : 0u) | ((m & 0xFF0000u) ? 4u : 0u) | ((m >> 24) ? 8u : 0u);
}

// A listed Gaussian (byte offset off) at the lane's pixels: e = exp(-q/2), oe = opacity e and
// alpha = min(0.99, oe).
template <int PP>
struct GroupAlpha {
  float2 alpha[PP], oe[PP], e[PP];
};
template <int PP, bool TALL, bool DUP>
__device__ __forceinline__ GroupAlpha<PP> group_alpha(const GroupGeo<DUP>& geo, uint32_t off,
                                                      const GroupCtx<PP, TALL>& c) {
  const GroupOperands q = geo.at(off);
  const f2 dx = add2(c.x2, q.nx);
  GroupAlpha<PP> r;
#pragma unroll
  for (int u = 0; u < PP; ++u) {
    const f2 dy = add2(c.y2[u], q.ny);
    const float2 E = unpack2(fma2(fma2(q.A, dx, mul2(q.Bc, dy)), dx, mul2(mul2(q.C, dy), dy)));
    r.e[u] = make_float2(ex2_approx(E.x), ex2_approx(E.y));
    r.oe[u] = unpack2(mul2(q.o, pack2(r.e[u].x, r.e[u].y)));
    r.alpha[u] = make_float2(min_nan(r.oe[u].x, kAlphaMax), min_nan(r.oe[u].y, kAlphaMax));
  }
  return r;
}

// Applies the alphas to the pixels' transmittances and returns the weights (0 where skipped). A pixel
// that stops gets T = 0, at which every later step stops again. COUNT: counts the steps taken in
// npairs. TEXP: T carries a factor 2^TEXP (from 2^TEXP down), so that the weights come out scaled by it, and the
// stop compares with the threshold scaled the same way: a power of two commutes with the roundings of these
// normal values, so the decisions and the scaled weights are exactly those of the unscaled step.
template <int PP>
struct GroupW {
  float2 v[PP];
};
template <bool COUNT = true, int TEXP = 0, int PP>
__device__ __forceinline__ GroupW<PP> group_take(const GroupAlpha<PP>& al, GroupT<PP>& T, uint32_t& npairs) {
  constexpr float kTMinScaled = kTMin * (float)(1 << TEXP);
  GroupW<PP> r;
#pragma unroll
  for (int u = 0; u < PP; ++u) {
    const float2 alpha = al.alpha[u];
    float2& t = T.v[u];
    const f2 a2 = pack2(alpha.x, alpha.y), T2 = pack2(t.x, t.y);
    const float2 tT = unpack2(mul2(T2, sub2(T.ones, a2)));  // T (1 - alpha)
    const float2 w = unpack2(mul2(a2, T2));
    const bool ok0 = alpha.x >= kAlphaMin, ok1 = alpha.y >= kAlphaMin;
    const bool keep0 = ok0 && !(tT.x < kTMinScaled), keep1 = ok1 && !(tT.y < kTMinScaled);
    if constexpr (COUNT) {
      npairs += keep0 ? 1u : 0u;
      npairs += keep1 ? 1u : 0u;
    }
    const float z0 = keep0 ? tT.x : 0.0f, z1 = keep1 ? tT.y : 0.0f;
    t.x = ok0 ? z0 : t.x;
    t.y = ok1 ? z1 : t.y;
    r.v[u] = make_float2(keep0 ? w.x : 0.0f, keep1 ? w.y : 0.0f);
  }
  return r;
}

}  // namespace walk
}  // namespace icgs
