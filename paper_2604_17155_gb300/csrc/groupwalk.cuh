// groupwalk.cuh -- the tile walk by 8-lane groups, shared by the CUDA-core kernels of blend.cu for few
// channels: two pixels a thread, and a depth-ordered hit list of its own for every 4x4 pixel block.
//
// What bounds these walks is instruction issue (85% of the cycles issued with one list per warp), so
// the layout is chosen for instructions per contributing (pixel, Gaussian) pair:
//   - A CTA of 128 threads takes a 16x16 tile. Its 16 groups of 8 lanes own a 4x4 block each, a thread
//     the pixels (x, y) and (x, y + 2) of its group's block. A warp's four groups step through their
//     own lists side by side, so a warp takes as many steps as its longest list has entries: measured
//     on the relight scene, 1.21 steps of 64 pixels per (Gaussian, tile) instance against 1.69 with
//     one list per 8x8 warp block (and 1.01 with 2x2 blocks, whose lists cost more to build).
//   - The two pixels' arithmetic is packed (add/mul/fma.rn.f32x2: two IEEE operations per issue). To
//     need no moves, a batch is staged with every scalar twice in a row.
//   - Lists hold byte offsets, are padded with a Gaussian of opacity 0 and so need no end test.
// The decisions and the weights are those of walk.cuh's blend_step, bit for bit: the same rounded
// operations in the same order (min.NaN keeps a NaN product NaN, so that it fails alpha >= 1/255, as
// it failed the fast reject).
#pragma once

#include <cuda_runtime.h>

#include "icgs_device.cuh"
#include "icgs_internal.h"
#include "walk.cuh"

namespace icgs {
namespace walk {

// ---- pairs of floats in a 64-bit register ----
using f2 = unsigned long long;
__device__ __forceinline__ f2 pack2(float a, float b) {
  f2 d;
  asm("mov.b64 %0, {%1, %2};" : "=l"(d) : "f"(a), "f"(b));
  return d;
}
__device__ __forceinline__ float2 unpack2(f2 v) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(v));
  return r;
}
__device__ __forceinline__ f2 add2(f2 a, f2 b) {
  f2 d;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 mul2(f2 a, f2 b) {
  f2 d;
  asm("mul.rn.f32x2 %0, %1, %2;" : "=l"(d) : "l"(a), "l"(b));
  return d;
}
__device__ __forceinline__ f2 fma2(f2 a, f2 b, f2 c) {
  f2 d;
  asm("fma.rn.f32x2 %0, %1, %2, %3;" : "=l"(d) : "l"(a), "l"(b), "l"(c));
  return d;
}
__device__ __forceinline__ float min_nan(float a, float b) {
  float d;
  asm("min.NaN.f32 %0, %1, %2;" : "=f"(d) : "f"(a), "f"(b));
  return d;
}

constexpr int kGThreads = 128;
constexpr int kGWarps = kGThreads / 32;
constexpr int kGroups = 16;                   // 4x4 pixel blocks of a tile
constexpr uint32_t kGPad = kBatch * 16;       // list entry of the padding Gaussian
constexpr int kGListStride = kBatch + 8;      // entries; 144 bytes: four groups' rows in distinct banks

struct GroupCtx {
  int j, t, px, py;        // camera, tile; the first pixel (the second is 2 rows below)
  bool in0, in1;           // the pixels inside the image
  float ox, oy;            // tile origin in image pixels
  f2 x2, y2;               // the two pixel centres, tile-relative
  float bx, by;            // origin of the warp's 8x8 block, tile-relative
  int group;               // this thread's group in the tile
  uint32_t b, len;
};

__device__ __forceinline__ GroupCtx group_ctx(const uint32_t* __restrict__ tile_off, uint32_t capacity, int tiles,
                                              int tiles_x, int width, int height) {
  GroupCtx c;
  const int bid = blockIdx.x;
  c.j = bid / tiles;
  c.t = bid - c.j * tiles;
  const int tyi = c.t / tiles_x, txi = c.t - tyi * tiles_x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gq = lane >> 3, l = lane & 7;
  const int bx = (warp & 1) * 8, by = (warp >> 1) * 8;
  const int lx = bx + (gq & 1) * 4 + (l & 3), ly = by + (gq >> 1) * 4 + (l >> 2);
  c.group = warp * 4 + gq;
  c.px = txi * kTile + lx;
  c.py = tyi * kTile + ly;
  c.in0 = c.px < width && c.py < height;
  c.in1 = c.px < width && c.py + 2 < height;
  c.ox = (float)(txi * kTile);
  c.oy = (float)(tyi * kTile);
  c.x2 = pack2((float)lx + 0.5f, (float)lx + 0.5f);
  c.y2 = pack2((float)ly + 0.5f, (float)ly + 2.5f);
  c.bx = (float)bx;
  c.by = (float)by;
  const uint32_t b = min(tile_off[bid], capacity);
  uint32_t e = min(tile_off[bid + 1], capacity);
  if (e < b) e = b;
  c.b = b;
  c.len = e - b;
  return c;
}

// A batch of kBatch Gaussians as the groups read it, every value twice (slot kBatch: the padding).
// The means are negated, so that the offset pixel - mean is one packed addition.
struct GroupBatch {
  float4 xy[kBatch + 1];   // (-mean_x, -mean_x, -mean_y, -mean_y), tile-relative
  float4 ab[kBatch + 1];   // (A, A, Bc, Bc): the scaled conic of walk.cuh
  float4 co[kBatch + 1];   // (C, C, opacity, opacity)
  float4 lim[kBatch];      // (E_thr - 1e-6, -Bc/(2C), -Bc/(2A), -): read by group_lists only
  uint32_t id[2][kBatch];  // Gaussian indices of this batch and of the one before
  uint16_t list[kGroups][kGListStride];
  uint8_t hits[kBatch][kGWarps];  // per Gaussian and warp: bit q set when group q of the warp lists it
};

__device__ __forceinline__ void group_batch_init(GroupBatch& s) {
  if (threadIdx.x == 0) {
    s.xy[kBatch] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    s.ab[kBatch] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    s.co[kBatch] = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  }
}

// Stages list[first, first + nb) with two threads a Gaussian: the even one the mean and (A, Bc), the
// odd one (C, opacity) and what the list test reads.
// Returns the Gaussian's index.
__device__ __forceinline__ uint32_t group_stage(const unsigned long long* list, uint32_t first, int nb,
                                                const ProjRec* __restrict__ rec_cam, int64_t n, float ox, float oy,
                                                GroupBatch& s, int buf) {
  const int g = threadIdx.x >> 1;
  if (g >= nb) return 0u;
  const uint32_t id = min((uint32_t)list[first + g], (uint32_t)(n - 1));
  const ProjRec* r = rec_cam + id;
  const float4 par = r->par;
  const float A = -kHalfLog2e * par.x, Bc = -2.0f * kHalfLog2e * par.y, C = -kHalfLog2e * par.z;
  if ((threadIdx.x & 1) == 0) {
    const float4 box = r->box;
    const float2 lo = unpack_half2(box.z);
    const float mx = __fadd_rn(__fsub_rn(box.x, ox), __fmul_rn(lo.x, kMeanLoScaleInv));
    const float my = __fadd_rn(__fsub_rn(box.y, oy), __fmul_rn(lo.y, kMeanLoScaleInv));
    s.id[buf][g] = id;
    s.xy[g] = make_float4(-mx, -mx, -my, -my);
    s.ab[g] = make_float4(A, A, Bc, Bc);
  } else {
    const float qthr = __fmaf_rn(2.0f * logf(255.0f * par.w), 1.0001f, 1e-4f);
    s.co[g] = make_float4(C, C, par.w, par.w);
    s.lim[g] = make_float4(__fmaf_rn(-kHalfLog2e, qthr, -1e-6f), __fdividef(-0.5f * Bc, C), __fdividef(-0.5f * Bc, A),
                           0.0f);
  }
  return id;
}

// Builds the warp's four hit lists of the batch and returns the longest one's length (warp-uniform).
// One Gaussian per lane is tested against the four 4x4 blocks: can E = A dx^2 + Bc dx dy + C dy^2
// (concave, 0 at the mean) reach the fast-reject threshold at a point of the rectangle of the block's
// pixel centres? Its peak over the rectangle lies on the edges that face the mean (or is the mean):
// the larger of E at the nearest x with its best y clamped to the rectangle, and E at the nearest y
// with its best x. Both are points of the rectangle, so neither overstates the peak. The test rejects
// only when that falls short of the threshold by more than a rounding margin, 2e-5 of
// |A dx^2| + |C dy^2|, which bounds half the sum of the three terms' magnitudes (the conic is positive
// definite); the per-pixel E is a few 2^-24 of those off. alive: bit q set while group q has a pixel
// that has not stopped.
__device__ __forceinline__ int group_lists(GroupBatch& s, const GroupCtx& c, int nb, uint32_t alive) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  uint16_t(*rows)[kGListStride] = s.list + warp * 4;
  // pad every entry first (144 bytes a row, four rows: 36 sixteen-byte stores)
  constexpr uint32_t kPad2 = kGPad | (kGPad << 16);
  uint4* flat = reinterpret_cast<uint4*>(rows);
  flat[lane] = make_uint4(kPad2, kPad2, kPad2, kPad2);
  if (lane < 4) flat[32 + lane] = make_uint4(kPad2, kPad2, kPad2, kPad2);
  __syncwarp();
  int cnt[4] = {0, 0, 0, 0};
  const uint32_t lt = (1u << lane) - 1u;
#pragma unroll
  for (int half = 0; half < kBatch / 32; ++half) {
    if (half * 32 >= nb) break;  // uniform
    const int g = half * 32 + lane;
    bool h[4] = {false, false, false, false};
    if (g < nb) {
      const float4 xy = s.xy[g], ab = s.ab[g], co = s.co[g], lim = s.lim[g];
      const f2 A = pack2(ab.x, ab.y), Bc = pack2(ab.z, ab.w), C = pack2(co.x, co.y);
      const f2 slack = pack2(-2e-5f, -2e-5f);
      float x0[2], x1[2], y0[2], y1[2], nx[2], ny[2], ty[2], tx[2];
#pragma unroll
      for (int u = 0; u < 2; ++u) {
        x0[u] = (c.bx + (4.0f * (float)u + 0.5f)) + xy.x;
        x1[u] = x0[u] + 3.0f;
        y0[u] = (c.by + (4.0f * (float)u + 0.5f)) + xy.z;
        y1[u] = y0[u] + 3.0f;
        nx[u] = fmaxf(x0[u], fminf(0.0f, x1[u]));
        ny[u] = fmaxf(y0[u], fminf(0.0f, y1[u]));
        ty[u] = lim.y * nx[u];  // the best dy at dx = nx
        tx[u] = lim.z * ny[u];  // the best dx at dy = ny
      }
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int u = q & 1, v = q >> 1;
        const f2 dx = pack2(nx[u], fminf(fmaxf(tx[v], x0[u]), x1[u]));
        const f2 dy = pack2(fminf(fmaxf(ty[u], y0[v]), y1[v]), ny[v]);
        const f2 sq = fma2(C, mul2(dy, dy), mul2(A, mul2(dx, dx)));
        const float2 e = unpack2(fma2(slack, sq, fma2(Bc, mul2(dx, dy), sq)));
        h[q] = fmaxf(e.x, e.y) >= lim.x && ((alive >> q) & 1u);
      }
      s.hits[g][warp] = (uint8_t)((h[0] ? 1 : 0) | (h[1] ? 2 : 0) | (h[2] ? 4 : 0) | (h[3] ? 8 : 0));
    }
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const uint32_t m = __ballot_sync(kFull, h[q]);
      if (h[q]) rows[q][cnt[q] + __popc(m & lt)] = (uint16_t)(g * 16);
      cnt[q] += __popc(m);
    }
  }
  __syncwarp();
  return max(max(cnt[0], cnt[1]), max(cnt[2], cnt[3]));
}

// Which of the warp's groups still have a pixel that has not stopped (bit q for group q).
__device__ __forceinline__ uint32_t group_alive(bool alive) {
  const uint32_t m = __ballot_sync(kFull, alive);
  return ((m & 0xFFu) ? 1u : 0u) | ((m & 0xFF00u) ? 2u : 0u) | ((m & 0xFF0000u) ? 4u : 0u) | ((m >> 24) ? 8u : 0u);
}

// A listed Gaussian (byte offset off) at the thread's two pixels: e = exp(-q/2), oe = opacity e and
// alpha = min(0.99, oe).
struct GroupAlpha {
  float2 alpha, oe, e;
};
__device__ __forceinline__ GroupAlpha group_alpha(const GroupBatch& s, uint32_t off, const GroupCtx& c) {
  const ulonglong2 xy = *reinterpret_cast<const ulonglong2*>(reinterpret_cast<const char*>(s.xy) + off);
  const ulonglong2 ab = *reinterpret_cast<const ulonglong2*>(reinterpret_cast<const char*>(s.ab) + off);
  const ulonglong2 co = *reinterpret_cast<const ulonglong2*>(reinterpret_cast<const char*>(s.co) + off);
  const f2 dx = add2(c.x2, xy.x), dy = add2(c.y2, xy.y);
  const float2 E = unpack2(fma2(fma2(ab.x, dx, mul2(ab.y, dy)), dx, mul2(mul2(co.x, dy), dy)));
  GroupAlpha r;
  r.e = make_float2(ex2_approx(E.x), ex2_approx(E.y));
  r.oe = unpack2(mul2(co.y, pack2(r.e.x, r.e.y)));
  r.alpha = make_float2(min_nan(r.oe.x, kAlphaMax), min_nan(r.oe.y, kAlphaMax));
  return r;
}

// Applies the two alphas to the two pixels' transmittances and returns the weights (0 where skipped).
// A pixel that stops keeps T = 0, at which every later step stops again; T starts at 0 outside the
// image. COUNT: counts the steps taken in npairs.
template <bool COUNT = true>
__device__ __forceinline__ float2 group_take(const float2 alpha, float2& T, uint32_t& npairs) {
  const f2 a2 = pack2(alpha.x, alpha.y), T2 = pack2(T.x, T.y);
  const float2 tT = unpack2(mul2(T2, fma2(a2, pack2(-1.0f, -1.0f), pack2(1.0f, 1.0f))));  // T (1 - alpha)
  const float2 w = unpack2(mul2(a2, T2));
  const bool ok0 = alpha.x >= kAlphaMin, ok1 = alpha.y >= kAlphaMin;
  const bool keep0 = ok0 && !(tT.x < kTMin), keep1 = ok1 && !(tT.y < kTMin);
  if constexpr (COUNT) {
    npairs += keep0 ? 1u : 0u;
    npairs += keep1 ? 1u : 0u;
  }
  if (ok0) T.x = keep0 ? tT.x : 0.0f;
  if (ok1) T.y = keep1 ? tT.y : 0.0f;
  return make_float2(keep0 ? w.x : 0.0f, keep1 ? w.y : 0.0f);
}

}  // namespace walk
}  // namespace icgs
