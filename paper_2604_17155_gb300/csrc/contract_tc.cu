// contract_tc.cu -- the blend-accumulate walk (Eq. 4-6) with its per-tile contraction on the
// 5th-generation tensor cores (tcgen05), for 16-bit targets with 16..64 channels.
//
// Per tile and batch of MG = 64 Gaussians (the MMA's M; 64 rather than 128 halves the weight
// operand, so that 3-4 CTAs fit on an SM), the S terms of Eq. 6 summed over the tile's 256 pixels
// form a dense product
//     D[g][n] = sum_p W[g][p] * B[n][p],   W[g][p] = alpha T of Gaussian g at pixel p (Eq. 4),
// with B's row 0 all ones, so that the same product also yields V = sum_p W[g][p] (Eq. 5), and rows 1..KT
// the tile's target channels. Four walker warps evaluate W by 8-lane groups (groupwalk.cuh, one
// pixel pair a lane) and store a pair as two FP16 values into a K-major, 128-byte-swizzled
// shared-memory operand; the tile's targets (BF16 or FP16) are transposed once into B as FP16. Both operands are scaled by powers of two -- W by 2^14 (the walk carries T scaled
// so), the targets so that the tile's largest magnitude lands in [2^14, 2^15) -- which makes every
// BF16 target exact in FP16, keeps small weights out of FP16's subnormal range, and is undone exactly
// in the epilogue. One thread issues 16 tcgen05.mma (kind::f16, M=MG, N=KT+8, K=16, FP32
// accumulation in TMEM) and commits them to an mbarrier. Four helper warps, one per K block of W and TMEM
// quarter, wait for them, clear the rows of W that were written, read D back with tcgen05.ld and add
// (V, S_0..S_{KT-1}) to the accumulator -- one atomic group per (Gaussian, tile) -- and stage the records
// and hit lists of the batch after next, all beside the walkers' next batch. The MMA's K index runs over
// each warp's 8x8 pixel block in turn, so a warp owns one K block of W. A batch costs one CTA barrier.
//
// What bounds it: instruction issue (about 70% of the cycles, with 31 warps per SM; the ALU pipe 56%), then the wait
// for a batch's MMAs and sums; shared memory takes 41% of its wavefronts besides the MMAs' own reads of W and B.
// Measured at 16 channels (3M Gaussians, 200 views of 1600 x 1060), each step against the tree before it: 101.8 ms
// with one list per 8x4 warp block and 256 threads; 94.3 with groups and 128 threads; 89.5 with one barrier a
// batch; 85.2 with the geometry stored once; 83 with only the written rows cleared; 80.4 with the helper warps, and
// 81.5 as it is now. 64 channels (1M Gaussians, 150 views): 47.6 -> 39.1, and 36.9 with the sums as fragments. Of the
// 80.4, the atomics take 1.5 and three quarters of the MMAs 6. Tried and slower: batches of 48 (84.8 against
// 81.9), alpha one pixel at a time (83.6 against 81.2).
//
// Every wait on the mbarrier is bounded in time (1 s by %globaltimer): past the limit the kernel
// sets kFlagTimeout in the status block (reported as ICGS_ERR_DEVICE_TIMEOUT), waits once more
// (also bounded) for the MMAs it issued, frees its TMEM and returns. A diagnostic entry point
// (icgs_debug_tc_wait) shortens the limit and can leave the MMAs unissued, so that a test drives a
// wait past its limit with nothing in flight.
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include "icgs_device.cuh"
#include "icgs_internal.h"
#include "groupwalk.cuh"
#include "walk.cuh"

namespace icgs {

namespace {

using namespace walk;

constexpr int kG = 128;                 // rows of the self-test MMA (the walk uses MG = 64)
constexpr int kKPix = 256;              // pixels per tile (MMA K in total, 16 instructions of 16)
constexpr uint64_t kWaitLimitNs = 1000000000ull;  // bounded mbarrier waits give up after 1 s
constexpr uint32_t kTmemCols = 128;     // TMEM columns of the self-test (N <= 80)

// ---- inline PTX ---------------------------------------------------------------------------
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

__device__ __forceinline__ void tmem_alloc(uint32_t* dst, uint32_t ncols) {
  asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_u32(dst)), "r"(ncols)
               : "memory");
}
__device__ __forceinline__ void tmem_relinquish() {
  asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
}
__device__ __forceinline__ void tmem_dealloc(uint32_t taddr, uint32_t ncols) {
  asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(taddr), "r"(ncols) : "memory");
}
__device__ __forceinline__ void tc_fence_before() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void tc_fence_after() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// Named barriers of some of the CTA's warps (barrier 0 is __syncthreads): wait with, or only announce, the
// count threads that take part.
template <int ID, int COUNT>
__device__ __forceinline__ void bar_sync() {
  asm volatile("barrier.cta.sync %0, %1;" ::"n"(ID), "n"(COUNT) : "memory");
}
template <int ID, int COUNT>
__device__ __forceinline__ void bar_arrive() {
  asm volatile("barrier.cta.arrive %0, %1;" ::"n"(ID), "n"(COUNT) : "memory");
}

__device__ __forceinline__ void mbar_init(uint64_t* mbar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_u32(mbar)), "r"(count) : "memory");
  asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
}
__device__ __forceinline__ bool mbar_try_wait(uint64_t* mbar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}\n"
      : "=r"(ok)
      : "r"(smem_u32(mbar)), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ uint64_t global_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
// Bounded wait; returns false (and the caller reports a timeout) once limit_ns have passed. The clock
// is read only after a first try has failed: a read costs more than the usual rest of the wait.
__device__ __forceinline__ bool mbar_wait_bounded(uint64_t* mbar, uint32_t parity, uint64_t limit_ns = kWaitLimitNs) {
  if (mbar_try_wait(mbar, parity)) return true;
  const uint64_t t0 = global_ns();
  while (!mbar_try_wait(mbar, parity))
    if (global_ns() - t0 > limit_ns) return false;
  return true;
}

// D[tmem] (+)= A[smem] * B[smem]^T, both operands K-major, kind::f16 (BF16 or FP16 in, FP32 out)
__device__ __forceinline__ void umma_f16(uint32_t d_tmem, uint64_t a_desc, uint64_t b_desc, uint32_t idesc,
                                         uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(a_desc), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive on the mbarrier once every MMA this thread issued has completed.
__device__ __forceinline__ void umma_commit(uint64_t* mbar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_u32(mbar))
               : "memory");
}
// 16 consecutive 32-bit columns of this warp's 32 TMEM lanes (one lane per thread).
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&r)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
        "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr)
      : "memory");
}
// 8 consecutive columns of 16 TMEM lanes by the whole warp, as an accumulator fragment: thread t gets columns
// 2 (t % 4), + 1 of lane t / 4 in r[0], r[1] and of lane t / 4 + 8 in r[2], r[3].
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, uint32_t* r) {
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x1.b32 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_wait_ld() { asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory"); }

// ---- operand layout -------------------------------------------------------------------------
// A [rows x 256] 16-bit matrix stored K-major with the 128-byte swizzle: four K blocks of 64
// elements, each block rows x 128 bytes, rows grouped by 8 into 1024-byte atoms, and the 16-byte
// chunk index of each row XOR-ed with the row's index inside its atom.
__device__ __forceinline__ uint32_t kmajor_sw128(int row, int k, int rows) {
  return (uint32_t)((k >> 6) * (rows * 128) + (row >> 3) * 1024 + (row & 7) * 128 +
                    ((((k & 63) >> 3) ^ (row & 7)) << 4) + ((k & 7) << 1));
}

// Shared-memory matrix descriptor (tcgen05 format): start address >> 4 in bits 0-13, leading byte
// offset >> 4 in bits 16-29 (unused for swizzled K-major; 1 by convention), stride byte offset
// >> 4 in bits 32-45 (1024 B between 8-row atoms), descriptor version 1 in bits 46-47, layout type
// in bits 61-63 (2 = 128-byte swizzle).
__device__ __forceinline__ uint64_t desc_kmajor_sw128(uint32_t saddr, uint32_t sbo = 1024) {
  return (uint64_t)((saddr & 0x3FFFFu) >> 4) | ((uint64_t)1 << 16) | ((uint64_t)(sbo >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

// Instruction descriptor of kind::f16: D format F32 (bits 4-5 = 1), A and B format (bits 7-9,
// 10-12: 0 = F16, 1 = BF16), both K-major (bits 15, 16 = 0), N >> 3 in bits 17-22, M >> 4 in
// bits 24-28.
__host__ __device__ constexpr uint32_t idesc_f16(int M, int N, bool bf16) {
  return (1u << 4) | ((bf16 ? 1u : 0u) << 7) | ((bf16 ? 1u : 0u) << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

constexpr int kWScaleExp = 14;  // W is stored as W * 2^14 (W < 1)

__device__ __forceinline__ uint16_t half_bits(float x) { return __half_as_ushort(__float2half_rn(x)); }
__device__ __forceinline__ float target_value(uint16_t raw, bool bf16) {
  return bf16 ? __uint_as_float((uint32_t)raw << 16) : __half2float(__ushort_as_half(raw));
}

// Issues the 16 MMAs of one batch (K = 256 pixels) and commits them to mbar.
template <int NB, int MG = kG>
__device__ __forceinline__ void issue_batch(uint32_t a_addr, uint32_t b_addr, uint32_t d_tmem, uint32_t idesc,
                                            uint64_t* mbar) {
  tc_fence_after();
#pragma unroll
  for (int ks = 0; ks < kKPix / 16; ++ks) {
    const int kb = ks >> 2, kk = ks & 3;
    const uint64_t ad = desc_kmajor_sw128(a_addr + kb * (MG * 128) + kk * 32);
    const uint64_t bd = desc_kmajor_sw128(b_addr + kb * (NB * 128) + kk * 32);
    umma_f16(d_tmem, ad, bd, idesc, ks > 0 ? 1u : 0u);
  }
  umma_commit(mbar);
}

// The accumulator row held in TMEM lane 32 q + l (the lane a thread l of a warp with quarter q
// reads), or -1: M = 128 puts row m in lane m; M = 64 puts row m in lane (m % 16) + 32 (m / 16),
// i.e. rows 16q..16q+15 in the first 16 lanes of quarter q.
template <int MG>
__device__ __forceinline__ int tmem_row_of_lane(int q, int l) {
  return MG == 128 ? q * 32 + l : (l < 16 ? q * 16 + l : -1);
}

// ---- self-test: D[M x N] = A[M x 256] B[N x 256]^T through the same layout and MMA path ----
// (M = 64 or 128). D_lanes, when given, receives the raw contents of all 128 TMEM lanes.
template <int NB, bool BF16, int MG>
__global__ void __launch_bounds__(256) k_tc_selftest(const uint16_t* __restrict__ A, const uint16_t* __restrict__ Bm,
                                                     float* __restrict__ D, float* __restrict__ D_lanes,
                                                     DevStatus* status) {
  extern __shared__ uint8_t smem_raw[];
  const uint32_t raw = smem_u32(smem_raw);
  uint8_t* base = smem_raw + (((raw + 1023u) & ~1023u) - raw);
  uint8_t* A_s = base;
  uint8_t* B_s = base + kG * kKPix * 2;
  uint64_t* mbar = reinterpret_cast<uint64_t*>(B_s + NB * kKPix * 2);
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(mbar + 1);
  for (int e = threadIdx.x; e < MG * kKPix; e += blockDim.x) {
    const int m = e / kKPix, k = e % kKPix;
    *reinterpret_cast<uint16_t*>(A_s + kmajor_sw128(m, k, MG)) = A[e];
  }
  for (int e = threadIdx.x; e < NB * kKPix; e += blockDim.x) {
    const int nn = e / kKPix, k = e % kKPix;
    *reinterpret_cast<uint16_t*>(B_s + kmajor_sw128(nn, k, NB)) = Bm[e];
  }
  if (threadIdx.x == 0) mbar_init(mbar, 1);
  if (threadIdx.x < 32) {
    tmem_alloc(tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  if (threadIdx.x == 0) issue_batch<NB, MG>(smem_u32(A_s), smem_u32(B_s), tmem, idesc_f16(MG, NB, BF16), mbar);
  const bool ok = __all_sync(0xFFFFFFFFu, mbar_wait_bounded(mbar, 0));  // warp-uniform for tcgen05.ld
  if (!ok && (threadIdx.x & 31) == 0) atomicOr(&status->flags, kFlagTimeout);
  tc_fence_after();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (warp < 4 && ok) {
    const int L = warp * 32 + lane;  // the TMEM lane this thread reads
    const int row = tmem_row_of_lane<MG>(warp, lane);
#pragma unroll
    for (int c0 = 0; c0 < NB; c0 += 16) {
      uint32_t r[16];
      tmem_ld16(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0, r);
      tmem_wait_ld();
#pragma unroll
      for (int q = 0; q < 16; ++q) {
        if (row >= 0) D[row * NB + c0 + q] = __uint_as_float(r[q]);
        if (D_lanes) D_lanes[L * NB + c0 + q] = __uint_as_float(r[q]);
      }
    }
  }
  if (!ok) mbar_wait_bounded(mbar, 0);
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

// ---- the accumulate walk with the tensor-core contraction --------------------------------------
// MG: Gaussians per batch, the MMA M. TMEM columns: the accumulator width rounded up to a power of two.
// Columns of B and of the accumulator: V, the KT target channels and zeros to a multiple of 8 (an M of 64
// takes N in steps of 8).
template <int KT>
__host__ __device__ constexpr int tc_cols() {
  return KT + 8;
}

template <int NB>
__host__ __device__ constexpr uint32_t tmem_cols() {
  return NB <= 32 ? 32u : (NB <= 64 ? 64u : 128u);
}

template <int KT, int MG>
__host__ __device__ constexpr int tc_ctas_per_sm() {
  return MG == 64 ? (KT <= 24 ? 4 : 3) : 2;
}

// What sits in front of the operands: the barrier and flags, the staged geometry and the hit lists of two
// batches. The geometry is stored once, not twice: the MMAs and the walk share the shared-memory
// bandwidth, and the moves cost less than the wider loads (masks walk 88.1 -> 85.2 ms).
constexpr int kTcWalkers = GroupCfg<1>::kThreads;  // warps 0-3
constexpr int kTcThreads = 2 * kTcWalkers;         // and the helpers, warps 4-7
struct TcBatch {
  uint64_t mbar;
  uint32_t tmem_slot;
  uint32_t timeout[2];   // set by a thread whose wait gave up, by the parity of the batch
  uint32_t tmax[8];
  uint32_t alive[2][4];  // by parity and walker warp: groups with a pixel that has not stopped
  uint32_t counts[2][kBatch / 4];  // list lengths by parity and group
  GroupGeo<false> geo[2];
  float2 lim[kBatch];
  GroupLists<1, true> lists[2];
};
constexpr uint32_t kTcFront = (sizeof(TcBatch) + 15) / 16 * 16;

template <int KT, bool BF16_TARGETS, int MG>
__global__ void __launch_bounds__(kTcThreads, tc_ctas_per_sm<KT, MG>()) k_blend_accumulate_tc(
    const uint32_t* __restrict__ tile_off, const uint64_t* __restrict__ entries, uint32_t capacity,
    const ProjRec* __restrict__ rec, int64_t n, int width, int height, int tiles_x, int tiles,
    const uint16_t* __restrict__ targets, int K, int cam0, float* __restrict__ acc, int RS,
    int64_t acc_cam_stride, DevStatus* status, uint64_t wait_limit_ns, bool issue_mma) {
  static_assert(MG == 64 && MG == kBatch, "staging and epilogue map Gaussian g to TMEM lane g % 16 of quarter g / 16");
  constexpr int NB = tc_cols<KT>();  // the row of ones (V), the target channels, rows of zeros
  extern __shared__ uint8_t smem_raw[];
  // The barrier, the flags and the staged batches sit in front of the operands, which start at the next
  // 1024-byte boundary. A base that is not 128-byte aligned is reported (kFlagLayout) before any work.
  const uint32_t raw = smem_u32(smem_raw);
  if (raw & 127u) {
    if (threadIdx.x == 0) atomicOr(&status->flags, kFlagLayout);
    return;
  }
  TcBatch& s = *reinterpret_cast<TcBatch*>(smem_raw);
  uint8_t* base = smem_raw + (((raw + kTcFront + 1023u) & ~1023u) - raw);
  uint8_t* A_s = base;                                 // MG x 256 (32 KB)
  uint8_t* B_s = base + MG * kKPix * 2;                // NB x 256

  // Walkers and helpers are numbered alike: tid, and warp 0-3 by K block and TMEM quarter.
  const bool walker = threadIdx.x < kTcWalkers;
  const int tid = threadIdx.x & (kTcWalkers - 1);
  const GroupCtx<1> c = group_ctx<1>(tile_off, capacity, tiles, tiles_x, width, height, tid);
  if (c.len == 0) return;  // uniform: nothing binned to this tile
  const int warp = tid >> 5, lane = tid & 31;
  // the MMA's K index of the thread's first pixel (the second is the next): 64 per warp block, row by row
  const int p = warp * 64 + ((c.py % kTile) & 7) * 8 + ((c.px % kTile) & 7);
  const unsigned long long* list = reinterpret_cast<const unsigned long long*>(entries);
  const ProjRec* rec_cam = rec + (int64_t)c.j * n;
  const uint32_t list_end = c.b + c.len;
  // helpers: the indices of the first four batches and the records of the first
  uint32_t id0 = 0, id1 = 0, id2 = 0, id3 = 0;
  GroupFetch fetch = {make_float4(0.0f, 0.0f, 0.0f, 0.0f), make_float4(0.0f, 0.0f, 0.0f, 0.0f)};
  if (!walker) {
    id0 = group_id<1>(list, c.b, list_end, n, tid);
    id1 = group_id<1>(list, c.b + MG, list_end, n, tid);
    id2 = group_id<1>(list, c.b + 2 * MG, list_end, n, tid);
    id3 = group_id<1>(list, c.b + 3 * MG, list_end, n, tid);
    fetch = group_fetch(id0, rec_cam);
  }

  // B: the tile's targets, transposed to [channel][pixel] and scaled by 2^sexp (the tile's largest
  // magnitude in [2^14, 2^15)) in rows 1..KT, below a row of ones, so that D's columns lie as the accumulator
  // row (V, S_0, S_1, ..) does; the rows left are zero. A walker takes the first half of its pixels' channels,
  // the helper of the same number the second.
  float t_scale_inv;
  {
    constexpr int KH = KT / 2;
    const int kh = walker ? 0 : KH;
    const uint16_t* src = targets + ((((int64_t)(cam0 + c.j) * height + c.py) * width + c.px) * K) + kh;
    // the two pixels' channels, loaded 16 (or, in halves of 12, 8) bytes at a time when the rows allow it
    uint32_t tv[KH];  // (first pixel's value, second pixel's value)
    if (KH % 8 == 0 && c.in1[0] && K == KT && (reinterpret_cast<uintptr_t>(src) & 15u) == 0) {
#pragma unroll
      for (int q = 0; q < KH / 8; ++q) {
        const uint4 u = __ldg(reinterpret_cast<const uint4*>(src) + q);
        const uint4 v = __ldg(reinterpret_cast<const uint4*>(src + K) + q);
        const uint32_t a[4] = {u.x, u.y, u.z, u.w}, b[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          tv[8 * q + 2 * h] = __byte_perm(a[h], b[h], 0x5410);
          tv[8 * q + 2 * h + 1] = __byte_perm(a[h], b[h], 0x7632);
        }
      }
    } else if (KH % 8 != 0 && c.in1[0] && K == KT && (reinterpret_cast<uintptr_t>(src) & 7u) == 0) {
#pragma unroll
      for (int q = 0; q < KH / 4; ++q) {
        const uint2 u = __ldg(reinterpret_cast<const uint2*>(src) + q);
        const uint2 v = __ldg(reinterpret_cast<const uint2*>(src + K) + q);
        tv[4 * q] = __byte_perm(u.x, v.x, 0x5410);
        tv[4 * q + 1] = __byte_perm(u.x, v.x, 0x7632);
        tv[4 * q + 2] = __byte_perm(u.y, v.y, 0x5410);
        tv[4 * q + 3] = __byte_perm(u.y, v.y, 0x7632);
      }
    } else {
#pragma unroll
      for (int k = 0; k < KH; ++k) {
        const uint32_t a = c.in0[0] && kh + k < K ? src[k] : 0u, b = c.in1[0] && kh + k < K ? src[K + k] : 0u;
        tv[k] = a | (b << 16);
      }
    }
    // the largest magnitude: non-negative floats order like their bit patterns, in 16 bits too
    uint32_t m16 = 0u;
#pragma unroll
    for (int k = 0; k < KH; ++k) m16 = __vmaxu2(m16, tv[k] & 0x7FFF7FFFu);
    uint32_t m = max(m16 & 0xFFFFu, m16 >> 16);
    if (m >= (BF16_TARGETS ? 0x7F80u : 0x7C00u)) atomicOr(&status->flags, kFlagNonfinite);
    m = __reduce_max_sync(0xFFFFFFFFu, m);
    if (lane == 0) s.tmax[threadIdx.x >> 5] = m;
    if (threadIdx.x == 0) {
      mbar_init(&s.mbar, 1);
      s.timeout[0] = s.timeout[1] = 0u;
    }
    if (threadIdx.x < 32) {
      tmem_alloc(&s.tmem_slot, tmem_cols<NB>());
      tmem_relinquish();
    }
    __syncthreads();
    m = s.tmax[0];
#pragma unroll
    for (int w = 1; w < 8; ++w) m = max(m, s.tmax[w]);
    const float gmax = target_value((uint16_t)m, BF16_TARGETS);
    int e = 0;
    if (gmax > 0.0f && isfinite(gmax)) frexpf(gmax, &e);  // gmax in [2^(e-1), 2^e)
    const int sexp = gmax > 0.0f ? 15 - e : 0;           // gmax * 2^sexp in [2^14, 2^15)
    t_scale_inv = ldexpf(1.0f, -(sexp + kWScaleExp));
    // 2^sexp as a product of two powers of two that are normal floats (sexp is in -113..148)
    const float s1 = ldexpf(1.0f, sexp / 2), s2 = ldexpf(1.0f, sexp - sexp / 2);
#pragma unroll
    for (int k = 0; k < KH; ++k) {
      const float x = target_value((uint16_t)(tv[k] & 0xFFFFu), BF16_TARGETS) * s1 * s2;
      const float y = target_value((uint16_t)(tv[k] >> 16), BF16_TARGETS) * s1 * s2;
      *reinterpret_cast<__half2*>(B_s + kmajor_sw128(1 + kh + k, p, NB)) = __floats2half2_rn(x, y);
    }
    if (walker) *reinterpret_cast<uint32_t*>(B_s + kmajor_sw128(0, p, NB)) = 0x3C003C00u;
    else
#pragma unroll
      for (int k = KT + 1; k < NB; ++k) *reinterpret_cast<uint32_t*>(B_s + kmajor_sw128(k, p, NB)) = 0u;
  }
  const float v_scale_inv = ldexpf(1.0f, -kWScaleExp);
  constexpr float kT0 = (float)(1 << kWScaleExp);  // the transmittance carries the factor 2^14 of W
  GroupT<1> T(c, kT0);
  uint32_t npairs = 0, phase = 0;
  bool ok = true;
  const int n_first = (int)min((uint32_t)MG, c.len);
  uint4* const w_block = reinterpret_cast<uint4*>(A_s + warp * (MG * 128));
  uint32_t listed0[2] = {0u, 0u}, listed1[2] = {0u, 0u};  // rows of W that the walk of this batch / the next writes
  if (!walker) {
    if (tid < 2) group_pad(s.geo[tid]);
    // the first two batches' geometry and lists, and W cleared (block w by helper warp w)
    group_put<1>(fetch, n_first, c.ox, c.oy, s.geo[0], s.lim, tid);
    fetch = group_fetch(id1, rec_cam);
#pragma unroll
    for (int i = 0; i < MG * 128 / 16; i += 32) w_block[i + lane] = make_uint4(0, 0, 0, 0);
    bar_sync<2, kTcWalkers>();
    group_lists(s.geo[0], s.lim, s.lists[0], c, n_first, 0xFu, tid, nullptr, listed0, s.counts[0]);
    if (MG < c.len) {
      const int n_second = (int)min((uint32_t)MG, c.len - MG);
      bar_sync<2, kTcWalkers>();  // lim has been read
      group_put<1>(fetch, n_second, c.ox, c.oy, s.geo[1], s.lim, tid);
      fetch = group_fetch(id2, rec_cam);
      bar_sync<2, kTcWalkers>();
      group_lists(s.geo[1], s.lim, s.lists[1], c, n_second, 0xFu, tid, nullptr, listed1, s.counts[1]);
    }
  }
  fence_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s.tmem_slot;

  // Whether a batch follows the one of parity buf that starts at start, from what every walker warp wrote
  // before the CTA barrier.
  auto more_after = [&](uint32_t start, uint32_t buf) -> bool {
    return start + MG < c.len && (s.alive[buf][0] | s.alive[buf][1] | s.alive[buf][2] | s.alive[buf][3]) != 0u;
  };

  if (walker) {
    // Walk the lists of a batch into W, hand W to the tensor cores, wait until it is clear again.
    const uint32_t a_addr = smem_u32(A_s), b_addr = smem_u32(B_s);
    constexpr uint32_t kIdesc = idesc_f16(MG, NB, false);
    // kmajor_sw128(g, p, MG) in terms of the list entry o = 16 g: 8 o + ((o & 0x70) ^ pixel part)
    char* const w_base = reinterpret_cast<char*>(A_s + warp * (MG * 128));
    const uint32_t w_pix = (uint32_t)((((p & 63) >> 3) << 4) | ((p & 7) << 1));
    for (uint32_t start = 0, buf = 0;; start += MG, buf ^= 1u) {
      // lists may still name groups whose pixels have all stopped since they were built
      const bool live = (group_alive(T.alive()) >> (lane >> 3)) & 1u;
      const int steps = (int)__reduce_max_sync(0xFFFFFFFFu, live ? s.counts[buf][c.group] : 0u);
      const GroupGeo<false>& geo = s.geo[buf];
      const uint16_t* const my_list = s.lists[buf].row[c.group];
      for (int i = 0; i < steps; i += 2) {
        const uint2 o = GroupLists<1, true>::pair(my_list, i);
        const uint32_t o1 = o.x, o2 = o.y;
        const GroupAlpha<1> a1 = group_alpha(geo, o1, c), a2 = group_alpha(geo, o2, c);  // independent of T
        const float2 w1 = group_take<true, kWScaleExp>(a1, T, npairs).v[0];
        const float2 w2 = group_take<true, kWScaleExp>(a2, T, npairs).v[0];
        if (o1 != kGPad)
          *reinterpret_cast<__half2*>(w_base + o1 * 8 + ((o1 & 0x70u) ^ w_pix)) = __floats2half2_rn(w1.x, w1.y);
        if (o2 != kGPad)
          *reinterpret_cast<__half2*>(w_base + o2 * 8 + ((o2 & 0x70u) ^ w_pix)) = __floats2half2_rn(w2.x, w2.y);
      }
      const uint32_t alive = group_alive(T.alive());
      if (lane == 0) s.alive[buf][warp] = alive;
      fence_async_smem();
      tc_fence_before();
      bar_sync<1, kTcWalkers>();  // W is written
      if (warp == 0) {
        if (start > 0) bar_sync<3, kTcWalkers + 32>();  // the helpers have read the last batch's sums
        if (lane == 0 && issue_mma) {
          issue_batch<NB, MG>(a_addr, b_addr, tmem, kIdesc, &s.mbar);
        }
        __syncwarp();
      }
      __syncthreads();
      if (s.timeout[buf] || !more_after(start, buf)) break;
    }
  } else {
    // Wait for a batch's MMAs, clear W, and then, beside the next batch's walk, add the sums and prepare the
    // geometry and lists of the batch after it.
    constexpr int kBlocks = KT / 8 + 1;                      // 8-column blocks of (V, S)
    const int ra = lane >> 2, rb = ra + 8, q2 = 2 * (lane & 3);  // the rows and columns of the thread's fragment
    float* acc_cam = acc + (int64_t)c.j * acc_cam_stride;
    const uint32_t trow = tmem + ((uint32_t)(warp * 32) << 16);
    for (uint32_t start = 0, buf = 0;; start += MG, buf ^= 1u) {
      // warp-uniform: tcgen05.ld needs whole warps
      ok = __all_sync(0xFFFFFFFFu, mbar_wait_bounded(&s.mbar, phase, wait_limit_ns));
      phase ^= 1u;
      tc_fence_after();
      if (ok) {  // the rows that the walk wrote (about a third), four of 128 bytes at a time
#pragma unroll
        for (int i = 0; i < MG * 128 / 16; i += 32)
          if ((listed0[i / 256] >> (lane >> 3)) & (1u << ((i / 8) & 31))) w_block[i + lane] = make_uint4(0, 0, 0, 0);
        fence_async_smem();
      } else {
        s.timeout[buf] = 1u;
      }
      __syncthreads();
      if (s.timeout[buf]) break;
      const bool more = more_after(start, buf);
      // The sums stream through registers 8 columns at a time as accumulator fragments: four neighbouring
      // threads hold 32 consecutive bytes of a row, so an instruction's 8-byte atomics fall in whole sectors
      // of 8 rows (with a row per thread, 16-byte atomics touched 16 rows: the 64-channel walk took
      // 39.1 ms, then 36.7; the 16-channel one, with a third of the sectors, 80.3 and 80.4).
      const int nb = (int)min((uint32_t)MG, c.len - start);
      const uint32_t id_a = __shfl_sync(0xFFFFFFFFu, id0, 2 * ra), id_b = __shfl_sync(0xFFFFFFFFu, id0, 2 * rb);
      float* const dst_a = acc_cam + (int64_t)id_a * RS + q2;
      float* const dst_b = acc_cam + (int64_t)id_b * RS + q2;
      bool add_a = false, add_b = false;
#pragma unroll
      for (int q = 0; q < kBlocks; q += 4) {
        uint32_t r[16];
#pragma unroll
        for (int h = 0; h < 4; ++h)
          if (q + h < kBlocks) tmem_ld_frag(trow + (uint32_t)(8 * (q + h)), r + 4 * h);
        tmem_wait_ld();
        if (q + 4 >= kBlocks && more) {  // every column is in registers: the next batch's MMAs may write
          tc_fence_before();
          bar_arrive<3, kTcWalkers + 32>();
        }
        if (q == 0) {  // V, column 0: a row that nothing reached is left alone
          const float va = __uint_as_float(__shfl_sync(0xFFFFFFFFu, r[0], lane & 28));
          const float vb = __uint_as_float(__shfl_sync(0xFFFFFFFFu, r[2], lane & 28));
          add_a = 16 * warp + ra < nb && va > 0.0f;
          add_b = 16 * warp + rb < nb && vb > 0.0f;
        }
#pragma unroll
        for (int h = 0; h < 4; ++h) {
          if (q + h >= kBlocks) continue;
          const int col = 8 * (q + h);
          const float s0 = q + h == 0 && q2 == 0 ? v_scale_inv : t_scale_inv;
          const bool in = col + q2 < RS;  // RS is even
          if (add_a && in)
            atomicAdd(reinterpret_cast<float2*>(dst_a + col),
                      make_float2(__uint_as_float(r[4 * h]) * s0, __uint_as_float(r[4 * h + 1]) * t_scale_inv));
          if (add_b && in)
            atomicAdd(reinterpret_cast<float2*>(dst_b + col),
                      make_float2(__uint_as_float(r[4 * h + 2]) * s0, __uint_as_float(r[4 * h + 3]) * t_scale_inv));
        }
        __syncwarp();
      }
      if (!more) break;
      listed0[0] = listed1[0];
      listed0[1] = listed1[1];
      listed1[0] = listed1[1] = 0u;
      const uint32_t after = start + 2 * MG;  // the batch that takes this one's buffers
      if (after < c.len) {
        const int na = (int)min((uint32_t)MG, c.len - after);
        group_put<1>(fetch, na, c.ox, c.oy, s.geo[buf], s.lim, tid);
        fetch = group_fetch(id3, rec_cam);
        const uint32_t alive = s.alive[buf][warp];
        bar_sync<2, kTcWalkers>();
        group_lists(s.geo[buf], s.lim, s.lists[buf], c, na, alive, tid, nullptr, listed1, s.counts[buf]);
      }
      id0 = id1;
      id1 = id2;
      id2 = id3;
      id3 = group_id<1>(list, c.b + start + 4 * MG, list_end, n, tid);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (s.timeout[0] | s.timeout[1]) {
    if (threadIdx.x == 0) atomicOr(&status->flags, kFlagTimeout);
    if (!ok) mbar_wait_bounded(&s.mbar, phase ^ 1u, wait_limit_ns);  // a last chance for the outstanding MMAs
  }
  if (walker) add_pair_count(npairs, status);
  tc_fence_before();
  __syncthreads();
  if (threadIdx.x < 32) {
    tc_fence_after();
    tmem_dealloc(tmem, tmem_cols<NB>());
  }
}

template <int NB>
constexpr size_t selftest_smem() {
  return 1024 + (size_t)kG * kKPix * 2 + (size_t)NB * kKPix * 2 + 16;
}
// the barrier, flags and staged batch with up to 1023 bytes of alignment, W, and B
template <int KT, int MG>
constexpr size_t tc_smem() {
  return kTcFront + 1023 + (size_t)MG * kKPix * 2 + (size_t)tc_cols<KT>() * kKPix * 2;
}
// CTAs per SM that the shared memory admits: each CTA's share rounded up to 1 KB, plus 1 KB the
// system reserves per CTA, out of the SM's 228 KB
template <int KT, int MG>
constexpr int tc_smem_ctas() {
  return (int)((228 * 1024) / ((tc_smem<KT, MG>() + 1023) / 1024 * 1024 + 1024));
}
static_assert(tc_smem_ctas<16, 64>() >= tc_ctas_per_sm<16, 64>(), "shared memory of the 16-channel walk");
static_assert(tc_smem_ctas<24, 64>() >= tc_ctas_per_sm<24, 64>(), "shared memory of the 24-channel walk");
static_assert(tc_smem_ctas<48, 64>() >= tc_ctas_per_sm<48, 64>(), "shared memory of the 48-channel walk");
static_assert(tc_smem_ctas<32, 64>() >= tc_ctas_per_sm<32, 64>(), "shared memory of the 32-channel walk");
static_assert(tc_smem_ctas<64, 64>() >= tc_ctas_per_sm<64, 64>(), "shared memory of the 64-channel walk");

// Diagnostic settings of this host thread (icgs_debug_tc_wait): the walk's wait limit and whether
// it issues its MMAs.
thread_local uint64_t g_wait_limit_ns = kWaitLimitNs;
thread_local bool g_issue_mma = true;

template <int KT, bool BF16_TARGETS>
void accumulate_tc(const Problem& p, int cb, int cam0, const void* targets, const Workspace& ws, cudaStream_t s) {
  constexpr int MG = 64;
  const size_t smem = tc_smem<KT, MG>();
  cudaFuncSetAttribute(k_blend_accumulate_tc<KT, BF16_TARGETS, MG>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                       (int)smem);
  cudaFuncSetAttribute(k_blend_accumulate_tc<KT, BF16_TARGETS, MG>, cudaFuncAttributePreferredSharedMemoryCarveout,
                       (int)cudaSharedmemCarveoutMaxShared);
  const int64_t stride = p.L == 0 ? 0 : p.n * (int64_t)p.acc_stride;
  k_blend_accumulate_tc<KT, BF16_TARGETS, MG><<<cb * p.tiles, kTcThreads, smem, s>>>(
      ws.tile_off, ws.entries, p.capacity, ws.rec, p.n, p.width, p.height, p.tiles_x, p.tiles,
      static_cast<const uint16_t*>(targets), p.K, cam0, ws.acc, p.acc_stride, stride, ws.status, g_wait_limit_ns,
      g_issue_mma);
  note_launches(1);
}

// The smallest operand that holds the channels: MMAs, shared memory and sums grow with its width, and up to 24
// four CTAs fit an SM. Against widths of 16, 32 and 64 only (300k Gaussians, 48 cameras of 800 x 600): 21
// channels 4.87 -> 4.30 ms, 24 5.07 -> 4.12, 33 6.09 -> 5.58, 48 7.24 -> 5.27.
template <bool BF16_TARGETS>
void accumulate_tc_dispatch(const Problem& p, int cb, int cam0, const void* targets, const Workspace& ws,
                            cudaStream_t s) {
  if (p.K <= 16) accumulate_tc<16, BF16_TARGETS>(p, cb, cam0, targets, ws, s);
  else if (p.K <= 24) accumulate_tc<24, BF16_TARGETS>(p, cb, cam0, targets, ws, s);
  else if (p.K <= 32) accumulate_tc<32, BF16_TARGETS>(p, cb, cam0, targets, ws, s);
  else if (p.K <= 48) accumulate_tc<48, BF16_TARGETS>(p, cb, cam0, targets, ws, s);
  else accumulate_tc<64, BF16_TARGETS>(p, cb, cam0, targets, ws, s);
}

}  // namespace

void set_tc_wait_diagnostic(int64_t limit_ns, bool issue_mma) {
  g_wait_limit_ns = limit_ns > 0 ? (uint64_t)limit_ns : kWaitLimitNs;
  g_issue_mma = issue_mma;
}

bool tc_accumulate_applies(const Problem& p, int dtype) {
  return p.precision == 1 && (dtype == 1 || dtype == 2) && p.K >= 16 && p.K <= 64;
}

void launch_blend_accumulate_tc(const Problem& p, int cb, int cam0, const void* targets, int dtype,
                                const Workspace& ws, cudaStream_t s) {
  if (dtype == 1) accumulate_tc_dispatch<true>(p, cb, cam0, targets, ws, s);
  else accumulate_tc_dispatch<false>(p, cb, cam0, targets, ws, s);
}

cudaError_t launch_tc_selftest(const uint16_t* A, int M, const uint16_t* B, int N, bool bf16, float* D, float* D_lanes,
                               DevStatus* status, cudaStream_t s) {
#define ICGS_ST(NB, BF, MG)                                                                                    \
  do {                                                                                                         \
    cudaFuncSetAttribute(k_tc_selftest<NB, BF, MG>, cudaFuncAttributeMaxDynamicSharedMemorySize,             \
                         (int)selftest_smem<NB>());                                                           \
    k_tc_selftest<NB, BF, MG><<<1, 256, selftest_smem<NB>(), s>>>(A, B, D, D_lanes, status);                   \
  } while (0)
#define ICGS_ST_M(NB, BF)                \
  do {                                   \
    if (M == 64) ICGS_ST(NB, BF, 64);    \
    else ICGS_ST(NB, BF, 128);           \
  } while (0)
  if (M != 64 && M != 128) return cudaErrorInvalidValue;
  if (N == 32 && bf16) ICGS_ST_M(32, true);
  else if (N == 32) ICGS_ST_M(32, false);
  else if (N == 80 && bf16) ICGS_ST_M(80, true);
  else if (N == 80) ICGS_ST_M(80, false);
  else return cudaErrorInvalidValue;
#undef ICGS_ST_M
#undef ICGS_ST
  return cudaGetLastError();
}

}  // namespace icgs
