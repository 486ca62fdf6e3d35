// Split-precision GEMM on the sm_103a tensor cores (tcgen05 + TMA + TMEM).
//
// C = op(A) op(B) for fp64 (or complex fp64) operands, computed as sums of
// low-precision slice products with fp32 accumulation, in one of two
// formats. bf16 x3 (CTM_PREC_SPLIT_BF16):
//   * every fp64 value x is split into three bf16 slices x = s0 + s1 + s2 + e
//     (the slices of x rounded to fp32, each the bf16 rounding of the
//     remainder; |e| <= 2^-24 |x|);
//   * a product keeps the six slice products of order >= 2^-16
//     (s0 t0, s0 t1, s1 t0, s0 t2, s1 t1, s2 t0); the leading s0 t0 is
//     accumulated in its own fp32 accumulator in tensor memory and the five
//     smaller ones in a second, so that their additions cost ulps of a
//     2^-8 smaller running sum, and the two are added once per partial;
// 3xTF32 (CTM_PREC_SPLIT_TF32): x = t0 + t1 + e with tf32 slices of the fp32
// rounding (|e| <= 2^-22 |x|), three products t0 u0 (own accumulator),
// t0 u1 + t1 u0 (second accumulator), tcgen05 kind::tf32 at half the bf16
// rate. Both formats stage 128-byte K rows (64 bf16 or 32 tf32 values), so
// tiles, swizzle and descriptors are shared.
//   * complex data uses the real embedding A_emb = [A_r | A_i] (M x 2K),
//     B_emb = [[B_r, B_i], [-B_i, B_r]] (2K x 2N), C_emb = [C_r | C_i];
//   * K is split over CTAs, at most KB_SPLIT_MAX K blocks of 64 each (the
//     error of an fp32 accumulator grows with the number of MMA steps it
//     takes); fp32 partials are reduced in fp64.
//
// Kernel: one CTA = 128 output rows x BNc (<= 160) output columns; A and B
// slices are K-major, staged by TMA in 64-element (128-byte, 128B-swizzled)
// K blocks through an mbarrier pipeline; one thread issues the
// tcgen05.mma instructions, eight warps drain the accumulator with
// tcgen05.ld. Every mbarrier wait is bounded (2 s of %globaltimer), after
// which the CTA records DEV_MBAR_TIMEOUT, skips its work, frees its tensor
// memory and returns.
#include <cuda.h>
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdio>
#include <cstring>
#include <string>
#include <type_traits>
#include <vector>

#include "common.cuh"
#include "kernels.h"
#include "split_gemm.h"

namespace ctm {

namespace {

constexpr int BM = 128;          // rows per CTA (tcgen05 M)
constexpr int BK = 64;           // bf16 K elements per stage (128 bytes)
constexpr int KROW = 128;        // bytes of one staged K row (either format)
constexpr int MAX_STAGES = 4;    // K blocks staged: as many as shared memory holds
constexpr size_t STAGE_SMEM = 225 * 1024;   // shared memory for stages
constexpr int MAX_BNC = 160;     // columns per CTA
constexpr int A_SLICE_BYTES = BM * KROW;     // 16 KB
constexpr uint64_t WAIT_NS = 2000000000ull;  // bound of every mbarrier wait
#ifndef CTM_KB_SPLIT_MAX
#define CTM_KB_SPLIT_MAX 8
#endif
constexpr int KB_SPLIT_MAX = CTM_KB_SPLIT_MAX;   // K blocks per fp32 partial

// ---------------------------------------------------------------- PTX
__device__ __forceinline__ uint32_t smem_u32(const void* p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}
__device__ __forceinline__ uint64_t globaltimer() {
  uint64_t t;
  asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t));
  return t;
}
__device__ __forceinline__ void mbar_init(uint32_t bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_expect_tx(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(bar), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
      " selp.u32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
// bounded wait for the completion of the phase with the given parity
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, int* err) {
  if (mbar_try(bar, parity)) return true;
  const uint64_t t0 = globaltimer();
  while (true) {
    if (mbar_try(bar, parity)) return true;
    if (globaltimer() - t0 > WAIT_NS) {
      atomicOr(err, DEV_MBAR_TIMEOUT);
      return false;
    }
  }
}
__device__ __forceinline__ void tma_load_3d(uint32_t dst, const CUtensorMap* map, int x, int y,
                                            int z, uint32_t bar) {
  asm volatile(
      "cp.async.bulk.tensor.3d.shared::cluster.global.tile.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4}], [%5];" ::"r"(dst),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(z), "r"(bar)
      : "memory");
}
// shared-memory matrix descriptor: K-major, 128-byte swizzle, 8-row groups
// 1024 bytes apart (sm_100 descriptor version 1)
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFFu) >> 4);
  d |= (uint64_t)1 << 16;               // leading byte offset (unused here)
  d |= (uint64_t)(1024 >> 4) << 32;     // stride byte offset
  d |= (uint64_t)1 << 46;               // descriptor version
  d |= (uint64_t)2 << 61;               // SWIZZLE_128B
  return d;
}
// instruction descriptor of kind::f16: bf16 x bf16 -> f32, both K-major
__host__ __device__ constexpr uint32_t idesc_bf16(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}
__device__ __forceinline__ void mma_bf16(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                         uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
__device__ __forceinline__ void mma_tf32(uint32_t tmem_d, uint64_t adesc, uint64_t bdesc,
                                         uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::tf32 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem_d),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// instruction descriptor of kind::tf32: tf32 x tf32 -> f32 (format code 2),
// both K-major
__host__ __device__ constexpr uint32_t idesc_tf32(int M, int N) {
  return (1u << 4) | (2u << 7) | (2u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

// slice formats: NS slices per operand, NP slice products (the first in its
// own accumulator), element bytes EB, K elements per 128-byte row KE
struct FmtBF16 {
  static constexpr int NS = 3, NP = 6, EB = 2, KE = 64;
};
struct FmtTF32 {
  static constexpr int NS = 2, NP = 3, EB = 4, KE = 32;
};

__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(bar)
      : "memory");
}
// 16 columns from each of two accumulators
__device__ __forceinline__ void tmem_ld16x2(uint32_t ta, uint32_t tb, uint32_t (&r)[16],
                                            uint32_t (&q)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%32];\n"
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31}, [%33];\n"
      "tcgen05.wait::ld.sync.aligned;"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15]),
        "=r"(q[0]), "=r"(q[1]), "=r"(q[2]), "=r"(q[3]), "=r"(q[4]), "=r"(q[5]), "=r"(q[6]), "=r"(q[7]), "=r"(q[8]), "=r"(q[9]), "=r"(q[10]), "=r"(q[11]), "=r"(q[12]), "=r"(q[13]), "=r"(q[14]), "=r"(q[15])
      : "r"(ta), "r"(tb)
      : "memory");
}

struct MmaParams {
  int M;          // output rows
  int Np;         // padded output columns (row length of the partials)
  int BNc;        // columns per CTA, multiple of 16, <= MAX_BNC
  int kb_total;   // K blocks of 64
  int kb_split;   // K blocks per split
  int mt, nchunks, nks;   // work items: row tiles x column chunks x splits
  int stages;     // staged K blocks, 2 .. MAX_STAGES
  float* part;    // [nks][M][Np] fp32 partial sums
  int* err;
};

// A persistent grid: CTA b takes the work items b, b + gridDim.x, ..., each one
// partial sum of a 128 x BNc tile. What bounds it is the operand stream from L2
// (6 slices of a K block, 84 KB at BNc = 96 and 108 KB at 160, feed 1150 and
// 1920 clocks of MMA), so the stream never stops: the producer runs on into the
// next item while the epilogue is at the last one, and the epilogue moves the
// accumulators to registers first, frees them for the next item's MMAs and only
// then stores. With one item per CTA, its start (barriers, tensor memory, the
// first loads) and its epilogue stood between the loads: a 5184 x 10368 corner
// times 298 columns took 193 us, now 144 (87 at the tensor rate), 2880 x 5760
// 63 us, now 50; a launch with one item per CTA is as before (15 us).
// Items are numbered with the chunk fastest, so that the tiles of A that the
// chunks share, and the splits of B that all row tiles share, are read together.
// Warp 0 loads, warp 1 issues, warps 2 to 9 drain (two per 32 lanes of tensor
// memory, alternate 16-column groups).
constexpr int MMA_THREADS = 320, MMA_EPI = 8, MMA_GROUPS = MAX_BNC / 32;

template <typename F>
__global__ void __launch_bounds__(MMA_THREADS, 1)
    split_mma_kernel(const __grid_constant__ CUtensorMap tmA,
                     const __grid_constant__ CUtensorMap tmB, MmaParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  const int BNc = p.BNc, nst = p.stages;
  const uint32_t b_slice_bytes = (uint32_t)BNc * KROW;
  const uint32_t stage_bytes = F::NS * A_SLICE_BYTES + F::NS * b_slice_bytes;
  __shared__ uint64_t bars[2 * MAX_STAGES + 2];
  __shared__ uint32_t tmem_slot;
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + MAX_STAGES),
                 done = smem_u32(bars + 2 * MAX_STAGES),
                 drained = smem_u32(bars + 2 * MAX_STAGES + 1);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  // two accumulators of BNc columns each: [0, acc1) for s0 t0, [acc1, ..)
  // for the five smaller slice products
  uint32_t acc1 = 32;
  while ((int)acc1 < BNc) acc1 <<= 1;
  const uint32_t ncols = 2 * acc1;

  if (threadIdx.x == 0) {
    for (int s = 0; s < nst; ++s) {
      mbar_init(full0 + 8 * s, 1);
      mbar_init(empty0 + 8 * s, 1);
    }
    mbar_init(done, 1);
    mbar_init(drained, MMA_EPI);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_slot)),
                 "r"(ncols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  const int items = p.mt * p.nchunks * p.nks;
  auto kblocks = [&](int item) {
    const int kb0 = item / (p.mt * p.nchunks) * p.kb_split;
    return min(p.kb_split, p.kb_total - kb0);
  };

  if (warp == 0) {
    if (lane == 0) {
      // TMA producer
      int s = 0, lap = 0;   // the stage, and how often it has been filled
      bool ok = true;
      for (int item = blockIdx.x; item < items && ok; item += gridDim.x) {
        const int chunk = item % p.nchunks, m_tile = item / p.nchunks % p.mt;
        const int kb0 = item / (p.mt * p.nchunks) * p.kb_split, nkb = kblocks(item);
        for (int kb = 0; kb < nkb; ++kb) {
          if (lap > 0 && !mbar_wait(empty0 + 8 * s, (lap - 1) & 1, p.err)) {
            ok = false;
            break;
          }
          const uint32_t full = full0 + 8 * s;
          mbar_expect_tx(full, stage_bytes);
          uint8_t* st = smem + s * stage_bytes;
          const int kx = (kb0 + kb) * F::KE;
          for (int sl = 0; sl < F::NS; ++sl)
            tma_load_3d(smem_u32(st + sl * A_SLICE_BYTES), &tmA, kx, m_tile * BM, sl, full);
          for (int sl = 0; sl < F::NS; ++sl)
            tma_load_3d(smem_u32(st + F::NS * A_SLICE_BYTES + sl * b_slice_bytes), &tmB, kx,
                        chunk * BNc, sl, full);
          if (++s == nst) s = 0, ++lap;
        }
      }
      // a CTA that gave up does not end before its copies have landed
      for (int i = 0; !ok && i < nst; ++i) {
        const int fills = lap + (i < s ? 1 : 0);
        if (fills > 0) mbar_wait(full0 + 8 * i, (fills - 1) & 1, p.err);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // MMA issuer: NP slice products per K block, four 32-byte K steps each
      const uint32_t idesc = F::EB == 2 ? idesc_bf16(BM, BNc) : idesc_tf32(BM, BNc);
      const int pa[6] = {0, 0, 1, 0, 1, 2};
      const int pb[6] = {0, 1, 0, 2, 1, 0};
      int s = 0, lap = 0, u = 0;
      bool ok = true;
      for (int item = blockIdx.x; item < items && ok; item += gridDim.x, ++u) {
        if (u > 0 && !mbar_wait(drained, (u - 1) & 1, p.err)) break;
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
        const int nkb = kblocks(item);
        for (int kb = 0; kb < nkb; ++kb) {
          if (!mbar_wait(full0 + 8 * s, lap & 1, p.err)) {
            ok = false;
            break;
          }
          asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          const uint32_t st = smem_u32(smem + s * stage_bytes);
          for (int pr = 0; pr < F::NP; ++pr) {
            const uint32_t a0 = st + pa[pr] * A_SLICE_BYTES;
            const uint32_t b0 = st + F::NS * A_SLICE_BYTES + pb[pr] * b_slice_bytes;
            const uint32_t d = pr == 0 ? tmem : tmem + acc1;
            const bool first = kb == 0 && (pr == 0 || pr == 1);
            for (int kk = 0; kk < KROW / 32; ++kk) {
              if (F::EB == 2)
                mma_bf16(d, smem_desc(a0 + kk * 32), smem_desc(b0 + kk * 32), idesc,
                         (first && kk == 0) ? 0u : 1u);
              else
                mma_tf32(d, smem_desc(a0 + kk * 32), smem_desc(b0 + kk * 32), idesc,
                         (first && kk == 0) ? 0u : 1u);
            }
          }
          mma_commit(empty0 + 8 * s);
          if (++s == nst) s = 0, ++lap;
        }
        if (ok) mma_commit(done);
      }
    }
  } else {
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31, rows of the tile
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    const uint32_t lanes = tmem + ((uint32_t)(quarter * 32) << 16);
    int u = 0;
    for (int item = blockIdx.x; item < items; item += gridDim.x, ++u) {
      if (!mbar_wait(done, u & 1, p.err)) break;
      asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
      const int chunk = item % p.nchunks, m_tile = item / p.nchunks % p.mt;
      const int ks = item / (p.mt * p.nchunks);
      const int row = m_tile * BM + quarter * 32 + lane;
      // 64 contiguous bytes of this thread's row per group (Np, BNc and c0 are
      // multiples of 16 floats, so the row segment is 64-byte aligned)
      float* out = p.part + ((size_t)ks * p.M + row) * p.Np + (size_t)chunk * BNc;
      auto load = [&](int c0, float (&v)[16]) {
        uint32_t r[16], q[16];
        tmem_ld16x2(lanes + (uint32_t)c0, lanes + acc1 + (uint32_t)c0, r, q);
        // one rounded addition joins the two accumulators
#pragma unroll
        for (int i = 0; i < 16; ++i)
          v[i] = __fadd_rn(__uint_as_float(r[i]), __uint_as_float(q[i]));
      };
      auto store = [&](int c0, const float (&v)[16]) {
        float4* o4 = reinterpret_cast<float4*>(out + c0);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          o4[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
      };
      if (item + (int)gridDim.x >= items) {
        // nothing waits for the accumulators: a short loop (the one below, unrolled,
        // costs a launch of one item per CTA 1 us of instruction fetches)
#pragma unroll 1
        for (int c0 = half * 16; c0 < BNc; c0 += 32) {
          float v[16];
          load(c0, v);
          if (row < p.M) store(c0, v);
        }
        break;
      }
      float v[MMA_GROUPS][16];
#pragma unroll
      for (int g = 0; g < MMA_GROUPS; ++g)
        if ((2 * g + half) * 16 < BNc) load((2 * g + half) * 16, v[g]);
      asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
      __syncwarp();
      if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(drained) : "memory");
      if (row < p.M) {
#pragma unroll
        for (int g = 0; g < MMA_GROUPS; ++g)
          if ((2 * g + half) * 16 < BNc) store((2 * g + half) * 16, v[g]);
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(ncols)
                 : "memory");
}

// ------------------------------------------------------------ slicing
// x -> three bf16 slices of its fp32 rounding xf: s0 + s1 + s2 = xf exactly
// (each remainder has at most 16, then 8 significant bits, so the fp32
// subtractions are exact); |x - xf| <= 2^-24 |x|. One fp64 operation per
// value: GB300's fp64 pipe is ~60x narrower than its fp32 pipe.
__device__ __forceinline__ void split3(double x, __nv_bfloat16& s0, __nv_bfloat16& s1,
                                       __nv_bfloat16& s2) {
  const float xf = f32_of(x);   // integer pipes, not the narrow fp64 pipe
  s0 = __float2bfloat16_rn(xf);
  const float r1 = xf - __bfloat162float(s0);
  s1 = __float2bfloat16_rn(r1);
  const float r2 = r1 - __bfloat162float(s1);
  s2 = __float2bfloat16_rn(r2);
}

// tf32 rounding of an fp32 value (nearest, ties away from zero): the 13 low
// mantissa bits are dropped after adding half of the last kept bit
__device__ __forceinline__ float tf32_rn(float x) {
  return __uint_as_float((__float_as_uint(x) + 0x1000u) & 0xffffe000u);
}

// the NS slices of x in format F (bf16: split3; tf32: t0 = tf32(xf),
// t1 = tf32(xf - t0), the subtraction exact in fp32)
template <typename F> struct SliceT;
template <> struct SliceT<FmtBF16> { using T = __nv_bfloat16; };
template <> struct SliceT<FmtTF32> { using T = float; };

__device__ __forceinline__ void slices_of(FmtBF16, double x, __nv_bfloat16* v) {
  split3(x, v[0], v[1], v[2]);
}
__device__ __forceinline__ void slices_of(FmtTF32, double x, float* v) {
  const float xf = f32_of(x);
  v[0] = tf32_rn(xf);
  v[1] = tf32_rn(xf - v[0]);
}
__device__ __forceinline__ __nv_bfloat16 negv(__nv_bfloat16 a) { return __hneg(a); }
__device__ __forceinline__ float negv(float a) { return -a; }
template <typename T> __device__ __forceinline__ T zero_slice();
template <> __device__ __forceinline__ __nv_bfloat16 zero_slice<__nv_bfloat16>() {
  return __float2bfloat16(0.0f);
}
template <> __device__ __forceinline__ float zero_slice<float>() { return 0.0f; }

template <typename F, typename T>
__device__ __forceinline__ void put_slices(T* out, long slice, long o, const T* v, bool neg) {
#pragma unroll
  for (int i = 0; i < F::NS; ++i) out[i * slice + o] = neg ? negv(v[i]) : v[i];
}


// A slices: out[s][m][kr], kr < K: Re op(A)(m, kr); K <= kr < 2K: Im
// (complex); zero up to Kp. The stored matrix (R x C, row-major) is read once, in
// PA x PA blocks, and each element sliced once; "direct" takes rows m = r and
// kr = c (op N and, conjugated, R), "trans" rows m = c and kr = r (op T and C),
// and both may be asked for. DRAM bounds it (16 bytes read and 12 written per
// complex element and orientation), so eight
// loads of a thread are in flight and the slices leave in eight bytes a lane. Both
// orientations of a complex 5184 x 5184 corner: 235 us (153 at the copy rate;
// two readings in 32 x 32 blocks with two-byte stores 310), one: 169 (156); at
// 2880 x 2880 72 (102), one 53.
struct PrepOut {
  void* out;   // null: not wanted
  int cj;      // conjugate
};
constexpr int PA_THREADS = 256;

// one slice of a value: the parts (re, im) side by side, so that both are rounded
// to bf16 by one instruction and stored by one
template <typename S, int PARTS>
struct alignas(sizeof(S) * PARTS) Cell { S p[PARTS]; };

__device__ __forceinline__ void cells_of(FmtBF16, cplx x, Cell<__nv_bfloat16, 2>* v) {
  float re = f32_of(x.x), im = f32_of(x.y);
#pragma unroll
  for (int i = 0; i < 3; ++i) {
    const __nv_bfloat162 s = __floats2bfloat162_rn(re, im);
    v[i].p[0] = s.x;
    v[i].p[1] = s.y;
    re -= __low2float(s);
    im -= __high2float(s);
  }
}
__device__ __forceinline__ void cells_of(FmtBF16, double x, Cell<__nv_bfloat16, 1>* v) {
  __nv_bfloat16 s[3];
  slices_of(FmtBF16(), x, s);
#pragma unroll
  for (int i = 0; i < 3; ++i) v[i].p[0] = s[i];
}
__device__ __forceinline__ void cells_of(FmtTF32, cplx x, Cell<float, 2>* v) {
  float a[2], b[2];
  slices_of(FmtTF32(), x.x, a);
  slices_of(FmtTF32(), x.y, b);
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    v[i].p[0] = a[i];
    v[i].p[1] = b[i];
  }
}
__device__ __forceinline__ void cells_of(FmtTF32, double x, Cell<float, 1>* v) {
  float s[2];
  slices_of(FmtTF32(), x, s);
#pragma unroll
  for (int i = 0; i < 2; ++i) v[i].p[0] = s[i];
}

template <typename T, typename F, int PA>
constexpr size_t prep_a_smem() {
  return (size_t)F::NS * PA * (PA + 1) * (sizeof(T) / 8) * sizeof(typename SliceT<F>::T);
}

template <typename T, typename F, int PA>
__global__ void __launch_bounds__(PA_THREADS)
    prep_a_kernel(const T* __restrict__ A, long lda, int R, int C, int KpD, int KpT, PrepOut direct,
                  PrepOut trans) {
  using S = typename SliceT<F>::T;
  constexpr int PARTS = sizeof(T) / 8, W = 8 / sizeof(S), PA_LD = PA + 1;
  using CellT = Cell<S, PARTS>;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  CellT* tile = reinterpret_cast<CellT*>(smem_raw);   // [slice][PA][PA_LD]
  const int tc = (C + PA - 1) / PA, tr = (R + PA - 1) / PA;
  for (int t = blockIdx.x; t < tc * tr; t += gridDim.x) {
    const int c0 = (t % tc) * PA, r0 = (t / tc) * PA;
    constexpr int STEP = PA_THREADS / PA, U = PA / STEP < 8 ? PA / STEP : 8;
    const int lc = threadIdx.x % PA, lr = threadIdx.x / PA;
#pragma unroll 1
    for (int b = 0; b < PA; b += U * STEP) {
      T v[U];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int r = r0 + lr + b + u * STEP, c = c0 + lc;
        v[u] = r < R && c < C ? __ldcs(A + (long)r * lda + c) : zero_of(T());
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        CellT sv[F::NS];
        cells_of(F(), v[u], sv);
#pragma unroll
        for (int i = 0; i < F::NS; ++i) tile[(i * PA + lr + b + u * STEP) * PA_LD + lc] = sv[i];
      }
    }
    __syncthreads();
    // rows of the output, eight bytes a lane and part: W slice values
    auto write = [&](const PrepOut& w, auto tr_, int m0, int M, int k0, int K, int Kp) {
      S* out = static_cast<S*>(w.out);
      const long slice = (long)M * Kp;
      constexpr int LPR = PA / W;   // lanes a row
      const int k = threadIdx.x % LPR * W, kc = k0 + k;
      const bool whole = kc + W <= K, cj = w.cj != 0, even = K % W == 0;
#pragma unroll 2
      for (int i = threadIdx.x / LPR; i < F::NS * PA; i += PA_THREADS / LPR) {
        const int sl = i / PA, m = i % PA;
        const CellT* src = tile + sl * PA * PA_LD;
        CellT e[W];
#pragma unroll
        for (int x = 0; x < W; ++x)
          e[x] = decltype(tr_)::value ? src[(k + x) * PA_LD + m] : src[m * PA_LD + k + x];
        if (m0 + m < M) {
          S* dst = out + sl * slice + (long)(m0 + m) * Kp + kc;
#pragma unroll
          for (int q = 0; q < PARTS; ++q, dst += K) {
            __align__(8) S o[W];
#pragma unroll
            for (int x = 0; x < W; ++x) o[x] = q == 1 && cj ? negv(e[x].p[q]) : e[x].p[q];
            if (whole && (q == 0 || even)) {
              *reinterpret_cast<uint2*>(dst) = *reinterpret_cast<const uint2*>(o);
            } else {
#pragma unroll
              for (int x = 0; x < W; ++x)
                if (kc + x < K) dst[x] = o[x];
            }
          }
        }
      }
    };
    if (direct.out) write(direct, std::false_type(), r0, R, c0, C, KpD);
    if (trans.out) write(trans, std::true_type(), c0, C, r0, R, KpT);
    __syncthreads();
  }
  // padding columns
  const long tid = (long)blockIdx.x * blockDim.x + threadIdx.x, nth = (long)gridDim.x * blockDim.x;
  auto pad = [&](const PrepOut& w, int M, int K, int Kp) {
    S* out = static_cast<S*>(w.out);
    const int Kr = PARTS * K, pc = Kp - Kr;
    for (long idx = tid; idx < (long)F::NS * M * pc; idx += nth)
      out[idx / pc * Kp + Kr + idx % pc] = zero_slice<S>();
  };
  if (direct.out) pad(direct, R, C, KpD);
  if (trans.out) pad(trans, C, R, KpT);
}

// B slices (K-major rows = output real columns): out[s][j][kr] = B_emb[kr][j]
// with B_emb = [[B_r, B_i], [-B_i, B_r]] for complex, B for real. A 32 x 32
// shared tile of op(B) is read along B's contiguous axis and written along
// kr; the padding rows and columns are zeroed.
template <typename T, typename F>
__global__ void prep_b_kernel(const T* B, long ldb, int op, int K, int N, int Kp, int Np,
                              typename SliceT<F>::T* out) {
  using S = typename SliceT<F>::T;
  __shared__ T tile[32][33];
  constexpr bool cx = sizeof(T) == 16;
  const int Kr = cx ? 2 * K : K;
  const int Nr = cx ? 2 * N : N;
  const long slice = (long)Np * Kp;
  const int tk = (K + 31) / 32, tn = (N + 31) / 32;
  const bool trans = (op == OP_T || op == OP_C);
  const bool cj = (op == OP_C || op == OP_R);
  for (int t = blockIdx.x; t < tk * tn; t += gridDim.x) {
    const int k0 = (t % tk) * 32, n0 = (t / tk) * 32;
    // tile[kk - k0][jj - n0] = op(B)(kk, jj) before conjugation
    for (int yy = threadIdx.y; yy < 32; yy += 8) {
      if (!trans) {
        const int kk = k0 + yy, jj = n0 + threadIdx.x;
        tile[yy][threadIdx.x] = (kk < K && jj < N) ? B[(long)kk * ldb + jj] : zero_of(T());
      } else {
        const int jj = n0 + yy, kk = k0 + threadIdx.x;
        tile[threadIdx.x][yy] = (kk < K && jj < N) ? B[(long)jj * ldb + kk] : zero_of(T());
      }
    }
    __syncthreads();
    for (int yy = threadIdx.y; yy < 32; yy += 8) {
      const int jj = n0 + yy, kk = k0 + threadIdx.x;
      if (jj < N && kk < K) {
        const T v = tile[threadIdx.x][yy];
        S re[3], im[3];
        if constexpr (cx) {
          // the slices of -x are the negated slices of x: each part is
          // sliced once
          slices_of(F(), v.x, re);
          slices_of(F(), v.y, im);
          put_slices<F>(out, slice, (long)jj * Kp + kk, re, false);
          put_slices<F>(out, slice, (long)jj * Kp + K + kk, im, !cj);
          put_slices<F>(out, slice, (long)(N + jj) * Kp + kk, im, cj);
          put_slices<F>(out, slice, (long)(N + jj) * Kp + K + kk, re, false);
        } else {
          slices_of(F(), v, re);
          put_slices<F>(out, slice, (long)jj * Kp + kk, re, false);
        }
      }
    }
    __syncthreads();
  }
  const S z = zero_slice<S>();
  const S zz[3] = {z, z, z};
  const long tid = (long)blockIdx.x * blockDim.x * blockDim.y + threadIdx.y * blockDim.x + threadIdx.x;
  const long nth = (long)gridDim.x * blockDim.x * blockDim.y;
  // padding rows j >= Nr
  for (long idx = tid; idx < (long)(Np - Nr) * Kp; idx += nth)
    put_slices<F>(out, slice, (long)Nr * Kp + idx, zz, false);
  // padding columns kr >= Kr of the rows j < Nr
  const int pc = Kp - Kr;
  for (long idx = tid; idx < (long)Nr * pc; idx += nth)
    put_slices<F>(out, slice, (idx / pc) * Kp + Kr + idx % pc, zz, false);
}

// error-free sum of two fp32 values (Knuth's TwoSum): hi + lo == a + b
__device__ __forceinline__ void two_sum_acc(float& hi, float& lo, float x) {
  const float s = hi + x;
  const float bb = s - hi;
  const float e = (hi - (s - bb)) + (x - bb);
  hi = s;
  lo += e;
}

// C[m][j] = sum over splits of the partials, complex from [C_r | C_i]. The
// sum is carried as an unevaluated fp32 pair (TwoSum on the fp32 pipe) and
// converted to fp64 once, because this GPU's fp64 pipe (conversions and
// additions alike) would bound the kernel; the pair is exact up to the
// rounding of its low part, ~2^-48 relative.
template <typename T>
__global__ void reduce_kernel(const float* part, int nks, int M, int N, int Np, T* C, long ldc) {
  for (unsigned idx = blockIdx.x * blockDim.x + threadIdx.x; idx < (unsigned)M * (unsigned)N;
       idx += gridDim.x * blockDim.x) {
    const unsigned m = idx / (unsigned)N, j = idx % (unsigned)N;
    const float* row = part + (size_t)m * Np + j;
    const size_t sstep = (size_t)M * Np;
    float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
    int s = 0;
    // eight splits' loads in flight at a time (the sum keeps the split order)
    for (; s + 8 <= nks; s += 8) {
      float a[8], b[8];
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        a[u] = __ldcs(row + (s + u) * sstep);
        if constexpr (sizeof(T) == 16) b[u] = __ldcs(row + (s + u) * sstep + N);
      }
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        two_sum_acc(rh, rl, a[u]);
        if constexpr (sizeof(T) == 16) two_sum_acc(ih, il, b[u]);
      }
    }
    for (; s < nks; ++s) {
      two_sum_acc(rh, rl, __ldcs(row + s * sstep));
      if constexpr (sizeof(T) == 16) two_sum_acc(ih, il, __ldcs(row + s * sstep + N));
    }
    const double re = f64_of(rh) + f64_of(rl);
    if constexpr (sizeof(T) == 16) C[(long)m * ldc + j] = make_double2(re, f64_of(ih) + f64_of(il));
    else C[(long)m * ldc + j] = re;
  }
}

// ------------------------------------------- fp64-accurate products (Ozaki)
// C = op(A) op(B) to fp64 accuracy on the bf16 tensor cores, for the
// products whose result must be fp64-accurate in split contexts (the Gram
// matrices of the CholeskyQR passes, rho = Z_L^H Z_R and the projectors
// Z_R v s^-1/2): an error-free splitting of the operands in the manner of
// Ozaki et al. (2012), "Error-free transformations of matrix multiplication
// by using fast routines of matrix multiplication and its applications".
//   * every row m of op(A) (every column n of op(B)) gets the exponent E of
//     its largest entry, |x| < 2^E; each entry is written as the 56-bit
//     fixed-point integer F = trunc(|x| 2^(56 - E)) and cut into eight 7-bit
//     digits d_0 .. d_7 (most significant first), stored with the sign of x
//     as bf16 (integers below 128 are exact in bf16);
//   * a digit product d_s e_t is an integer below 2^14, exact in fp32; the
//     products of equal weight w = s + t (w <= 7; the dropped ones are below
//     2^-53 of the row / column maxima) are accumulated in tensor memory,
//     one fp32 accumulator per weight, over at most OZ_KB_DRAIN K blocks of
//     64: at most 8 * 128 * 127^2 < 2^24, so every partial sum is an exact
//     integer;
//   * each accumulator is drained after OZ_KB_DRAIN K blocks and added,
//     scaled by 2^-7w, into an unevaluated fp32 pair (TwoSum) per output;
//     the pairs of the K splits are summed the same way and the result is
//     hi + lo scaled by 2^(E_m + E_n - 14), to about 2^-48 relative.
// One matrix instruction multiplies digit s of A with up to four digits t of B: B's
// digits lie one after the other in shared memory, and so do the accumulators of
// the weights s + t in tensor memory, so the digits of B are simply more columns
// (N up to 256; all sums are exact integers, so their order is free).
// The digits are staged in four groups, each with its own buffer: A's 0-3 and
// 4-7, B's 0-3 and 4-7. A K block uses (A 0-3, B 4-7), (A 0-3, B 0-3) and
// (A 4-7, B 0-3), in this order: every weight is started by digit 0 of A, and the
// groups are free again one after the other, so that the next K block's loads
// run beside the rest of this one's products.
// A persistent grid: CTA b takes the work items b, b + gridDim.x, ... (a split of
// a tile each), the loads running ahead into the next item. Complex, against 36
// single digit products of N = 64 per K block from three staged quarters (a third
// more loads), one item per CTA and four draining warps: 1024 x 1024 times 69
// columns 64 us -> 31, 65536 x 16 times 16 63 -> 26, one K block 24 -> 14.
constexpr int OZ_NS = 8;          // digits per operand
constexpr int OZ_BITS = 7;        // bits per digit
constexpr int OZ_BN = 64;         // output columns per CTA (one accumulator width) at most
constexpr int OZ_KB_DRAIN = 2;    // K blocks per exact accumulation
constexpr int OZ_GA = 4 * A_SLICE_BYTES, OZ_GB = 4 * OZ_BN * KROW;   // bytes of a group
constexpr int OZ_THREADS = 320, OZ_EPI = 8;

struct OzParams {
  int M;          // output rows (real-embedded)
  int Np;         // padded output columns
  int BNc;        // output columns per CTA, a multiple of 16, <= OZ_BN
  int kb_total;   // K blocks of 64
  int kb_split;   // K blocks per work item
  int mt, nchunks, nks;   // work items: row tiles x column chunks x splits
  float2* part;   // [nks][M][Np] (hi, lo)
  int* err;
};

// two_sum_acc of scale * x, scale a power of two (the product is exact)
__device__ __forceinline__ void two_sum_scaled(float& hi, float& lo, float x, float scale) {
  const float s = fmaf(x, scale, hi);
  const float bb = s - hi;
  const float e = (hi - (s - bb)) + fmaf(x, scale, -bb);
  hi = s;
  lo += e;
}

__global__ void __launch_bounds__(OZ_THREADS, 1)
    oz_mma_kernel(const __grid_constant__ CUtensorMap tmA,
                  const __grid_constant__ CUtensorMap tmB, OzParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>(
      (reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~(uintptr_t)1023);
  // groups in the order of their loads: B 4-7, A 0-3, B 0-3, A 4-7
  const uint32_t base = smem_u32(smem);
  const uint32_t gaddr[4] = {base + 2 * OZ_GA, base, base + 2 * OZ_GA + OZ_GB, base + OZ_GA};
  __shared__ uint64_t bars[10];
  __shared__ uint32_t tmem_slot;
  const uint32_t full0 = smem_u32(bars), empty0 = smem_u32(bars + 4), cdone = smem_u32(bars + 8),
                 drained = smem_u32(bars + 9);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int BN = p.BNc;
  if (threadIdx.x == 0) {
    for (int g = 0; g < 4; ++g) {
      mbar_init(full0 + 8 * g, 1);
      mbar_init(empty0 + 8 * g, 1);
    }
    mbar_init(cdone, 1);
    mbar_init(drained, OZ_EPI);
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(
                     smem_u32(&tmem_slot)),
                 "r"(512)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
  const uint32_t tmem = tmem_slot;
  const int items = p.mt * p.nchunks * p.nks;
  auto kblocks = [&](int item) {
    return min(p.kb_split, p.kb_total - item / (p.mt * p.nchunks) * p.kb_split);
  };

  if (warp == 0) {
    if (lane == 0) {
      // TMA producer
      bool ok = true;
      int t = 0, g = 0;   // K blocks and groups of the current one loaded
      for (int item = blockIdx.x; item < items && ok; item += gridDim.x) {
        const int chunk = item % p.nchunks, m_tile = item / p.nchunks % p.mt;
        const int kb0 = item / (p.mt * p.nchunks) * p.kb_split, nkb = kblocks(item);
        for (int kb = 0; kb < nkb && ok; ++kb) {
          const int kx = (kb0 + kb) * BK;
          for (g = 0; g < 4; ++g) {
            if (t > 0 && !mbar_wait(empty0 + 8 * g, (t - 1) & 1, p.err)) {
              ok = false;
              break;
            }
            const bool is_a = g & 1;
            const uint32_t full = full0 + 8 * g, step = is_a ? A_SLICE_BYTES : BN * KROW;
            mbar_expect_tx(full, 4 * step);
            const int d0 = g == 0 || g == 3 ? 4 : 0;
            for (int i = 0; i < 4; ++i)
              tma_load_3d(gaddr[g] + i * step, is_a ? &tmA : &tmB, kx,
                          is_a ? m_tile * BM : chunk * BN, d0 + i, full);
          }
          if (ok) ++t, g = 0;
        }
      }
      // a CTA that gave up does not end before its copies have landed
      for (int i = 0; !ok && i < 4; ++i) {
        const int fills = t + (i < g ? 1 : 0);
        if (fills > 0) mbar_wait(full0 + 8 * i, (fills - 1) & 1, p.err);
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // MMA issuer; a chunk of OZ_KB_DRAIN K blocks starts each accumulator afresh
      // once the epilogue has drained the last one
      bool ok = true;
      int t = 0, cc = 0;
      // digits d of A (at a) with the first nj of a group of B (at b) into the weights from w
      auto mma = [&](uint32_t a, uint32_t b, int nj, int w, bool fresh) {
        const uint32_t idesc = idesc_bf16(BM, nj * BN);
        const uint64_t da = smem_desc(a), db = smem_desc(b);
        const uint32_t d = tmem + (uint32_t)(w * BN);
        mma_bf16(d, da, db, idesc, fresh ? 0u : 1u);
#pragma unroll
        for (int kk = 1; kk < KROW / 32; ++kk) mma_bf16(d, da + 2 * kk, db + 2 * kk, idesc, 1u);
      };
      for (int item = blockIdx.x; item < items && ok; item += gridDim.x) {
        const int nkb = kblocks(item);
        for (int kb = 0; kb < nkb && ok; ++kb, ++t) {
          const bool first = kb % OZ_KB_DRAIN == 0;
          if (first) {
            if (cc > 0 && !mbar_wait(drained, (cc - 1) & 1, p.err)) ok = false;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
          }
          for (int q = 0; q < 3 && ok; ++q) {
            // groups that this quarter is the first to use
            const int g0 = q == 0 ? 0 : q + 1;
            for (int g = g0; g <= q + 1 && ok; ++g) ok = mbar_wait(full0 + 8 * g, t & 1, p.err);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
            const uint32_t a = gaddr[q == 2 ? 3 : 1], b = gaddr[q == 0 ? 0 : 2];
#pragma unroll 1
            for (int i = 0; i < 4; ++i)
              mma(a + i * A_SLICE_BYTES, b, q == 1 ? 4 : 4 - i, q == 1 ? i : 4 + i,
                  first && i == 0 && q < 2);
            if (q == 0) {
              mma_commit(empty0);
            } else if (q == 1) {
              mma_commit(empty0 + 8);
            } else {
              mma_commit(empty0 + 16);
              mma_commit(empty0 + 24);
            }
          }
          if (ok && (kb % OZ_KB_DRAIN == OZ_KB_DRAIN - 1 || kb == nkb - 1)) {
            mma_commit(cdone);
            ++cc;
          }
        }
      }
    }
  } else {
    // epilogue: warp w reads TMEM lanes 32 (w % 4) .. + 31 and alternate groups of
    // 16 columns
    const int quarter = warp & 3, half = (warp - 2) >> 2;
    const uint32_t lanes = tmem + ((uint32_t)(quarter * 32) << 16);
    bool ok = true;
    int cc = 0;
    for (int item = blockIdx.x; item < items && ok; item += gridDim.x) {
      float hi[2][16], lo[2][16];
#pragma unroll
      for (int g = 0; g < 2; ++g)
#pragma unroll
        for (int i = 0; i < 16; ++i) hi[g][i] = lo[g][i] = 0.f;
      const int nkb = kblocks(item);
      for (int kb = 0; kb < nkb; kb += OZ_KB_DRAIN, ++cc) {
        if (!mbar_wait(cdone, cc & 1, p.err)) {
          ok = false;
          break;
        }
        asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory");
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          const int c0 = (2 * g + half) * 16;
          if (c0 < BN) {
            float scale = 1.f;
#pragma unroll 1
            for (int w = 0; w < OZ_NS; w += 2) {
              uint32_t r[16], q[16];
              tmem_ld16x2(lanes + (uint32_t)(w * BN + c0), lanes + (uint32_t)((w + 1) * BN + c0), r, q);
#pragma unroll
              for (int i = 0; i < 16; ++i)
                two_sum_scaled(hi[g][i], lo[g][i], __uint_as_float(r[i]), scale);
              scale *= 0.0078125f;   // 2^-7
#pragma unroll
              for (int i = 0; i < 16; ++i)
                two_sum_scaled(hi[g][i], lo[g][i], __uint_as_float(q[i]), scale);
              scale *= 0.0078125f;
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
        __syncwarp();
        if (lane == 0) asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(drained) : "memory");
      }
      const int chunk = item % p.nchunks, m_tile = item / p.nchunks % p.mt;
      const int ks = item / (p.mt * p.nchunks);
      const int row = m_tile * BM + quarter * 32 + lane;
      if (ok && row < p.M) {
        float2* out = p.part + ((size_t)ks * p.M + row) * p.Np + (size_t)chunk * BN;
#pragma unroll
        for (int g = 0; g < 2; ++g) {
          const int c0 = (2 * g + half) * 16;
          if (c0 < BN) {
            float4* o4 = reinterpret_cast<float4*>(out + c0);
#pragma unroll
            for (int i = 0; i < 8; ++i)
              o4[i] = make_float4(hi[g][2 * i], lo[g][2 * i], hi[g][2 * i + 1], lo[g][2 * i + 1]);
          }
        }
      }
    }
  }
  __syncwarp();
  asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory");
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(512)
                 : "memory");
}

// biased exponent field of |x| (0 for zero and subnormals)
__device__ __forceinline__ int bexp(double x) {
  return (int)(((unsigned)__double2hiint(x) >> 20) & 0x7ffu);
}

// One operand of an exact-digit product: V vectors (rows of op(A), columns of
// op(B)) of K entries, stored as rows ("rows", the entries side by side) or as
// columns of a row-major matrix.
template <typename T>
struct OzOperand {
  const T* p;
  long ld;
  int V, K;
  int rows;          // vectors are stored rows
  int cj;            // conjugate
  int* e;            // exponent field of each vector's largest entry
  __nv_bfloat16* out;   // digits [8][rows of out][Kp]
  int Vp;            // rows of out: V for A, the padded real columns for B
  int tiles_c, tiles;   // 32 x 32 blocks of the stored matrix: per row, in all
};
constexpr int OZ_T = 32, OZ_PREP = 256, OZ_U = OZ_T * OZ_T / OZ_PREP;

// this thread's four entries of block t: rows r + 8 u, column c
template <typename T>
__device__ __forceinline__ void oz_load(const OzOperand<T>& o, int t, int& r, int& c, T (&v)[OZ_U]) {
  const int R = o.rows ? o.V : o.K, C = o.rows ? o.K : o.V;
  c = t % o.tiles_c * OZ_T + threadIdx.x % OZ_T;
  r = t / o.tiles_c * OZ_T + threadIdx.x / OZ_T;
#pragma unroll
  for (int u = 0; u < OZ_U; ++u)
    v[u] = r + 8 * u < R && c < C ? o.p[(long)(r + 8 * u) * o.ld + c] : zero_of(T());
}

// exponent fields of both operands' vectors: the maximum over each block, one
// atomicMax per vector and block
template <typename T>
__global__ void __launch_bounds__(OZ_PREP) oz_exp_kernel(OzOperand<T> a, OzOperand<T> b) {
  __shared__ int part[OZ_PREP / 32][32];
  for (int t = blockIdx.x; t < a.tiles + b.tiles; t += gridDim.x) {
    const OzOperand<T>& o = t < a.tiles ? a : b;
    T v[OZ_U];
    int r, c;
    oz_load(o, t < a.tiles ? t : t - a.tiles, r, c, v);
    int e[OZ_U], m = 0;
#pragma unroll
    for (int u = 0; u < OZ_U; ++u) {
      if constexpr (sizeof(T) == 16) e[u] = max(bexp(v[u].x), bexp(v[u].y));
      else e[u] = bexp(v[u]);
      m = max(m, e[u]);
    }
    if (o.rows) {
#pragma unroll
      for (int u = 0; u < OZ_U; ++u) {
        const int x = __reduce_max_sync(0xffffffffu, e[u]);
        if ((threadIdx.x & 31) == 0 && r + 8 * u < o.V && x > 0) atomicMax(o.e + r + 8 * u, x);
      }
    } else {
      part[threadIdx.x >> 5][threadIdx.x & 31] = m;
      __syncthreads();
      if (threadIdx.x < 32) {
#pragma unroll
        for (int w = 1; w < OZ_PREP / 32; ++w) m = max(m, part[w][threadIdx.x]);
        if (c < o.V && m > 0) atomicMax(o.e + c, m);
      }
      __syncthreads();
    }
  }
}

// the 56-bit fixed-point magnitude of x against the exponent field eb of its row /
// column maximum: trunc(|x| 2^(56 - E)), E = eb - 1022
__device__ __forceinline__ unsigned long long oz_fixed(double x, int eb) {
  const unsigned hi = (unsigned)__double2hiint(x), lo = (unsigned)__double2loint(x);
  const int ex = (int)((hi >> 20) & 0x7ffu);
  if (ex == 0) return 0ull;
  const unsigned long long m = ((unsigned long long)((hi & 0xfffffu) | 0x100000u) << 32) | lo;
  const int sh = ex - eb + 3;   // <= 3 since ex <= eb
  return sh >= 0 ? (m << sh) : (sh > -64 ? (m >> -sh) : 0ull);
}
// bits 7 (7 - s) .. + 6 of F as an fp32 integer (its low half is zero: a bf16 on top)
__device__ __forceinline__ unsigned oz_digit(unsigned long long F, int s) {
  const unsigned v = (unsigned)(F >> (OZ_BITS * (OZ_NS - 1 - s))) & 127u;
  return __float_as_uint(__uint_as_float(0x4b000000u | v) - 8388608.0f);
}

// signed digits of both operands, as prep_a_kernel and prep_b_kernel lay their
// slices out (rows of A: [Re | Im]; rows of B: [Re | -Im], then [Im | Re]). One
// launch for both: most products here are small, and the operands' blocks fill
// the GPU together. A value's digits are cut once, the real and imaginary one side
// by side, and leave in eight bytes a lane. Four launches with two-byte stores
// took 24 us of kernel time for a 69 x 69 product of 1024 rows, and an exact
// iteration 24.4 ms at 1x2, D = 4, chi = 33 (22.2 now), 12.7 at 2x1, D = 3,
// chi = 19 (11.9).
template <typename T>
__global__ void __launch_bounds__(OZ_PREP) oz_prep_kernel(OzOperand<T> a, OzOperand<T> b, int Kp) {
  constexpr int PARTS = sizeof(T) / 8, LD = OZ_T + 1, W = 4, LPR = OZ_T / W;
  using CellT = Cell<unsigned short, PARTS>;
  __shared__ CellT tile[OZ_NS * OZ_T * LD];   // [digit][row][column]
  for (int t = blockIdx.x; t < a.tiles + b.tiles; t += gridDim.x) {
    const bool is_b = t >= a.tiles;
    const OzOperand<T>& o = is_b ? b : a;
    const int tt = is_b ? t - a.tiles : t;
    T v[OZ_U];
    int r, c;
    oz_load(o, tt, r, c, v);
#pragma unroll
    for (int u = 0; u < OZ_U; ++u) {
      const int vec = o.rows ? r + 8 * u : c;
      const int eb = vec < o.V ? o.e[vec] : 0;
      CellT* d = tile + (threadIdx.x / OZ_T + 8 * u) * LD + threadIdx.x % OZ_T;
      if constexpr (PARTS == 2) {
        const unsigned long long fr = oz_fixed(v[u].x, eb), fi = oz_fixed(v[u].y, eb);
        const unsigned sign = ((unsigned)__double2hiint(v[u].x) >> 31 << 15) |
                              ((unsigned)__double2hiint(v[u].y) & 0x80000000u);
#pragma unroll
        for (int s = 0; s < OZ_NS; ++s)
          *reinterpret_cast<unsigned*>(d + s * OZ_T * LD) =
              __byte_perm(oz_digit(fr, s), oz_digit(fi, s), 0x7632) | sign;
      } else {
        const unsigned long long f = oz_fixed(v[u], eb);
        const unsigned sign = (unsigned)__double2hiint(v[u]) >> 31 << 15;
#pragma unroll
        for (int s = 0; s < OZ_NS; ++s)
          d[s * OZ_T * LD].p[0] = (unsigned short)((oz_digit(f, s) >> 16) | sign);
      }
    }
    __syncthreads();
    const int tr0 = tt / o.tiles_c * OZ_T, tc0 = tt % o.tiles_c * OZ_T;
    const int v0 = o.rows ? tr0 : tc0, k0 = o.rows ? tc0 : tr0;
    const int k = threadIdx.x % LPR * W, kc = k0 + k;
    const bool whole = kc + W <= o.K, even = o.K % W == 0;
    const long slice = (long)o.Vp * Kp;
    // four values of a part at kc of row m, the second half (h) at K + kc
    auto put = [&](int s, int m, int h, const CellT (&e)[W], int part, bool neg) {
      unsigned short* dst = reinterpret_cast<unsigned short*>(o.out) + s * slice + (long)m * Kp +
                            (h ? o.K : 0) + kc;
      const unsigned short x = neg ? 0x8000 : 0;
      if (whole && (!h || even)) {
        *reinterpret_cast<ushort4*>(dst) =
            make_ushort4(e[0].p[part] ^ x, e[1].p[part] ^ x, e[2].p[part] ^ x, e[3].p[part] ^ x);
      } else {
#pragma unroll
        for (int y = 0; y < W; ++y)
          if (kc + y < o.K) dst[y] = e[y].p[part] ^ x;
      }
    };
#pragma unroll 2
    for (int i = threadIdx.x / LPR; i < OZ_NS * OZ_T; i += OZ_PREP / LPR) {
      const int s = i / OZ_T, m = i % OZ_T;
      CellT e[W];
#pragma unroll
      for (int y = 0; y < W; ++y)
        e[y] = tile[s * OZ_T * LD + (o.rows ? m * LD + k + y : (k + y) * LD + m)];
      if (v0 + m < o.V) {
        put(s, v0 + m, 0, e, 0, false);
        if constexpr (PARTS == 2) {
          put(s, v0 + m, 1, e, 1, is_b ? !o.cj : o.cj != 0);
          if (is_b) {
            put(s, o.V + v0 + m, 0, e, 1, o.cj != 0);
            put(s, o.V + v0 + m, 1, e, 0, false);
          }
        }
      }
    }
    __syncthreads();
  }
  // padding: the columns from PARTS K to Kp of the rows in use, then B's rows beyond them
  const int tid = blockIdx.x * blockDim.x + threadIdx.x, nth = gridDim.x * blockDim.x;
  const int Kr = PARTS * a.K, pc = Kp - Kr, Nr = PARTS * b.V, pr = b.Vp - Nr;
  const __nv_bfloat16 z = __float2bfloat16(0.0f);
  for (long i = tid; i < (long)OZ_NS * a.V * pc; i += nth)
    a.out[i / pc * Kp + Kr + i % pc] = z;
  for (long i = tid; i < (long)OZ_NS * Nr * pc; i += nth) {
    const long row = i / pc;
    b.out[(row / Nr * b.Vp + row % Nr) * Kp + Kr + i % pc] = z;
  }
  const int q = Kp / 8;   // sixteen bytes
  for (long i = tid; i < (long)OZ_NS * pr * q; i += nth) {
    const long row = i / q;
    reinterpret_cast<uint4*>(b.out + (row / pr * b.Vp + Nr + row % pr) * Kp)[i % q] =
        make_uint4(0u, 0u, 0u, 0u);
  }
}

// C[m][j] = (sum over K splits of the pairs) 2^(E_m + E_j - 14), complex
// from [C_r | C_i]; the pairs are summed with TwoSum and converted to fp64
// once, and the power of two is applied to the exponent field
template <typename T>
__global__ void oz_reduce_kernel(const float2* part, int nks, int M, int N, int Np,
                                 const int* ea, const int* ebx, T* C, long ldc) {
  for (long idx = blockIdx.x * (long)blockDim.x + threadIdx.x; idx < (long)M * N;
       idx += (long)gridDim.x * blockDim.x) {
    const int m = (int)(idx / N), j = (int)(idx % N);
    const size_t sstep = (size_t)M * Np;
    const float2* row = part + (size_t)m * Np + j;
    float rh = 0.f, rl = 0.f, ih = 0.f, il = 0.f;
    for (int s = 0; s < nks; ++s) {
      const float2 a = row[s * sstep];
      two_sum_acc(rh, rl, a.x);
      two_sum_acc(rh, rl, a.y);
      if constexpr (sizeof(T) == 16) {
        const float2 b = row[s * sstep + N];
        two_sum_acc(ih, il, b.x);
        two_sum_acc(ih, il, b.y);
      }
    }
    const int e1 = ea[m], e2 = ebx[j];
    // 2^(E_m + E_j - 14) with E = field - 1022
    const int sc = (e1 > 0 && e2 > 0) ? e1 + e2 - 2044 - 14 : -2000;
    const double f = sc > -1022 && sc < 1023 ? __hiloint2double((sc + 1023) << 20, 0) : 0.0;
    const double re = (f64_of(rh) + f64_of(rl)) * f;
    if constexpr (sizeof(T) == 16)
      C[(long)m * ldc + j] = make_double2(re, (f64_of(ih) + f64_of(il)) * f);
    else
      C[(long)m * ldc + j] = re;
  }
}

unsigned grid_cap(long n, long cap = 152L * 8) {
  long g = (n + 255) / 256;
  if (g < 1) g = 1;
  if (g > cap) g = cap;
  return (unsigned)g;
}

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*,
                                  const cuuint64_t*, const cuuint64_t*, const cuuint32_t*,
                                  const cuuint32_t*, CUtensorMapInterleave, CUtensorMapSwizzle,
                                  CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

EncodeTiledFn get_encoder() {
  static const EncodeTiledFn fn = [] {
    void* p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      return reinterpret_cast<EncodeTiledFn>(p);
    return (EncodeTiledFn) nullptr;
  }();
  return fn;
}

// 3-D map over [ns][rows][Kp] slices (bf16 or tf32-in-fp32) with a
// (128 bytes, box_rows, 1) box, 128B swizzle; ns = 0: the format's count
bool make_map(CUtensorMap* map, const void* base, int rows, int Kp, int box_rows, bool tf32,
              int ns = 0) {
  EncodeTiledFn enc = get_encoder();
  if (!enc) return false;
  const int eb = tf32 ? 4 : 2;
  cuuint64_t dims[3] = {(cuuint64_t)Kp, (cuuint64_t)rows,
                        (cuuint64_t)(ns > 0 ? ns : (tf32 ? 2 : 3))};
  cuuint64_t strides[2] = {(cuuint64_t)Kp * eb, (cuuint64_t)Kp * eb * rows};
  cuuint32_t box[3] = {(cuuint32_t)(KROW / eb), (cuuint32_t)box_rows, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, tf32 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT32 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 3,
             const_cast<void*>(base), dims, strides,
             box, estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) ==
         CUDA_SUCCESS;
}

}  // namespace

// ------------------------------------------------------------ context
struct SplitCtx {
  bool cx = false;
  bool tf32 = false;        // 3xTF32 slices instead of bf16 x3
  int N = 0, k = 0;
  std::string msg;
  SplitMemory mem;
  // cached corner operands: [corner][op N / op H] slices, and their sources
  void* corner_src[4] = {nullptr};
  void* cslices[4][2] = {{nullptr}};
  int corner_Kp = 0;
  bool borrowed = false;    // cslices belong to another context
  // operand and partial-sum buffers (grown on demand). fp64-accurate products: digits
  // of both operands, exponent fields, partials
  struct Buf {
    void* p = nullptr;
    size_t bytes = 0;
    size_t want = 0;        // the most that a product asked for while noting
  };
  enum { ABUF, BBUF, PART, OZ_A, OZ_B, OZ_E, OZ_PART, NBUF };
  Buf buf[NBUF];
  bool noting = false;
  long oz_launches = 0;
  int* err = nullptr;       // device error flag of the owning context
  // per-launch CUDA events around the tensor-core kernel (profiling)
  bool prof = false;
  std::vector<cudaEvent_t> ev;
  size_t ev_used = 0;
  long prof_launches = 0;
  double prof_flops = 0.0, prof_bytes = 0.0, prof_ms = 0.0;
};

namespace {

ctm_status sfail(SplitCtx* sc, ctm_status st, const char* m) {
  sc->msg = m;
  return st;
}

bool mem_alloc(SplitCtx* sc, void** p, size_t bytes) {
  const cudaError_t e =
      sc->mem.alloc ? sc->mem.alloc(sc->mem.owner, p, bytes) : cudaMalloc(p, bytes);
  if (e == cudaSuccess) return true;
  cudaGetLastError();
  *p = nullptr;
  return false;
}

void mem_release(SplitCtx* sc, void** p, size_t bytes) {
  if (!*p) return;
  if (sc->mem.release) sc->mem.release(sc->mem.owner, *p, bytes);
  else cudaFree(*p);
  *p = nullptr;
}

ctm_status grow(SplitCtx* sc, int which, size_t need) {
  SplitCtx::Buf& b = sc->buf[which];
  if (sc->noting) b.want = std::max(b.want, need);
  if (b.bytes >= need) return CTM_OK;
  mem_release(sc, &b.p, b.bytes);
  b.bytes = 0;
  if (!mem_alloc(sc, &b.p, need))
    return sfail(sc, CTM_ENOMEM, "split-precision buffer allocation failed");
  b.bytes = need;
  return CTM_OK;
}

int pad_to(int x, int m) { return (x + m - 1) / m * m; }

// column chunking of Nr real output columns into CTAs of <= MAX_BNC columns
void chunking(int Nr, int* nchunks, int* BNc) {
  int nc = (Nr + MAX_BNC - 1) / MAX_BNC;
  if (nc < 1) nc = 1;
  int b = pad_to((Nr + nc - 1) / nc, 16);
  if (b < 16) b = 16;
  *nchunks = nc;
  *BNc = b;
}

int choose_splits(int tiles, int kb_total, int kb_max) {
  int best = 1;
  double best_t = 1e30;
  const int smin = (kb_total + kb_max - 1) / kb_max;
  const int smax = std::max(smin, std::min(std::max(32, smin), kb_total / 4));
  for (int s = smin; s <= smax; ++s) {
    const int per = (kb_total + s - 1) / s;
    const int used = (kb_total + per - 1) / per;
    const long ctas = (long)tiles * used;
    const long waves = (ctas + 151) / 152;
    const double t = (double)waves * (per + 2);
    if (t < best_t - 1e-9) { best_t = t; best = used; }
  }
  return best;
}

// real K of the current problem (set by the caller before run_mma)
thread_local int g_kr_real = 0;
inline double Kr_used(int Kp, const SplitCtx*) { return g_kr_real > 0 ? g_kr_real : Kp; }

// slices per operand, K elements per 128-byte row, bytes per slice element
inline int ns_of(const SplitCtx* sc) { return sc->tf32 ? 2 : 3; }
inline int ke_of(const SplitCtx* sc) { return sc->tf32 ? 32 : 64; }
inline int eb_of(const SplitCtx* sc) { return sc->tf32 ? 4 : 2; }

// bytes of a corner's slices in one orientation
size_t slice_bytes(const SplitCtx* sc, int N, int Kp) {
  return (size_t)ns_of(sc) * N * Kp * eb_of(sc);
}

// run the tensor-core kernel on prepared slices: A [ns][M][Kp], B [ns][Np][Kp]
ctm_status run_mma(SplitCtx* sc, const void* As, const void* Bs, int M, int Kp,
                   int Nr, int nchunks, int BNc, void* C, long ldc, int Nout, cudaStream_t s,
                   long* launches) {
  const int Np = nchunks * BNc;
  const int kb_total = Kp / ke_of(sc);
  const int mt = (M + BM - 1) / BM;
  // the same K elements per fp32 partial in both formats
  const int nks = choose_splits(mt * nchunks, kb_total, KB_SPLIT_MAX * BK / ke_of(sc));
  const int kb_split = (kb_total + nks - 1) / nks;
  {
    ctm_status st = grow(sc, SplitCtx::PART, (size_t)nks * M * Np * 4);
    if (st != CTM_OK) return st;
  }
  CUtensorMap ta, tb;
  if (!make_map(&ta, As, M, Kp, BM, sc->tf32) || !make_map(&tb, Bs, Np, Kp, BNc, sc->tf32))
    return sfail(sc, CTM_ECUDA, "cuTensorMapEncodeTiled failed");
  MmaParams p;
  p.M = M;
  p.Np = Np;
  p.BNc = BNc;
  p.kb_total = kb_total;
  p.kb_split = kb_split;
  p.mt = mt;
  p.nchunks = nchunks;
  p.nks = nks;
  float* const part = static_cast<float*>(sc->buf[SplitCtx::PART].p);
  p.part = part;
  p.err = sc->err;
  const int ns = ns_of(sc);
  const size_t stage = ns * A_SLICE_BYTES + ns * (size_t)BNc * KROW;
  p.stages = (int)std::min<size_t>(MAX_STAGES, STAGE_SMEM / stage);
  const size_t smem = 1024 + p.stages * stage;
  static size_t configured_bf16 = 0, configured_tf32 = 0;
  const void* kfn = sc->tf32 ? (const void*)split_mma_kernel<FmtTF32>
                             : (const void*)split_mma_kernel<FmtBF16>;
  if (raise_smem(kfn, sc->tf32 ? configured_tf32 : configured_bf16, smem) != cudaSuccess)
    return sfail(sc, CTM_ECUDA, "cannot reserve shared memory for the tensor-core kernel");
  const unsigned grid = (unsigned)std::min<long>(152, (long)mt * nchunks * nks);
  if (sc->prof && sc->ev_used + 2 > sc->ev.size()) {
    // every launch of the profiled region is timed: the event pool grows
    const size_t old = sc->ev.size();
    sc->ev.resize(old + 8192);
    for (size_t i = old; i < sc->ev.size(); ++i)
      if (cudaEventCreate(&sc->ev[i]) != cudaSuccess) {
        sc->ev.resize(i);
        break;
      }
  }
  const bool timed = sc->prof && sc->ev_used + 2 <= sc->ev.size();
  if (timed) cudaEventRecord(sc->ev[sc->ev_used], s);
  if (sc->tf32) split_mma_kernel<FmtTF32><<<grid, MMA_THREADS, smem, s>>>(ta, tb, p);
  else split_mma_kernel<FmtBF16><<<grid, MMA_THREADS, smem, s>>>(ta, tb, p);
  if (timed) {
    cudaEventRecord(sc->ev[sc->ev_used + 1], s);
    sc->ev_used += 2;
    // tensor-pipe work: the slice products (six bf16 or three tf32) of the
    // real-embedded (unpadded) problem; bytes: all slices of both operands
    // once, plus the fp32 partials
    sc->prof_launches += 1;
    const double np = sc->tf32 ? 3.0 : 6.0;
    sc->prof_flops += np * 2.0 * (double)M * (double)Nr * (double)Kr_used(Kp, sc);
    sc->prof_bytes += (double)ns * eb_of(sc) * ((double)M * Kp + (double)nchunks * BNc * Kp) +
                      4.0 * (double)nks * M * Np;
  }
  if (launches) ++*launches;
  if (sc->cx)
    reduce_kernel<cplx><<<grid_cap((long)M * Nout), 256, 0, s>>>(part, nks, M, Nout, Np,
                                                                 (cplx*)C, ldc);
  else
    reduce_kernel<double><<<grid_cap((long)M * Nout), 256, 0, s>>>(part, nks, M, Nout, Np,
                                                                   (double*)C, ldc);
  if (launches) ++*launches;
  if (cudaGetLastError() != cudaSuccess) return sfail(sc, CTM_ECUDA, "split GEMM launch failed");
  (void)Nr;
  return CTM_OK;
}

template <typename T, typename F, int PA>
cudaError_t launch_prep_a_tiles(const void* A, long lda, int R, int C, int KpD, int KpT, PrepOut direct,
                          PrepOut trans, cudaStream_t s) {
  static size_t configured = 0;
  constexpr size_t smem = prep_a_smem<T, F, PA>();
  cudaError_t e = raise_smem((const void*)prep_a_kernel<T, F, PA>, configured, smem);
  if (e != cudaSuccess) return e;
  const long tiles = (long)((R + PA - 1) / PA) * ((C + PA - 1) / PA);
  const unsigned g = (unsigned)std::max<long>(1, std::min<long>(tiles, 152L * 16));
  prep_a_kernel<T, F, PA><<<g, PA_THREADS, smem, s>>>(static_cast<const T*>(A), lda, R, C, KpD, KpT,
                                                      direct, trans);
  return cudaGetLastError();
}

// blocks of 64 x 64, or of 32 x 32 where those would leave SMs without a block (an
// edge of 41 x 1025: 17 blocks of 64)
template <typename T, typename F>
cudaError_t launch_prep_a(const void* A, long lda, int R, int C, int KpD, int KpT, PrepOut direct,
                          PrepOut trans, cudaStream_t s) {
  if ((long)((R + 63) / 64) * ((C + 63) / 64) < 152)
    return launch_prep_a_tiles<T, F, 32>(A, lda, R, C, KpD, KpT, direct, trans, s);
  return launch_prep_a_tiles<T, F, 64>(A, lda, R, C, KpD, KpT, direct, trans, s);
}

// slices of the stored R x C matrix A in either orientation
ctm_status prep_a_both(SplitCtx* sc, const void* A, long lda, int R, int C, int KpD, int KpT,
                       PrepOut direct, PrepOut trans, cudaStream_t s, long* launches) {
  cudaError_t e;
  if (sc->tf32)
    e = sc->cx ? launch_prep_a<cplx, FmtTF32>(A, lda, R, C, KpD, KpT, direct, trans, s)
               : launch_prep_a<double, FmtTF32>(A, lda, R, C, KpD, KpT, direct, trans, s);
  else
    e = sc->cx ? launch_prep_a<cplx, FmtBF16>(A, lda, R, C, KpD, KpT, direct, trans, s)
               : launch_prep_a<double, FmtBF16>(A, lda, R, C, KpD, KpT, direct, trans, s);
  if (launches) ++*launches;
  return e == cudaSuccess ? CTM_OK : sfail(sc, CTM_ECUDA, "slice launch failed");
}

ctm_status prep_a(SplitCtx* sc, const void* A, long lda, int op, int M, int K, int Kp,
                  void* out, cudaStream_t s, long* launches) {
  const PrepOut none{nullptr, 0}, o{out, op == OP_C || op == OP_R};
  if (op == OP_T || op == OP_C)
    return prep_a_both(sc, A, lda, K, M, Kp, Kp, none, o, s, launches);
  return prep_a_both(sc, A, lda, M, K, Kp, Kp, o, none, s, launches);
}

ctm_status prep_b(SplitCtx* sc, const void* B, long ldb, int op, int K, int N, int Kp, int Np,
                  void* out, cudaStream_t s, long* launches) {
  long tiles = (long)((K + 31) / 32) * ((N + 31) / 32);
  if (tiles > 152L * 8) tiles = 152L * 8;
  if (tiles < 1) tiles = 1;
  const dim3 blk(32, 8);
  const unsigned g = (unsigned)tiles;
  if (sc->tf32) {
    float* o = static_cast<float*>(out);
    if (sc->cx) prep_b_kernel<cplx, FmtTF32><<<g, blk, 0, s>>>((const cplx*)B, ldb, op, K, N, Kp, Np, o);
    else prep_b_kernel<double, FmtTF32><<<g, blk, 0, s>>>((const double*)B, ldb, op, K, N, Kp, Np, o);
  } else {
    __nv_bfloat16* o = static_cast<__nv_bfloat16*>(out);
    if (sc->cx) prep_b_kernel<cplx, FmtBF16><<<g, blk, 0, s>>>((const cplx*)B, ldb, op, K, N, Kp, Np, o);
    else prep_b_kernel<double, FmtBF16><<<g, blk, 0, s>>>((const double*)B, ldb, op, K, N, Kp, Np, o);
  }
  if (launches) ++*launches;
  return cudaGetLastError() == cudaSuccess ? CTM_OK : sfail(sc, CTM_ECUDA, "slice launch failed");
}

}  // namespace

ctm_status split_create(SplitCtx** out, bool cx, bool tf32, int N, int k, int* err,
                        cudaStream_t s, const SplitMemory& mem) {
  (void)s;
  *out = nullptr;
  if (!get_encoder()) return CTM_EUNSUPPORTED;
  SplitCtx* sc = new SplitCtx();
  sc->cx = cx;
  sc->tf32 = tf32;
  sc->N = N;
  sc->k = k;
  sc->err = err;
  sc->mem = mem;
  *out = sc;
  return CTM_OK;
}

ctm_status split_profile(SplitCtx* sc, int on, double* ms, long* launches, double* flops,
                         double* bytes) {
  if (on >= 0) {
    if (on && sc->ev.empty()) {
      sc->ev.resize(8192);
      for (auto& e : sc->ev)
        if (cudaEventCreate(&e) != cudaSuccess) return sfail(sc, CTM_ECUDA, "event creation failed");
    }
    sc->prof = on != 0;
    sc->ev_used = 0;
    sc->prof_launches = 0;
    sc->prof_flops = sc->prof_bytes = sc->prof_ms = 0.0;
    return CTM_OK;
  }
  // read: fold the recorded pairs into the totals
  for (size_t i = 0; i + 1 < sc->ev_used; i += 2) {
    if (cudaEventSynchronize(sc->ev[i + 1]) != cudaSuccess)
      return sfail(sc, CTM_ECUDA, "event synchronisation failed");
    float t = 0.f;
    cudaEventElapsedTime(&t, sc->ev[i], sc->ev[i + 1]);
    sc->prof_ms += t;
  }
  sc->ev_used = 0;
  if (ms) *ms = sc->prof_ms;
  if (launches) *launches = sc->prof_launches;
  if (flops) *flops = sc->prof_flops;
  if (bytes) *bytes = sc->prof_bytes;
  return CTM_OK;
}

void split_destroy(SplitCtx* sc) {
  if (!sc) return;
  for (auto& e : sc->ev) cudaEventDestroy(e);
  for (int i = 0; i < 4 && !sc->borrowed; ++i)
    for (int o = 0; o < 2; ++o)
      mem_release(sc, &sc->cslices[i][o], slice_bytes(sc, sc->N, sc->corner_Kp));
  for (auto& b : sc->buf) mem_release(sc, &b.p, b.bytes);
  delete sc;
}

ctm_status split_prepare_corners(SplitCtx* sc, void* const* Q, int N, unsigned mask,
                                 unsigned ops, cudaStream_t s, long* launches) {
  const int Kr = sc->cx ? 2 * N : N;
  const int Kp = pad_to(Kr, ke_of(sc));
  sc->corner_Kp = Kp;
  for (int i = 0; i < 4; ++i) {
    if (!(mask >> i & 1u)) continue;
    sc->corner_src[i] = Q[i];
    for (int o = 0; o < 2; ++o)
      if ((ops >> o & 1u) && !sc->cslices[i][o] &&
          !mem_alloc(sc, &sc->cslices[i][o], slice_bytes(sc, N, Kp)))
        return sfail(sc, CTM_ENOMEM, "corner slice allocation failed");
    // both orientations from one reading
    const PrepOut direct{ops & 1u ? sc->cslices[i][0] : nullptr, 0};
    const PrepOut trans{ops & 2u ? sc->cslices[i][1] : nullptr, sc->cx ? 1 : 0};
    ctm_status st = prep_a_both(sc, Q[i], N, N, N, Kp, Kp, direct, trans, s, launches);
    if (st != CTM_OK) return st;
  }
  return CTM_OK;
}

void split_borrow_corners(SplitCtx* sc, const SplitCtx* src) {
  sc->borrowed = true;
  sc->corner_Kp = src->corner_Kp;
  for (int i = 0; i < 4; ++i) {
    sc->corner_src[i] = src->corner_src[i];
    for (int o = 0; o < 2; ++o) sc->cslices[i][o] = src->cslices[i][o];
  }
}

void split_note(SplitCtx* sc, bool on) { sc->noting = on; }

size_t split_reserve_bytes(const SplitCtx* sc, const SplitCtx* like) {
  size_t n = 0;
  for (int i = 0; i < SplitCtx::NBUF; ++i)
    if (like->buf[i].want > (sc ? sc->buf[i].bytes : 0)) n += device_bytes(like->buf[i].want);
  return n;
}

ctm_status split_reserve(SplitCtx* sc, const SplitCtx* like) {
  for (int i = 0; i < SplitCtx::NBUF; ++i) {
    const ctm_status st = grow(sc, i, like->buf[i].want);
    if (st != CTM_OK) return st;
  }
  return CTM_OK;
}

ctm_status split_apply(SplitCtx* sc, const void* Q, bool herm, const void* Zin, void* Zout, int N,
                       int k, cudaStream_t s, long* launches) {
  int ci = -1;
  for (int i = 0; i < 4; ++i)
    if (sc->corner_src[i] == Q) ci = i;
  if (ci < 0) return sfail(sc, CTM_EINVAL, "corner was not prepared");
  const int Kp = sc->corner_Kp;
  const int Nr = sc->cx ? 2 * k : k;
  g_kr_real = sc->cx ? 2 * N : N;
  int nchunks, BNc;
  chunking(Nr, &nchunks, &BNc);
  const int Np = nchunks * BNc;
  ctm_status st = grow(sc, SplitCtx::BBUF, (size_t)ns_of(sc) * Np * Kp * eb_of(sc));
  if (st != CTM_OK) return st;
  void* const bbuf = sc->buf[SplitCtx::BBUF].p;
  st = prep_b(sc, Zin, k, OP_N, N, k, Kp, Np, bbuf, s, launches);
  if (st != CTM_OK) return st;
  return run_mma(sc, sc->cslices[ci][herm ? 1 : 0], bbuf, N, Kp, Nr, nchunks, BNc, Zout, k, k,
                 s, launches);
}

ctm_status split_gemm(SplitCtx* sc, int opA, const void* A, long lda, int opB, const void* B,
                      long ldb, int M, int N, int K, void* C, long ldc, cudaStream_t s,
                      long* launches) {
  const int Kr = sc->cx ? 2 * K : K;
  const int Kp = pad_to(Kr, ke_of(sc));
  const int Nr = sc->cx ? 2 * N : N;
  g_kr_real = Kr;
  int nchunks, BNc;
  chunking(Nr, &nchunks, &BNc);
  const int Np = nchunks * BNc;
  const size_t per = (size_t)ns_of(sc) * eb_of(sc);
  ctm_status st = grow(sc, SplitCtx::ABUF, per * M * Kp);
  if (st != CTM_OK) return st;
  st = grow(sc, SplitCtx::BBUF, per * Np * Kp);
  if (st != CTM_OK) return st;
  void *const abuf = sc->buf[SplitCtx::ABUF].p, *const bbuf = sc->buf[SplitCtx::BBUF].p;
  st = prep_a(sc, A, lda, opA, M, K, Kp, abuf, s, launches);
  if (st != CTM_OK) return st;
  st = prep_b(sc, B, ldb, opB, K, N, Kp, Np, bbuf, s, launches);
  if (st != CTM_OK) return st;
  return run_mma(sc, abuf, bbuf, M, Kp, Nr, nchunks, BNc, C, ldc, N, s, launches);
}

ctm_status oz_gemm(SplitCtx* sc, int opA, const void* A, long lda, int opB, const void* B,
                   long ldb, int M, int N, int K, void* C, long ldc, cudaStream_t s,
                   long* launches) {
  if (M <= 0 || N <= 0 || K <= 0) return sfail(sc, CTM_EINVAL, "empty fp64-accurate product");
  const bool cx = sc->cx;
  const int Kr = cx ? 2 * K : K;
  const int Kp = pad_to(Kr, BK);
  const int Nr = cx ? 2 * N : N;
  const int nchunks = (Nr + OZ_BN - 1) / OZ_BN;
  const int BNc = pad_to((Nr + nchunks - 1) / nchunks, 16);
  const int Np = nchunks * BNc;
  const int mt = (M + BM - 1) / BM;
  const int kb_total = Kp / BK;
  // about two waves of CTAs, at least OZ_KB_DRAIN K blocks each
  const long tiles = (long)mt * nchunks;
  int nks = (int)std::max<long>(1, std::min<long>((2 * 152 + tiles - 1) / tiles,
                                                  (kb_total + OZ_KB_DRAIN - 1) / OZ_KB_DRAIN));
  const int kb_split = (kb_total + nks - 1) / nks;
  nks = (kb_total + kb_split - 1) / kb_split;
  ctm_status st = grow(sc, SplitCtx::OZ_A, (size_t)OZ_NS * M * Kp * 2);
  if (st == CTM_OK) st = grow(sc, SplitCtx::OZ_B, (size_t)OZ_NS * Np * Kp * 2);
  if (st == CTM_OK) st = grow(sc, SplitCtx::OZ_E, (size_t)(M + N) * sizeof(int));
  if (st == CTM_OK) st = grow(sc, SplitCtx::OZ_PART, (size_t)nks * M * Np * 8);
  if (st != CTM_OK) return st;
  void *const oz_a = sc->buf[SplitCtx::OZ_A].p, *const oz_b = sc->buf[SplitCtx::OZ_B].p;
  int* const ea = static_cast<int*>(sc->buf[SplitCtx::OZ_E].p);
  int* const ebx = ea + M;
  if (cudaMemsetAsync(ea, 0, (size_t)(M + N) * sizeof(int), s) != cudaSuccess)
    return sfail(sc, CTM_ECUDA, "exponent reset failed");
  auto prepare = [&](auto zero) {
    using T = decltype(zero);
    OzOperand<T> a, b;
    a.p = static_cast<const T*>(A);
    a.ld = lda;
    a.V = M;
    a.rows = opA == OP_N || opA == OP_R;
    a.cj = opA == OP_C || opA == OP_R;
    a.e = ea;
    a.out = static_cast<__nv_bfloat16*>(oz_a);
    a.Vp = M;
    b.p = static_cast<const T*>(B);
    b.ld = ldb;
    b.V = N;
    b.rows = opB == OP_T || opB == OP_C;
    b.cj = opB == OP_C || opB == OP_R;
    b.e = ebx;
    b.out = static_cast<__nv_bfloat16*>(oz_b);
    b.Vp = Np;
    for (OzOperand<T>* o : {&a, &b}) {
      o->K = K;
      o->tiles_c = ((o->rows ? K : o->V) + OZ_T - 1) / OZ_T;
      o->tiles = o->tiles_c * (((o->rows ? o->V : K) + OZ_T - 1) / OZ_T);
    }
    const unsigned g = (unsigned)std::min<long>((long)a.tiles + b.tiles, 152L * 16);
    oz_exp_kernel<T><<<g, OZ_PREP, 0, s>>>(a, b);
    oz_prep_kernel<T><<<g, OZ_PREP, 0, s>>>(a, b, Kp);
  };
  if (cx) prepare(cplx());
  else prepare(0.0);
  if (launches) *launches += 2;
  CUtensorMap ta, tb;
  if (!make_map(&ta, oz_a, M, Kp, BM, false, OZ_NS) ||
      !make_map(&tb, oz_b, Np, Kp, BNc, false, OZ_NS))
    return sfail(sc, CTM_ECUDA, "cuTensorMapEncodeTiled failed");
  OzParams p;
  p.M = M;
  p.Np = Np;
  p.kb_total = kb_total;
  p.kb_split = kb_split;
  p.BNc = BNc;
  p.mt = mt;
  p.nchunks = nchunks;
  p.nks = nks;
  p.part = static_cast<float2*>(sc->buf[SplitCtx::OZ_PART].p);
  p.err = sc->err;
  const size_t smem = 1024 + 2 * OZ_GA + 2 * OZ_GB;
  static size_t configured = 0;
  if (raise_smem((const void*)oz_mma_kernel, configured, smem) != cudaSuccess)
    return sfail(sc, CTM_ECUDA, "cannot reserve shared memory for the fp64-accurate product");
  const unsigned grid = (unsigned)std::min<long>(152, tiles * nks);
  oz_mma_kernel<<<grid, OZ_THREADS, smem, s>>>(ta, tb, p);
  ++sc->oz_launches;
  if (cx)
    oz_reduce_kernel<cplx><<<grid_cap((long)M * N), 256, 0, s>>>(
        p.part, nks, M, N, Np, ea, ebx, (cplx*)C, ldc);
  else
    oz_reduce_kernel<double><<<grid_cap((long)M * N), 256, 0, s>>>(
        p.part, nks, M, N, Np, ea, ebx, (double*)C, ldc);
  if (launches) *launches += 2;
  if (cudaGetLastError() != cudaSuccess) return sfail(sc, CTM_ECUDA, "fp64-accurate product launch failed");
  return CTM_OK;
}

size_t split_partial_splits(size_t N, bool cx) {
  const size_t kb = ((cx ? 2 : 1) * N + BK - 1) / BK;
  return std::max<size_t>(32, (kb + KB_SPLIT_MAX - 1) / KB_SPLIT_MAX);
}

const char* split_last_error(const SplitCtx* sc) {
  return sc ? sc->msg.c_str() : "split precision not initialised";
}

}  // namespace ctm
