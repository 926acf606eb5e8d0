// Tensor-core GEMM on the fifth-generation tensor cores (tcgen05) for the
// U-Net's contractions whose operands are both K-contiguous:
//   C[m][n] = epilogue(alpha * sum_k A[m][k] * B[n][k])
// (A: activations [M][lda], B: weights [N][ldb], BF16, FP32 accumulation).
//
// One CTA computes a 128 x BN tile (BN = 32, 64, 128 or 256) with eight warps:
//   warp 0 (one lane)  streams 128 x 64 and BN x 64 operand tiles into a
//                      shared-memory ring of up to four stages with TMA
//                      (128-byte swizzle, zero fill outside the matrices);
//   warp 1 (one lane)  issues tcgen05.mma (kind::f16, M = 128, N = BN,
//                      K = 16 per instruction) accumulating in tensor memory
//                      and releases each stage with tcgen05.commit;
//   warp 2             allocates and frees the BN tensor-memory columns;
//   all eight warps    read the accumulator back (tcgen05.ld, 32 rows and
//                      half the columns per warp) into shared memory, then
//                      write coalesced rows through the epilogue (bias,
//                      residual, GELU with the pre-activation copy or GELU',
//                      FP32 or BF16 output).
// Every wait on an mbarrier has an iteration limit; on expiry the kernel sets
// the library's timeout flag, skips its stores, waits (again bounded) for its
// own copies and products still in flight and frees its tensor memory.
#include <cuda.h>
#include <cuda_bf16.h>

#include <atomic>
#include <cstring>

#include "nn_gemm.cuh"
#include "pe_internal.cuh"

namespace {

typedef __nv_bfloat16 bf16;
typedef __nv_bfloat162 bf162;

constexpr int TC_BM = 128, TC_BK = 64, TC_STAGES = 4, TC_THREADS = 256;
constexpr uint32_t kWaitLimit = 1u << 22;

template <int BN>
struct tc_cfg {
  static constexpr int A_BYTES = TC_BM * TC_BK * 2;  // 16 KB, 1024-byte multiple
  static constexpr int B_BYTES = BN * TC_BK * 2;     // 4/8/16/32 KB
  static constexpr int STAGE = A_BYTES + B_BYTES;
  static constexpr int C_LD = BN + 4;                        // FP32 staging row (floats)
  static constexpr int C_BYTES = TC_BM * C_LD * 4;
  // ring of `stages` operand stages, reused for the FP32 output tile; then
  // the barriers; plus slack to align the base to 1024 bytes
  static int smem(int stages) {
    const int ring = stages * STAGE > C_BYTES ? stages * STAGE : C_BYTES;
    return ((ring + 1023) / 1024) * 1024 + 1024 + 1024;
  }
  // instruction descriptor, kind::f16: D = F32 (bits 4-5), A = B = BF16
  // (bits 7-9, 10-12), both K-major (bits 15, 16 clear), N >> 3 (bits
  // 17-22), M >> 4 (bits 24-28)
  static constexpr uint32_t IDESC = (1u << 4) | (1u << 7) | (1u << 10) |
                                    ((uint32_t)(BN >> 3) << 17) | ((uint32_t)(TC_BM >> 4) << 24);
};

__device__ __forceinline__ uint32_t sm_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// Shared-memory matrix descriptor of a K-major tile with the 128-byte
// swizzle: start address >> 4 (bits 0-13), leading offset 16 B (unused for
// this layout), stride offset 1024 B between 8-row groups (bits 32-45),
// descriptor version 1 (bits 46-47), swizzle mode 2 = 128 B (bits 61-63).
__device__ __forceinline__ uint64_t kmajor_sw128_desc(uint32_t saddr) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)1 << 16) | ((uint64_t)(1024 >> 4) << 32) |
         ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

__device__ __forceinline__ void mbar_init(uint64_t *bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(sm_u32(bar)), "r"(count));
}
__device__ __forceinline__ void mbar_expect_tx(uint64_t *bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(sm_u32(bar)),
               "r"(bytes)
               : "memory");
}
// Bounded wait for the phase with the given parity to complete: at most
// `limit` polls (each mbarrier.try_wait may itself suspend the thread for a
// short, system-dependent time); false if the phase has not completed.
__device__ __forceinline__ bool mbar_wait(uint64_t *bar, uint32_t parity,
                                          uint32_t limit = kWaitLimit) {
  const uint32_t a = sm_u32(bar);
  for (uint32_t i = 0; i < limit; ++i) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void tma_load_2d(void *dst, const CUtensorMap *map, int x, int y,
                                            uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.2d.shared::cluster.global.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3}], [%4];\n" ::"r"(sm_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(x), "r"(y), "r"(sm_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tc_fence_before() {
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
}
__device__ __forceinline__ void tc_fence_after() {
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
}

__device__ __forceinline__ void tc_mma(uint32_t tmem, uint64_t adesc, uint64_t bdesc,
                                       uint32_t idesc, uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
      "l"(adesc), "l"(bdesc), "r"(idesc), "r"(accumulate)
      : "memory");
}
// Arrive on `bar` once every tcgen05 operation issued so far by this thread
// has completed.
__device__ __forceinline__ void tc_commit(uint64_t *bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
          sm_u32(bar))
      : "memory");
}

__device__ __forceinline__ void tc_ld16(uint32_t taddr, float (&v)[16]) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
  for (int i = 0; i < 16; ++i) v[i] = __uint_as_float(r[i]);
}

template <int BN>
__global__ void __launch_bounds__(TC_THREADS, 3)
    gemm_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                   const pe_gemm_args g, int stages, uint32_t wait_limit, unsigned int *err) {
  // wait_limit bounds the waits of the main loop and of the epilogue; the
  // clean-up after a failed wait always waits the full kWaitLimit for the
  // copies and products already issued (they complete in microseconds)
  using cfg = tc_cfg<BN>;
  extern __shared__ __align__(1024) uint8_t tc_smem_raw[];
  // 1024-byte aligned base for the swizzled tiles
  uint8_t *base = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  const int ring = stages * cfg::STAGE > cfg::C_BYTES ? stages * cfg::STAGE : cfg::C_BYTES;
  uint64_t *full = reinterpret_cast<uint64_t *>(base + ((ring + 1023) / 1024) * 1024);
  uint64_t *empty = full + TC_STAGES;
  uint64_t *accum = empty + TC_STAGES;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(accum + 1);
  __shared__ int s_fail;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m0 = blockIdx.x * TC_BM, n0 = blockIdx.y * BN;
  const int nk = (int)((g.K + TC_BK - 1) / TC_BK);

  if (threadIdx.x == 0) {
    s_fail = 0;
    for (int s = 0; s < stages; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    mbar_init(accum, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    asm volatile("prefetch.tensormap [%0];\n" ::"l"(reinterpret_cast<uint64_t>(&tmA)) : "memory");
    asm volatile("prefetch.tensormap [%0];\n" ::"l"(reinterpret_cast<uint64_t>(&tmB)) : "memory");
  }
  if (warp == 2) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     sm_u32(tmem_slot)),
                 "r"((uint32_t)BN)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  int issued = 0;  // k-blocks whose loads were issued (producer lane)
  if (warp == 0 && lane == 0) {
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % stages;
      const uint32_t ph = (uint32_t)(kb / stages) & 1u;
      if (!mbar_wait(empty + s, ph ^ 1u, wait_limit)) {
        atomicOr(&s_fail, 1);
        break;
      }
      uint8_t *sa = base + s * cfg::STAGE;
      mbar_expect_tx(full + s, (uint32_t)cfg::STAGE);
      tma_load_2d(sa, &tmA, kb * TC_BK, m0, full + s);
      tma_load_2d(sa + cfg::A_BYTES, &tmB, kb * TC_BK, n0, full + s);
      issued = kb + 1;
    }
  } else if (warp == 1 && lane == 0) {
    int kb = 0;
    for (; kb < nk; ++kb) {
      const int s = kb % stages;
      const uint32_t ph = (uint32_t)(kb / stages) & 1u;
      if (!mbar_wait(full + s, ph, wait_limit)) {
        atomicOr(&s_fail, 1);
        break;
      }
      tc_fence_after();
      const uint32_t sa = sm_u32(base + s * cfg::STAGE);
      const uint64_t ad = kmajor_sw128_desc(sa), bd = kmajor_sw128_desc(sa + cfg::A_BYTES);
#pragma unroll
      for (int k = 0; k < TC_BK / 16; ++k)  // +32 bytes per K step inside the swizzled row
        tc_mma(tmem, ad + (uint64_t)(2 * k), bd + (uint64_t)(2 * k), cfg::IDESC,
               (kb > 0 || k > 0) ? 1u : 0u);
      tc_commit(empty + s);
    }
    tc_commit(accum);  // all products issued above are complete
  }
  // epilogue: the accumulator goes through shared memory (the operand ring
  // is free once every product has completed), then all threads write
  // coalesced rows.  Warp w reads tensor-memory lanes 32 (w % 4) .. + 31
  // (its rows) for half of the columns.
  const bool ready = mbar_wait(accum, 0u, wait_limit);
  if (!ready) atomicOr(&s_fail, 1);
  tc_fence_after();
  __syncwarp();
  // a warp-uniform decision: tcgen05.ld needs the whole warp
  const bool ok = __all_sync(0xffffffffu, ready && !s_fail);
  float *Cs = reinterpret_cast<float *>(base);
  if (ok) {
    const int quad = warp & 3, half = warp >> 2;
    const int r = quad * 32 + lane;
    const uint32_t row = tmem + ((uint32_t)(quad * 32) << 16);
    for (int c = half * (BN / 2); c < (half + 1) * (BN / 2); c += 16) {
      float v[16];
      tc_ld16(row + (uint32_t)c, v);
      float4 *dst = reinterpret_cast<float4 *>(Cs + r * cfg::C_LD + c);
#pragma unroll
      for (int q = 0; q < 4; ++q)
        dst[q] = make_float4(v[4 * q] * g.alpha, v[4 * q + 1] * g.alpha, v[4 * q + 2] * g.alpha,
                             v[4 * q + 3] * g.alpha);
    }
  }
  __syncthreads();
  if (!s_fail) {
    for (int c = threadIdx.x; c < TC_BM * BN / 8; c += TC_THREADS) {
      const int r = c / (BN / 8), cc = (c % (BN / 8)) * 8;
      const int m = m0 + r, n = n0 + cc;
      if (m >= g.M || n >= g.N) continue;
      float v[8];
      const float4 a = *reinterpret_cast<const float4 *>(Cs + r * cfg::C_LD + cc);
      const float4 b = *reinterpret_cast<const float4 *>(Cs + r * cfg::C_LD + cc + 4);
      v[0] = a.x; v[1] = a.y; v[2] = a.z; v[3] = a.w;
      v[4] = b.x; v[5] = b.y; v[6] = b.z; v[7] = b.w;
      pe_gemm_store8(g, m, n, v);
    }
  }
  __syncthreads();
  if (s_fail) {
    // Let the copies issued by the producer land before the shared memory is
    // released: each issued stage's full barrier completes when its bytes
    // have arrived (bounded wait), and the products were committed above.
    if (threadIdx.x == 0) {
      atomicOr(err, PE_ERR_TIMEOUT);
    }
    if (warp == 0 && lane == 0) {
      for (int kb = (issued > stages ? issued - stages : 0); kb < issued; ++kb)
        mbar_wait(full + kb % stages, (uint32_t)(kb / stages) & 1u);
    }
    if (warp == 1 && lane == 0) mbar_wait(accum, 0u);
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 2) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"((uint32_t)BN)
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// The streaming form: BF16 output rows, persistent CTAs.
//
// Most of the U-Net's contractions are narrow (K, N = 32..512 over millions of
// pixels): they are bound by moving rows through the SM, so the kernel is
// built around that.  A CTA walks its share of the output tiles; one lane
// loads operand blocks (TMA ring), one issues the products of tile i + 1 into
// one half of the tensor memory while the epilogue warps drain tile i from the
// other.  Two groups of four epilogue warps take alternate tiles; each warp
// owns 32 rows (its tensor-memory lanes) and goes through 32-column slabs:
// registers -> its own 64-byte-row staging slab (64-byte swizzle, conflict
// free for a row per lane) -> TMA store.  The residual or the pre-activation a
// mode reads arrives the same way (TMA load into the slab, prefetched), is
// replaced in place by the result and stored from there, so global memory
// sees only whole-row bulk copies and no CTA-wide barrier stands between
// tiles.
//   MODE 0  C = acc (+ bias)            MODE 1  C = acc (+ bias) + X
//   MODE 2  Z = acc (+ bias), C = GELU  MODE 3  C = (acc (+ bias)) GELU'(X)
//   MODE 4  FP32 C = acc (+ bias) (+ R), N <= 8: the heads, whose rows are too
//           short to stage; a lane writes its row's few values itself (1048576
//           rows, K = 32: 37 us, 70 us through the staged kernel)
// The arithmetic per element is pe_gemm_store8's, in the same order.
//
// Against the kernel above on the same contractions (which holds a 128 x 256
// FP32 tile in shared memory, so one CTA per SM loads, multiplies and stores in
// turn), 64 channels, 524288 pixels: 1x1 expansion with GELU 375 -> 159 us (603
// MB: 89 us of copy bandwidth; the erf of 134M values bounds it), data gradient
// through GELU' 542 -> 239 us (603 MB; erf and exp), projection with residual
// 110 -> 70 us (402 MB, 59 us of copy bandwidth), data gradient 75 -> 50 us (336
// MB, 49 us).  All results equal bit for bit.  Column tiles of 128 at most: two
// CTAs per SM, whose tensor memory (2 x 128 columns each) fills the SM's 512.
// ---------------------------------------------------------------------------
constexpr int ST_THREADS = 320;  // producer, issuer, eight epilogue warps
constexpr int ST_MAX_BIAS = 1024;  // columns whose bias is kept in shared memory

// GELU' of a BF16 pre-activation, for MODE 3: the kernel tabulates it for
// 2^-11 <= |z| < 8 (two signs of 14 binades of 128 values, 15 KB of shared
// memory per CTA, filled once by pe_gelu_grad itself) and computes the rest.
// One shared-memory load in place of an erf and an exp per value, which had
// bounded it: the data gradient of 64 -> 256 channels at 524288 pixels (603 MB, 89
// us of copy bandwidth), 239 -> 143 us.  The negative half starts 2048 floats in,
// a shift of the sign bit; rows with a value outside the table (found by packed
// 16-bit minima and maxima) are recomputed value by value.
constexpr uint32_t DG_LO = 116u << 7, DG_N = 14u * 128u, DG_NEG = 2048u;
constexpr uint32_t DG_FLOATS = DG_NEG + DG_N + 1u;
__device__ __noinline__ float dg_outside(float z) { return pe_gelu_grad(z); }

template <int BN, int MODE, bool WIDE>
struct st_cfg {
  static constexpr int STAGES = WIDE ? 1 : (BN == 128 ? 2 : 3);
  static constexpr int NB = (MODE == 1 && BN == 32) ? 3 : 2;  // staging slabs per warp
  static constexpr int COLS = WIDE ? 64 : 32;                  // columns of a slab
  static constexpr int SLAB = 32 * COLS * 2;
  static constexpr int A_BYTES = TC_BM * TC_BK * 2, B_BYTES = BN * TC_BK * 2;
  static constexpr int STAGE = A_BYTES + B_BYTES;
  static constexpr int STAGING = 8 * NB * SLAB;
  // barriers (an even number of 8-byte words, so that the bias after them and
  // the two words that follow is 16-byte aligned)
  static constexpr int BARS = (2 * STAGES + 4 + 8 * NB + 1 + 1) & ~1;
  static_assert((STAGES * STAGE) % 1024 == 0 && STAGING % 1024 == 0 && (BARS * 8) % 16 == 0,
                "alignment of the slabs, the barriers and the bias");
  static constexpr uint32_t IDESC = tc_cfg<BN>::IDESC;
  // the bias of N columns takes whole slabs: the epilogue reads a slab's width of
  // it also where the columns end inside the slab
  static __host__ __device__ constexpr int bias_floats(int n) { return (n + COLS - 1) / COLS * COLS; }
  static int smem(int n_bias) {
    return 1024 + STAGES * STAGE + STAGING + BARS * 8 + 16 + bias_floats(n_bias) * 4 +
           (MODE == 3 ? DG_FLOATS * 4 : 0);
  }
};

// The image behind an im2col operand: element (p, tap C + c) of the matrix is
// channel c of the pixel that tap (3 ky + kx) reads at pixel p.
struct conv_img {
  int C, W, H;  // C = 0: a plain matrix
};

struct st_args {
  int M, N, K;
  int tiles_n;
  int items;  // output tiles
  float alpha;
  const float *bias;
  conv_img img;  // of A
  float *c32;    // MODE 4
  int64_t ldc, ldr;
  const bf16 *r;
  uint32_t wait_limit;
  unsigned int *err;
};

// Bounded wait that also gives up once another role of the CTA has.
__device__ __forceinline__ bool st_wait(uint64_t *bar, uint32_t parity, uint32_t limit,
                                        volatile int *fail) {
  const uint32_t a = sm_u32(bar);
  for (uint32_t i = 0; i < limit; ++i) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(a), "r"(parity)
        : "memory");
    if (done) return true;
    if ((i & 63u) == 63u && *fail) return false;
  }
  return false;
}

__device__ __forceinline__ void mbar_arrive(uint64_t *bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(sm_u32(bar)) : "memory");
}
__device__ __forceinline__ void tma_store_2d(const CUtensorMap *map, const void *src, int x, int y) {
  asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%1, %2}], [%3];\n" ::"l"(
                   reinterpret_cast<uint64_t>(map)),
               "r"(x), "r"(y), "r"(sm_u32(src))
               : "memory");
}
// A column of the 3x3 neighbourhood matrix: consecutive pixels in raster order
// from (w, h, n) on, each moved by (ow, oh), channels c .. c + 63; pixels outside
// the image read as zero (a TMA load in im2col mode).
__device__ __forceinline__ void tma_load_im2col(void *dst, const CUtensorMap *map, int c, int w,
                                                int h, int n, uint16_t ow, uint16_t oh,
                                                uint64_t *bar) {
  asm volatile(
      "cp.async.bulk.tensor.4d.shared::cluster.global.im2col.mbarrier::complete_tx::bytes"
      " [%0], [%1, {%2, %3, %4, %5}], [%6], {%7, %8};\n" ::"r"(sm_u32(dst)),
      "l"(reinterpret_cast<uint64_t>(map)), "r"(c), "r"(w), "r"(h), "r"(n), "r"(sm_u32(bar)),
      "h"(ow), "h"(oh)
      : "memory");
}

__device__ __forceinline__ void load_conv_box(void *dst, const CUtensorMap *map, const conv_img &im,
                                              int k0, int p, uint64_t *bar) {
  int tap = k0 / im.C, c = k0 - tap * im.C;
  if (tap > 8) {  // past the matrix: channels outside the image are zero
    tap = 8;
    c = im.C;
  }
  const int x = p % im.W, y = p / im.W;
  tma_load_im2col(dst, map, c, x - 1, y % im.H - 1, y / im.H, (uint16_t)(tap % 3),
                  (uint16_t)(tap / 3), bar);
}

__device__ __forceinline__ void bulk_commit() {
  asm volatile("cp.async.bulk.commit_group;\n" ::: "memory");
}
template <int N>
__device__ __forceinline__ void bulk_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read %0;\n" ::"n"(N) : "memory");
}
__device__ __forceinline__ void bulk_wait_all() {
  asm volatile("cp.async.bulk.wait_group 0;\n" ::: "memory");
}
__device__ __forceinline__ void async_fence() {
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
}

__device__ __forceinline__ void tc_ld32(uint32_t taddr, float (&v)[32]) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]),
        "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]), "=r"(r[19]), "=r"(r[20]),
        "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]), "=r"(r[25]), "=r"(r[26]), "=r"(r[27]),
        "=r"(r[28]), "=r"(r[29]), "=r"(r[30]), "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
  for (int i = 0; i < 32; ++i) v[i] = __uint_as_float(r[i]);
}

template <int BN, int MODE, bool WIDE>
__global__ void __launch_bounds__(ST_THREADS, 2)
    gemm_stream_kernel(const __grid_constant__ CUtensorMap tmA,
                       const __grid_constant__ CUtensorMap tmB,
                       const __grid_constant__ CUtensorMap tmC,
                       const __grid_constant__ CUtensorMap tmX, const st_args g) {
  using cfg = st_cfg<BN, MODE, WIDE>;
  constexpr int S = cfg::STAGES, NB = cfg::NB, CW = cfg::COLS, SLABS = BN / CW, SLAB = cfg::SLAB;
  constexpr bool XIN = MODE == 1 || MODE == 3;
  extern __shared__ __align__(1024) uint8_t tc_smem_raw[];
  uint8_t *base = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  uint8_t *staging = base + S * cfg::STAGE;
  uint64_t *full = reinterpret_cast<uint64_t *>(staging + cfg::STAGING);
  uint64_t *empty = full + S, *tfull = empty + S, *tempty = tfull + 2, *xbar = tempty + 2;
  uint64_t *drain = xbar + 8 * NB;
  uint32_t *tmem_slot = reinterpret_cast<uint32_t *>(full + cfg::BARS);
  volatile int *s_fail = reinterpret_cast<volatile int *>(tmem_slot + 1);
  float *s_bias = reinterpret_cast<float *>(tmem_slot + 4);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int nk = (g.K + TC_BK - 1) / TC_BK;

  if (threadIdx.x == 0) {
    *s_fail = 0;
    for (int s = 0; s < S; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, 1);
    }
    for (int s = 0; s < 2; ++s) {
      mbar_init(tfull + s, 1);
      mbar_init(tempty + s, 4);  // the four warps of a group
    }
    for (int s = 0; s < 8 * NB; ++s) mbar_init(xbar + s, 1);
    mbar_init(drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  const int n_pad = g.bias ? cfg::bias_floats(g.N) : 0;
  if (g.bias)
    for (int i = threadIdx.x; i < n_pad; i += ST_THREADS) s_bias[i] = i < g.N ? g.bias[i] : 0.0f;
  float *s_dg = s_bias + n_pad;  // [DG_N], 1 for z > 0; from DG_NEG on for z < 0
  if (MODE == 3)
    for (uint32_t i = threadIdx.x; i < 2 * (DG_N + 1u); i += ST_THREADS) {
      const uint32_t k = i % (DG_N + 1u), neg = i / (DG_N + 1u);
      s_dg[k + neg * DG_NEG] =
          k < DG_N ? pe_gelu_grad(__uint_as_float((DG_LO + k + neg * 0x8000u) << 16)) : 1.0f;
    }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     sm_u32(tmem_slot)),
                 "r"((uint32_t)(2 * BN))
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;

  uint32_t c = 0;  // k-blocks whose loads the producer issued
  if (warp == 0) {
    if (lane == 0) {
      // ---- producer ------------------------------------------------------
      bool ok = true;
      for (int it = blockIdx.x; ok && it < g.items; it += gridDim.x) {
        const int m0 = (it / g.tiles_n) * TC_BM, n0 = (it % g.tiles_n) * BN;
        for (int kb = 0; kb < nk; ++kb, ++c) {
          const int s = (int)(c % S);
          if (!st_wait(empty + s, ((c / S) & 1u) ^ 1u, g.wait_limit, s_fail)) {
            *s_fail = 1;
            ok = false;
            break;
          }
          uint8_t *sa = base + s * cfg::STAGE;
          mbar_expect_tx(full + s, (uint32_t)cfg::STAGE);
          if (MODE == 0 && g.img.C) load_conv_box(sa, &tmA, g.img, kb * TC_BK, m0, full + s);
          else tma_load_2d(sa, &tmA, kb * TC_BK, m0, full + s);
          tma_load_2d(sa + cfg::A_BYTES, &tmB, kb * TC_BK, n0, full + s);
        }
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // ---- product issuer ------------------------------------------------
      uint32_t i = 0;
      bool ok = true;
      for (int it = blockIdx.x; ok && it < g.items; it += gridDim.x, ++i) {
        const uint32_t st = i & 1u;
        if (!st_wait(tempty + st, ((i >> 1) & 1u) ^ 1u, g.wait_limit, s_fail)) {
          *s_fail = 1;
          ok = false;
          break;
        }
        tc_fence_after();
        for (int kb = 0; kb < nk; ++kb, ++c) {
          const int s = (int)(c % S);
          if (!st_wait(full + s, (c / S) & 1u, g.wait_limit, s_fail)) {
            *s_fail = 1;
            ok = false;
            break;
          }
          tc_fence_after();
          const uint32_t sa = sm_u32(base + s * cfg::STAGE);
          const uint64_t ad = kmajor_sw128_desc(sa), bd = kmajor_sw128_desc(sa + cfg::A_BYTES);
          const int steps = min(TC_BK / 16, (g.K - kb * TC_BK + 15) / 16);
          for (int k = 0; k < steps; ++k)
            tc_mma(tmem + st * BN, ad + (uint64_t)(2 * k), bd + (uint64_t)(2 * k), cfg::IDESC,
                   (kb > 0 || k > 0) ? 1u : 0u);
          tc_commit(empty + s);
        }
        if (ok) tc_commit(tfull + st);
      }
    }
  } else {
    // ---- epilogue ----------------------------------------------------------
    const int ew = warp - 2, grp = ew >> 2, quad = warp & 3;
    uint8_t *slabs = staging + ew * NB * SLAB;
    uint64_t *xb = xbar + ew * NB;
    // this lane's row in a slab: chunk q (16 bytes) at row + ((q ^ sw) << 4)
    const uint32_t row = (uint32_t)lane * (CW * 2u);
    const uint32_t sw = WIDE ? (uint32_t)lane & 7u : ((uint32_t)lane >> 1) & 3u;
    const uint32_t tlane = tmem + (uint32_t)(grp * BN) + ((uint32_t)(quad * 32) << 16);
    // a cursor over this warp's slabs: tiles of its parity, the slabs that
    // hold rows and columns of the matrix
    struct cursor {
      int it, j;
    };
    auto inside = [&](const cursor &k) {
      return (k.it / g.tiles_n) * TC_BM + quad * 32 < g.M &&
             (k.it % g.tiles_n) * BN + k.j * CW < g.N;
    };
    auto step = [&](cursor &k) {
      do {
        if (++k.j == SLABS) {
          k.j = 0;
          k.it += 2 * (int)gridDim.x;
        }
      } while (k.it < g.items && !inside(k));
    };
    auto load_x = [&](const cursor &k, uint32_t seq) {
      const uint32_t b = seq % NB;
      mbar_expect_tx(xb + b, SLAB);
      tma_load_2d(slabs + b * SLAB, &tmX, (k.it % g.tiles_n) * BN + k.j * CW,
                  (k.it / g.tiles_n) * TC_BM + quad * 32, xb + b);
    };
    const int first = (int)(blockIdx.x + grp * gridDim.x);
    cursor ld = {first, -1};
    uint32_t ld_seq = 0;
    if (XIN) {
      step(ld);
      for (int k = 0; k < NB - 1 && ld.it < g.items; ++k, ++ld_seq, step(ld))
        if (lane == 0) load_x(ld, ld_seq);
    }
    uint32_t seq = 0, u = 0;
    bool ok = true;
    for (int it = first; ok && it < g.items; it += 2 * (int)gridDim.x, ++u) {
      const int m0 = (it / g.tiles_n) * TC_BM + quad * 32, n0 = (it % g.tiles_n) * BN;
      bool ready = st_wait(tfull + grp, u & 1u, g.wait_limit, s_fail);
      ok = __all_sync(0xffffffffu, ready);
      if (!ok) break;
      tc_fence_after();
      if (MODE == 4 && m0 < g.M) {
        float v[16];
        tc_ld16(tlane, v);
        const int m = m0 + lane;
#pragma unroll
        for (int n = 0; n < 8; ++n)
          if (m < g.M && n < g.N) {
            float x = __fmul_rn(v[n], g.alpha);
            if (g.bias) x += s_bias[n];
            if (g.r) x += __bfloat162float(g.r[(int64_t)m * g.ldr + n]);
            g.c32[(int64_t)m * g.ldc + n] = x;
          }
      }
#pragma unroll 1
      for (int j = 0; j < (MODE == 4 ? 0 : SLABS); ++j) {
        const int c0 = n0 + CW * j;
        if (m0 >= g.M || c0 >= g.N) continue;
        const uint32_t b = seq % NB;
        uint8_t *slab = slabs + b * SLAB;
        if (XIN) {
          // the slab read ahead: its buffer's last store has been read out
          if (ld.it < g.items) {
            if (lane == 0) {
              bulk_wait_read<0>();
              load_x(ld, ld_seq);
            }
            ++ld_seq;
            step(ld);
          }
          ready = st_wait(xb + b, (seq / NB) & 1u, g.wait_limit, s_fail);
          ok = __all_sync(0xffffffffu, ready);
          if (!ok) break;
        }
#pragma unroll 1
        for (int h = 0; h < CW / 32; ++h) {  // 32 columns at a time
          float v[32];
          tc_ld32(tlane + (uint32_t)(CW * j + 32 * h), v);
          if (g.alpha != 1.0f) {
#pragma unroll
            for (int e = 0; e < 32; ++e) v[e] = __fmul_rn(v[e], g.alpha);
          }
          if (g.bias) {
            const float4 *bp = reinterpret_cast<const float4 *>(s_bias + c0 + 32 * h);
#pragma unroll
            for (int q = 0; q < 8; ++q) {
              const float4 t = bp[q];
              v[4 * q] += t.x;
              v[4 * q + 1] += t.y;
              v[4 * q + 2] += t.z;
              v[4 * q + 3] += t.w;
            }
          }
          if (MODE == 1) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint4 xv = *reinterpret_cast<const uint4 *>(slab + row + (((q + 4 * h) ^ sw) << 4));
              const uint32_t xw[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                v[8 * q + 2 * e] += __uint_as_float(xw[e] << 16);
                v[8 * q + 2 * e + 1] += __uint_as_float(xw[e] & 0xffff0000u);
              }
            }
          }
          if (MODE == 3) {
            uint32_t lo = 0xffffffffu, hi = 0u;  // of the row's |z|, as 16-bit pairs
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const uint4 xv = *reinterpret_cast<const uint4 *>(slab + row + (((q + 4 * h) ^ sw) << 4));
              const uint32_t xw[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const uint32_t mag = xw[e] & 0x7fff7fffu;
                lo = __vminu2(lo, mag);
                hi = __vmaxu2(hi, mag);
                const uint32_t k0 = min((mag & 0xffffu) - DG_LO, DG_N);
                const uint32_t k1 = min((mag >> 16) - DG_LO, DG_N);
                v[8 * q + 2 * e] *= s_dg[k0 + ((xw[e] >> 4) & DG_NEG)];
                v[8 * q + 2 * e + 1] *= s_dg[k1 + ((xw[e] >> 20) & DG_NEG)];
              }
            }
            const uint32_t least = min(lo & 0xffffu, lo >> 16), most = max(hi & 0xffffu, hi >> 16);
            if (least < DG_LO || most >= DG_LO + DG_N) {
              // (their factor so far is the entry 1 past the table's end)
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const bf16 *zp = reinterpret_cast<const bf16 *>(slab + row + (((q + 4 * h) ^ sw) << 4));
#pragma unroll
                for (int e = 0; e < 8; ++e) {
                  const float z = __bfloat162float(zp[e]);
                  if (!(fabsf(z) >= 0.00048828125f && fabsf(z) < 8.0f)) v[8 * q + e] *= dg_outside(z);
                }
              }
            }
          }
          auto put = [&](uint8_t *dst) {
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              uint4 o;
              bf162 *op = reinterpret_cast<bf162 *>(&o);
#pragma unroll
              for (int e = 0; e < 4; ++e)
                op[e] = __floats2bfloat162_rn(v[8 * q + 2 * e], v[8 * q + 2 * e + 1]);
              *reinterpret_cast<uint4 *>(dst + row + (((q + 4 * h) ^ sw) << 4)) = o;
            }
          };
          if (MODE == 2) {
            // both slabs of the warp: the pre-activation, then the result
            if (h == 0) {
              if (lane == 0) bulk_wait_read<0>();
              __syncwarp();
            }
            put(slabs);
#pragma unroll
            for (int e = 0; e < 32; ++e) v[e] = pe_gelu(v[e]);
            put(slabs + SLAB);
          } else {
            if (!XIN && h == 0) {
              if (lane == 0) bulk_wait_read<NB - 1>();
              __syncwarp();
            }
            put(slab);
          }
        }
        async_fence();
        __syncwarp();
        if (lane == 0) {
          if (MODE == 2) {
            tma_store_2d(&tmX, slabs, c0, m0);
            tma_store_2d(&tmC, slabs + SLAB, c0, m0);
          } else {
            tma_store_2d(&tmC, slab, c0, m0);
          }
          bulk_commit();
        }
        ++seq;
      }
      if (!ok) break;
      // this half of the tensor memory may take the group's next tile
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(tempty + grp);
    }
    if (!ok) {
      *s_fail = 1;
      if (XIN && lane == 0)  // loads in flight land before the memory is released
        for (uint32_t k = seq; k < ld_seq; ++k) mbar_wait(xb + k % NB, (k / NB) & 1u);
    }
    if (lane == 0) bulk_wait_all();
  }
  __syncthreads();
  if (*s_fail) {
    // whichever role gave up: the copies in flight land before the shared memory
    // is released (each block's full barrier completes when its bytes arrived),
    // the products in flight complete before the tensor memory is freed
    if (warp == 0 && lane == 0) {
      atomicOr(g.err, PE_ERR_TIMEOUT);
      for (uint32_t k = c > (uint32_t)S ? c - S : 0; k < c; ++k)
        mbar_wait(full + k % S, (k / S) & 1u);
    }
    if (warp == 1 && lane == 0) {
      tc_commit(drain);
      mbar_wait(drain, 0u);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"((uint32_t)(2 * BN))
                 : "memory");
  }
}

// ---------------------------------------------------------------------------
// Weight gradients of a linear layer: dW[n][k] = sum_p dY[p][n] X[p][k] and
// db[n] = sum_p dY[p][n] in one pass over both matrices.
//
// Both operands are contiguous along their channels, so their tiles (64 pixels
// x 64 channels, TMA with the 128-byte swizzle) are MN-major for the tensor
// cores and the products accumulate over pixels in tensor memory: up to four
// accumulators of 128 rows (channels of the wider operand) by up to 256
// columns (the narrower one), so at the network's narrow levels each pixel is
// read once.  Four more warps add up dY's columns from the same shared-memory
// tiles (one column-sum kernel and one read of dY fewer) and write the partial
// results at the end.  A CTA takes one tile of the result over one stretch of
// pixels; part[split][N K + N] is then added in split order.
//
// The tensor cores truncate where an FP32 addition rounds, so a sum drifts with
// the number of products added into one accumulator (1e-6 of the result after
// 1024 pixels, 2.3e-6 after 2048, against 64 bits).  Where a tile leaves room,
// pixel blocks take several copies of its accumulators in turn, and there are at
// least as many sums over the pixels as the split mma.sync kernel makes.
// Bound by reading X and dY: 64 channels, 524288 pixels, both layers of a
// block (671 MB, 99 us of copy bandwidth) take 153 us with their partials'
// sums, against 296 us for the split mma.sync kernel and 150 us for the column
// sums.  Over the gradient of a 32 x 256^2 batch: 14.2 -> 4.8 ms.
// ---------------------------------------------------------------------------
constexpr int WG_PX = 64, WG_THREADS = 192, WG_BOX = WG_PX * 128, WG_STAGES = 4;

struct wg_args {
  int N, K;           // dW is [N][K]
  int mt, nt;         // accumulators of a tile, columns of each
  int sets;           // copies of the accumulators, taken in turn by pixel blocks
  int nbx;            // 64-channel boxes of the column operand per stage
  int tiles_n;
  int a_is_dy;        // rows of the accumulators: dY's channels, else X's
  int64_t P;
  int px_per_split;   // a multiple of WG_PX
  int stages;
  float *part;
  int want_db;
  conv_img img;       // of X
  uint32_t cols;      // tensor-memory columns
  uint32_t wait_limit;
  unsigned int *err;
};

// MN-major tile with the 128-byte swizzle: 64 channels (128 bytes) by 8 pixels
// per 1024-byte atom, `lbo` bytes to the next 64 channels, 1024 to the next 8
// pixels.
__device__ __forceinline__ uint64_t mnmajor_sw128_desc(uint32_t saddr, uint32_t lbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)(lbo >> 4) << 16) |
         ((uint64_t)(1024 >> 4) << 32) | ((uint64_t)1 << 46) | ((uint64_t)2 << 61);
}

__global__ void __launch_bounds__(WG_THREADS)
    wgrad_tc_kernel(const __grid_constant__ CUtensorMap tmA, const __grid_constant__ CUtensorMap tmB,
                    const wg_args g) {
  extern __shared__ __align__(1024) uint8_t tc_smem_raw[];
  uint8_t *base = reinterpret_cast<uint8_t *>(
      (reinterpret_cast<uintptr_t>(tc_smem_raw) + 1023) & ~static_cast<uintptr_t>(1023));
  __shared__ uint64_t full[WG_STAGES], empty[WG_STAGES], accum, drain;
  __shared__ uint32_t tmem_slot;
  __shared__ volatile int s_fail;
  __shared__ float s_db[4][512];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tm = blockIdx.y / g.tiles_n, tn = blockIdx.y % g.tiles_n;
  const int m0 = tm * g.mt * 128, n0 = tn * g.nt;
  const int a_boxes = 2 * g.mt;
  const uint32_t stage_bytes = (uint32_t)(a_boxes + g.nbx) * WG_BOX;
  const int64_t p0 = (int64_t)blockIdx.x * g.px_per_split;
  const int64_t pe = p0 + g.px_per_split < g.P ? p0 + g.px_per_split : g.P;
  const int nk = (int)((pe - p0 + WG_PX - 1) / WG_PX);
  // the tile whose other operand is its first adds up dY's columns
  const bool sums = g.want_db && (g.a_is_dy ? tn == 0 : tm == 0);

  if (threadIdx.x == 0) {
    s_fail = 0;
    for (int s = 0; s < g.stages; ++s) {
      mbar_init(full + s, 1);
      mbar_init(empty + s, sums ? 5 : 1);
    }
    mbar_init(&accum, 1);
    mbar_init(&drain, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     sm_u32(&tmem_slot)),
                 "r"(g.cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  int issued = 0;  // pixel blocks whose loads the producer issued
  if (warp == 0) {
    if (lane == 0) {
      for (int kb = 0; kb < nk; ++kb) {
        const int s = kb % g.stages;
        if (!st_wait(empty + s, ((uint32_t)(kb / g.stages) & 1u) ^ 1u, g.wait_limit, &s_fail)) {
          s_fail = 1;
          break;
        }
        uint8_t *sa = base + (size_t)s * stage_bytes;
        const int px = (int)(p0 + (int64_t)kb * WG_PX);
        mbar_expect_tx(full + s, stage_bytes);
        const bool ca = g.img.C && !g.a_is_dy, cb = g.img.C && g.a_is_dy;  // where X is
        for (int b = 0; b < a_boxes; ++b) {
          if (ca) load_conv_box(sa + b * WG_BOX, &tmA, g.img, m0 + 64 * b, px, full + s);
          else tma_load_2d(sa + b * WG_BOX, &tmA, m0 + 64 * b, px, full + s);
        }
        for (int b = 0; b < g.nbx; ++b) {
          uint8_t *d = sa + (a_boxes + b) * WG_BOX;
          if (cb) load_conv_box(d, &tmB, g.img, n0 + 64 * b, px, full + s);
          else tma_load_2d(d, &tmB, n0 + 64 * b, px, full + s);
        }
        issued = kb + 1;
      }
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // both operands MN-major (bits 15 and 16), as tc_cfg::IDESC otherwise
      const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) |
                             ((uint32_t)(g.nt >> 3) << 17) | ((uint32_t)(128 >> 4) << 24);
      bool ok = true;
      for (int kb = 0; kb < nk; ++kb) {
        const int s = kb % g.stages;
        if (!st_wait(full + s, (uint32_t)(kb / g.stages) & 1u, g.wait_limit, &s_fail)) {
          s_fail = 1;
          ok = false;
          break;
        }
        tc_fence_after();
        const uint32_t sa = sm_u32(base + (size_t)s * stage_bytes);
        const uint32_t sb = sa + (uint32_t)a_boxes * WG_BOX;
        for (int i = 0; i < g.mt; ++i) {
          const uint64_t ad = mnmajor_sw128_desc(sa + (uint32_t)(2 * i) * WG_BOX, WG_BOX);
          const uint64_t bd = mnmajor_sw128_desc(sb, WG_BOX);
#pragma unroll
          for (int k = 0; k < WG_PX / 16; ++k)  // 16 pixels: two atoms of 1024 bytes
            tc_mma(tmem + (uint32_t)((kb % g.sets * g.mt + i) * g.nt), ad + (uint64_t)(128 * k),
                   bd + (uint64_t)(128 * k), idesc, (kb >= g.sets || k > 0) ? 1u : 0u);
        }
        tc_commit(empty + s);
      }
      if (ok) tc_commit(&accum);
    }
  } else {
    const int t = threadIdx.x - 64, j = t & 7, r0 = t >> 3;
    bool ok = true;
    float *out = g.part + (int64_t)blockIdx.x * ((int64_t)g.N * g.K + g.N);
    if (sums) {
      // dY's columns: thread t adds chunk j (eight channels) of every box at
      // pixels r0, r0 + 16, ...: a block's four values, then the blocks' sums
      // with the error of each addition kept (Knuth's two-sum), so that a long
      // stretch costs no precision: plain chains over up to thousands of pixels
      // were less exact than the column sums of 256 pixels that they replace.
      const int nd = g.a_is_dy ? a_boxes : g.nbx, d0 = g.a_is_dy ? 0 : a_boxes;
      float sum[8][8], lost[8][8];
#pragma unroll
      for (int b = 0; b < 8; ++b)
#pragma unroll
        for (int e = 0; e < 8; ++e) sum[b][e] = lost[b][e] = 0.0f;
      for (int kb = 0; kb < nk; ++kb) {
        const int s = kb % g.stages;
        ok = __all_sync(0xffffffffu,
                        st_wait(full + s, (uint32_t)(kb / g.stages) & 1u, g.wait_limit, &s_fail));
        if (!ok) break;
        const uint8_t *sd = base + (size_t)s * stage_bytes + (size_t)d0 * WG_BOX + r0 * 128 +
                            ((j ^ (r0 & 7)) << 4);
#pragma unroll
        for (int b = 0; b < 8; ++b) {
          if (b < nd) {
            float v[8];
#pragma unroll
            for (int r = 0; r < WG_PX / 16; ++r) {
              const uint4 u = *reinterpret_cast<const uint4 *>(sd + b * WG_BOX + r * 16 * 128);
              const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
              for (int e = 0; e < 4; ++e) {
                const float v0 = __uint_as_float(w[e] << 16), v1 = __uint_as_float(w[e] & 0xffff0000u);
                v[2 * e] = r ? v[2 * e] + v0 : v0;
                v[2 * e + 1] = r ? v[2 * e + 1] + v1 : v1;
              }
            }
#pragma unroll
            for (int e = 0; e < 8; ++e) {
              const float a = sum[b][e], t = __fadd_rn(a, v[e]), z = __fsub_rn(t, a);
              lost[b][e] += __fadd_rn(__fsub_rn(a, __fsub_rn(t, z)), __fsub_rn(v[e], z));
              sum[b][e] = t;
            }
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty + s);
      }
#pragma unroll
      for (int b = 0; b < 8; ++b)
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          // (the error of an infinite sum is NaN)
          float v = fabsf(lost[b][e]) < INFINITY ? sum[b][e] + lost[b][e] : sum[b][e];
          v += __shfl_xor_sync(0xffffffffu, v, 8);
          v += __shfl_xor_sync(0xffffffffu, v, 16);
          if (lane < 8) s_db[warp - 2][64 * b + 8 * j + e] = v;
        }
      asm volatile("bar.sync 1, 128;\n" ::: "memory");
      const int w0 = g.a_is_dy ? m0 : n0, wn = g.a_is_dy ? g.mt * 128 : g.nt;
      if (ok)
        for (int c = t; c < wn; c += 128)
          if (w0 + c < g.N)
            out[(int64_t)g.N * g.K + w0 + c] = (s_db[0][c] + s_db[1][c]) + (s_db[2][c] + s_db[3][c]);
    }
    ok = __all_sync(0xffffffffu, ok && st_wait(&accum, 0u, g.wait_limit, &s_fail));
    if (!ok) {
      s_fail = 1;
    } else {
      tc_fence_after();
      const int quad = warp & 3, na = g.a_is_dy ? g.N : g.K, nb = g.a_is_dy ? g.K : g.N;
      for (int i = 0; i < g.mt; ++i) {
        const int m = m0 + i * 128 + quad * 32 + lane;
        for (int c = 0; c < g.nt; c += 16) {
          float v[16];
          tc_ld16(tmem + (uint32_t)(i * g.nt + c) + ((uint32_t)(quad * 32) << 16), v);
          for (int z = 1; z < g.sets && z < nk; ++z) {
            float a[16];
            tc_ld16(tmem + (uint32_t)((z * g.mt + i) * g.nt + c) + ((uint32_t)(quad * 32) << 16), a);
#pragma unroll
            for (int e = 0; e < 16; ++e) v[e] += a[e];
          }
          if (m >= na) continue;
          if (g.a_is_dy) {
            float *dst = out + (int64_t)m * g.K + n0 + c;
            if (n0 + c + 16 <= nb && (reinterpret_cast<uintptr_t>(dst) & 15) == 0) {
#pragma unroll
              for (int e = 0; e < 4; ++e)
                reinterpret_cast<float4 *>(dst)[e] =
                    make_float4(v[4 * e], v[4 * e + 1], v[4 * e + 2], v[4 * e + 3]);
            } else {
#pragma unroll
              for (int e = 0; e < 16; ++e)
                if (n0 + c + e < nb) dst[e] = v[e];
            }
          } else {  // transposed: consecutive lanes write consecutive k
            float *dst = out + (int64_t)(n0 + c) * g.K + m;
#pragma unroll
            for (int e = 0; e < 16; ++e)
              if (n0 + c + e < nb) dst[(int64_t)e * g.K] = v[e];
          }
        }
      }
    }
  }
  __syncthreads();
  if (s_fail) {  // as in gemm_stream_kernel: nothing is left in flight
    if (warp == 0 && lane == 0) {
      atomicOr(g.err, PE_ERR_TIMEOUT);
      for (int k = issued > g.stages ? issued - g.stages : 0; k < issued; ++k)
        mbar_wait(full + k % g.stages, (uint32_t)(k / g.stages) & 1u);
    }
    if (warp == 1 && lane == 0) {
      tc_commit(&drain);
      mbar_wait(&drain, 0u);
    }
  }
  tc_fence_before();
  __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(g.cols)
                 : "memory");
  }
}

// dW, db = the partials added in split order: eight lanes take splits z, z + 8,
// ..., and their sums are added in order.
__global__ void wgrad_reduce_kernel(const float *__restrict__ part, int splits, int64_t nw,
                                    int64_t n_all, float *__restrict__ dW, float *__restrict__ db) {
  __shared__ float red[8][33];
  const int64_t t = (int64_t)blockIdx.x * 32 + threadIdx.x;
  float v = 0.0f;
  if (t < n_all)
    for (int z = threadIdx.y; z < splits; z += 8) v += part[(int64_t)z * n_all + t];
  red[threadIdx.y][threadIdx.x] = v;
  __syncthreads();
  if (threadIdx.y == 0 && t < n_all) {
    float s = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += red[k][threadIdx.x];
    if (t < nw) dW[t] = s;
    else if (db) db[t - nw] = s;
  }
}

typedef CUresult (*encode_tiled_fn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                    const cuuint64_t *, const cuuint64_t *, const cuuint32_t *,
                                    const cuuint32_t *, CUtensorMapInterleave, CUtensorMapSwizzle,
                                    CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

encode_tiled_fn encoder() {
  static encode_tiled_fn fn = nullptr;
  static bool tried = false;
  if (!tried) {
    tried = true;
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    if (cudaGetDriverEntryPointByVersion("cuTensorMapEncodeTiled", &p, 12000, cudaEnableDefault,
                                         &q) == cudaSuccess &&
        q == cudaDriverEntryPointSuccess)
      fn = reinterpret_cast<encode_tiled_fn>(p);
  }
  return fn;
}

// Row-major [rows][ld] BF16 matrix, K = inner extent; box 64 x box_rows,
// 128-byte swizzle, zero fill outside.
bool make_map(CUtensorMap *map, const void *ptr, int64_t rows, int64_t K, int64_t ld, int box_rows) {
  encode_tiled_fn enc = encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)K, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)TC_BK, (cuuint32_t)box_rows};
  cuuint32_t estr[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

typedef CUresult (*encode_im2col_fn)(CUtensorMap *, CUtensorMapDataType, cuuint32_t, void *,
                                     const cuuint64_t *, const cuuint64_t *, const int *,
                                     const int *, cuuint32_t, cuuint32_t, const cuuint32_t *,
                                     CUtensorMapInterleave, CUtensorMapSwizzle,
                                     CUtensorMapL2promotion, CUtensorMapFloatOOBfill);

encode_im2col_fn im2col_encoder() {
  static const encode_im2col_fn fn = []() -> encode_im2col_fn {
    void *p = nullptr;
    cudaDriverEntryPointQueryResult q;
    const bool ok = cudaGetDriverEntryPointByVersion("cuTensorMapEncodeIm2col", &p, 12000,
                                                     cudaEnableDefault, &q) == cudaSuccess &&
                    q == cudaDriverEntryPointSuccess;
    return ok ? reinterpret_cast<encode_im2col_fn>(p) : nullptr;
  }();
  return fn;
}

// BF16 [B][H][W][C] as the neighbourhood matrix of a 3x3 convolution with zero
// padding 1: boxes of `pixels` pixels by 64 channels.
bool make_conv_map(CUtensorMap *map, const void *ptr, int B, int H, int W, int C, int pixels) {
  encode_im2col_fn enc = im2col_encoder();
  if (!enc) return false;
  cuuint64_t dims[4] = {(cuuint64_t)C, (cuuint64_t)W, (cuuint64_t)H, (cuuint64_t)B};
  cuuint64_t strides[3] = {(cuuint64_t)C * 2, (cuuint64_t)W * C * 2, (cuuint64_t)H * W * C * 2};
  int lower[2] = {-1, -1}, upper[2] = {-1, -1};
  cuuint32_t estr[4] = {1, 1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 4, const_cast<void *>(ptr), dims, strides, lower,
             upper, 64, (cuuint32_t)pixels, estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

// Polls of the kernel's main-loop waits (pe_nn_set_wait_limit).
std::atomic<uint32_t> g_wait_limit{kWaitLimit};

template <int BN>
pe_status launch_bn(const pe_gemm_args &g, cudaStream_t s) {
  using cfg = tc_cfg<BN>;
  CUtensorMap ma, mb;
  if (!make_map(&ma, g.A, g.M, g.K, g.sam, TC_BM) || !make_map(&mb, g.B, g.N, g.K, g.sbn, BN))
    return PE_EUNSUPPORTED;  // the caller takes the other kernel
  // as many stages as K-blocks, up to four; the shared memory this takes
  // also caps the CTAs per SM so their tensor memory (BN columns each)
  // stays within the SM's 512 columns
  const int nk = (int)((g.K + TC_BK - 1) / TC_BK);
  const int stages = nk < TC_STAGES ? nk : TC_STAGES;
  const int smem = cfg::smem(stages);
  static bool attr = false;
  if (!attr) {
    PE_TRY_CUDA(cudaFuncSetAttribute(gemm_tc_kernel<BN>, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     cfg::smem(TC_STAGES)));
    // the whole unified L1 as shared memory: up to three CTAs of the
    // narrow shapes side by side (registers are capped for three as well)
    PE_TRY_CUDA(cudaFuncSetAttribute(gemm_tc_kernel<BN>, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     (int)cudaSharedmemCarveoutMaxShared));
    attr = true;
  }
  dim3 grid((unsigned)((g.M + TC_BM - 1) / TC_BM), (unsigned)((g.N + BN - 1) / BN));
  gemm_tc_kernel<BN><<<grid, TC_THREADS, smem, s>>>(ma, mb, g, stages, g_wait_limit.load(),
                                                     pe_err_word());
  PE_TRY_LAUNCH("gemm_tc_kernel");
  return PE_OK;
}

// Row-major BF16 [rows][ld] in slabs of 32 rows by 32 or 64 columns, swizzled
// over their row's bytes, for the streaming kernel's output rows and the rows
// its epilogue reads.
bool make_slab_map(CUtensorMap *map, const void *ptr, int64_t rows, int64_t cols, int64_t ld,
                   int width) {
  encode_tiled_fn enc = encoder();
  if (!enc) return false;
  cuuint64_t dims[2] = {(cuuint64_t)cols, (cuuint64_t)rows};
  cuuint64_t strides[1] = {(cuuint64_t)ld * 2};
  cuuint32_t box[2] = {(cuuint32_t)width, 32};
  cuuint32_t estr[2] = {1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void *>(ptr), dims, strides, box,
             estr, CU_TENSOR_MAP_INTERLEAVE_NONE,
             width == 64 ? CU_TENSOR_MAP_SWIZZLE_128B : CU_TENSOR_MAP_SWIZZLE_64B,
             CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

int tc_sms() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

// `conv`: A is the neighbourhood matrix of that image (batch images of it).
template <int BN, int MODE, bool WIDE>
pe_status launch_stream(const pe_gemm_args &g, cudaStream_t s, const conv_img *conv = nullptr,
                        int batch = 0) {
  using cfg = st_cfg<BN, MODE, WIDE>;
  CUtensorMap ma, mb, mc, mx;
  const int64_t items = (int64_t)((g.M + TC_BM - 1) / TC_BM) * ((g.N + BN - 1) / BN);
  if (items >= (1ll << 30)) return PE_EUNSUPPORTED;  // (tile numbers are 32-bit)
  if (!(conv ? make_conv_map(&ma, g.A, batch, conv->H, conv->W, conv->C, TC_BM)
             : make_map(&ma, g.A, g.M, g.K, g.sam, TC_BM)) ||
      !make_map(&mb, g.B, g.N, g.K, g.sbn, BN) ||
      (MODE != 4 && !make_slab_map(&mc, g.C, g.M, g.N, g.ldc, cfg::COLS)))
    return PE_EUNSUPPORTED;
  if (MODE == 4) mx = mc = ma;  // (unused)
  else if (MODE == 0) mx = mc;
  else if (!make_slab_map(&mx, MODE == 1 ? g.R : g.Z, g.M, g.N, MODE == 1 ? g.ldr : g.ldz,
                          cfg::COLS))
    return PE_EUNSUPPORTED;
  static bool attr = false;
  if (!attr) {
    PE_TRY_CUDA(cudaFuncSetAttribute(gemm_stream_kernel<BN, MODE, WIDE>,
                                     cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     cfg::smem(ST_MAX_BIAS)));
    PE_TRY_CUDA(cudaFuncSetAttribute(gemm_stream_kernel<BN, MODE, WIDE>,
                                     cudaFuncAttributePreferredSharedMemoryCarveout,
                                     (int)cudaSharedmemCarveoutMaxShared));
    attr = true;
  }
  st_args a;
  memset(&a, 0, sizeof(a));
  a.M = g.M;
  a.N = g.N;
  a.K = (int)g.K;
  a.tiles_n = (g.N + BN - 1) / BN;
  a.items = (int)items;
  a.alpha = g.alpha;
  a.bias = g.bias;
  if (conv) a.img = *conv;
  if (MODE == 4) {
    a.c32 = static_cast<float *>(g.C);
    a.ldc = g.ldc;
    a.r = g.R;
    a.ldr = g.ldr;
  }
  a.wait_limit = g_wait_limit.load();
  a.err = pe_err_word();
  const int most = 2 * tc_sms();  // two CTAs per SM
  gemm_stream_kernel<BN, MODE, WIDE><<<a.items < most ? a.items : most, ST_THREADS,
                                 cfg::smem(g.bias ? g.N : 0), s>>>(ma, mb, mc, mx,
                                                                                    a);
  PE_TRY_LAUNCH("gemm_stream_kernel");
  return PE_OK;
}

// The streaming kernel's mode for these arguments, -1 when it does not apply:
// a TMA store writes BF16 rows on 16-byte boundaries, so wider FP32 outputs and
// unaligned rows stay with the other kernel, as does an epilogue
// outside the four forms.  Where both apply the streaming kernel was the
// faster one at every shape of the network (gradients of a 32 x 256^2 batch:
// 21.4 -> 11.7 ms over its 113 contractions).
int stream_mode(const pe_gemm_args &g) {
  if (g.c_f32 && g.N <= 8 && g.gelu == 0 && g.beta == 0.0f && g.K < (1ll << 30)) return 4;
  if (g.c_f32 || !g.vec_c || g.K >= (1ll << 30) || (g.bias && g.N > ST_MAX_BIAS)) return -1;
  if (g.gelu == 0) return g.R ? 1 : 0;
  if (g.R) return -1;
  if (g.gelu == 1) return g.Z ? 2 : -1;
  return 3;
}

template <int BN>
pe_status launch_stream_mode(int mode, const pe_gemm_args &g, cudaStream_t s) {
  switch (mode) {
    case 0: return launch_stream<BN, 0, false>(g, s);
    case 1: return launch_stream<BN, 1, false>(g, s);
    case 2: return launch_stream<BN, 2, false>(g, s);
    default: return launch_stream<BN, 3, false>(g, s);
  }
}

// Column tile and slab width.  The GELU modes move two rows of N per row of K
// (N = 4 K): their slabs take 64 columns, half the rows for the TMA unit, where
// one operand block is the whole of K and so a single ring stage makes room (GELU'
// form, 64 channels, 524288 pixels: 174 -> 161 us before the packed range test).
pe_status launch_stream_shape(int mode, const pe_gemm_args &g, cudaStream_t s) {
  if (mode == 4) return launch_stream<32, 4, false>(g, s);
  if (g.N > 64 && g.K <= TC_BK && mode == 2) return launch_stream<128, 2, true>(g, s);
  if (g.N > 64 && g.K <= TC_BK && mode == 3) return launch_stream<128, 3, true>(g, s);
  if (g.N <= 32) return launch_stream_mode<32>(mode, g, s);
  if (g.N <= 64) return launch_stream_mode<64>(mode, g, s);
  return launch_stream_mode<128>(mode, g, s);
}

// Tile and split of a weight gradient.  The wider operand gives the rows; its
// 128-row accumulators share a tile as far as tensor memory (512 columns) and
// shared memory allow.  About 304 CTAs (two per SM where their tensor memory
// fits; a constant, so that sums do not depend on the device), at least 512
// pixels each unless the mma.sync kernel makes more sums.
struct wg_plan {
  int a_is_dy, mt, nt, nbx, sets, tiles_m, tiles_n, stages, smem;
  int64_t px, splits;
  uint32_t cols;
};
wg_plan plan_wgrad(int64_t P, int N, int K) {
  wg_plan w;
  w.a_is_dy = N >= K;
  const int na = w.a_is_dy ? N : K, nb = w.a_is_dy ? K : N;
  const int t = (na + 127) / 128;
  w.nt = nb >= 256 ? 256 : (nb + 15) / 16 * 16;
  w.nbx = (w.nt + 63) / 64;
  w.tiles_n = (nb + w.nt - 1) / w.nt;
  const int most = w.nt > 128 ? 2 : (w.nt > 64 ? 3 : 4);  // <= 512 columns, 64-80 KB a stage
  w.tiles_m = (t + most - 1) / most;
  w.mt = (t + w.tiles_m - 1) / w.tiles_m;
  w.sets = 256 / (w.mt * w.nt);
  w.sets = w.sets < 1 ? 1 : (w.sets > 8 ? 8 : w.sets);
  w.cols = 32;
  while ((int)w.cols < w.sets * w.mt * w.nt) w.cols *= 2;
  const int stage = (2 * w.mt + w.nbx) * WG_BOX;
  const int room = w.cols <= 256 ? 100 * 1024 : 208 * 1024;  // two CTAs per SM, or one
  w.stages = room / stage;
  w.stages = w.stages < 2 ? 2 : (w.stages > WG_STAGES ? WG_STAGES : w.stages);
  w.smem = w.stages * stage + 1024;
  const int64_t tiles = (int64_t)w.tiles_m * w.tiles_n;
  int64_t splits = ((w.cols <= 256 ? 304 : 152) + tiles - 1) / tiles;
  const int64_t most_splits = (P + 511) / 512;
  if (splits > most_splits) splits = most_splits;
  // at least the sums of the mma.sync kernel (one per 256 pixels at most)
  const int64_t least = (pe_gemm_split(N, K, P) + w.sets - 1) / w.sets;
  if (splits < least) splits = least;
  w.px = (P + splits - 1) / splits;
  w.px = (w.px + WG_PX - 1) / WG_PX * WG_PX;
  if (w.px > WG_PX && (P + w.px - 1) / w.px < least) w.px -= WG_PX;
  w.splits = (P + w.px - 1) / w.px;
  return w;
}

}  // namespace

bool pe_gemm_tc_eligible(const pe_gemm_args &g) {
  auto al16 = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  return g.sak == 1 && g.sbk == 1 && g.sam % 8 == 0 && g.sbn % 8 == 0 && al16(g.A) && al16(g.B) &&
         g.K >= 16 && g.M >= 1 && g.N >= 1 && (int64_t)g.M + TC_BM < (1ll << 31) && encoder();
}

pe_status pe_gemm_tc(const pe_gemm_args &g, cudaStream_t s) {
  const int mode = stream_mode(g);
  if (mode >= 0) {
    const pe_status st = launch_stream_shape(mode, g, s);
    if (st != PE_EUNSUPPORTED) return st;
  }
  if (g.N <= 32) return launch_bn<32>(g, s);
  if (g.N <= 64) return launch_bn<64>(g, s);
  if (g.N <= 128) return launch_bn<128>(g, s);
  return launch_bn<256>(g, s);
}

pe_status pe_wgrad_reduce(const float *part, int splits, int64_t nw, int64_t n_all, float *dW, float *db,
                          cudaStream_t s) {
  wgrad_reduce_kernel<<<(unsigned)((n_all + 31) / 32), dim3(32, 8), 0, s>>>(part, splits, nw, n_all,
                                                                          dW, db);
  PE_TRY_LAUNCH("wgrad_reduce_kernel");
  return PE_OK;
}

bool pe_wgrad_tc_eligible(const void *dY, int64_t ldy, const void *X, int64_t ldx, int64_t P, int32_t N,
                          int32_t K) {
  auto al16 = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  return ldy % 8 == 0 && ldx % 8 == 0 && al16(dY) && al16(X) && N >= 8 && K >= 8 && P >= 16 &&
         P < (1ll << 31) - 4096 && encoder();
}

bool pe_conv3_tc_sizes(int32_t B, int32_t H, int32_t W, int32_t C, int32_t N) {
  return C % 64 == 0 && N > 64 && N <= ST_MAX_BIAS && N % 8 == 0 && W < 32768 && H < 32768 &&
         (int64_t)B * H * W >= 16 && (int64_t)B * H * W < (1ll << 31) - 4096 && encoder() &&
         im2col_encoder();
}

pe_status pe_conv3_tc(const pe_gemm_args &g, int32_t B, int32_t H, int32_t W, int32_t C,
                      cudaStream_t s) {
  const conv_img im = {C, W, H};
  return launch_stream<128, 0, false>(g, s, &im, B);
}

size_t pe_wgrad_tc_workspace(int64_t P, int32_t N, int32_t K) {
  return (size_t)plan_wgrad(P, N, K).splits * ((size_t)N * K + N) * sizeof(float);
}

pe_status pe_wgrad_tc(const void *dY, int64_t ldy, const void *X, int64_t ldx, int64_t P, int32_t N,
                      int32_t K, float *dW, float *db, float *part, cudaStream_t s,
                      const int32_t *conv) {
  const wg_plan w = plan_wgrad(P, N, K);
  CUtensorMap my, mx;
  if (!make_map(&my, dY, P, N, ldy, WG_PX) ||
      !(conv ? make_conv_map(&mx, X, conv[0], conv[1], conv[2], K / 9, WG_PX)
             : make_map(&mx, X, P, K, ldx, WG_PX)))
    return PE_EUNSUPPORTED;
  static bool attr = false;
  if (!attr) {
    PE_TRY_CUDA(cudaFuncSetAttribute(wgrad_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize,
                                     209 * 1024));
    PE_TRY_CUDA(cudaFuncSetAttribute(wgrad_tc_kernel, cudaFuncAttributePreferredSharedMemoryCarveout,
                                     (int)cudaSharedmemCarveoutMaxShared));
    attr = true;
  }
  wg_args g;
  memset(&g, 0, sizeof(g));
  g.N = N;
  g.K = K;
  g.mt = w.mt;
  g.nt = w.nt;
  g.nbx = w.nbx;
  g.sets = w.sets;
  g.tiles_n = w.tiles_n;
  g.a_is_dy = w.a_is_dy;
  g.P = P;
  g.px_per_split = (int)w.px;
  g.stages = w.stages;
  g.part = part;
  g.want_db = db != nullptr;
  g.cols = w.cols;
  if (conv) g.img = conv_img{K / 9, conv[2], conv[1]};
  g.wait_limit = g_wait_limit.load();
  g.err = pe_err_word();
  const dim3 grid((unsigned)w.splits, (unsigned)(w.tiles_m * w.tiles_n));
  wgrad_tc_kernel<<<grid, WG_THREADS, w.smem, s>>>(w.a_is_dy ? my : mx, w.a_is_dy ? mx : my, g);
  PE_TRY_LAUNCH("wgrad_tc_kernel");
  return pe_wgrad_reduce(part, (int)w.splits, (int64_t)N * K, (int64_t)N * K + N, dW, db, s);
}

extern "C" pe_status pe_nn_set_wait_limit(int64_t polls) {
  if (polls > (int64_t)UINT32_MAX) return pe_fail(PE_EINVAL, "pe_nn_set_wait_limit: at most 2^32 - 1");
  g_wait_limit.store(polls < 0 ? kWaitLimit : (uint32_t)polls);
  return PE_OK;
}
