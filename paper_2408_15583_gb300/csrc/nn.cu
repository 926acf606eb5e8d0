// Layer kernels of the learned GFB completion network (a8): BF16 activations
// in NHWC layout, FP32 accumulation, FP32 master weights.
//
//   GEMM (tensor cores, mma.sync m16n8k16 BF16 -> FP32) with fused bias,
//   residual, GELU epilogues and deterministic split-K; im2col / col2im for
//   3x3 convolutions; depthwise 7x7; LayerNorm over channels; max-pool 2x2;
//   pixel shuffle x2; channel copies for concatenation; bias / LayerNorm /
//   depthwise weight reductions in a fixed order; the losses of Eq. 17-21 with
//   their gradients; AdamW.
#include <cuda_bf16.h>

#include <cstring>
#include <type_traits>

#include "pe_internal.cuh"
#include "nn_gemm.cuh"

typedef __nv_bfloat16 bf16;
typedef __nv_bfloat162 bf162;

namespace {

__device__ __forceinline__ float b2f(bf16 x) { return __bfloat162float(x); }
__device__ __forceinline__ bf16 f2b(float x) { return __float2bfloat16_rn(x); }

int n_sms() {
  static int n = 0;
  if (!n) {
    int dev = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&n, cudaDevAttrMultiProcessorCount, dev);
    if (n <= 0) n = 1;
  }
  return n;
}

int grid1(int64_t n, int threads, int per_sm = 16) {
  int64_t b = (n + threads - 1) / threads;
  int64_t cap = (int64_t)n_sms() * per_sm;
  if (b < 1) b = 1;
  return (int)(b < cap ? b : cap);
}

// ---------------------------------------------------------------------------
// GEMM
// ---------------------------------------------------------------------------


// Block tile 128 (M) x 64 (N) x 32 (K), eight warps of 32 x 32, a
// three-stage cp.async pipeline; fragments by ldmatrix (transposed for the
// operands whose M or N index is the contiguous one, as in the weight
// gradients).  Shared-memory rows are padded by 16 bytes so the eight row
// addresses of an ldmatrix fall in distinct banks.
constexpr int TM = 128, TN = 64, TK = 32, STAGES = 3, GEMM_THREADS = 256;
constexpr int A_STAGE = TM * (TK + 8);  // >= TK * (TM + 8)
constexpr int B_STAGE = TN * (TK + 8);  // >= TK * (TN + 8)
static_assert(A_STAGE >= TK * (TM + 8) && B_STAGE >= TK * (TN + 8), "stage sizes");
constexpr int GEMM_SMEM = STAGES * (A_STAGE + B_STAGE) * 2;
constexpr int C_LD = TN + 4;  // FP32 staging of the output tile
static_assert(TM * C_LD * 4 <= GEMM_SMEM, "epilogue staging fits the pipeline buffers");

__device__ __forceinline__ uint32_t smem_u32(const void *p) {
  return static_cast<uint32_t>(__cvta_generic_to_shared(p));
}

// 16-byte asynchronous copy; bytes < 16 zero-fills the rest (0: all zeros,
// the source is then not read).
__device__ __forceinline__ void cp16(void *dst, const void *src, int bytes) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem_u32(dst)), "l"(src),
               "r"(bytes));
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;\n" ::); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;\n" ::"n"(N));
}

__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const void *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const void *p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];\n"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem_u32(p)));
}

// Stage one operand tile.  ROWS x TK with K contiguous (KC: S[row][k], row
// stride TK + 8) or TK x ROWS with the row index contiguous (S[k][row], row
// stride ROWS + 8).  X(row, k) = X[row * s_r + k * s_k]; rows >= n_rows and
// k >= k_end read as zero.  vec: 16-byte copies are legal (aligned base,
// contiguous stride 1 and the other stride a multiple of 8 elements).
template <bool KC, int ROWS>
__device__ __forceinline__ void stage_tile(bf16 *S, const bf16 *__restrict__ X, int64_t s_r,
                                           int64_t s_k, int row0, int64_t k0, int n_rows,
                                           int64_t k_end, bool vec) {
  const bf16 zero = f2b(0.0f);
  if (KC) {
    constexpr int CH = ROWS * TK / 8;
    for (int c = threadIdx.x; c < CH; c += GEMM_THREADS) {
      const int r = c >> 2, kc = (c & 3) * 8;
      const int gr = row0 + r;
      const int64_t gk = k0 + kc;
      bf16 *d = S + r * (TK + 8) + kc;
      if (vec) {
        int64_t left = k_end - gk;
        int bytes = (gr < n_rows && left > 0) ? (int)(left >= 8 ? 16 : 2 * left) : 0;
        cp16(d, bytes ? X + (int64_t)gr * s_r + gk : X, bytes);
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e)
          d[e] = (gr < n_rows && gk + e < k_end) ? X[(int64_t)gr * s_r + (gk + e) * s_k] : zero;
      }
    }
  } else {
    constexpr int CH = ROWS * TK / 8, PER_K = ROWS / 8;
    for (int c = threadIdx.x; c < CH; c += GEMM_THREADS) {
      const int k = c / PER_K, rc = (c % PER_K) * 8;
      const int64_t gk = k0 + k;
      const int gr = row0 + rc;
      bf16 *d = S + k * (ROWS + 8) + rc;
      if (vec) {
        int left = n_rows - gr;
        int bytes = (gk < k_end && left > 0) ? (left >= 8 ? 16 : 2 * left) : 0;
        cp16(d, bytes ? X + gk * s_k + gr : X, bytes);
      } else {
#pragma unroll
        for (int e = 0; e < 8; ++e)
          d[e] = (gk < k_end && gr + e < n_rows) ? X[(int64_t)(gr + e) * s_r + gk * s_k] : zero;
      }
    }
  }
}

// C = epilogue(alpha * A B) over one 128 x 64 tile and the K range of split
// blockIdx.z; with split-K the raw products go to part[z][M][N].
template <bool AK, bool BK>
__global__ void __launch_bounds__(GEMM_THREADS, 3) gemm_kernel(const pe_gemm_args g) {
  __shared__ __align__(128) bf16 smem[STAGES * (A_STAGE + B_STAGE)];
  bf16 *As = smem, *Bs = smem + STAGES * A_STAGE;
  const int m0 = blockIdx.x * TM, n0 = blockIdx.y * TN;
  const int64_t kb = (int64_t)blockIdx.z * g.k_per_split;
  int64_t ke = kb + g.k_per_split;
  if (ke > g.K) ke = g.K;
  const int nk = (int)((ke - kb + TK - 1) / TK);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wm = (warp & 3) * 32, wn = (warp >> 2) * 32;
  const int gq = lane >> 2, tq = lane & 3;
  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[i][j][e] = 0.0f;

  auto load = [&](int st, int kt) {
    if (kt < nk) {
      const int64_t k0 = kb + (int64_t)kt * TK;
      stage_tile<AK, TM>(As + st * A_STAGE, g.A, g.sam, g.sak, m0, k0, g.M, ke, g.vec_a);
      stage_tile<BK, TN>(Bs + st * B_STAGE, g.B, g.sbn, g.sbk, n0, k0, g.N, ke, g.vec_b);
    }
    cp_commit();
  };
#pragma unroll
  for (int st = 0; st < STAGES - 1; ++st) load(st, st);
  for (int kt = 0; kt < nk; ++kt) {
    cp_wait<STAGES - 2>();
    __syncthreads();
    const bf16 *A = As + (kt % STAGES) * A_STAGE, *B = Bs + (kt % STAGES) * B_STAGE;
#pragma unroll
    for (int kk = 0; kk < TK; kk += 16) {
      uint32_t a[2][4], b[4][2];
#pragma unroll
      for (int i = 0; i < 2; ++i) {
        if (AK) {
          const int r = wm + 16 * i + (lane & 7) + ((lane >> 3) & 1) * 8;
          ldsm4(a[i], A + r * (TK + 8) + kk + (lane >> 4) * 8);
        } else {
          const int k = kk + (lane >> 4) * 8 + (lane & 7);
          ldsm4t(a[i], A + k * (TM + 8) + wm + 16 * i + ((lane >> 3) & 1) * 8);
        }
      }
#pragma unroll
      for (int j = 0; j < 4; j += 2) {
        uint32_t r[4];
        if (BK) {
          const int n = wn + 8 * (j + (lane >> 4)) + (lane & 7);
          ldsm4(r, B + n * (TK + 8) + kk + ((lane >> 3) & 1) * 8);
        } else {
          const int q = lane >> 3;
          const int k = kk + (q & 1) * 8 + (lane & 7);
          ldsm4t(r, B + k * (TN + 8) + wn + 8 * (j + (q >> 1)));
        }
        b[j][0] = r[0];
        b[j][1] = r[1];
        b[j + 1][0] = r[2];
        b[j + 1][1] = r[3];
      }
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          asm volatile(
              "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, "
              "{%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
              : "+f"(acc[i][j][0]), "+f"(acc[i][j][1]), "+f"(acc[i][j][2]), "+f"(acc[i][j][3])
              : "r"(a[i][0]), "r"(a[i][1]), "r"(a[i][2]), "r"(a[i][3]), "r"(b[j][0]),
                "r"(b[j][1]));
    }
    load((kt + STAGES - 1) % STAGES, kt + STAGES - 1);
  }
  cp_wait<0>();
  __syncthreads();
  // stage alpha * acc as FP32 in shared memory, then write rows of eight
  float *Cs = reinterpret_cast<float *>(smem);
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const int r = wm + 16 * i + gq + 8 * h, c = wn + 8 * j + 2 * tq;
        *reinterpret_cast<float2 *>(Cs + r * C_LD + c) =
            make_float2(acc[i][j][2 * h] * g.alpha, acc[i][j][2 * h + 1] * g.alpha);
      }
  __syncthreads();
  const bool split = g.part != nullptr;
  for (int c = threadIdx.x; c < TM * TN / 8; c += GEMM_THREADS) {
    const int r = c >> 3, cc = (c & 7) * 8;
    const int m = m0 + r, n = n0 + cc;
    if (m >= g.M || n >= g.N) continue;
    float v[8];
#pragma unroll
    for (int e = 0; e < 8; ++e) v[e] = Cs[r * C_LD + cc + e];
    if (split) {
      float *dst = g.part + ((int64_t)blockIdx.z * g.M + m) * g.N + n;
      for (int e = 0; e < 8 && n + e < g.N; ++e) dst[e] = v[e];
      continue;
    }
    pe_gemm_store8(g, m, n, v);
  }
}

// C[m][n] = alpha A[m] B[n] (K = 1: the data gradient of a one-output head), BF16,
// eight columns per thread.  The one product is exact in FP32, so this is what
// the contraction kernels give.  (157 us there for 2.1M x 32, 134 MB.)
__global__ void outer_kernel(const bf16 *__restrict__ A, int64_t sam, const bf16 *__restrict__ Bv,
                             int64_t sbn, int64_t M, int NV, float alpha, bf16 *__restrict__ Cm,
                             int64_t ldc) {
  const int64_t total = M * NV;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int n = (int)(t % NV) * 8;
    const int64_t m = t / NV;
    const float a = b2f(A[m * sam]);
    uint4 u;
    bf162 *e = reinterpret_cast<bf162 *>(&u);
#pragma unroll
    for (int k = 0; k < 4; ++k)  // (+ 0: a product of -0 is a sum of +0 there)
      e[k] = __floats2bfloat162_rn(
          __fmul_rn(__fadd_rn(__fmul_rn(a, b2f(Bv[(n + 2 * k) * sbn])), 0.0f), alpha),
          __fmul_rn(__fadd_rn(__fmul_rn(a, b2f(Bv[(n + 2 * k + 1) * sbn])), 0.0f), alpha));
    *reinterpret_cast<uint4 *>(Cm + m * ldc + n) = u;
  }
}

// Sum of the split-K partials in a fixed order (lane ty of a (32, 8) block
// takes splits ty, ty + 8, ...; the eight are added in order), then the
// epilogue.
__global__ void gemm_splitk_reduce(const pe_gemm_args g, int split) {
  __shared__ float red[8][33];
  const int64_t total = (int64_t)g.M * g.N;
  const int64_t t = (int64_t)blockIdx.x * 32 + threadIdx.x;
  float v = 0.0f;
  if (t < total)
    for (int z = threadIdx.y; z < split; z += 8) v += g.part[(int64_t)z * total + t];
  red[threadIdx.y][threadIdx.x] = v;
  __syncthreads();
  if (threadIdx.y == 0 && t < total) {
    float s = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += red[k][threadIdx.x];
    pe_gemm_store(g, (int)(t / g.N), (int)(t % g.N), s);
  }
}

// The same sums for at most eight splits (one per lane ty above, so they are
// added in order), a thread taking eight columns of a row: 16-byte accesses and
// no thread without a split.  16384 x 256, two splits: 134 us above, 11 us here.
__global__ void __launch_bounds__(256) gemm_splitk_reduce8(const pe_gemm_args g, int split) {
  const int64_t total = (int64_t)g.M * g.N;
  for (int64_t t = ((int64_t)blockIdx.x * blockDim.x + threadIdx.x) * 8; t < total;
       t += (int64_t)gridDim.x * blockDim.x * 8) {
    float v[8] = {0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f, 0.0f};
    for (int z = 0; z < split; ++z) {
      const float4 *q = reinterpret_cast<const float4 *>(g.part + (int64_t)z * total + t);
      const float4 a = __ldcs(q), b = __ldcs(q + 1);
      v[0] += a.x;
      v[1] += a.y;
      v[2] += a.z;
      v[3] += a.w;
      v[4] += b.x;
      v[5] += b.y;
      v[6] += b.z;
      v[7] += b.w;
    }
    pe_gemm_store8(g, (int)(t / g.N), (int)(t % g.N), v);
  }
}

// ---------------------------------------------------------------------------
// 3x3 convolution helpers (NHWC, zero padding 1): col[p][(ky*3+kx)*C + c]
// ---------------------------------------------------------------------------
// VEC channels per thread: 8 (one 16-byte load and store) when C is a
// multiple of 8 and the buffers are 16-byte aligned, else 1.  The index
// arithmetic runs once per VEC channels.
template <int VEC>
struct chunk_of;
template <>
struct chunk_of<1> {
  using T = bf16;
};
template <>
struct chunk_of<8> {
  using T = uint4;
};

template <int VEC>
__global__ void im2col3_kernel(const bf16 *__restrict__ X, int B, int H, int W, int C,
                               bf16 *__restrict__ col) {
  using T = typename chunk_of<VEC>::T;
  const int CV = C / VEC;
  const T *Xv = reinterpret_cast<const T *>(X);
  T *colv = reinterpret_cast<T *>(col);
  const int64_t total = (int64_t)B * H * W * 9 * CV;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int cv = (int)(t % CV);
    const int64_t r = t / CV;
    const int tap = (int)(r % 9);
    const int64_t p = r / 9;
    const int x = (int)(p % W);
    const int64_t q = p / W;
    const int y = (int)(q % H), b = (int)(q / H);
    const int yy = y + tap / 3 - 1, xx = x + tap % 3 - 1;
    T v;
    if (yy >= 0 && yy < H && xx >= 0 && xx < W) {
      v = Xv[(((int64_t)b * H + yy) * W + xx) * CV + cv];
    } else {
      memset(&v, 0, sizeof(T));  // bf16 zero is all-zero bits
    }
    colv[t] = v;
  }
}

// dX[b,y,x,c] = sum over taps of dcol at the pixel that read (y, x) through
// that tap (taps in order 0..8, FP32 sums).
template <int VEC>
__global__ void col2im3_kernel(const bf16 *__restrict__ dcol, int B, int H, int W, int C,
                               bf16 *__restrict__ dX) {
  const int CV = C / VEC;
  const int64_t total = (int64_t)B * H * W * CV;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int cv = (int)(t % CV);
    const int64_t p = t / CV;
    const int x = (int)(p % W);
    const int64_t q = p / W;
    const int y = (int)(q % H), b = (int)(q / H);
    float s[VEC];
#pragma unroll
    for (int k = 0; k < VEC; ++k) s[k] = 0.0f;
    for (int tap = 0; tap < 9; ++tap) {
      const int py = y - (tap / 3 - 1), px = x - (tap % 3 - 1);
      if (py < 0 || py >= H || px < 0 || px >= W) continue;
      const bf16 *src = dcol + ((((int64_t)b * H + py) * W + px) * 9 + tap) * C + (int64_t)cv * VEC;
      if (VEC == 8) {
        const uint4 u = *reinterpret_cast<const uint4 *>(src);
        const bf16 *e = reinterpret_cast<const bf16 *>(&u);
#pragma unroll
        for (int k = 0; k < VEC; ++k) s[k] += b2f(e[k]);
      } else {
        s[0] += b2f(src[0]);
      }
    }
    bf16 *dst = dX + p * C + (int64_t)cv * VEC;
    if (VEC == 8) {
      uint4 u;
      bf16 *e = reinterpret_cast<bf16 *>(&u);
#pragma unroll
      for (int k = 0; k < VEC; ++k) e[k] = f2b(s[k]);
      *reinterpret_cast<uint4 *>(dst) = u;
    } else {
      dst[0] = f2b(s[0]);
    }
  }
}

// ---------------------------------------------------------------------------
// depthwise 7x7 (zero padding 3), weights w[ky][kx][c] FP32; C even, rows of
// channel pairs (bf16x2).
// ---------------------------------------------------------------------------
// Both kernels work on channel pairs as packed FP32 pairs (one fma.f32x2 per
// tap and pixel: the pipe's rate is that of two FMAs, but one issue slot) and
// are laid out so that a converted input serves many taps: the FMAs, 49 per
// value, bound them.  Threads of a block share cpb channel pairs (the block's
// y index picks which); thread t takes pair t % cpb at position t / cpb.
constexpr int DW_PX = 8;        // pixels of a row per thread
constexpr int DW_THREADS = 256;
constexpr int DWG_THREADS = 256;  // two halves: tap rows 0..3 and 4..6

__device__ __forceinline__ float2 unpack2(uint32_t u) {
  return make_float2(__uint_as_float(u << 16), __uint_as_float(u & 0xffff0000u));
}

// Y = bias + sum_taps w * X (FLIP = 0), or the data gradient dX = sum_taps
// w[6-ky][6-kx] * dY[y+ky-3][x+kx-3] (FLIP = 1, X = dY, no bias).  A thread
// owns eight pixels of R consecutive rows: each input row is loaded and
// converted once (14 values) and serves the up to R output rows it reaches,
// 56 packed FMAs each, taps in order (ky, then kx) per output, so the sums
// are those of one output computed alone.  CT: the channel count when known
// (the loads' offsets are then immediates), else 0.
// 64 channels, 32 x 128^2 (33.5M values; 42 us of FMAs, 20 us of copy
// bandwidth): 96 us, half of its issue slots empty on the weights' shared-memory
// loads; 240 us with one row per thread, scalar FMAs and a bounds check per
// load.  Four rows take the registers of two resident blocks (three rows 105,
// two rows at three blocks 114 us); one row is for images whose positions do
// not fill the GPU at four rows per thread.
template <bool FLIP, int R, int CT>
__global__ void __launch_bounds__(DW_THREADS, 2)
    dw7_kernel(const uint32_t *__restrict__ X, const float *__restrict__ w,
               const float *__restrict__ bias, int B, int H, int W, int C_, int cpb_,
               uint32_t *__restrict__ Y) {
  const int C = CT ? CT : C_;
  const int cpb = CT ? (CT / 2 < 32 ? CT / 2 : 32) : cpb_;
  const int cp2 = C >> 1;
  extern __shared__ float2 s_w[];  // [49][cpb], tap order of the sum
  const int cp0 = blockIdx.y * cpb;
  for (int i = threadIdx.x; i < 49 * cpb; i += DW_THREADS) {
    const int tap = i / cpb, c = cp0 + i % cpb;
    s_w[i] = c < cp2 ? __ldg(reinterpret_cast<const float2 *>(w + (FLIP ? 48 - tap : tap) * C) + c)
                     : make_float2(0.f, 0.f);
  }
  __syncthreads();
  const int slots = DW_THREADS / cpb;
  const int slot = threadIdx.x / cpb, lc = threadIdx.x - slot * cpb, cp = cp0 + lc;
  if (slot >= slots || cp >= cp2) return;
  const int gx = (W + DW_PX - 1) / DW_PX, gy = (H + R - 1) / R;
  const int64_t npos = (int64_t)B * gy * gx;
  const float2 *wl = s_w + lc;
  const float2 b0 = bias ? make_float2(bias[2 * cp], bias[2 * cp + 1]) : make_float2(0.f, 0.f);
  for (int64_t pos = (int64_t)blockIdx.x * slots + slot; pos < npos;
       pos += (int64_t)gridDim.x * slots) {
    const int x0 = (int)(pos % gx) * DW_PX;
    const int64_t rr = pos / gx;
    const int y0 = (int)(rr % gy) * R, b = (int)(rr / gy);
    uint32_t in_x = 0;  // which of the 14 columns lie in the image
#pragma unroll
    for (int k = 0; k < DW_PX + 6; ++k)
      in_x |= (unsigned)(x0 + k - 3) < (unsigned)W ? 1u << k : 0u;
    float2 acc[R][DW_PX];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int i = 0; i < DW_PX; ++i) acc[r][i] = b0;
    // input rows ylo..yhi lie in the image; the next row's loads are issued
    // before the current row's FMAs
    const int ylo = max(y0 - 3, 0), yhi = min(y0 + R + 2, H - 1);
    uint32_t raw[DW_PX + 6];
    auto load_row = [&](int yy) {
      const uint32_t *row = X + ((int64_t)(b * H + yy) * W + (x0 - 3)) * cp2 + cp;
      if (in_x == (1u << (DW_PX + 6)) - 1u) {  // no checks away from the image's sides
#pragma unroll
        for (int k = 0; k < DW_PX + 6; ++k) raw[k] = __ldg(row + k * cp2);
      } else {
#pragma unroll
        for (int k = 0; k < DW_PX + 6; ++k) raw[k] = (in_x >> k) & 1u ? __ldg(row + k * cp2) : 0u;
      }
    };
    load_row(ylo);
#pragma unroll 1
    for (int yy = ylo; yy <= yhi; ++yy) {
      float2 in[DW_PX + 6];
#pragma unroll
      for (int k = 0; k < DW_PX + 6; ++k) in[k] = unpack2(raw[k]);
      if (yy < yhi) load_row(yy + 1);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int ky = yy - y0 - r + 3;
        if (ky < 0 || ky > 6) continue;
        const float2 *wr = wl + ky * 7 * cpb;
#pragma unroll
        for (int kx = 0; kx < 7; ++kx) {
          const float2 wv = wr[kx * cpb];
#pragma unroll
          for (int i = 0; i < DW_PX; ++i) acc[r][i] = __ffma2_rn(wv, in[i + kx], acc[r][i]);
        }
      }
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      if (y0 + r >= H) break;
      uint32_t *out = Y + ((int64_t)(b * H + y0 + r) * W + x0) * cp2 + cp;
#pragma unroll
      for (int i = 0; i < DW_PX; ++i)
        if (x0 + i < W) {
          const bf162 v = __floats2bfloat162_rn(acc[r][i].x, acc[r][i].y);
          out[i * cp2] = *reinterpret_cast<const uint32_t *>(&v);
        }
    }
  }
}

// Partial weight / bias gradients: part[blockIdx.x][50][C] (tap 49 = bias).  A
// thread keeps the sums of its tap rows and channel pair and walks stretches of `seg`
// pixels of an input row: per pixel one new value of X (a window of seven in
// registers) meets the seven values of dY above and below it, 49 packed FMAs
// for eight loads, split over two halves of the block by tap rows (28 sums
// fit 128 registers; all 49 in one thread measured 264 us, the loads of its
// 12 warps per SM in the open).  The block's positions are then added in
// order.  The loads run four pixels ahead: a pixel's FMAs are far shorter than
// its loads, and 16 warps per SM leave little else to cover them.  64 channels,
// 32 x 128^2: 203 us with a thread per tap row, which read a pixel's dY and X for
// seven FMAs, 127 us one pixel ahead, 101 us now; 32 channels, 32 x 256^2: 330 us
// one pixel ahead, 212 us now.
template <int K0, int NK, int CT>
__device__ __forceinline__ void dw7_wgrad_rows(const uint32_t *__restrict__ X,
                                               const uint32_t *__restrict__ dY, int B, int H, int W,
                                               int cp2_, int cp, int seg, int64_t first,
                                               int64_t stride, float2 (&acc)[28], float2 &accb) {
  const int cp2 = CT ? CT / 2 : cp2_;
  const int nseg = (W + seg - 1) / seg;
  const int64_t items = (int64_t)B * H * nseg, grow = (int64_t)W * cp2;
  for (int64_t it = first; it < items; it += stride) {
    const int xs = (int)(it % nseg) * seg, xe = min(W, xs + seg);
    const int64_t r = it / nseg;
    const int yy = (int)(r % H);
    const uint32_t *xr = X + r * grow + cp;
    // dY row of tap row K0 + k: yy - K0 - k + 3 (outside the image: some row
    // of it, whose products are left out: zeros in their place would make NaN of
    // an infinite X)
    const uint32_t *gp[NK];
    bool row_in[NK], rows_in = true;
#pragma unroll
    for (int k = 0; k < NK; ++k) {
      row_in[k] = (unsigned)(yy - K0 - k + 3) < (unsigned)H;
      rows_in = rows_in && row_in[k];
      gp[k] = dY + (r + (row_in[k] ? 3 - K0 - k : 0)) * grow + cp;
    }
    float2 win[8];  // the value at column x + k - 3 in slot k mod 8
#pragma unroll
    for (int k = 0; k < 6; ++k) {
      const int xx = xs + k - 3;
      win[k] = unpack2(xx >= 0 && xx < W ? __ldg(xr + (int64_t)xx * cp2) : 0u);
    }
    // dY and the window's new X of the next D pixels (pixel x in slot x mod D)
    constexpr int D = 4;
    uint32_t raw[D][NK + 1];
    auto load_px = [&](int j, int xx) {
#pragma unroll
      for (int k = 0; k < NK; ++k) raw[j][k] = xx < xe ? __ldg(gp[k] + (int64_t)xx * cp2) : 0u;
      raw[j][NK] = xx < xe && xx + 3 < W ? __ldg(xr + (int64_t)(xx + 3) * cp2) : 0u;
    };
    // (checked rows only at the image's upper and lower sides: the checks' registers
    // in every pixel's FMAs took 18 of 100 us at 64 channels, 32 x 128^2)
    auto walk = [&](auto all) {
      constexpr bool ALL = decltype(all)::value;
      auto pixel = [&](int u, bool on, auto &&load_next) {  // on: inside the stretch
        float2 g[NK];
#pragma unroll
        for (int k = 0; k < NK; ++k) g[k] = unpack2(raw[u % D][k]);
        win[(u + 6) % 8] = unpack2(raw[u % D][NK]);
        load_next();
        if (!on) return;
        if (K0 <= 3 && 3 < K0 + NK) {
          accb.x += g[3 - K0 < NK ? 3 - K0 : 0].x;
          accb.y += g[3 - K0 < NK ? 3 - K0 : 0].y;
        }
#pragma unroll
        for (int k = 0; k < NK; ++k)
          if (ALL || row_in[k]) {
#pragma unroll
            for (int kx = 0; kx < 7; ++kx)
              acc[k * 7 + kx] = __ffma2_rn(g[k], win[(u + kx) % 8], acc[k * 7 + kx]);
          }
      };
#pragma unroll
      for (int j = 0; j < D; ++j) load_px(j, xs + j);
      int x = xs;
      // every load in the stretch and the row (or read by no pixel, when these
      // eight end the stretch): no checks
#pragma unroll 1
      for (; (x + 8 + D <= xe || x + 8 == xe) && x + 10 + D < W; x += 8) {
        const uint32_t *xp = xr + (int64_t)(x + D + 3) * cp2;
        const uint32_t *gx[NK];
#pragma unroll
        for (int k = 0; k < NK; ++k) gx[k] = gp[k] + (int64_t)(x + D) * cp2;
#pragma unroll
        for (int u = 0; u < 8; ++u)
          pixel(u, true, [&] {
#pragma unroll
            for (int k = 0; k < NK; ++k) raw[u % D][k] = __ldg(gx[k] + u * cp2);
            raw[u % D][NK] = __ldg(xp + u * cp2);
          });
      }
#pragma unroll 1
      for (; x < xe; x += 8)
#pragma unroll
        for (int u = 0; u < 8; ++u) pixel(u, x + u < xe, [&] { load_px(u % D, x + u + D); });
    };
    if (rows_in) walk(std::true_type());
    else walk(std::false_type());
  }
}

template <int CT>
__global__ void __launch_bounds__(DWG_THREADS, 2)
    dw7_wgrad_kernel(const uint32_t *__restrict__ X, const uint32_t *__restrict__ dY, int B, int H,
                     int W, int C_, int cpb_, int seg, int reps, float *__restrict__ part) {
  const int C = CT ? CT : C_;
  const int cpb = CT ? (CT / 2 < 32 ? CT / 2 : 32) : cpb_;
  const int cp2 = C >> 1;
  const int half = threadIdx.x / (DWG_THREADS / 2), t = threadIdx.x % (DWG_THREADS / 2);
  const int slots = DWG_THREADS / 2 / cpb;
  const int slot = t / cpb, lc = t - slot * cpb;
  const int cp = blockIdx.y * cpb + lc;
  const bool on = slot < slots && cp < cp2;
  float2 acc[28], accb = make_float2(0.f, 0.f);
#pragma unroll
  for (int k = 0; k < 28; ++k) acc[k] = make_float2(0.f, 0.f);
  const int64_t first = (int64_t)blockIdx.x * slots + slot, stride = (int64_t)gridDim.x * slots;
  if (on) {
    if (half == 0)
      dw7_wgrad_rows<0, 4, CT>(X, dY, B, H, W, cp2, cp, seg, first, stride, acc, accb);
    else
      dw7_wgrad_rows<4, 3, CT>(X, dY, B, H, W, cp2, cp, seg, first, stride, acc, accb);
  }
  // positions of the block, added in a fixed order in shared memory: `reps` of
  // them side by side, then by halves (one after the other, the 32 positions of 8
  // channels and the 128 of two were most of a small image's time and of its
  // rounding)
  extern __shared__ float2 s_w[];  // [reps][50][cpb]
  const int n_w = 50 * cpb;
  for (int i = threadIdx.x; i < reps * n_w; i += DWG_THREADS) s_w[i] = make_float2(0.f, 0.f);
  for (int k = 0; k < slots; k += reps) {
    __syncthreads();
    if (on && slot >= k && slot < k + reps) {
      const int t0 = half * 28, n = half ? 21 : 28;
      float2 *w = s_w + (slot - k) * n_w + lc;
#pragma unroll
      for (int j = 0; j < 28; ++j) {
        if (j >= n) break;
        float2 v = w[(t0 + j) * cpb];
        v.x += acc[j].x;
        v.y += acc[j].y;
        w[(t0 + j) * cpb] = v;
      }
      if (!half) {
        float2 v = w[49 * cpb];
        v.x += accb.x;
        v.y += accb.y;
        w[49 * cpb] = v;
      }
    }
  }
  for (int o = reps / 2; o > 0; o /= 2) {
    __syncthreads();
    for (int i = threadIdx.x; i < o * n_w; i += DWG_THREADS) {
      s_w[i].x += s_w[i + o * n_w].x;
      s_w[i].y += s_w[i + o * n_w].y;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 50 * cpb; i += DWG_THREADS) {
    const int k = i / cpb, c = blockIdx.y * cpb + i % cpb;
    if (c < cp2) {
      float *dst = part + ((size_t)blockIdx.x * 50 + k) * C + 2 * c;
      dst[0] = s_w[i].x;
      dst[1] = s_w[i].y;
    }
  }
}

// out[i] = (accumulate ? out[i] : 0) + sum over chunks of part[chunk][i],
// i < n, in a fixed order: lane ty of the block sums chunks ty, ty + 8, ...
// and the eight partial sums are added in order.  Block (32, 8).
__global__ void __launch_bounds__(1024) sum_chunks_kernel(const float *part, int chunks,
                                                          int64_t n, float *out,
                                                          int accumulate) {
  // 32 outputs per block, 32 threads per output walking the chunks in a
  // fixed interleave, then their 32 sums in a fixed order (deterministic).
  // out may be part itself (chunk 0 overwritten): a block reads only its own
  // 32 columns, all of them before the barrier, and writes them after it
  // (hence no __restrict__ here).
  __shared__ float red[32][33];
  const int64_t i = (int64_t)blockIdx.x * 32 + threadIdx.x;
  float s = 0.0f;
  if (i < n)
    for (int k = threadIdx.y; k < chunks; k += 32) s += part[(int64_t)k * n + i];
  red[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y == 0 && i < n) {
    float t = 0.0f;
#pragma unroll
    for (int k = 0; k < 32; ++k) t += red[k][threadIdx.x];
    out[i] = accumulate ? out[i] + t : t;
  }
}

// ---------------------------------------------------------------------------
// LayerNorm over the C channels of each pixel (one warp per pixel)
// ---------------------------------------------------------------------------
__global__ void ln_fwd_kernel(const bf16 *__restrict__ X, const float *__restrict__ gam,
                              const float *__restrict__ bet, int64_t P, int C, float eps,
                              bf16 *__restrict__ Y, float *__restrict__ mean,
                              float *__restrict__ rstd) {
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t p = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); p < P; p += warps) {
    const bf16 *x = X + p * C;
    float v[8];  // C <= 256: channel lane + 32 i
    float s = 0.0f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int c = lane + 32 * i;
      v[i] = c < C ? b2f(x[c]) : 0.0f;
      s += v[i];
    }
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    const float mu = s / C;
    float var = 0.0f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float d = lane + 32 * i < C ? v[i] - mu : 0.0f;
      var += d * d;
    }
    for (int o = 16; o > 0; o >>= 1) var += __shfl_xor_sync(0xffffffffu, var, o);
    const float rs = rsqrtf(var / C + eps);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int c = lane + 32 * i;
      if (c < C) Y[p * C + c] = f2b((v[i] - mu) * rs * gam[c] + bet[c]);
    }
    if (lane == 0) {
      mean[p] = mu;
      rstd[p] = rs;
    }
  }
}

// LayerNorm for narrow pixels (C a multiple of 8, used for C = 32): one thread per
// pixel, its C channels in registers through 16-byte loads and stores, the
// mean and variance summed in channel order (no shuffles).
template <int C>
__global__ void __launch_bounds__(256) ln_fwd_narrow_kernel(
    const bf16 *__restrict__ X, const float *__restrict__ gam, const float *__restrict__ bet,
    int64_t P, float eps, bf16 *__restrict__ Y, float *__restrict__ mean,
    float *__restrict__ rstd) {
  static_assert(C % 8 == 0 && C <= 64, "narrow LayerNorm: C a multiple of 8, at most 64");
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < P;
       p += (int64_t)gridDim.x * blockDim.x) {
    float v[C];
    const uint4 *x = reinterpret_cast<const uint4 *>(X + p * C);
#pragma unroll
    for (int k = 0; k < C / 8; ++k) {
      const uint4 u = x[k];
      const bf16 *e = reinterpret_cast<const bf16 *>(&u);
#pragma unroll
      for (int m = 0; m < 8; ++m) v[8 * k + m] = b2f(e[m]);
    }
    float s = 0.0f;
#pragma unroll
    for (int c = 0; c < C; ++c) s += v[c];
    const float mu = s / C;
    float var = 0.0f;
#pragma unroll
    for (int c = 0; c < C; ++c) {
      const float d = v[c] - mu;
      var += d * d;
    }
    const float rs = rsqrtf(var / C + eps);
    uint4 *y = reinterpret_cast<uint4 *>(Y + p * C);
#pragma unroll
    for (int k = 0; k < C / 8; ++k) {
      uint4 u;
      bf16 *e = reinterpret_cast<bf16 *>(&u);
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const int c = 8 * k + m;
        e[m] = f2b((v[c] - mu) * rs * __ldg(gam + c) + __ldg(bet + c));
      }
      y[k] = u;
    }
    mean[p] = mu;
    rstd[p] = rs;
  }
}

// LayerNorm for C = 32 NI channels, four threads per pixel: thread q holds, of
// every 32 channels, the eight from 8 q on (16-byte loads; a warp reads eight
// pixels' 64-byte pieces).  The sums are those of a warp per pixel with lane l
// on channels l, l + 32, ...: over i in the thread, then the butterfly 16, 8
// (two shuffles of the eight values) and 4, 2, 1 (in the thread), so the
// results are the same bit for bit.  64 channels, 524288 pixels: forward 28 us
// (134 MB, 20 us of copy bandwidth), backward 41 us (201 MB, 30 us); a warp per
// pixel took 224 instructions a pixel over 2-byte loads, 118 and 130 us.
template <int NI>
struct ln_quad {
  // the butterfly sum of the 32 per-lane values whose eight this thread holds
  static __device__ __forceinline__ float tree(float (&t)[8]) {
#pragma unroll
    for (int o = 2; o > 0; o >>= 1)
#pragma unroll
      for (int m = 0; m < 8; ++m) t[m] += __shfl_xor_sync(0xffffffffu, t[m], o);
    return ((t[0] + t[4]) + (t[2] + t[6])) + ((t[1] + t[5]) + (t[3] + t[7]));
  }
  static __device__ __forceinline__ void load(const bf16 *__restrict__ x, float (&v)[NI * 8]) {
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      const uint4 u = __ldg(reinterpret_cast<const uint4 *>(x + 32 * i));
      const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
      for (int m = 0; m < 4; ++m) {
        v[8 * i + 2 * m] = __uint_as_float(w[m] << 16);
        v[8 * i + 2 * m + 1] = __uint_as_float(w[m] & 0xffff0000u);
      }
    }
  }
  static __device__ __forceinline__ void store(bf16 *__restrict__ y, const float (&v)[NI * 8]) {
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      uint4 u;
      bf162 *e = reinterpret_cast<bf162 *>(&u);
#pragma unroll
      for (int m = 0; m < 4; ++m) e[m] = __floats2bfloat162_rn(v[8 * i + 2 * m], v[8 * i + 2 * m + 1]);
      *reinterpret_cast<uint4 *>(y + 32 * i) = u;
    }
  }
  // eight of a row of C floats in shared memory
  static __device__ __forceinline__ void row8(const float *s, float (&g)[8]) {
    const float4 a = *reinterpret_cast<const float4 *>(s), b = *reinterpret_cast<const float4 *>(s + 4);
    g[0] = a.x; g[1] = a.y; g[2] = a.z; g[3] = a.w;
    g[4] = b.x; g[5] = b.y; g[6] = b.z; g[7] = b.w;
  }
};

constexpr int LN_THREADS = 256;

template <int NI>
__global__ void __launch_bounds__(LN_THREADS)
    ln_fwd_quad_kernel(const bf16 *__restrict__ X, const float *__restrict__ gam,
                       const float *__restrict__ bet, int64_t P, float eps, bf16 *__restrict__ Y,
                       float *__restrict__ mean, float *__restrict__ rstd) {
  constexpr int C = 32 * NI;
  using Q = ln_quad<NI>;
  __shared__ __align__(16) float s_g[C], s_b[C];
  for (int c = threadIdx.x; c < C; c += LN_THREADS) {
    s_g[c] = gam[c];
    s_b[c] = bet[c];
  }
  __syncthreads();
  const int q = threadIdx.x & 3;
  const int64_t step = (int64_t)gridDim.x * (LN_THREADS / 4);
  for (int64_t p0 = (int64_t)blockIdx.x * (LN_THREADS / 4); p0 < P; p0 += step) {
    const int64_t p = p0 + (threadIdx.x >> 2);
    const bool on = p < P;  // (the shuffles take the whole warp)
    float v[NI * 8];
    Q::load(X + (on ? p : P - 1) * C + 8 * q, v);
    float t[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      float s = 0.0f;
#pragma unroll
      for (int i = 0; i < NI; ++i) s += v[8 * i + m];
      t[m] = s;
    }
    const float mu = Q::tree(t) / C;
#pragma unroll
    for (int m = 0; m < 8; ++m) {
      float var = 0.0f;
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const float d = v[8 * i + m] - mu;
        var += d * d;
      }
      t[m] = var;
    }
    const float rs = rsqrtf(Q::tree(t) / C + eps);
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      float g[8], b[8];
      Q::row8(s_g + 32 * i + 8 * q, g);
      Q::row8(s_b + 32 * i + 8 * q, b);
#pragma unroll
      for (int m = 0; m < 8; ++m) v[8 * i + m] = (v[8 * i + m] - mu) * rs * g[m] + b[m];
    }
    if (on) {
      Q::store(Y + p * C + 8 * q, v);
      if (q == 0) {
        mean[p] = mu;
        rstd[p] = rs;
      }
    }
  }
}

// dX (as ln_bwd_kernel's, bit for bit) and per-block partials of dgamma, dbeta:
// part[block][2][C].  A thread keeps its channels' sums over its pixels; the
// eight pixels of a warp and the block's warps are added at the end.
template <int NI>
__global__ void __launch_bounds__(LN_THREADS, NI == 4 ? 1 : 2)
    ln_bwd_quad_kernel(const bf16 *__restrict__ dY, const bf16 *__restrict__ X,
                       const float *__restrict__ gam, const float *__restrict__ mean,
                       const float *__restrict__ rstd, int64_t P, bf16 *__restrict__ dX,
                       float *__restrict__ part) {
  constexpr int C = 32 * NI;
  using Q = ln_quad<NI>;
  __shared__ __align__(16) float s_g[C];
  __shared__ float s_sum[LN_THREADS / 32][2][C];
  for (int c = threadIdx.x; c < C; c += LN_THREADS) s_g[c] = gam[c];
  __syncthreads();
  const int q = threadIdx.x & 3;
  float dg[NI * 8], db[NI * 8];
#pragma unroll
  for (int k = 0; k < NI * 8; ++k) dg[k] = db[k] = 0.0f;
  const int64_t step = (int64_t)gridDim.x * (LN_THREADS / 4);
  for (int64_t p0 = (int64_t)blockIdx.x * (LN_THREADS / 4); p0 < P; p0 += step) {
    const int64_t p = p0 + (threadIdx.x >> 2);
    const bool on = p < P;
    const int64_t pc = on ? p : P - 1;
    const float mu = __ldg(mean + pc), rs = __ldg(rstd + pc);
    float xh[NI * 8], gg[NI * 8];
    Q::load(X + pc * C + 8 * q, xh);
    Q::load(dY + pc * C + 8 * q, gg);
    float t1[8], t2[8];
#pragma unroll
    for (int m = 0; m < 8; ++m) t1[m] = t2[m] = 0.0f;
#pragma unroll
    for (int i = 0; i < NI; ++i) {
      float g[8];
      Q::row8(s_g + 32 * i + 8 * q, g);
#pragma unroll
      for (int m = 0; m < 8; ++m) {
        const int k = 8 * i + m;
        xh[k] = (xh[k] - mu) * rs;
        const float gy = gg[k];
        gg[k] = gy * g[m];
        t1[m] += gg[k];
        t2[m] += gg[k] * xh[k];
        if (on) {
          dg[k] += gy * xh[k];
          db[k] += gy;
        }
      }
    }
    const float s1 = Q::tree(t1) / C, s2 = Q::tree(t2) / C;
#pragma unroll
    for (int k = 0; k < NI * 8; ++k) gg[k] = rs * (gg[k] - s1 - xh[k] * s2);
    if (on) Q::store(dX + p * C + 8 * q, gg);
  }
#pragma unroll
  for (int k = 0; k < NI * 8; ++k)
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) {
      dg[k] += __shfl_xor_sync(0xffffffffu, dg[k], o);
      db[k] += __shfl_xor_sync(0xffffffffu, db[k], o);
    }
  const int warp = threadIdx.x >> 5;
  if ((threadIdx.x & 31) < 4) {
#pragma unroll
    for (int k = 0; k < NI * 8; ++k) {
      const int c = 32 * (k / 8) + 8 * q + k % 8;
      s_sum[warp][0][c] = dg[k];
      s_sum[warp][1][c] = db[k];
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < 2 * C; i += LN_THREADS) {
    float t = 0.0f;
#pragma unroll
    for (int w = 0; w < LN_THREADS / 32; ++w) t += s_sum[w][i / C][i % C];
    part[(size_t)blockIdx.x * 2 * C + i] = t;
  }
}

// dX and per-warp partials of dgamma, dbeta: part[warp][2][C].
__global__ void __launch_bounds__(256, 4) ln_bwd_kernel(const bf16 *__restrict__ dY, const bf16 *__restrict__ X,
                              const float *__restrict__ gam, const float *__restrict__ mean,
                              const float *__restrict__ rstd, int64_t P, int C,
                              bf16 *__restrict__ dX, float *__restrict__ part) {
  const int lane = threadIdx.x & 31;
  const int64_t gw = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  float dg[8], db[8];  // C <= 256
#pragma unroll
  for (int i = 0; i < 8; ++i) dg[i] = db[i] = 0.0f;
  for (int64_t p = gw; p < P; p += warps) {
    const float mu = mean[p], rs = rstd[p];
    float xh[8], gg[8];
    float s1 = 0.0f, s2 = 0.0f;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      int c = lane + 32 * i;
      xh[i] = gg[i] = 0.0f;
      if (c >= C) continue;
      xh[i] = (b2f(X[p * C + c]) - mu) * rs;
      float gy = b2f(dY[p * C + c]);
      gg[i] = gy * gam[c];
      s1 += gg[i];
      s2 += gg[i] * xh[i];
      dg[i] += gy * xh[i];
      db[i] += gy;
    }
    for (int o = 16; o > 0; o >>= 1) {
      s1 += __shfl_xor_sync(0xffffffffu, s1, o);
      s2 += __shfl_xor_sync(0xffffffffu, s2, o);
    }
    s1 /= C;
    s2 /= C;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      int c = lane + 32 * i;
      if (c < C) dX[p * C + c] = f2b(rs * (gg[i] - s1 - xh[i] * s2));
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    int c = lane + 32 * i;
    if (c >= C) break;
    part[(gw * 2 + 0) * C + c] = dg[i];
    part[(gw * 2 + 1) * C + c] = db[i];
  }
}

// Column sums of a [M][ld] BF16 matrix in a fixed order: block (32, 8) owns
// 32 columns (PAIR: 32 column pairs) of chunk blockIdx.y; lane ty sums rows
// r0 + ty, r0 + ty + 8, ...; the eight lanes are added in order into
// part[chunk][N].
template <bool PAIR>
__global__ void colsum_kernel(const bf16 *__restrict__ Xs, int64_t M, int N, int64_t ld,
                              int64_t rows_per_chunk, float *__restrict__ part) {
  __shared__ float2 red[8][33];
  const int c = (blockIdx.x * 32 + threadIdx.x) * (PAIR ? 2 : 1);
  const int64_t r0 = (int64_t)blockIdx.y * rows_per_chunk;
  int64_t r1 = r0 + rows_per_chunk;
  if (r1 > M) r1 = M;
  float2 s = make_float2(0.f, 0.f);
  if (c < N) {
    for (int64_t r = r0 + threadIdx.y; r < r1; r += 8) {
      if (PAIR) {
        const float2 v = __bfloat1622float2(*reinterpret_cast<const bf162 *>(Xs + r * ld + c));
        s.x += v.x;
        s.y += v.y;
      } else {
        s.x += b2f(Xs[r * ld + c]);
      }
    }
  }
  red[threadIdx.y][threadIdx.x] = s;
  __syncthreads();
  if (threadIdx.y == 0 && c < N) {
    float2 t = make_float2(0.f, 0.f);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      t.x += red[k][threadIdx.x].x;
      t.y += red[k][threadIdx.x].y;
    }
    part[(int64_t)blockIdx.y * N + c] = t.x;
    if (PAIR) part[(int64_t)blockIdx.y * N + c + 1] = t.y;
  }
}

// ---------------------------------------------------------------------------
// elementwise
// ---------------------------------------------------------------------------
__global__ void gelu_bwd_kernel(const bf16 *__restrict__ dA, const bf16 *__restrict__ Z, int64_t n,
                                bf16 *__restrict__ dZ) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    dZ[i] = f2b(b2f(dA[i]) * pe_gelu_grad(b2f(Z[i])));
  }
}

__global__ void maxpool2_fwd_kernel(const bf16 *__restrict__ X, int B, int H, int W, int C,
                                    bf16 *__restrict__ Y, uint8_t *__restrict__ arg) {
  const int Ho = H / 2, Wo = W / 2;
  const int64_t total = (int64_t)B * Ho * Wo * C;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    int c = (int)(t % C);
    int64_t p = t / C;
    int x = (int)(p % Wo), y = (int)((p / Wo) % Ho), b = (int)(p / ((int64_t)Wo * Ho));
    float best = -INFINITY;
    int bi = 0;
    for (int k = 0; k < 4; ++k) {
      float v = b2f(X[(((int64_t)b * H + 2 * y + (k >> 1)) * W + 2 * x + (k & 1)) * C + c]);
      if (v > best) {
        best = v;
        bi = k;
      }
    }
    Y[t] = f2b(best);
    arg[t] = (uint8_t)bi;
  }
}

__global__ void maxpool2_bwd_kernel(const bf16 *__restrict__ dY, const uint8_t *__restrict__ arg,
                                    int B, int H, int W, int C, bf16 *__restrict__ dX) {
  const int64_t total = (int64_t)B * H * W * C;
  const int Ho = H / 2, Wo = W / 2;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    int c = (int)(t % C);
    int64_t p = t / C;
    int x = (int)(p % W), y = (int)((p / W) % H), b = (int)(p / ((int64_t)W * H));
    int64_t q = (((int64_t)b * Ho + y / 2) * Wo + x / 2) * C + c;
    dX[t] = (arg[q] == (uint8_t)(((y & 1) << 1) | (x & 1))) ? dY[q] : f2b(0.0f);
  }
}

// Eight channels per thread (16-byte activations, 8-byte argument words); the
// backward thread owns a pooled pixel and writes the four under it.  (One channel
// per thread: 218 us backward for 134 + 34 MB.)
__global__ void maxpool2_wide_kernel(const uint4 *__restrict__ X, int B, int H, int W, int CV,
                                     uint4 *__restrict__ Y, uint2 *__restrict__ arg, int backward) {
  const int Ho = H / 2, Wo = W / 2;
  const int64_t total = (int64_t)B * Ho * Wo * CV;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(t % CV);
    const int64_t p = t / CV;
    const int x = (int)(p % Wo);
    const int64_t by = p / Wo;  // b Ho + y
    const int64_t g = ((2 * by) * W + 2 * x) * CV + c, row = (int64_t)W * CV;
    if (!backward) {
      uint4 in[4];
#pragma unroll
      for (int k = 0; k < 4; ++k) in[k] = __ldg(X + g + (k >> 1) * row + (k & 1) * CV);
      uint4 o;
      uint32_t am[2] = {0u, 0u};
      bf16 *out = reinterpret_cast<bf16 *>(&o);
#pragma unroll
      for (int e = 0; e < 8; ++e) {
        float best = -INFINITY;
        uint32_t bi = 0;
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const float v = b2f(reinterpret_cast<const bf16 *>(&in[k])[e]);
          if (v > best) {
            best = v;
            bi = k;
          }
        }
        out[e] = f2b(best);
        am[e >> 2] |= bi << (8 * (e & 3));
      }
      Y[t] = o;
      arg[t] = make_uint2(am[0], am[1]);
    } else {
      const uint4 d = __ldg(X + t);
      const uint2 aw = __ldg(arg + t);
      const bf16 *dv = reinterpret_cast<const bf16 *>(&d);
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint4 o;
        bf16 *out = reinterpret_cast<bf16 *>(&o);
#pragma unroll
        for (int e = 0; e < 8; ++e) {
          const uint32_t a = ((e < 4 ? aw.x : aw.y) >> (8 * (e & 3))) & 0xffu;
          out[e] = a == (uint32_t)k ? dv[e] : f2b(0.0f);
        }
        Y[g + (k >> 1) * row + (k & 1) * CV] = o;
      }
    }
  }
}

// out[b, 2y+i, 2x+j, off + c] = in[b, y, x, 4c + 2i + j]; dir 1: the reverse.
// One thread per pixel (Y, X) of the 2H x 2W image and VEC consecutive
// channels c: the small image's element [b, Y/2, X/2][4c + 2(Y&1) + (X&1)]
// moves to / from the large image's [b, Y, X][off + c] (VEC = 8: the large
// side as one 16-byte access).
template <int VEC>
__global__ void pixel_shuffle2_kernel(const bf16 *__restrict__ src, int B, int H, int W, int C,
                                      bf16 *__restrict__ dst, int64_t ld_big, int off, int dir) {
  const int CV = C / VEC;
  const int W2 = 2 * W, H2 = 2 * H;
  const int64_t total = (int64_t)B * H2 * W2 * CV;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int c0 = (int)(t % CV) * VEC;
    const int64_t P = t / CV;                 // large-image pixel
    const int X = (int)(P % W2);
    const int64_t q = P / W2;
    const int Y = (int)(q % H2), b = (int)(q / H2);
    const int sub = 2 * (Y & 1) + (X & 1);
    const int64_t small = ((int64_t)b * H + (Y >> 1)) * W + (X >> 1);
    const int64_t sbase = small * 4 * C + 4 * (int64_t)c0 + sub;   // stride 4 over c
    const int64_t bbase = P * ld_big + off + c0;
    if (VEC == 8) {
      if (dir == 0) {
        uint4 u;
        bf16 *e = reinterpret_cast<bf16 *>(&u);
#pragma unroll
        for (int k = 0; k < 8; ++k) e[k] = src[sbase + 4 * k];
        *reinterpret_cast<uint4 *>(dst + bbase) = u;
      } else {
        const uint4 u = *reinterpret_cast<const uint4 *>(src + bbase);
        const bf16 *e = reinterpret_cast<const bf16 *>(&u);
#pragma unroll
        for (int k = 0; k < 8; ++k) dst[sbase + 4 * k] = e[k];
      }
    } else {
      if (dir == 0)
        dst[bbase] = src[sbase];
      else
        dst[sbase] = src[bbase];
    }
  }
}

// The same with everything in 16-byte accesses: a thread moves eight channels of
// the four pixels under one small pixel, 64 contiguous bytes on the small side
// and 16 per pixel on the large one.  (The form above touches the small side two
// bytes at a time: 66 us against 20 for 134 MB each way.)
__global__ void pixel_shuffle2_wide_kernel(const bf16 *__restrict__ src, int B, int H, int W, int C,
                                           bf16 *__restrict__ dst, int64_t ld_big, int off,
                                           int dir) {
  const int CV = C / 8;
  const int64_t total = (int64_t)B * H * W * CV;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int c0 = (int)(t % CV) * 8;
    const int64_t small = t / CV;
    const int x = (int)(small % W);
    const int64_t q = small / W;
    const int64_t big0 = (2 * q * (2 * W) + 2 * x) * ld_big + off + c0;  // (q = b H + y)
    const int64_t row = 2 * (int64_t)W * ld_big;
    uint4 s4[4], b4[4];
    uint4 *sp = reinterpret_cast<uint4 *>(const_cast<bf16 *>(dir == 0 ? src : dst) + small * 4 * C +
                                          4 * c0);
    bf16 *bp = const_cast<bf16 *>(dir == 0 ? dst : src) + big0;
    // s4 holds elements 4 k + sub (channel k, sub-pixel sub), b4[sub] channels k
    if (dir == 0) {
#pragma unroll
      for (int k = 0; k < 4; ++k) s4[k] = __ldg(sp + k);
      const uint32_t *sw = reinterpret_cast<const uint32_t *>(s4);
#pragma unroll
      for (int sub = 0; sub < 4; ++sub) {
        uint32_t w[4];
#pragma unroll
        for (int k = 0; k < 4; ++k)  // channels 2 k, 2 k + 1
          w[k] = __byte_perm(sw[4 * k + (sub >> 1)], sw[4 * k + 2 + (sub >> 1)],
                             (sub & 1) ? 0x7632 : 0x5410);
        b4[sub] = make_uint4(w[0], w[1], w[2], w[3]);
      }
#pragma unroll
      for (int sub = 0; sub < 4; ++sub)
        *reinterpret_cast<uint4 *>(bp + (sub >> 1) * row + (sub & 1) * ld_big) = b4[sub];
    } else {
#pragma unroll
      for (int sub = 0; sub < 4; ++sub)
        b4[sub] = __ldg(reinterpret_cast<const uint4 *>(bp + (sub >> 1) * row + (sub & 1) * ld_big));
      const uint32_t *bw = reinterpret_cast<const uint32_t *>(b4);
      uint32_t w[16];
#pragma unroll
      for (int k = 0; k < 8; ++k)  // channel k: sub-pixels 0, 1 and 2, 3
#pragma unroll
        for (int h = 0; h < 2; ++h)
          w[2 * k + h] = __byte_perm(bw[4 * (2 * h) + (k >> 1)], bw[4 * (2 * h + 1) + (k >> 1)],
                                     (k & 1) ? 0x7632 : 0x5410);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        sp[k] = make_uint4(w[4 * k], w[4 * k + 1], w[4 * k + 2], w[4 * k + 3]);
    }
  }
}

// dst[p][doff + c] (=|+=) src[p][soff + c] for c < C; VEC = 8: 16-byte
// chunks (sums per element in FP32, as for VEC = 1).
template <int VEC>
__global__ void copy_channels_kernel(const bf16 *__restrict__ src, int64_t lds, int soff,
                                     bf16 *__restrict__ dst, int64_t ldd, int doff, int64_t P,
                                     int C, int accumulate) {
  const int CV = C / VEC;
  const int64_t total = P * CV;
  for (int64_t t = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; t < total;
       t += (int64_t)gridDim.x * blockDim.x) {
    const int c = (int)(t % CV) * VEC;
    const int64_t p = t / CV;
    const bf16 *sp = src + p * lds + soff + c;
    bf16 *d = dst + p * ldd + doff + c;
    if (VEC == 8) {
      uint4 u = *reinterpret_cast<const uint4 *>(sp);
      if (accumulate) {
        const uint4 w = *reinterpret_cast<const uint4 *>(d);
        bf16 *e = reinterpret_cast<bf16 *>(&u);
        const bf16 *f = reinterpret_cast<const bf16 *>(&w);
#pragma unroll
        for (int k = 0; k < 8; ++k) e[k] = f2b(b2f(f[k]) + b2f(e[k]));
      }
      *reinterpret_cast<uint4 *>(d) = u;
    } else {
      const float v = b2f(*sp);
      *d = f2b(accumulate ? b2f(*d) + v : v);
    }
  }
}

// dst[c][r] = src[r][c] (BF16), 32 x 32 tiles through shared memory.
__global__ void transpose_kernel(const bf16 *__restrict__ src, int R, int Cc,
                                 bf16 *__restrict__ dst) {
  __shared__ bf16 t[32][33];
  const int r0 = blockIdx.y * 32, c0 = blockIdx.x * 32;
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int r = r0 + i, c = c0 + threadIdx.x;
    if (r < R && c < Cc) t[i][threadIdx.x] = src[(int64_t)r * Cc + c];
  }
  __syncthreads();
  for (int i = threadIdx.y; i < 32; i += blockDim.y) {
    const int c = c0 + i, r = r0 + threadIdx.x;
    if (c < Cc && r < R) dst[(int64_t)c * R + r] = t[threadIdx.x][i];
  }
}

__global__ void f32_to_bf16_kernel(const float *__restrict__ x, int64_t n, bf16 *__restrict__ y) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x)
    y[i] = f2b(x[i]);
}

__global__ void adamw_kernel(float *__restrict__ p, const float *__restrict__ g,
                             float *__restrict__ m, float *__restrict__ v, bf16 *__restrict__ pb,
                             int64_t n, float lr, float b1, float b2, float eps, float wd,
                             float bc1, float bc2) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    float gi = g[i];
    float mi = b1 * m[i] + (1.0f - b1) * gi;
    float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    float pi = p[i] * (1.0f - lr * wd) - lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
    p[i] = pi;
    if (pb) pb[i] = f2b(pi);
  }
}

// ---------------------------------------------------------------------------
// Losses of Eq. 17-21 and their gradients.  Outputs are FP32 head outputs:
// depth [P], normal [P][3], mask logit [P].  Ground truth: d_gt [P],
// n_gt [P][3], m_gt [P] (0/1).  counts[0] = hit pixels, [1] = L4 pixels,
// [2] = all pixels (set by loss_count_kernel).
// ---------------------------------------------------------------------------
struct loss_args {
  const float *d, *n, *z, *d_gt, *n_gt, *m_gt;
  int B, H, W;
  float alpha, gamma, w1, w2, w3, w4;
  const float *counts;
  float *g_d, *g_n, *g_z;  // gradients of the total loss
  float *c4u, *c4v;        // per pixel dL4/d(gu), dL4/d(gv) (scratch)
  float *part;             // [blocks][4] loss partial sums
};

__device__ __forceinline__ bool hit_at(const loss_args &a, int b, int y, int x) {
  return a.m_gt[((int64_t)b * a.H + y) * a.W + x] > 0.5f;
}

__device__ __forceinline__ bool l4_valid(const loss_args &a, int b, int y, int x) {
  if (x < 1 || y < 1 || x > a.W - 2 || y > a.H - 2) return false;
  return hit_at(a, b, y, x) && hit_at(a, b, y, x - 1) && hit_at(a, b, y, x + 1) &&
         hit_at(a, b, y - 1, x) && hit_at(a, b, y + 1, x);
}

// f = |a x b| / (|a| |b| + e) with |a x b| = sqrt(|a x b|^2 + 1e-12); returns f
// and df/da.
__device__ __forceinline__ float cross_ratio(const float a[3], const float b[3], float ga[3]) {
  float c[3] = {a[1] * b[2] - a[2] * b[1], a[2] * b[0] - a[0] * b[2], a[0] * b[1] - a[1] * b[0]};
  float cn = sqrtf(c[0] * c[0] + c[1] * c[1] + c[2] * c[2] + 1e-12f);
  float na = sqrtf(a[0] * a[0] + a[1] * a[1] + a[2] * a[2]);
  float nb = sqrtf(b[0] * b[0] + b[1] * b[1] + b[2] * b[2]);
  float den = na * nb + 1e-8f;
  float bxc[3] = {b[1] * c[2] - b[2] * c[1], b[2] * c[0] - b[0] * c[2], b[0] * c[1] - b[1] * c[0]};
  for (int k = 0; k < 3; ++k)
    ga[k] = (bxc[k] / cn) / den - cn * nb * (na > 0.0f ? a[k] / na : 0.0f) / (den * den);
  return cn / den;
}

// Hit pixels and valid L4 centres, as exact integer counts (cnt zeroed first).
__global__ void loss_count_kernel(const loss_args a, unsigned long long *cnt) {
  const int64_t P = (int64_t)a.B * a.H * a.W;
  unsigned c0 = 0, c1 = 0;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < P;
       p += (int64_t)gridDim.x * blockDim.x) {
    const int x = (int)(p % a.W), y = (int)((p / a.W) % a.H), b = (int)(p / ((int64_t)a.W * a.H));
    c0 += hit_at(a, b, y, x) ? 1u : 0u;
    c1 += l4_valid(a, b, y, x) ? 1u : 0u;
  }
  for (int o = 16; o > 0; o >>= 1) {
    c0 += __shfl_xor_sync(0xffffffffu, c0, o);
    c1 += __shfl_xor_sync(0xffffffffu, c1, o);
  }
  if ((threadIdx.x & 31) == 0) {
    if (c0) atomicAdd(cnt, (unsigned long long)c0);
    if (c1) atomicAdd(cnt + 1, (unsigned long long)c1);
  }
}

__global__ void loss_count_finish(const unsigned long long *cnt, int64_t P, float *counts) {
  counts[0] = fmaxf((float)cnt[0], 1.0f);
  counts[1] = fmaxf((float)cnt[1], 1.0f);
  counts[2] = (float)P;
}

__device__ __forceinline__ void grads_at(const loss_args &a, const float *d, int b, int y, int x,
                                         float g[3]) {
  const int64_t row = ((int64_t)b * a.H + y) * a.W;
  g[0] = 0.5f * (d[row + x + 1] - d[row + x - 1]);
  g[1] = 0.5f * (d[row + a.W + x] - d[row - a.W + x]);
  g[2] = 1.0f;
}

// Pass 1: per-pixel terms of L1, L2, L3 with their gradients, and the L4
// partials with respect to the centre's (gu, gv).
__global__ void __launch_bounds__(256) loss_pass1_kernel(const loss_args a) {
  __shared__ float red[4][256];
  const int64_t P = (int64_t)a.B * a.H * a.W;
  const float nh = a.counts[0], n4 = a.counts[1], na = a.counts[2];
  float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < P;
       p += (int64_t)gridDim.x * blockDim.x) {
    int x = (int)(p % a.W), y = (int)((p / a.W) % a.H), b = (int)(p / ((int64_t)a.W * a.H));
    const bool hit = a.m_gt[p] > 0.5f;
    // L1
    float gd = 0.0f;
    if (hit) {
      float e = a.d[p] - a.d_gt[p];
      s[0] += e * e / nh;
      gd = a.w1 * 2.0f * e / nh;
    }
    a.g_d[p] = gd;
    // L2
    float gn[3] = {0.0f, 0.0f, 0.0f};
    if (hit) {
      float np_[3] = {a.n[3 * p], a.n[3 * p + 1], a.n[3 * p + 2]};
      float ng[3] = {a.n_gt[3 * p], a.n_gt[3 * p + 1], a.n_gt[3 * p + 2]};
      float ga[3];
      s[1] += cross_ratio(np_, ng, ga) / nh;
      for (int k = 0; k < 3; ++k) gn[k] = a.w2 * ga[k] / nh;
    }
    for (int k = 0; k < 3; ++k) a.g_n[3 * p + k] = gn[k];
    // L3 (focal, alpha-balanced)
    {
      float z = a.z[p];
      float pr = 1.0f / (1.0f + expf(-z));
      float lp = -(fmaxf(-z, 0.0f) + log1pf(expf(-fabsf(z))));   // log p
      float l1p = -(fmaxf(z, 0.0f) + log1pf(expf(-fabsf(z))));   // log (1 - p)
      float l, dl;
      if (hit) {
        float q = powf(1.0f - pr, a.gamma);
        l = -a.alpha * q * lp;
        dl = -a.alpha * q * (-a.gamma * pr * lp + (1.0f - pr));
      } else {
        float q = powf(pr, a.gamma);
        l = -(1.0f - a.alpha) * q * l1p;
        dl = -(1.0f - a.alpha) * q * (a.gamma * (1.0f - pr) * l1p - pr);
      }
      s[2] += l / na;
      a.g_z[p] = a.w3 * dl / na;
    }
    // L4 partials at valid centres
    float cu = 0.0f, cv = 0.0f;
    if (l4_valid(a, b, y, x)) {
      float gp[3], gg[3], ga[3];
      grads_at(a, a.d, b, y, x, gp);
      grads_at(a, a.d_gt, b, y, x, gg);
      s[3] += cross_ratio(gp, gg, ga) / n4;
      cu = a.w4 * ga[0] / n4;
      cv = a.w4 * ga[1] / n4;
    }
    a.c4u[p] = cu;
    a.c4v[p] = cv;
  }
  for (int k = 0; k < 4; ++k) red[k][threadIdx.x] = s[k];
  __syncthreads();
  if (threadIdx.x == 0) {
    for (int k = 0; k < 4; ++k) {
      float t = 0.0f;
      for (int i = 0; i < (int)blockDim.x; ++i) t += red[k][i];
      a.part[blockIdx.x * 4 + k] = t;
    }
  }
}

// Pass 2: scatter the L4 centre partials to the depths they were made of
// (gather form): d(x+1) gets +0.5 cu(x), d(x-1) gets -0.5 cu(x), likewise v.
__global__ void loss_pass2_kernel(const loss_args a) {
  const int64_t P = (int64_t)a.B * a.H * a.W;
  for (int64_t p = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; p < P;
       p += (int64_t)gridDim.x * blockDim.x) {
    int x = (int)(p % a.W), y = (int)((p / a.W) % a.H);
    float g = 0.0f;
    if (x >= 1) g += 0.5f * a.c4u[p - 1];
    if (x <= a.W - 2) g -= 0.5f * a.c4u[p + 1];
    if (y >= 1) g += 0.5f * a.c4v[p - a.W];
    if (y <= a.H - 2) g -= 0.5f * a.c4v[p + a.W];
    a.g_d[p] += g;
  }
}

__global__ void loss_total_kernel(const float *part, int blocks, float w1, float w2, float w3,
                                  float w4, float *out) {
  if (threadIdx.x != 0 || blockIdx.x != 0) return;
  float s[4] = {0, 0, 0, 0};
  for (int b = 0; b < blocks; ++b)
    for (int k = 0; k < 4; ++k) s[k] += part[b * 4 + k];
  out[0] = w1 * s[0] + w2 * s[1] + w3 * s[2] + w4 * s[3];
  for (int k = 0; k < 4; ++k) out[1 + k] = s[k];
}

}  // namespace

// ===========================================================================
// C ABI
// ===========================================================================
#define NN_CHECK_STREAM cudaStream_t s = static_cast<cudaStream_t>(stream)

// 0: tcgen05 kernel where it applies (K-contiguous operands, no split-K),
// else the mma.sync kernel; 1: the mma.sync kernel only.
static int g_gemm_path = 0;

extern "C" int32_t pe_nn_gemm_path(int32_t path) {
  const int prev = g_gemm_path;
  if (path == 0 || path == 1) g_gemm_path = path;
  return prev;
}

// Split-K factor: enough blocks for the whole GPU (about 1024, fixed so the
// summation order does not depend on the device), at least 8 K-steps each.
static int64_t gemm_split(int32_t M, int32_t N, int64_t K, int64_t *kps_out) {
  const int64_t tiles = (int64_t)((N + TN - 1) / TN) * ((M + TM - 1) / TM);
  int64_t split = tiles >= 1024 ? 1 : (1024 + tiles - 1) / tiles;
  const int64_t max_split = (K + 8 * TK - 1) / (8 * TK);
  if (split > max_split) split = max_split;
  if (split > 4096) split = 4096;
  if (split < 1) split = 1;
  int64_t kps = (K + split - 1) / split;
  kps = (kps + TK - 1) / TK * TK;
  split = (K + kps - 1) / kps;
  if (kps_out) *kps_out = kps;
  return split;
}

int64_t pe_gemm_split(int32_t M, int32_t N, int64_t K) { return gemm_split(M, N, K, nullptr); }

extern "C" size_t pe_nn_gemm_workspace(int32_t M, int32_t N, int64_t K) {
  if (M <= 0 || N <= 0 || K <= 0) return 0;
  const int64_t split = gemm_split(M, N, K, nullptr);
  if (split <= 1) return 256;
  return (size_t)split * M * N * sizeof(float) + 256;
}

extern "C" pe_status pe_nn_gemm(int32_t M, int32_t N, int64_t K, const void *A, int64_t sam,
                                int64_t sak, const void *B, int64_t sbk, int64_t sbn, void *C,
                                int64_t ldc, int32_t c_f32, const float *bias, const void *R,
                                int64_t ldr, void *Z, int64_t ldz, int32_t gelu, float alpha,
                                float beta, void *ws, size_t ws_bytes, void *stream) {
  NN_CHECK_STREAM;
  if (M <= 0 || N <= 0 || K <= 0 || !A || !B || !C || gelu < 0 || gelu > 2 || (gelu == 2 && !Z))
    return pe_fail(PE_EINVAL, "pe_nn_gemm: bad sizes, null operands or gelu mode");
  pe_gemm_args g;
  memset(&g, 0, sizeof(g));
  g.M = M;
  g.N = N;
  g.K = K;
  g.A = static_cast<const bf16 *>(A);
  g.sam = sam;
  g.sak = sak;
  g.B = static_cast<const bf16 *>(B);
  g.sbk = sbk;
  g.sbn = sbn;
  g.C = C;
  g.ldc = ldc;
  g.c_f32 = c_f32;
  g.bias = bias;
  g.R = static_cast<const bf16 *>(R);
  g.ldr = ldr;
  g.Z = static_cast<bf16 *>(Z);
  g.ldz = ldz;
  g.gelu = gelu;
  g.alpha = alpha;
  g.beta = beta;
  const bool ak = sak == 1, bk = sbk == 1;
  // 16-byte copies need aligned bases and rows along the contiguous dimension
  auto al = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  g.vec_a = al(A) && (ak ? (sam % 8 == 0) : (sam == 1 && sak % 8 == 0));
  g.vec_b = al(B) && (bk ? (sbn % 8 == 0) : (sbn == 1 && sbk % 8 == 0));
  g.vec_c = al(C) && (c_f32 ? ldc % 4 == 0 : ldc % 8 == 0) && (!R || (al(R) && ldr % 8 == 0)) &&
            (!Z || (al(Z) && ldz % 8 == 0)) && (!bias || (reinterpret_cast<uintptr_t>(bias) & 3) == 0);
  int64_t kps = 0;
  const int64_t split = gemm_split(M, N, K, &kps);
  g.k_per_split = kps;
  if (split > 1) {
    size_t need = (size_t)split * M * N * sizeof(float);
    if (!ws || ws_bytes < need) return pe_fail(PE_ENOMEM, "pe_nn_gemm: workspace needs %zu", need);
    g.part = static_cast<float *>(ws);
  }
  if ((N + TN - 1) / TN > 65535) return pe_fail(PE_EINVAL, "pe_nn_gemm: N too large");
  if (g_gemm_path == 0 && K == 1 && !c_f32 && !bias && !R && gelu == 0 && g.vec_c && N % 8 == 0) {
    outer_kernel<<<grid1((int64_t)M * (N / 8), 256), 256, 0, s>>>(g.A, sam, g.B, sbn, M, N / 8, alpha,
                                                                  static_cast<bf16 *>(C), ldc);
    PE_TRY_LAUNCH("outer_kernel");
    return PE_OK;
  }
  if (split == 1 && g_gemm_path == 0 && pe_gemm_tc_eligible(g)) {
    const pe_status st = pe_gemm_tc(g, s);
    if (st != PE_EUNSUPPORTED) return st;
  }
  dim3 grid((M + TM - 1) / TM, (N + TN - 1) / TN, (unsigned)split);
  if (ak && bk) gemm_kernel<true, true><<<grid, GEMM_THREADS, 0, s>>>(g);
  else if (ak && !bk) gemm_kernel<true, false><<<grid, GEMM_THREADS, 0, s>>>(g);
  else if (!ak && bk) gemm_kernel<false, true><<<grid, GEMM_THREADS, 0, s>>>(g);
  else gemm_kernel<false, false><<<grid, GEMM_THREADS, 0, s>>>(g);
  PE_TRY_LAUNCH("gemm_kernel");
  if (split > 1) {
    const int64_t total = (int64_t)M * N;
    if (split <= 8 && N % 8 == 0 && al(ws)) {
      gemm_splitk_reduce8<<<grid1(total / 8, 256), 256, 0, s>>>(g, (int)split);
      PE_TRY_LAUNCH("gemm_splitk_reduce8");
      return PE_OK;
    }
    gemm_splitk_reduce<<<(unsigned)((total + 31) / 32), dim3(32, 8), 0, s>>>(g, (int)split);
    PE_TRY_LAUNCH("gemm_splitk_reduce");
  }
  return PE_OK;
}

extern "C" pe_status pe_nn_im2col3(const void *X, int32_t B, int32_t H, int32_t W, int32_t C,
                                   void *col, int32_t backward, void *stream) {
  NN_CHECK_STREAM;
  if (!X || !col || B <= 0 || H <= 0 || W <= 0 || C <= 0)
    return pe_fail(PE_EINVAL, "pe_nn_im2col3: bad arguments");
  const bool v8 = (C % 8) == 0 && (reinterpret_cast<uintptr_t>(X) & 15) == 0 &&
                  (reinterpret_cast<uintptr_t>(col) & 15) == 0;
  const bf16 *x = static_cast<const bf16 *>(X);
  bf16 *y = static_cast<bf16 *>(col);
  if (!backward) {
    const int64_t n = (int64_t)B * H * W * 9 * (v8 ? C / 8 : C);
    if (v8) im2col3_kernel<8><<<grid1(n, 256), 256, 0, s>>>(x, B, H, W, C, y);
    else im2col3_kernel<1><<<grid1(n, 256), 256, 0, s>>>(x, B, H, W, C, y);
    PE_TRY_LAUNCH("im2col3_kernel");
  } else {  // X is dcol [P][9C], col is dX [P][C]
    const int64_t n = (int64_t)B * H * W * (v8 ? C / 8 : C);
    if (v8) col2im3_kernel<8><<<grid1(n, 256), 256, 0, s>>>(x, B, H, W, C, y);
    else col2im3_kernel<1><<<grid1(n, 256), 256, 0, s>>>(x, B, H, W, C, y);
    PE_TRY_LAUNCH("col2im3_kernel");
  }
  return PE_OK;
}

static bool al4(const void *p) { return (reinterpret_cast<uintptr_t>(p) & 3) == 0; }

// Channel pairs a depthwise block shares.
static int dw_cpb(int32_t C) { return C / 2 < 32 ? C / 2 : 32; }

template <bool FLIP, int R>
static pe_status launch_dw7_rows(const void *X, const float *w, const float *bias, int B, int H,
                                 int W, int C, void *Y, cudaStream_t s) {
  const int cpb = dw_cpb(C), slots = DW_THREADS / cpb, gy = (C / 2 + cpb - 1) / cpb;
  const int64_t npos = (int64_t)B * ((H + R - 1) / R) * ((W + DW_PX - 1) / DW_PX);
  int64_t gx = (npos + slots - 1) / slots;
  const int64_t cap = ((int64_t)n_sms() * 8 + gy - 1) / gy;  // a few positions per weight load
  if (gx > cap) gx = cap;
  const dim3 grid((unsigned)gx, (unsigned)gy);
  const size_t smem = sizeof(float2) * 49 * cpb;
  const uint32_t *x = static_cast<const uint32_t *>(X);
  uint32_t *y = static_cast<uint32_t *>(Y);
  switch (C) {
    case 32: dw7_kernel<FLIP, R, 32><<<grid, DW_THREADS, smem, s>>>(x, w, bias, B, H, W, C, cpb, y); break;
    case 64: dw7_kernel<FLIP, R, 64><<<grid, DW_THREADS, smem, s>>>(x, w, bias, B, H, W, C, cpb, y); break;
    case 128: dw7_kernel<FLIP, R, 128><<<grid, DW_THREADS, smem, s>>>(x, w, bias, B, H, W, C, cpb, y); break;
    case 256: dw7_kernel<FLIP, R, 256><<<grid, DW_THREADS, smem, s>>>(x, w, bias, B, H, W, C, cpb, y); break;
    default: dw7_kernel<FLIP, R, 0><<<grid, DW_THREADS, smem, s>>>(x, w, bias, B, H, W, C, cpb, y);
  }
  PE_TRY_LAUNCH("dw7_kernel");
  return PE_OK;
}

// Four rows per thread when that still gives every SM its two blocks of
// threads, else one.
template <bool FLIP>
static pe_status launch_dw7(const void *X, const float *w, const float *bias, int B, int H, int W,
                            int C, void *Y, cudaStream_t s) {
  const int64_t threads4 = (int64_t)B * ((H + 3) / 4) * ((W + DW_PX - 1) / DW_PX) * (C / 2);
  return threads4 >= (int64_t)n_sms() * 2 * DW_THREADS
             ? launch_dw7_rows<FLIP, 4>(X, w, bias, B, H, W, C, Y, s)
             : launch_dw7_rows<FLIP, 1>(X, w, bias, B, H, W, C, Y, s);
}

extern "C" pe_status pe_nn_dwconv7(const void *X, const float *w, const float *bias, int32_t B,
                                   int32_t H, int32_t W, int32_t C, void *Y, void *stream) {
  NN_CHECK_STREAM;
  if (!X || !w || !Y || B <= 0 || H <= 0 || W <= 0 || C <= 0 || (C & 1) || !al4(X) || !al4(Y) ||
      (reinterpret_cast<uintptr_t>(w) & 7))
    return pe_fail(PE_EINVAL, "pe_nn_dwconv7: bad arguments (C even, aligned buffers)");
  return launch_dw7<false>(X, w, bias, B, H, W, C, Y, s);
}

// The weight gradient's split (by constants and sizes only, so that the order of
// the sums does not depend on the device): the stretch of a row a thread walks
// at a time, shorter where the image has too few of them for the threads; the
// partials per channel chunk, about 304 blocks over the chunks (two per SM), or
// a multiple of that where a thread's chain of additions would be longer than that
// of one thread for every 1024th row (128 and 256 channels; FP32's rounding grows
// with the chain: error against 64 bits, 32 x 32^2 by 256, 8.5e-8 -> 8.0e-8, the
// whole backward 79 -> 94 us; 32 x 64^2 by 128 120 -> 131 us); and the positions
// added side by side, two turns within 26 KB.
struct dw_plan {
  int seg, chunks, reps;
};
static dw_plan plan_dw(int32_t B, int32_t H, int32_t W, int32_t C) {
  dw_plan w;
  const int cpb = dw_cpb(C), slots = DWG_THREADS / 2 / cpb, gy = (C / 2 + cpb - 1) / cpb;
  const int64_t rows = (int64_t)B * H, most = (304 + gy - 1) / gy;
  w.seg = W >= 128 ? 64 : (W >= 64 ? 32 : 16);
  while (w.seg > 8 && rows * ((W + w.seg - 1) / w.seg) < most * slots) w.seg /= 2;
  const int64_t items = rows * ((W + w.seg - 1) / w.seg), need = (items + slots - 1) / slots;
  const int64_t per = (rows + 1023) / 1024 * W / (W < w.seg ? W : w.seg);  // (at least one)
  const int64_t least = ((items + per - 1) / per + slots - 1) / slots;
  const int64_t chunks = (least + most - 1) / most * most;
  w.chunks = (int)(need < chunks ? need : chunks);
  w.reps = 1;
  while (2 * w.reps <= slots && 2 * w.reps * 50 * cpb * (int)sizeof(float2) <= 26 * 1024) w.reps *= 2;
  return w;
}

extern "C" size_t pe_nn_dwconv7_bwd_workspace(int32_t B, int32_t H, int32_t W, int32_t C) {
  if (B <= 0 || H <= 0 || W <= 0 || C < 2) return 0;
  return (size_t)plan_dw(B, H, W, C).chunks * 50 * C * sizeof(float) + 256;
}

// dX (nullable), dw [7][7][C] and db [C] (FP32, overwritten).
extern "C" pe_status pe_nn_dwconv7_bwd(const void *X, const void *dY, const float *w, int32_t B,
                                       int32_t H, int32_t W, int32_t C, void *dX, float *dw,
                                       float *db, void *ws, size_t ws_bytes, void *stream) {
  NN_CHECK_STREAM;
  if (!X || !dY || !w || B <= 0 || H <= 0 || W <= 0 || C <= 0 || (C & 1) || !al4(X) ||
      !al4(dY) || (dX && !al4(dX)) || (reinterpret_cast<uintptr_t>(w) & 7))
    return pe_fail(PE_EINVAL, "pe_nn_dwconv7_bwd: bad arguments (C even, aligned buffers)");
  if (dX) {
    const pe_status st = launch_dw7<true>(dY, w, nullptr, B, H, W, C, dX, s);
    if (st != PE_OK) return st;
  }
  if (dw || db) {
    const dw_plan p = plan_dw(B, H, W, C);
    const int chunks = p.chunks;
    size_t need = (size_t)chunks * 50 * C * sizeof(float);
    if (!ws || ws_bytes < need) return pe_fail(PE_ENOMEM, "pe_nn_dwconv7_bwd: workspace");
    float *part = static_cast<float *>(ws);
    const int cpb = dw_cpb(C);
    const dim3 grid((unsigned)chunks, (unsigned)((C / 2 + cpb - 1) / cpb));
    const size_t smem = sizeof(float2) * 50 * cpb * p.reps;
    const uint32_t *x = static_cast<const uint32_t *>(X), *g = static_cast<const uint32_t *>(dY);
    switch (C) {
      case 32: dw7_wgrad_kernel<32><<<grid, DWG_THREADS, smem, s>>>(x, g, B, H, W, C, cpb, p.seg, p.reps, part); break;
      case 64: dw7_wgrad_kernel<64><<<grid, DWG_THREADS, smem, s>>>(x, g, B, H, W, C, cpb, p.seg, p.reps, part); break;
      case 128: dw7_wgrad_kernel<128><<<grid, DWG_THREADS, smem, s>>>(x, g, B, H, W, C, cpb, p.seg, p.reps, part); break;
      case 256: dw7_wgrad_kernel<256><<<grid, DWG_THREADS, smem, s>>>(x, g, B, H, W, C, cpb, p.seg, p.reps, part); break;
      default: dw7_wgrad_kernel<0><<<grid, DWG_THREADS, smem, s>>>(x, g, B, H, W, C, cpb, p.seg, p.reps, part);
    }
    PE_TRY_LAUNCH("dw7_wgrad_kernel");
    // part[chunk][50][C]: taps 0..48 -> dw, 49 -> db; sum the chunks in
    // order into chunk 0 (a block reads only the columns it writes)
    sum_chunks_kernel<<<(unsigned)((50 * C + 31) / 32), dim3(32, 32), 0, s>>>(part, chunks,
                                                                          50 * (int64_t)C, part, 0);
    PE_TRY_LAUNCH("sum_chunks_kernel");
    if (dw) PE_TRY_CUDA(cudaMemcpyAsync(dw, part, sizeof(float) * 49 * C, cudaMemcpyDeviceToDevice, s));
    if (db)
      PE_TRY_CUDA(cudaMemcpyAsync(db, part + 49 * C, sizeof(float) * C, cudaMemcpyDeviceToDevice, s));
  }
  return PE_OK;
}

extern "C" pe_status pe_nn_layernorm(const void *X, const float *gamma, const float *beta,
                                     int64_t P, int32_t C, float eps, void *Y, float *mean,
                                     float *rstd, void *stream) {
  NN_CHECK_STREAM;
  if (!X || !gamma || !beta || !Y || !mean || !rstd || P <= 0 || C <= 0 || C > 256)
    return pe_fail(PE_EINVAL, "pe_nn_layernorm: bad arguments (C <= 256)");
  const bool al16 = (reinterpret_cast<uintptr_t>(X) & 15) == 0 &&
                    (reinterpret_cast<uintptr_t>(Y) & 15) == 0;
  if (al16 && C == 32) {   // (64 channels in registers would cap a thread at 255 registers)
    ln_fwd_narrow_kernel<32><<<grid1(P, 256), 256, 0, s>>>(
        static_cast<const bf16 *>(X), gamma, beta, P, eps, static_cast<bf16 *>(Y), mean, rstd);
    PE_TRY_LAUNCH("ln_fwd_narrow_kernel");
  } else if (al16 && (C == 64 || C == 128 || C == 256)) {
    // (the widths of the network's levels; the kernel takes any multiple of 32, an
    // instance each, and the other widths have a warp per pixel and 2-byte loads,
    // which took four times as long at 64 channels)
    const bf16 *x = static_cast<const bf16 *>(X);
    bf16 *y = static_cast<bf16 *>(Y);
    const int blocks = grid1(P, LN_THREADS / 4, 8);
    if (C == 64) ln_fwd_quad_kernel<2><<<blocks, LN_THREADS, 0, s>>>(x, gamma, beta, P, eps, y, mean, rstd);
    else if (C == 128) ln_fwd_quad_kernel<4><<<blocks, LN_THREADS, 0, s>>>(x, gamma, beta, P, eps, y, mean, rstd);
    else ln_fwd_quad_kernel<8><<<blocks, LN_THREADS, 0, s>>>(x, gamma, beta, P, eps, y, mean, rstd);
    PE_TRY_LAUNCH("ln_fwd_quad_kernel");
  } else {
    ln_fwd_kernel<<<grid1(P * 32, 256), 256, 0, s>>>(static_cast<const bf16 *>(X), gamma, beta, P,
                                                     C, eps, static_cast<bf16 *>(Y), mean, rstd);
    PE_TRY_LAUNCH("ln_fwd_kernel");
  }
  return PE_OK;
}

// Blocks of the quad backward: 64 pixels each, 608 at most (four per SM; a
// constant, so that the order of the sums does not depend on the device).
static int ln_bwd_blocks(int64_t P) {
  const int64_t b = (P + LN_THREADS / 4 - 1) / (LN_THREADS / 4);
  return (int)(b < 608 ? b : 608);
}

extern "C" size_t pe_nn_layernorm_bwd_workspace(int64_t P, int32_t C) {
  int64_t warps = (int64_t)grid1(P * 32, 256) * 8;  // (the quad kernels: fewer, one per block)
  return (size_t)warps * 2 * C * sizeof(float) + 256;
}

// dX and dgamma, dbeta (FP32, overwritten).
extern "C" pe_status pe_nn_layernorm_bwd(const void *dY, const void *X, const float *gamma,
                                         const float *mean, const float *rstd, int64_t P, int32_t C,
                                         void *dX, float *dgamma, float *dbeta, void *ws,
                                         size_t ws_bytes, void *stream) {
  NN_CHECK_STREAM;
  if (!dY || !X || !gamma || !mean || !rstd || !dX || P <= 0 || C <= 0 || C > 256)
    return pe_fail(PE_EINVAL, "pe_nn_layernorm_bwd: bad arguments (C <= 256)");
  int blocks = grid1(P * 32, 256);
  int64_t warps = (int64_t)blocks * 8;
  size_t need = (size_t)warps * 2 * C * sizeof(float);
  if (!ws || ws_bytes < need) return pe_fail(PE_ENOMEM, "pe_nn_layernorm_bwd: workspace");
  float *part = static_cast<float *>(ws);
  auto al16 = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  if (al16(X) && al16(dY) && al16(dX) && (C == 32 || C == 64 || C == 128)) {
    // (as forward, but 256 channels would hold 256 values and sums per thread)
    const bf16 *x = static_cast<const bf16 *>(X), *dy = static_cast<const bf16 *>(dY);
    bf16 *dx = static_cast<bf16 *>(dX);
    const int nb = ln_bwd_blocks(P);
    if (C == 32) ln_bwd_quad_kernel<1><<<nb, LN_THREADS, 0, s>>>(dy, x, gamma, mean, rstd, P, dx, part);
    else if (C == 64) ln_bwd_quad_kernel<2><<<nb, LN_THREADS, 0, s>>>(dy, x, gamma, mean, rstd, P, dx, part);
    else ln_bwd_quad_kernel<4><<<nb, LN_THREADS, 0, s>>>(dy, x, gamma, mean, rstd, P, dx, part);
    PE_TRY_LAUNCH("ln_bwd_quad_kernel");
    warps = nb;  // one partial per block
  } else {
  ln_bwd_kernel<<<blocks, 256, 0, s>>>(static_cast<const bf16 *>(dY), static_cast<const bf16 *>(X),
                                       gamma, mean, rstd, P, C, static_cast<bf16 *>(dX), part);
  PE_TRY_LAUNCH("ln_bwd_kernel");
  }
  // part[warp or block][2][C]: summed in order
  sum_chunks_kernel<<<(unsigned)((2 * C + 31) / 32), dim3(32, 32), 0, s>>>(part, (int)warps,
                                                                        2 * (int64_t)C, part, 0);
  PE_TRY_LAUNCH("sum_chunks_kernel");
  if (dgamma) PE_TRY_CUDA(cudaMemcpyAsync(dgamma, part, sizeof(float) * C, cudaMemcpyDeviceToDevice, s));
  if (dbeta) PE_TRY_CUDA(cudaMemcpyAsync(dbeta, part + C, sizeof(float) * C, cudaMemcpyDeviceToDevice, s));
  return PE_OK;
}

// Row chunks of a column sum: fixed by M.
static int64_t colsum_chunks(int64_t M) {
  int64_t c = (M + 255) / 256;
  return c < 1 ? 1 : (c > 1024 ? 1024 : c);
}

extern "C" size_t pe_nn_colsum_workspace(int64_t M, int32_t N) {
  return (size_t)colsum_chunks(M) * N * sizeof(float) + 256;
}

// out[n] = (accumulate ? out[n] : 0) + sum_m X[m * ld + n] (fixed order).
extern "C" pe_status pe_nn_colsum(const void *X, int64_t M, int32_t N, int64_t ld, float *out,
                                  int32_t accumulate, void *ws, size_t ws_bytes, void *stream) {
  NN_CHECK_STREAM;
  if (!X || !out || M <= 0 || N <= 0 || ld < N) return pe_fail(PE_EINVAL, "pe_nn_colsum: bad arguments");
  const int64_t chunks = colsum_chunks(M);
  size_t need = (size_t)chunks * N * sizeof(float);
  if (!ws || ws_bytes < need) return pe_fail(PE_ENOMEM, "pe_nn_colsum: workspace");
  float *part = static_cast<float *>(ws);
  const int64_t rpc = (M + chunks - 1) / chunks;
  const bool pair = (N % 2 == 0) && (ld % 2 == 0) && al4(X);
  const bf16 *x = static_cast<const bf16 *>(X);
  if (pair) {
    colsum_kernel<true><<<dim3((N / 2 + 31) / 32, (unsigned)chunks), dim3(32, 8), 0, s>>>(
        x, M, N, ld, rpc, part);
  } else {
    colsum_kernel<false><<<dim3((N + 31) / 32, (unsigned)chunks), dim3(32, 8), 0, s>>>(
        x, M, N, ld, rpc, part);
  }
  PE_TRY_LAUNCH("colsum_kernel");
  sum_chunks_kernel<<<(unsigned)((N + 31) / 32), dim3(32, 32), 0, s>>>(part, (int)chunks, N, out,
                                                                      accumulate);
  PE_TRY_LAUNCH("sum_chunks_kernel");
  return PE_OK;
}

// Weight and bias gradient of a layer with N <= 4 outputs (the heads: rows of dY
// too short for a TMA row): a thread owns eight inputs and strides over the
// pixels, N x 8 sums in registers; the block's threads of the same inputs are
// added in order.  part[block][N K + N].  (The mma.sync kernel spent a 128-row
// tile on one row: 355 us for 2.1M pixels of 32 inputs, 134 MB.)
namespace {
constexpr int THIN_THREADS = 256;
template <int N>
__global__ void __launch_bounds__(THIN_THREADS)
    wgrad_thin_kernel(const bf16 *__restrict__ dY, int64_t ldy, const bf16 *__restrict__ X,
                      int64_t ldx, int64_t P, int K, float *__restrict__ part) {
  extern __shared__ float s_red[];  // [THIN_THREADS][N * 8 + N]
  constexpr int NV = N * 8 + N;
  const int kv = K / 8, j = threadIdx.x % kv, r = threadIdx.x / kv, rows = THIN_THREADS / kv;
  float acc[NV];
#pragma unroll
  for (int i = 0; i < NV; ++i) acc[i] = 0.0f;
  for (int64_t p = (int64_t)blockIdx.x * rows + r; p < P; p += (int64_t)gridDim.x * rows) {
    const uint4 u = __ldg(reinterpret_cast<const uint4 *>(X + p * ldx) + j);
    const uint32_t w[4] = {u.x, u.y, u.z, u.w};
#pragma unroll
    for (int n = 0; n < N; ++n) {
      const float g = b2f(dY[p * ldy + n]);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        acc[n * 8 + 2 * e] = fmaf(g, __uint_as_float(w[e] << 16), acc[n * 8 + 2 * e]);
        acc[n * 8 + 2 * e + 1] = fmaf(g, __uint_as_float(w[e] & 0xffff0000u), acc[n * 8 + 2 * e + 1]);
      }
      acc[N * 8 + n] += g;
    }
  }
#pragma unroll
  for (int i = 0; i < NV; ++i) s_red[threadIdx.x * NV + i] = acc[i];
  __syncthreads();
  float *out = part + (size_t)blockIdx.x * (N * K + N);
  for (int o = threadIdx.x; o < N * K + N; o += THIN_THREADS) {
    const int n = o < N * K ? o / K : o - N * K, k = o < N * K ? o % K : 0;
    const int i = o < N * K ? n * 8 + k % 8 : N * 8 + n;
    float t = 0.0f;
    for (int q = 0; q < rows; ++q) t += s_red[(q * kv + k / 8) * NV + i];
    out[o] = t;
  }
}
}  // namespace

constexpr int kThinBlocks = 608;  // four per SM; a constant, as for the other sums
static bool thin_wgrad(const void *X, int64_t ldx, int32_t N, int32_t K) {
  return N <= 4 && K % 8 == 0 && K <= 256 && THIN_THREADS % (K / 8) == 0 && ldx % 8 == 0 &&
         (reinterpret_cast<uintptr_t>(X) & 15) == 0;
}

// Workspace of pe_nn_linear_wgrad: either path's.
extern "C" size_t pe_nn_linear_wgrad_workspace(int64_t P, int32_t N, int32_t K) {
  if (P <= 0 || N <= 0 || K <= 0) return 0;
  size_t a = pe_wgrad_tc_workspace(P, N, K), b = pe_nn_gemm_workspace(N, K, P),
         c = pe_nn_colsum_workspace(P, N);
  const size_t d = N <= 4 ? (size_t)kThinBlocks * ((size_t)N * K + N) * sizeof(float) : 0;
  a = a > b ? a : b;
  a = a > d ? a : d;
  return (a > c ? a : c) + 256;
}

extern "C" pe_status pe_nn_linear_wgrad(const void *dY, int64_t ldy, const void *X, int64_t ldx,
                                        int64_t P, int32_t N, int32_t K, float *dW, float *db,
                                        void *ws, size_t ws_bytes, void *stream) {
  NN_CHECK_STREAM;
  if (!dY || !X || !dW || P <= 0 || N <= 0 || K <= 0 || ldy < N || ldx < K)
    return pe_fail(PE_EINVAL, "pe_nn_linear_wgrad: bad arguments");
  if (!ws || ws_bytes < pe_nn_linear_wgrad_workspace(P, N, K))
    return pe_fail(PE_ENOMEM, "pe_nn_linear_wgrad: workspace");
  if (g_gemm_path == 0 && pe_wgrad_tc_eligible(dY, ldy, X, ldx, P, N, K)) {
    const pe_status st = pe_wgrad_tc(dY, ldy, X, ldx, P, N, K, dW, db, static_cast<float *>(ws), s);
    if (st != PE_EUNSUPPORTED) return st;
  }
  if (g_gemm_path == 0 && thin_wgrad(X, ldx, N, K)) {
    const int64_t need = (P + THIN_THREADS / (K / 8) - 1) / (THIN_THREADS / (K / 8));
    const int blocks = (int)(need < kThinBlocks ? need : kThinBlocks);
    const size_t smem = sizeof(float) * THIN_THREADS * 9 * N;
    const bf16 *y = static_cast<const bf16 *>(dY), *x = static_cast<const bf16 *>(X);
    float *part = static_cast<float *>(ws);
    if (N == 1) wgrad_thin_kernel<1><<<blocks, THIN_THREADS, smem, s>>>(y, ldy, x, ldx, P, K, part);
    else if (N == 2) wgrad_thin_kernel<2><<<blocks, THIN_THREADS, smem, s>>>(y, ldy, x, ldx, P, K, part);
    else if (N == 3) wgrad_thin_kernel<3><<<blocks, THIN_THREADS, smem, s>>>(y, ldy, x, ldx, P, K, part);
    else wgrad_thin_kernel<4><<<blocks, THIN_THREADS, smem, s>>>(y, ldy, x, ldx, P, K, part);
    PE_TRY_LAUNCH("wgrad_thin_kernel");
    return pe_wgrad_reduce(part, blocks, (int64_t)N * K, (int64_t)N * K + N, dW, db, s);
  }
  const pe_status st = pe_nn_gemm(N, K, P, dY, 1, ldy, X, ldx, 1, dW, K, 1, nullptr, nullptr, 0,
                                  nullptr, 0, 0, 1.0f, 0.0f, ws, ws_bytes, stream);
  if (st != PE_OK || !db) return st;
  return pe_nn_colsum(dY, P, N, ldy, db, 0, ws, ws_bytes, stream);
}

// One input channel (the network's first layer): K = 9 is too short for a TMA
// row.  Forward: a warp takes 16 pixels by 32 outputs, its lanes read the taps of
// their mma.sync fragment from the image, and the products are those of
// gemm_kernel on the neighbourhood matrix (one k-step of 16, taps 9..15 zero, and
// one of zeros), so are the bits.  16 x 256^2 by 32: 126 us with the
// matrix written, 39 us now (writing y takes 10; the taps' index arithmetic most of
// the rest).
namespace {
struct stem_img {
  const bf16 *x;
  int W, H;
  // tap (3 ky + kx) at pixel (px, py) of the image that starts at row0 rows
  __device__ __forceinline__ uint32_t tap(int64_t p, int px, int py, int t) const {
    const int dy = t / 3 - 1, dx = t % 3 - 1;
    const bool in = (unsigned)(py + dy) < (unsigned)H && (unsigned)(px + dx) < (unsigned)W;
    return in ? (uint32_t)__ldg(reinterpret_cast<const unsigned short *>(x) + p + dy * W + dx) : 0u;
  }
};

__global__ void __launch_bounds__(256)
    stem_fwd_kernel(const stem_img im, int64_t P, const bf16 *__restrict__ w,
                    const float *__restrict__ bias, bf16 *__restrict__ y, int N) {
  const int lane = threadIdx.x & 31, gq = lane >> 2, tq = lane & 3, n0 = blockIdx.y * 32;
  const bool vec = (reinterpret_cast<uintptr_t>(y) & 15) == 0;
  uint32_t b[4][2];
  float bs[8];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const unsigned short *r = reinterpret_cast<const unsigned short *>(w) + (int64_t)(n0 + 8 * j + gq) * 9;
    b[j][0] = (uint32_t)r[2 * tq] | (uint32_t)r[2 * tq + 1] << 16;
    b[j][1] = tq == 0 ? (uint32_t)r[8] : 0u;
  }
#pragma unroll
  for (int e = 0; e < 8; ++e) bs[e] = bias ? bias[n0 + 8 * tq + e] : 0.0f;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  for (int64_t m0 = ((int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5)) * 16; m0 < P;
       m0 += warps * 16) {
    uint32_t a[4] = {0u, 0u, 0u, 0u};
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t p = m0 + gq + 8 * h;
      if (p < P) {
        const uint32_t q = (uint32_t)p / (uint32_t)im.W;  // (P < 2^31)
        const int px = (int)((uint32_t)p - q * (uint32_t)im.W), py = (int)(q % (uint32_t)im.H);
        a[h] = im.tap(p, px, py, 2 * tq) | im.tap(p, px, py, 2 * tq + 1) << 16;
        if (tq == 0) a[2 + h] = im.tap(p, px, py, 8);
      }
    }
    uint32_t out[2][4];  // [row half][8-column block]: this lane's two columns
    float acc[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int e = 0; e < 4; ++e) acc[j][e] = 0.0f;
#pragma unroll
      for (int k = 0; k < 2; ++k)
        asm volatile(
            "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, "
            "{%4,%5,%6,%7}, {%8,%9}, {%0,%1,%2,%3};\n"
            : "+f"(acc[j][0]), "+f"(acc[j][1]), "+f"(acc[j][2]), "+f"(acc[j][3])
            : "r"(k ? 0u : a[0]), "r"(k ? 0u : a[1]), "r"(k ? 0u : a[2]), "r"(k ? 0u : a[3]),
              "r"(k ? 0u : b[j][0]), "r"(k ? 0u : b[j][1]));
    }
    // the four lanes of a row exchange their pairs of columns, so that each holds
    // the eight columns from 8 tq on: lane tq keeps block tq of every partner
    float v[2][8];
#pragma unroll
    for (int h = 0; h < 2; ++h)
#pragma unroll
      for (int r = 0; r < 4; ++r) {  // from lane tq ^ r, which sends its block (its tq) ^ r
        const int send = tq ^ r;
        float s0 = acc[0][2 * h], s1 = acc[0][2 * h + 1];
#pragma unroll
        for (int j = 1; j < 4; ++j) {
          s0 = send == j ? acc[j][2 * h] : s0;
          s1 = send == j ? acc[j][2 * h + 1] : s1;
        }
        s0 = __shfl_xor_sync(0xffffffffu, s0, r);
        s1 = __shfl_xor_sync(0xffffffffu, s1, r);
#pragma unroll
        for (int e = 0; e < 4; ++e)
          if (e == send) {
            v[h][2 * e] = s0;
            v[h][2 * e + 1] = s1;
          }
      }
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int64_t p = m0 + gq + 8 * h;
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        float c0 = v[h][2 * e], c1 = v[h][2 * e + 1];
        if (bias) {
          c0 += bs[2 * e];
          c1 += bs[2 * e + 1];
        }
        const bf162 o = __floats2bfloat162_rn(c0, c1);
        out[h][e] = *reinterpret_cast<const uint32_t *>(&o);
      }
      bf16 *dst = y + p * N + n0 + 8 * tq;
      if (p < P && vec) {
        *reinterpret_cast<uint4 *>(dst) = make_uint4(out[h][0], out[h][1], out[h][2], out[h][3]);
      } else if (p < P) {
#pragma unroll
        for (int e = 0; e < 8; ++e)
          reinterpret_cast<unsigned short *>(dst)[e] = (unsigned short)(out[h][e / 2] >> (16 * (e & 1)));
      }
    }
  }
}

// Weight and bias gradient of that layer: dW[n][tap] = sum_p dY[p][n] x[p + tap].
// LPP = N / 8 lanes per pixel, eight outputs and 8 x 9 + 8 sums each, so dY is
// read once in 16-byte accesses and x through the caches.  part[block][9 N + N].
// 32 x 256^2 by 32: 361 us with the matrix written and a 128-row mma.sync tile of
// which 32 rows held outputs, 117 us now.
// VEC: rows of dY on 16-byte boundaries.
constexpr int kStemBlocks = 304, STEM_THREADS = 256;
template <int LPP, bool VEC>
__global__ void __launch_bounds__(STEM_THREADS, 2)
    stem_wgrad_kernel(const stem_img im, int64_t P, const bf16 *__restrict__ dY,
                      float *__restrict__ part) {
  constexpr int PPW = 32 / LPP, N = 8 * LPP, WARPS = STEM_THREADS / 32;
  __shared__ float s_sum[WARPS][10 * 8][LPP];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, c = lane % LPP;
  float acc[10][8];
#pragma unroll
  for (int t = 0; t < 10; ++t)
#pragma unroll
    for (int e = 0; e < 8; ++e) acc[t][e] = 0.0f;
  const int64_t step = (int64_t)gridDim.x * WARPS * PPW;
  for (int64_t p = ((int64_t)blockIdx.x * WARPS + warp) * PPW + lane / LPP; p < P; p += step) {
    uint32_t wd[4];
    if (VEC) {
      const uint4 u = __ldg(reinterpret_cast<const uint4 *>(dY + p * N) + c);
      wd[0] = u.x;
      wd[1] = u.y;
      wd[2] = u.z;
      wd[3] = u.w;
    } else {
      const unsigned short *r = reinterpret_cast<const unsigned short *>(dY + p * N) + 8 * c;
#pragma unroll
      for (int e = 0; e < 4; ++e) wd[e] = (uint32_t)__ldg(r + 2 * e) | (uint32_t)__ldg(r + 2 * e + 1) << 16;
    }
    const uint32_t q = (uint32_t)p / (uint32_t)im.W;
    const int px = (int)((uint32_t)p - q * (uint32_t)im.W), py = (int)(q % (uint32_t)im.H);
    float xt[9], d[8];
#pragma unroll
    for (int t = 0; t < 9; ++t) xt[t] = __uint_as_float(im.tap(p, px, py, t) << 16);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      d[2 * e] = __uint_as_float(wd[e] << 16);
      d[2 * e + 1] = __uint_as_float(wd[e] & 0xffff0000u);
    }
#pragma unroll
    for (int e = 0; e < 8; ++e) {
#pragma unroll
      for (int t = 0; t < 9; ++t) acc[t][e] = fmaf(d[e], xt[t], acc[t][e]);
      acc[9][e] += d[e];
    }
  }
#pragma unroll
  for (int t = 0; t < 10; ++t)
#pragma unroll
    for (int e = 0; e < 8; ++e) {
#pragma unroll
      for (int o = 16; o >= LPP; o >>= 1) acc[t][e] += __shfl_xor_sync(0xffffffffu, acc[t][e], o);
      if (lane < LPP) s_sum[warp][t * 8 + e][lane] = acc[t][e];
    }
  __syncthreads();
  float *out = part + (size_t)blockIdx.x * (10 * N);
  for (int o = threadIdx.x; o < 10 * N; o += STEM_THREADS) {
    const int n = o < 9 * N ? o / 9 : o - 9 * N, t = o < 9 * N ? o % 9 : 9;
    float v = 0.0f;
    for (int k = 0; k < WARPS; ++k) v += s_sum[k][t * 8 + n % 8][n / 8];
    out[o] = v;
  }
}

template <int LPP>
pe_status launch_stem_wgrad(const stem_img &im, int64_t P, const bf16 *dY, float *dW, float *db,
                            float *part, cudaStream_t s) {
  constexpr int per_block = STEM_THREADS / LPP;
  const int64_t need = (P + per_block - 1) / per_block;
  const int blocks = (int)(need < kStemBlocks ? need : kStemBlocks);
  if ((reinterpret_cast<uintptr_t>(dY) & 15) == 0)
    stem_wgrad_kernel<LPP, true><<<blocks, STEM_THREADS, 0, s>>>(im, P, dY, part);
  else
    stem_wgrad_kernel<LPP, false><<<blocks, STEM_THREADS, 0, s>>>(im, P, dY, part);
  PE_TRY_LAUNCH("stem_wgrad_kernel");
  return pe_wgrad_reduce(part, blocks, 72 * LPP, 80 * LPP, dW, db, s);
}
}  // namespace

// 3x3 convolution, y = col(x) w^T + bias with col the neighbourhood matrix.  The
// TMA loads gather it from the image itself (im2col mode) where its channels
// fill whole 64-channel blocks and the contraction would run unsplit on the
// tcgen05 kernel anyway (same products in the same order, same bits); else col is
// written to the workspace.  Writing and reading col, nine times the image, was
// a tenth of the network's forward pass: 16 x 256^2 images, 6.15 -> 5.32 ms
// together with the heads' rows written from registers (nn_tc.cu, MODE 4).
static pe_gemm_args conv_args(const void *x, int32_t B, int32_t H, int32_t W, int32_t Cin,
                              const void *w, const float *bias, void *y, int32_t Cout) {
  pe_gemm_args g;
  memset(&g, 0, sizeof(g));
  g.M = B * H * W;
  g.N = Cout;
  g.K = 9 * (int64_t)Cin;
  g.A = static_cast<const bf16 *>(x);
  g.sak = g.sbk = 1;
  g.sam = 9 * (int64_t)Cin;
  g.B = static_cast<const bf16 *>(w);
  g.sbn = 9 * (int64_t)Cin;
  g.C = y;
  g.ldc = Cout;
  g.bias = bias;
  g.alpha = 1.0f;
  auto al = [](const void *p) { return (reinterpret_cast<uintptr_t>(p) & 15) == 0; };
  g.vec_c = al(y) && Cout % 8 == 0 && (!bias || (reinterpret_cast<uintptr_t>(bias) & 3) == 0);
  return g;
}

static bool conv_sizes(int32_t B, int32_t H, int32_t W, int32_t Cin, int32_t Cout) {
  return B > 0 && H > 0 && W > 0 && Cin > 0 && Cout > 0 && (int64_t)B * H * W < (1ll << 31) - 4096;
}

// Whether both passes gather (then no col is written and the workspace holds none).
static bool conv_gathered(int32_t B, int32_t H, int32_t W, int32_t Cin, int32_t Cout) {
  return g_gemm_path == 0 && gemm_split(B * H * W, Cout, 9 * (int64_t)Cin, nullptr) == 1 &&
         pe_conv3_tc_sizes(B, H, W, Cin, Cout);
}

// Whether the one-channel kernels above take a layer's forward pass, its gradient.
static bool stem_fwd_sizes(int32_t Cin, int32_t Cout) {
  return Cin == 1 && Cout % 32 == 0 && Cout / 32 <= 65535;
}
static bool stem_wgrad_sizes(int32_t Cin, int32_t Cout) {
  return Cin == 1 && (Cout == 8 || Cout == 16 || Cout == 32 || Cout == 64 || Cout == 128);
}

extern "C" size_t pe_nn_conv3_workspace(int32_t B, int32_t H, int32_t W, int32_t Cin, int32_t Cout) {
  if (!conv_sizes(B, H, W, Cin, Cout)) return 0;
  const int64_t P = (int64_t)B * H * W;
  const size_t col = ((size_t)P * 9 * Cin * sizeof(bf16) + 255) & ~size_t(255);
  const size_t a = pe_nn_gemm_workspace((int32_t)P, Cout, 9 * (int64_t)Cin),
               b = pe_nn_linear_wgrad_workspace(P, Cout, 9 * Cin);
  const size_t c = Cin == 1 ? (size_t)kStemBlocks * 10 * Cout * sizeof(float) : 0;
  if (stem_fwd_sizes(Cin, Cout) && stem_wgrad_sizes(Cin, Cout)) return c + 512;  // neither writes col
  const size_t most = a > b ? (a > c ? a : c) : (b > c ? b : c);
  return (conv_gathered(B, H, W, Cin, Cout) ? 0 : col) + most + 512;
}

// col in the workspace (256-byte aligned), with the rest of it after col.
static bf16 *conv_col(const void *x, int32_t B, int32_t H, int32_t W, int32_t Cin, void *ws,
                      size_t ws_bytes, char **rest, size_t *rest_bytes, cudaStream_t s,
                      pe_status *st) {
  const uintptr_t p = (reinterpret_cast<uintptr_t>(ws) + 255) & ~uintptr_t(255);
  const size_t skip = p - reinterpret_cast<uintptr_t>(ws);
  const size_t bytes = ((size_t)B * H * W * 9 * Cin * sizeof(bf16) + 255) & ~size_t(255);
  if (ws_bytes < skip + bytes) {
    *st = pe_fail(PE_ENOMEM, "pe_nn_conv3: workspace");
    return nullptr;
  }
  *rest = reinterpret_cast<char *>(p) + bytes;
  *rest_bytes = ws_bytes - skip - bytes;
  *st = pe_nn_im2col3(x, B, H, W, Cin, reinterpret_cast<void *>(p), 0, s);
  return reinterpret_cast<bf16 *>(p);
}

extern "C" pe_status pe_nn_conv3(const void *x, int32_t B, int32_t H, int32_t W, int32_t Cin,
                                 const void *w, const float *bias, void *y, int32_t Cout, void *ws,
                                 size_t ws_bytes, void *stream) {
  NN_CHECK_STREAM;
  if (!x || !w || !y || !conv_sizes(B, H, W, Cin, Cout))
    return pe_fail(PE_EINVAL, "pe_nn_conv3: bad arguments");
  if (!ws || ws_bytes < pe_nn_conv3_workspace(B, H, W, Cin, Cout))
    return pe_fail(PE_ENOMEM, "pe_nn_conv3: workspace");
  const pe_gemm_args g = conv_args(x, B, H, W, Cin, w, bias, y, Cout);
  if (conv_gathered(B, H, W, Cin, Cout)) {
    if (((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(w)) & 15) != 0 || !g.vec_c)
      return pe_fail(PE_EINVAL, "pe_nn_conv3: pointers on 16-byte boundaries");
    return pe_conv3_tc(g, B, H, W, Cin, s);
  }
  if (stem_fwd_sizes(Cin, Cout)) {
    const stem_img im = {g.A, W, H};
    const int64_t P = (int64_t)B * H * W;
    stem_fwd_kernel<<<dim3(grid1((P + 127) / 128, 1, 8), Cout / 32), 256, 0, s>>>(
        im, P, g.B, bias, static_cast<bf16 *>(y), Cout);
    PE_TRY_LAUNCH("stem_fwd_kernel");
    return PE_OK;
  }
  pe_status st;
  char *rest;
  size_t rest_bytes;
  const bf16 *col = conv_col(x, B, H, W, Cin, ws, ws_bytes, &rest, &rest_bytes, s, &st);
  if (st != PE_OK) return st;
  return pe_nn_gemm(g.M, Cout, g.K, col, g.K, 1, w, 1, g.K, y, Cout, 0, bias, nullptr, 0, nullptr, 0,
                    0, 1.0f, 0.0f, rest, rest_bytes, stream);
}

extern "C" pe_status pe_nn_conv3_wgrad(const void *dY, const void *x, int32_t B, int32_t H, int32_t W,
                                       int32_t Cin, int32_t Cout, float *dW, float *db, void *ws,
                                       size_t ws_bytes, void *stream) {
  NN_CHECK_STREAM;
  if (!dY || !x || !dW || !conv_sizes(B, H, W, Cin, Cout))
    return pe_fail(PE_EINVAL, "pe_nn_conv3_wgrad: bad arguments");
  if (!ws || ws_bytes < pe_nn_conv3_workspace(B, H, W, Cin, Cout))
    return pe_fail(PE_ENOMEM, "pe_nn_conv3_wgrad: workspace");
  const int64_t P = (int64_t)B * H * W;
  if (conv_gathered(B, H, W, Cin, Cout)) {
    if (((reinterpret_cast<uintptr_t>(x) | reinterpret_cast<uintptr_t>(dY)) & 15) != 0)
      return pe_fail(PE_EINVAL, "pe_nn_conv3_wgrad: pointers on 16-byte boundaries");
    const int32_t img[3] = {B, H, W};
    return pe_wgrad_tc(dY, Cout, x, 9 * (int64_t)Cin, P, Cout, 9 * Cin, dW, db,
                       static_cast<float *>(ws), s, img);
  }
  if (stem_wgrad_sizes(Cin, Cout)) {
    const stem_img im = {static_cast<const bf16 *>(x), W, H};
    const bf16 *d = static_cast<const bf16 *>(dY);
    float *part = reinterpret_cast<float *>((reinterpret_cast<uintptr_t>(ws) + 255) & ~uintptr_t(255));
    switch (Cout) {
      case 8: return launch_stem_wgrad<1>(im, P, d, dW, db, part, s);
      case 16: return launch_stem_wgrad<2>(im, P, d, dW, db, part, s);
      case 32: return launch_stem_wgrad<4>(im, P, d, dW, db, part, s);
      case 64: return launch_stem_wgrad<8>(im, P, d, dW, db, part, s);
      default: return launch_stem_wgrad<16>(im, P, d, dW, db, part, s);
    }
  }
  pe_status st;
  char *rest;
  size_t rest_bytes;
  const bf16 *col = conv_col(x, B, H, W, Cin, ws, ws_bytes, &rest, &rest_bytes, s, &st);
  if (st != PE_OK) return st;
  return pe_nn_linear_wgrad(dY, Cout, col, 9 * (int64_t)Cin, P, Cout, 9 * Cin, dW, db, rest,
                            rest_bytes, stream);
}

extern "C" pe_status pe_nn_gelu_bwd(const void *dA, const void *Z, int64_t n, void *dZ,
                                    void *stream) {
  NN_CHECK_STREAM;
  if (!dA || !Z || !dZ || n <= 0) return pe_fail(PE_EINVAL, "pe_nn_gelu_bwd: bad arguments");
  gelu_bwd_kernel<<<grid1(n, 256), 256, 0, s>>>(static_cast<const bf16 *>(dA),
                                                static_cast<const bf16 *>(Z), n,
                                                static_cast<bf16 *>(dZ));
  PE_TRY_LAUNCH("gelu_bwd_kernel");
  return PE_OK;
}

extern "C" pe_status pe_nn_maxpool2(const void *X, int32_t B, int32_t H, int32_t W, int32_t C,
                                    void *Y, uint8_t *arg, int32_t backward, void *stream) {
  NN_CHECK_STREAM;
  if (!X || !Y || !arg || B <= 0 || H < 2 || W < 2 || C <= 0 || (H & 1) || (W & 1))
    return pe_fail(PE_EINVAL, "pe_nn_maxpool2: bad arguments (even H, W)");
  if (C % 8 == 0 && ((reinterpret_cast<uintptr_t>(X) | reinterpret_cast<uintptr_t>(Y)) & 15) == 0 &&
      (reinterpret_cast<uintptr_t>(arg) & 7) == 0) {
    maxpool2_wide_kernel<<<grid1((int64_t)B * H * W * C / 32, 256), 256, 0, s>>>(
        static_cast<const uint4 *>(X), B, H, W, C / 8, static_cast<uint4 *>(Y),
        reinterpret_cast<uint2 *>(arg), backward ? 1 : 0);
    PE_TRY_LAUNCH("maxpool2_wide_kernel");
    return PE_OK;
  }
  if (!backward) {
    maxpool2_fwd_kernel<<<grid1((int64_t)B * H * W * C / 4, 256), 256, 0, s>>>(
        static_cast<const bf16 *>(X), B, H, W, C, static_cast<bf16 *>(Y), arg);
    PE_TRY_LAUNCH("maxpool2_fwd_kernel");
  } else {  // X = dY (pooled), Y = dX (full)
    maxpool2_bwd_kernel<<<grid1((int64_t)B * H * W * C, 256), 256, 0, s>>>(
        static_cast<const bf16 *>(X), arg, B, H, W, C, static_cast<bf16 *>(Y));
    PE_TRY_LAUNCH("maxpool2_bwd_kernel");
  }
  return PE_OK;
}

// Forward: src [B][H][W][4C] -> dst [B][2H][2W][ld_big] at channel offset off.
// Backward: src = the big gradient, dst = [B][H][W][4C].
extern "C" pe_status pe_nn_pixel_shuffle2(const void *src, int32_t B, int32_t H, int32_t W,
                                          int32_t C, void *dst, int64_t ld_big, int32_t off,
                                          int32_t backward, void *stream) {
  NN_CHECK_STREAM;
  if (!src || !dst || B <= 0 || H <= 0 || W <= 0 || C <= 0 || off < 0 || off + C > ld_big)
    return pe_fail(PE_EINVAL, "pe_nn_pixel_shuffle2: bad arguments");
  {
    const bf16 *big = static_cast<const bf16 *>(backward ? src : dst);
    const bool v8 = C % 8 == 0 && off % 8 == 0 && ld_big % 8 == 0 &&
                    (reinterpret_cast<uintptr_t>(big) & 15) == 0;
    const int64_t n = (int64_t)B * 4 * H * W * (v8 ? C / 8 : C);
    if (v8 && (reinterpret_cast<uintptr_t>(backward ? dst : src) & 15) == 0)
      pixel_shuffle2_wide_kernel<<<grid1(n / 4, 256), 256, 0, s>>>(
          static_cast<const bf16 *>(src), B, H, W, C, static_cast<bf16 *>(dst), ld_big, off,
          backward ? 1 : 0);
    else if (v8)
      pixel_shuffle2_kernel<8><<<grid1(n, 256), 256, 0, s>>>(
          static_cast<const bf16 *>(src), B, H, W, C, static_cast<bf16 *>(dst), ld_big, off,
          backward ? 1 : 0);
    else
      pixel_shuffle2_kernel<1><<<grid1(n, 256), 256, 0, s>>>(
          static_cast<const bf16 *>(src), B, H, W, C, static_cast<bf16 *>(dst), ld_big, off,
          backward ? 1 : 0);
  }
  PE_TRY_LAUNCH("pixel_shuffle2_kernel");
  return PE_OK;
}

extern "C" pe_status pe_nn_copy_channels(const void *src, int64_t lds, int32_t soff, void *dst,
                                         int64_t ldd, int32_t doff, int64_t P, int32_t C,
                                         int32_t accumulate, void *stream) {
  NN_CHECK_STREAM;
  if (!src || !dst || P <= 0 || C <= 0) return pe_fail(PE_EINVAL, "pe_nn_copy_channels: bad arguments");
  const bool v8 = C % 8 == 0 && soff % 8 == 0 && doff % 8 == 0 && lds % 8 == 0 && ldd % 8 == 0 &&
                  (reinterpret_cast<uintptr_t>(src) & 15) == 0 &&
                  (reinterpret_cast<uintptr_t>(dst) & 15) == 0;
  if (v8)
    copy_channels_kernel<8><<<grid1(P * (C / 8), 256), 256, 0, s>>>(
        static_cast<const bf16 *>(src), lds, soff, static_cast<bf16 *>(dst), ldd, doff, P, C,
        accumulate);
  else
    copy_channels_kernel<1><<<grid1(P * C, 256), 256, 0, s>>>(
        static_cast<const bf16 *>(src), lds, soff, static_cast<bf16 *>(dst), ldd, doff, P, C,
        accumulate);
  PE_TRY_LAUNCH("copy_channels_kernel");
  return PE_OK;
}

extern "C" pe_status pe_nn_transpose(const void *src, int32_t R, int32_t Cc, void *dst,
                                     void *stream) {
  NN_CHECK_STREAM;
  if (!src || !dst || R <= 0 || Cc <= 0) return pe_fail(PE_EINVAL, "pe_nn_transpose: bad arguments");
  if ((R + 31) / 32 > 65535) return pe_fail(PE_EINVAL, "pe_nn_transpose: too many rows");
  dim3 grid((unsigned)((Cc + 31) / 32), (unsigned)((R + 31) / 32));
  transpose_kernel<<<grid, dim3(32, 8), 0, s>>>(static_cast<const bf16 *>(src), R, Cc,
                                                static_cast<bf16 *>(dst));
  PE_TRY_LAUNCH("transpose_kernel");
  return PE_OK;
}

extern "C" pe_status pe_nn_to_bf16(const float *x, int64_t n, void *y, void *stream) {
  NN_CHECK_STREAM;
  if (!x || !y || n <= 0) return pe_fail(PE_EINVAL, "pe_nn_to_bf16: bad arguments");
  f32_to_bf16_kernel<<<grid1(n, 256), 256, 0, s>>>(x, n, static_cast<bf16 *>(y));
  PE_TRY_LAUNCH("f32_to_bf16_kernel");
  return PE_OK;
}

extern "C" pe_status pe_nn_adamw(float *p, const float *g, float *m, float *v, void *p_bf16,
                                 int64_t n, float lr, float beta1, float beta2, float eps,
                                 float weight_decay, int32_t step, void *stream) {
  NN_CHECK_STREAM;
  if (!p || !g || !m || !v || n <= 0 || step < 1) return pe_fail(PE_EINVAL, "pe_nn_adamw: bad arguments");
  float bc1 = 1.0f - powf(beta1, (float)step), bc2 = 1.0f - powf(beta2, (float)step);
  adamw_kernel<<<grid1(n, 256), 256, 0, s>>>(p, g, m, v, static_cast<bf16 *>(p_bf16), n, lr, beta1,
                                             beta2, eps, weight_decay, bc1, bc2);
  PE_TRY_LAUNCH("adamw_kernel");
  return PE_OK;
}

static int loss_blocks(int64_t P) { return grid1(P, 256, 4); }

extern "C" size_t pe_nn_unet_losses_workspace(int32_t B, int32_t H, int32_t W) {
  int64_t P = (int64_t)B * H * W;
  return (size_t)(2 * P + 4 * loss_blocks(P) + 8) * sizeof(float) + 1024;
}

// Eq. 17-21: loss[0] = L, loss[1..4] = L1..L4 (device FP32); gradients of L
// with respect to the head outputs (FP32, overwritten).
extern "C" pe_status pe_nn_unet_losses(const float *depth, const float *normal, const float *logit,
                                       const float *d_gt, const float *n_gt, const float *m_gt,
                                       int32_t B, int32_t H, int32_t W, float alpha, float gamma,
                                       const float *lambdas, float *loss, float *g_depth,
                                       float *g_normal, float *g_logit, void *ws, size_t ws_bytes,
                                       void *stream) {
  NN_CHECK_STREAM;
  if (!depth || !normal || !logit || !d_gt || !n_gt || !m_gt || !lambdas || !loss || !g_depth ||
      !g_normal || !g_logit || B <= 0 || H < 3 || W < 3)
    return pe_fail(PE_EINVAL, "pe_nn_unet_losses: bad arguments");
  int64_t P = (int64_t)B * H * W;
  if (!ws || ws_bytes < pe_nn_unet_losses_workspace(B, H, W))
    return pe_fail(PE_ENOMEM, "pe_nn_unet_losses: workspace");
  float *f = static_cast<float *>(ws);
  loss_args a;
  memset(&a, 0, sizeof(a));
  a.d = depth;
  a.n = normal;
  a.z = logit;
  a.d_gt = d_gt;
  a.n_gt = n_gt;
  a.m_gt = m_gt;
  a.B = B;
  a.H = H;
  a.W = W;
  a.alpha = alpha;
  a.gamma = gamma;
  a.w1 = lambdas[0];
  a.w2 = lambdas[1];
  a.w3 = lambdas[2];
  a.w4 = lambdas[3];
  a.g_d = g_depth;
  a.g_n = g_normal;
  a.g_z = g_logit;
  a.c4u = f;
  a.c4v = f + P;
  int blocks = loss_blocks(P);
  a.part = f + 2 * P;
  float *counts = f + 2 * P + 4 * blocks;
  a.counts = counts;
  // two 64-bit counters after the three counts (the offset is a multiple of 8 bytes)
  unsigned long long *cnt = reinterpret_cast<unsigned long long *>(counts + 4);
  PE_TRY_CUDA(cudaMemsetAsync(cnt, 0, 2 * sizeof(unsigned long long), s));
  loss_count_kernel<<<grid1(P, 256), 256, 0, s>>>(a, cnt);
  PE_TRY_LAUNCH("loss_count_kernel");
  loss_count_finish<<<1, 1, 0, s>>>(cnt, P, counts);
  PE_TRY_LAUNCH("loss_count_finish");
  loss_pass1_kernel<<<blocks, 256, 0, s>>>(a);
  PE_TRY_LAUNCH("loss_pass1_kernel");
  loss_pass2_kernel<<<grid1(P, 256), 256, 0, s>>>(a);
  PE_TRY_LAUNCH("loss_pass2_kernel");
  loss_total_kernel<<<1, 32, 0, s>>>(a.part, blocks, a.w1, a.w2, a.w3, a.w4, loss);
  PE_TRY_LAUNCH("loss_total_kernel");
  return PE_OK;
}
