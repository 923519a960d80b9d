// mlp_tc.cu -- the MLP's products on the 5th-generation tensor cores.
//
// Forward and input gradient: out[M x N] = act(A[M x K] . B[N x K]^T + bias),
// BF16 operands, FP32 accumulation in tensor memory (TMEM), N and K in {64,
// 256}; act 1 applies GELU, act 2 multiplies by GELU'(g) of a stored
// pre-activation g (the input gradient through the activation).  Weight
// gradient: a split-K product D[M x N] = A[K x M]^T . B[K x N] with K the
// batch (gemm_tn_splitk_tc below).  Persistent
// CTAs (one per SM): each loads B once into shared memory and then walks
// 128-row tiles of A.  Per tile: one thread issues K/16 tcgen05.mma (128 x N
// x 16) on the A tile in shared memory and commits them to an mbarrier, all
// threads wait on it (bounded), start copying the next A tile into the now
// free buffer (cp.async), and meanwhile each warp reads a 16-column piece
// of its lane group's 32 accumulator rows from TMEM (tcgen05.ld) and applies
// bias, GELU and the BF16/FP32 stores; sixteen warps, four per lane group,
// because the piece loop is a chain of waits (tensor memory, the stored
// pre-activation).  A gradient of 16384 rows of the surrogate network took
// 3154 us with serial column sums, ten transposed copies and four-warp
// epilogues, and takes 189 us (with a fused forward and grouped weight
// gradients).
//
// Shared-memory operand layout: 128-byte swizzle, 1024-byte atoms of eight rows
// of 128 bytes whose 16-byte chunk c of row r sits in place c ^ (r % 8).
// K-major (gemm_tc_kernel): an atom is 8 rows x 64 K; atoms of neighbouring
// row groups are 1024 bytes apart (the descriptor's stride offset), K blocks
// of 64 follow one another.  MN-major (the weight gradient): an atom is 8 K x
// 64 columns; neighbouring K groups are 1024 bytes apart (stride offset), the
// next 64 columns KC * 128 bytes (leading offset).  Lanes then copy along a
// row, 128 to 512 contiguous bytes, and eight of them fill a row of an atom,
// all banks once.  (Unswizzled core matrices want eight rows per eight lanes:
// 16 bytes of each: a gradient of 16384 rows took 228 us, of 65536 rows 549
// us, against 189 and 441.)
#include <cuda_bf16.h>

#include <algorithm>

#include "pg_host.h"

namespace pg {

namespace {

constexpr int TM = 128;
constexpr int kTcThreads = 512;
constexpr int kTcWarps = kTcThreads / 32;
constexpr int kColGroups = kTcWarps / 4;     // warps that share a lane group split the columns
constexpr long long kSpinLimit = 20000000;   // mbarrier polls before giving up

__device__ __forceinline__ uint32_t su32(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// GELU in its tanh form, 0.5 x (1 + tanh(sqrt(2/pi) (x + 0.044715 x^3))),
// written as h + h t with h = x / 2 and the tanh argument x (c0 + c1 x^2);
// hardware tanh approximation.  The same expression as mlp.cu and the fused
// forward (mlp_fused.cu).
__device__ __forceinline__ float gelu_tc(float x) {
  const float p = fmaf(x * x, 0.035677408136300125f, 0.7978845608028654f);
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(x * p));
  const float h = 0.5f * x;
  return fmaf(h, t, h);
}

// Its derivative, as mlp.cu's gelu_grad.
__device__ __forceinline__ float gelu_grad_tc(float x) {
  const float u = 0.7978845608028654f * (x + 0.044715f * x * x * x);
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(u));
  return 0.5f * (1.0f + t) +
         0.5f * x * (1.0f - t * t) * 0.7978845608028654f * (1.0f + 0.134145f * x * x);
}

// 64-bit shared-memory matrix descriptor: start address, leading and stride
// byte offsets (all >> 4), the fixed 0b001 at bits 46-48, 128-byte swizzle (2
// at bits 61-63).
__device__ __forceinline__ uint64_t smem_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);
  d |= (uint64_t)((lbo & 0x3FFFF) >> 4) << 16;
  d |= (uint64_t)((sbo & 0x3FFFF) >> 4) << 32;
  d |= (uint64_t)1 << 46;
  d |= (uint64_t)2 << 61;
  return d;
}

// Byte offset of 16-byte chunk c of row r in a swizzled atom column.
__device__ __forceinline__ uint32_t swizzled(int r, int c) {
  return (uint32_t)((r >> 3) * 1024 + (r & 7) * 128 + (((c & 7) ^ (r & 7)) << 4));
}

// Instruction descriptor, kind::f16: D FP32, A and B BF16, both K-major.
__host__ __device__ constexpr uint32_t instr_desc(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(m >> 4) << 24);
}

// 32 bytes in one store or load (dst, src 32-byte aligned): a lane of these
// kernels has a row's columns to itself, so 16-byte accesses touch every
// 32-byte sector of the row twice.
__device__ __forceinline__ void store32(void *dst, const uint32_t (&w)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"l"(dst), "r"(w[0]),
               "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}
__device__ __forceinline__ void load32(const void *src, uint32_t (&w)[8]) {
  asm volatile("ld.global.v8.b32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];\n"
               : "=r"(w[0]), "=r"(w[1]), "=r"(w[2]), "=r"(w[3]), "=r"(w[4]), "=r"(w[5]),
                 "=r"(w[6]), "=r"(w[7])
               : "l"(src)
               : "memory");
}

// 16 FP32 values rounded to BF16 (nearest even, in pairs), one 32-byte store.
__device__ __forceinline__ void store_bf16x16(__nv_bfloat16 *dst, const float (&v)[16]) {
  uint32_t w[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    w[j] = *reinterpret_cast<const uint32_t *>(&h);
  }
  store32(dst, w);
}

// 16 FP32 values in two 32-byte stores.
__device__ __forceinline__ void store_f32x16(float *dst, const float (&v)[16]) {
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    uint32_t w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) w[j] = __float_as_uint(v[8 * h + j]);
    store32(dst + 8 * h, w);
  }
}

// Sums over the warp's 32 lanes of 16 values per lane: a reduce-scatter of 16
// shuffles (five per value as 16 separate sums would be 80).  Lane l returns
// the sum of column col(l) = 8 b4 + 4 b3 + 2 b2 + b1 (the bits of l); v is
// used up.  Fixed order, so the result does not depend on timing.
__device__ __forceinline__ float warp_column_sums16(float (&v)[16], int lane) {
#pragma unroll
  for (int w = 8, bit = 16; w >= 1; w >>= 1, bit >>= 1) {
    const bool up = (lane & bit) != 0;
#pragma unroll
    for (int j = 0; j < w; ++j) {
      const float keep = up ? v[j + w] : v[j], send = up ? v[j] : v[j + w];
      v[j] = keep + __shfl_xor_sync(0xffffffffu, send, bit);
    }
  }
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}

// copy rows [0, rows) of a K-wide BF16 matrix (row stride ld) into the K-major
// layout; rows in [rows, R) are zero-filled (R a multiple of 8)
template <int K>
__device__ __forceinline__ void load_tile(uint8_t *dst, const __nv_bfloat16 *src, int ld, int rows,
                                          int R) {
  constexpr int KC = K / 8;   // 16-byte chunks per row
  for (int idx = threadIdx.x; idx < R * KC; idx += kTcThreads) {
    const int r = idx / KC, c = idx % KC;
    const uint32_t off = (uint32_t)((c >> 3) * (R * 128)) + swizzled(r, c);
    const bool ok = r < rows;
    const __nv_bfloat16 *s = src + (size_t)(ok ? r : 0) * ld + c * 8;
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(su32(dst + off)),
                 "l"(s), "r"(ok ? 16 : 0));
  }
}

// Poll the mbarrier for the given phase parity at most kSpinLimit times.
__device__ __forceinline__ bool wait_parity_bounded(uint64_t *mbar, uint32_t phase) {
  uint32_t done = 0;
  long long spins = 0;
  while (!done) {
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(su32(mbar)), "r"(phase));
    if (!done && ++spins > kSpinLimit) break;
  }
  return done != 0;
}

template <int N, int K>
__global__ void __launch_bounds__(kTcThreads, 1)
gemm_tc_kernel(const __nv_bfloat16 *__restrict__ A, int lda, const __nv_bfloat16 *__restrict__ B,
               int ldb, int64_t M, const float *__restrict__ bias, int act, float *out_f32,
               __nv_bfloat16 *out_bf16, __nv_bfloat16 *pre_bf16,
               const __nv_bfloat16 *gin, int ldc, float *colpart, int *err) {
  constexpr int NCOLS = N < 32 ? 32 : N;       // TMEM columns (power of two >= 32)
  constexpr uint32_t SB = N * K * 2, SA = TM * K * 2;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint8_t *sB = smem;
  uint8_t *sA = smem + SB;
  uint64_t *mbar = reinterpret_cast<uint64_t *>(smem + SB + SA);
  uint32_t *tslot = reinterpret_cast<uint32_t *>(smem + SB + SA + 8);
  // column sums of the CTA's rows, one row per lane group: [4][N]
  float *sCol = reinterpret_cast<float *>(smem + SB + SA + 16);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int64_t ntiles = (M + TM - 1) / TM;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     su32(tslot)), "r"(NCOLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(su32(mbar)));
    asm volatile("fence.mbarrier_init.release.cluster;\n");
  }
  for (int i = threadIdx.x; i < 4 * N; i += kTcThreads) sCol[i] = 0.f;
  load_tile<K>(sB, B, ldb, N, N);
  asm volatile("cp.async.commit_group;\n");
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n");
  const uint32_t tmem = *tslot;
  const uint32_t idesc = instr_desc(TM, N);
  uint32_t phase = 0;
  bool failed = false;

  // The A tile of the next iteration is copied while this tile's epilogue
  // runs: once the MMA has completed (mbarrier), the shared A buffer is free.
  auto copy_a = [&](int64_t t) {
    const int64_t m = t * TM;
    load_tile<K>(sA, A + (size_t)m * lda, lda, (int)((M - m) < TM ? (M - m) : TM), TM);
    asm volatile("cp.async.commit_group;\n");
  };
  if ((int64_t)blockIdx.x < ntiles) copy_a(blockIdx.x);
  for (int64_t tile = blockIdx.x; tile < ntiles && !failed; tile += gridDim.x) {
    const int64_t m0 = tile * TM;
    asm volatile("cp.async.wait_group 0;\n");
    asm volatile("fence.proxy.async.shared::cta;\n");
    __syncthreads();
    if (threadIdx.x == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;\n");
#pragma unroll
      for (int ks = 0; ks < K / 16; ++ks) {
        // 16 K-columns: 32 bytes along an atom's rows, four to a K block
        const uint64_t da = smem_desc(su32(sA) + (ks >> 2) * (TM * 128) + (ks & 3) * 32, 16, 1024);
        const uint64_t db = smem_desc(su32(sB) + (ks >> 2) * (N * 128) + (ks & 3) * 32, 16, 1024);
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
            "l"(da), "l"(db), "r"(idesc), "r"(ks));
      }
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
              su32(mbar)));
    }
    // wait for the accumulator (bounded).  The CTA decides together whether
    // the wait failed, so every thread leaves the loop at the same point and
    // no aligned tcgen05 instruction or barrier is reached by part of it.
    {
      const bool done = wait_parity_bounded(mbar, phase);
      failed = __syncthreads_or(!done) != 0;
      if (failed) {
        if (threadIdx.x == 0) atomicCAS(err, 0, 1);
        // the MMAs may still be running: give them a second bounded wait
        // before the TMEM is released below, and let the copies in flight land
        wait_parity_bounded(mbar, phase);
        asm volatile("cp.async.wait_group 0;\n");
        __syncthreads();
      }
    }
    phase ^= 1u;
    if (failed) break;
    if (tile + gridDim.x < ntiles) copy_a(tile + gridDim.x);
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    // a warp reaches the 32 accumulator rows of its lane group (warp % 4); the
    // warps of a group take 16-column pieces in turn
    const int lg = warp & 3;
    const int64_t row = m0 + lg * 32 + lane;
#pragma unroll 1
    for (int c0 = (warp >> 2) * 16; c0 < N; c0 += 16 * kColGroups) {
      uint32_t r[16];
      const uint32_t taddr = tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)c0;
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
          "%14,%15}, [%16];\n"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
            "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
            "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
          : "r"(taddr));
      asm volatile("tcgen05.wait::ld.sync.aligned;\n");
      float v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = row < M ? __uint_as_float(r[j]) : 0.f;
      if (row < M) {
        // 16 consecutive columns of this thread's row
        const size_t o = (size_t)row * ldc + c0;
        if (bias) {
#pragma unroll
          for (int j = 0; j < 16; j += 4) {
            const float4 b4 = *reinterpret_cast<const float4 *>(bias + c0 + j);
            v[j] += b4.x; v[j + 1] += b4.y; v[j + 2] += b4.z; v[j + 3] += b4.w;
          }
        }
        if (pre_bf16) store_bf16x16(pre_bf16 + o, v);
        if (act == 1) {
#pragma unroll
          for (int j = 0; j < 16; ++j) v[j] = gelu_tc(v[j]);
        } else if (act == 2) {
          // times GELU'(g): 16 BF16 pre-activations in one load
          uint32_t gw[8];
          load32(gin + o, gw);
#pragma unroll
          for (int j = 0; j < 8; ++j) {
            const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162 *>(&gw[j]);
            v[2 * j] *= gelu_grad_tc(__low2float(h));
            v[2 * j + 1] *= gelu_grad_tc(__high2float(h));
          }
        }
        if (out_f32) store_f32x16(out_f32 + o, v);
        if (out_bf16) store_bf16x16(out_bf16 + o, v);
      }
      if (colpart) {
        const float cs = warp_column_sums16(v, lane);
        const int c = ((lane >> 4) & 1) * 8 + ((lane >> 3) & 1) * 4 + ((lane >> 2) & 1) * 2 +
                      ((lane >> 1) & 1);
        if (!(lane & 1)) sCol[lg * N + c0 + c] += cs;   // this warp's cells alone
      }
    }
    asm volatile("tcgen05.fence::before_thread_sync;\n");
    __syncthreads();
  }
  __syncthreads();
  if (colpart) {
    for (int c = threadIdx.x; c < N; c += kTcThreads)
      colpart[(size_t)blockIdx.x * N + c] =
          (sCol[c] + sCol[N + c]) + (sCol[2 * N + c] + sCol[3 * N + c]);
  }
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"(NCOLS));
  }
}

template <int N, int K>
cudaError_t launch_tc(const __nv_bfloat16 *A, int lda, const __nv_bfloat16 *B, int ldb, int64_t M,
                      const float *bias, int act, float *out_f32, __nv_bfloat16 *out_bf16,
                      __nv_bfloat16 *pre_bf16, const __nv_bfloat16 *gin, int ldc, float *colpart,
                      int *nparts, cudaStream_t st, int *err) {
  constexpr size_t smem = (size_t)N * K * 2 + (size_t)TM * K * 2 + 16 + 4 * (size_t)N * 4;
  // the attribute belongs to the current device's context: set it on every
  // launch (cheap), so a first launch on another device is configured too
  cudaError_t e = cudaFuncSetAttribute(gemm_tc_kernel<N, K>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  const int64_t ntiles = (M + TM - 1) / TM;
  const int grid = (int)(ntiles < sms ? ntiles : sms);
  gemm_tc_kernel<N, K><<<grid, kTcThreads, smem, st>>>(
      A, lda, B, ldb, M, bias, act, out_f32, out_bf16, pre_bf16, gin, ldc, colpart, err);
  if (nparts) *nparts = grid;
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace

// CTAs of a gemm_nt_tc launch at most: the rows of its column-sum partials.
int gemm_tc_max_ctas() {
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  return sms;
}

// Products of the MLP on tcgen05; N and K must be 64 or 256, all row
// strides multiples of 8 elements (ldc of 16), bias 16-byte and outputs 32-byte
// aligned.
// out_bf16 may be gin: an element is read before it is written, by the same
// thread.  colpart (may be null): column sums of the result over each CTA's rows,
// [*nparts][N] FP32, from the values before they are rounded to BF16.  *err
// (device) is set to 1 if a CTA gave up waiting for its accumulator.
cudaError_t gemm_nt_tc(const __nv_bfloat16 *A, int lda, const __nv_bfloat16 *B, int ldb,
                       int64_t M, int N, int K, const float *bias, int act, float *out_f32,
                       __nv_bfloat16 *out_bf16, __nv_bfloat16 *pre_bf16, int ldc, cudaStream_t st,
                       int *err, const __nv_bfloat16 *gin, float *colpart, int *nparts) {
  if (M == 0) return cudaSuccess;
  if (lda % 8 || ldb % 8 || ldc % 16 || !err || (act == 2 && !gin)) return cudaErrorInvalidValue;
  if ((uintptr_t)bias % 16 || ((uintptr_t)out_f32 | (uintptr_t)out_bf16 | (uintptr_t)pre_bf16 |
                               (uintptr_t)gin) % 32)
    return cudaErrorInvalidValue;
  if (N == 256 && K == 256)
    return launch_tc<256, 256>(A, lda, B, ldb, M, bias, act, out_f32, out_bf16, pre_bf16, gin, ldc, colpart, nparts, st, err);
  if (N == 256 && K == 64)
    return launch_tc<256, 64>(A, lda, B, ldb, M, bias, act, out_f32, out_bf16, pre_bf16, gin, ldc, colpart, nparts, st, err);
  if (N == 64 && K == 256)
    return launch_tc<64, 256>(A, lda, B, ldb, M, bias, act, out_f32, out_bf16, pre_bf16, gin, ldc, colpart, nparts, st, err);
  if (N == 64 && K == 64)
    return launch_tc<64, 64>(A, lda, B, ldb, M, bias, act, out_f32, out_bf16, pre_bf16, gin, ldc, colpart, nparts, st, err);
  return cudaErrorNotSupported;
}

// ------------------------------------------------------ split-K product ---
namespace {

constexpr int KC = 64;           // K elements (batch rows) per pipeline chunk

// Instruction descriptor with both operands MN-major (bits 15 and 16): the
// batch is the contraction and memory holds a batch row's columns side by
// side, so the operands come from the row-major matrices as they are, with no
// transposed copies.
__host__ __device__ constexpr uint32_t instr_desc_mn(int m, int n) {
  return instr_desc(m, n) | (1u << 15) | (1u << 16);
}

// copy batch rows [k0, k0 + KC) of columns [0, cols) of a BF16 matrix (row
// stride ld, K valid rows, CC chunks of 8 columns) into the MN-major layout;
// columns >= cols and rows >= K are zero-filled
template <int CC>
__device__ __forceinline__ void load_chunk_mn(uint8_t *dst, const __nv_bfloat16 *src, int64_t ld,
                                              int cols, int64_t k0, int64_t K) {
  for (int idx = threadIdx.x; idx < KC * CC; idx += kTcThreads) {
    const int c = idx % CC, k = idx / CC;
    const uint32_t off = (uint32_t)((c >> 3) * (KC * 128)) + swizzled(k, c);
    const int64_t m = k0 + k;
    const bool ok = m < K && c * 8 < cols;
    const __nv_bfloat16 *s = src + (ok ? (size_t)m * ld + (size_t)c * 8 : 0);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(su32(dst + off)),
                 "l"(s), "r"(ok ? 16 : 0));
  }
}

// The weight gradients of one or more layers in one launch.  Group g (a layer)
// has mtiles * splits CTAs from CTA `first`; CTA (m-tile mt, split s) forms D_s
// = A[K slice, mt columns]^T . B[K slice, :] in TMEM over chunks [c0, c1)
// through a ring of kStages buffers, then the FP32 partial [128 x N] to
// part[s][mt * 128 + row][col].  All layers together, because one layer's
// products fill the chip only when they are cut into 64 splits whose partials
// cost as much again to write and sum (16384 rows: five launches and five sums
// 88 us, one of each 25).
constexpr int kStages = 4;
constexpr int kMaxGroups = 20;
struct SplitGroup {
  const __nv_bfloat16 *A, *B;
  int64_t lda, ldb;
  int Mrows, N, mtiles, first;
  float *part, *out;
  const float *bpart;
  int nparts, rblock;          // rblock: first block of its sums
  float *bout;
};
struct SplitGroups {
  SplitGroup g[kMaxGroups];
  int n, cps, splits;
  int64_t K;
  int *err;
};

__global__ void __launch_bounds__(kTcThreads, 1)
gemm_splitk_tc_kernel(const __grid_constant__ SplitGroups args) {
  constexpr int NCOLS = 256;
  constexpr uint32_t SA = TM * KC * 2, SB = NCOLS * KC * 2;
  extern __shared__ __align__(1024) uint8_t smem[];
  // stage st: A at smem + st * (SA + SB), B behind it
  auto sA = [&](int st) { return smem + st * (SA + SB); };
  auto sB = [&](int st) { return smem + st * (SA + SB) + SA; };
  uint64_t *mbar = reinterpret_cast<uint64_t *>(smem + kStages * (SA + SB));
  uint32_t *tslot = reinterpret_cast<uint32_t *>(smem + kStages * (SA + SB) + kStages * 8);
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  int gi = 0;
  while (gi + 1 < args.n && (int)blockIdx.x >= args.g[gi + 1].first) ++gi;
  const SplitGroup &G = args.g[gi];
  const int N = G.N, local = (int)blockIdx.x - G.first;
  const int mt = local % G.mtiles, sp = local / G.mtiles, mtiles = G.mtiles;
  const int64_t K = args.K, nchunks = (K + KC - 1) / KC;
  const int64_t c0 = (int64_t)sp * args.cps;
  const int64_t c1 = c0 + args.cps < nchunks ? c0 + args.cps : nchunks;
  const int rows = G.Mrows - mt * TM < TM ? G.Mrows - mt * TM : TM;
  const __nv_bfloat16 *Am = G.A + (size_t)mt * TM;
  int *err = args.err;

  // one copy group per chunk, empty past the last one, so that group counts
  // and chunks agree
  auto copy_chunk = [&](int64_t c) {
    if (c < c1) {
      const int st = (int)((c - c0) % kStages);
      load_chunk_mn<TM / 8>(sA(st), Am, G.lda, rows, c * KC, K);
      if (N == 256) load_chunk_mn<32>(sB(st), G.B, G.ldb, N, c * KC, K);
      else load_chunk_mn<8>(sB(st), G.B, G.ldb, N, c * KC, K);
    }
    asm volatile("cp.async.commit_group;\n");
  };
  for (int q = 0; q < kStages - 1; ++q) copy_chunk(c0 + q);
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     su32(tslot)), "r"(NCOLS));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (threadIdx.x == 0) {
    for (int q = 0; q < kStages; ++q)
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(su32(&mbar[q])));
    asm volatile("fence.mbarrier_init.release.cluster;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n");
  const uint32_t tmem = *tslot;
  const uint32_t idesc = instr_desc_mn(TM, N);
  bool failed = false;
  int last_stage = -1;
  uint32_t last_phase = 0u;

  for (int64_t c = c0; c < c1; ++c) {
    const int64_t i = c - c0;
    const int st = (int)(i % kStages);
    if (c > c0) {
      // the stage of chunk c + kStages - 1 held chunk c - 1, whose products
      // must be done (its commit: use (i - 1) / kStages of that stage)
      const bool ok = c + kStages - 1 >= c1 || wait_parity_bounded(&mbar[last_stage], last_phase);
      failed = __syncthreads_or(!ok) != 0;
      if (failed) break;       // the wait below retries this phase
    }
    copy_chunk(c + kStages - 1);
    asm volatile("cp.async.wait_group %0;\n" ::"n"(kStages - 1));   // chunk c has landed
    asm volatile("fence.proxy.async.shared::cta;\n");
    __syncthreads();
    if (threadIdx.x == 0) {
      asm volatile("tcgen05.fence::after_thread_sync;\n");
#pragma unroll
      for (int ks = 0; ks < KC / 16; ++ks) {
        // 16 batch rows: two K groups of an atom column
        const uint64_t da = smem_desc(su32(sA(st)) + ks * 2048, KC * 128, 1024);
        const uint64_t db = smem_desc(su32(sB(st)) + ks * 2048, KC * 128, 1024);
        const uint32_t accum = (c > c0 || ks > 0) ? 1u : 0u;
        asm volatile(
            "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
            " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
            "l"(da), "l"(db), "r"(idesc), "r"(accum));
      }
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
              su32(&mbar[st])));
    }
    last_stage = st;
    last_phase = (uint32_t)((i / kStages) & 1);
  }
  if (!failed && last_stage >= 0) {
    // the last commit covers every product issued before it
    const bool ok = wait_parity_bounded(&mbar[last_stage], last_phase);
    failed = __syncthreads_or(!ok) != 0;
  }
  if (failed) {
    if (threadIdx.x == 0) atomicCAS(err, 0, 1);
    // give products still in flight a second bounded wait before the TMEM
    // is released, and let the copies land
    if (last_stage >= 0) wait_parity_bounded(&mbar[last_stage], last_phase);
    asm volatile("cp.async.wait_group 0;\n");
  } else if (last_stage >= 0) {
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    const int lg = warp & 3;
    float *out = G.part + ((size_t)sp * mtiles * TM + (size_t)mt * TM + lg * 32 + lane) * N;
#pragma unroll 1
    for (int cc = (warp >> 2) * 16; cc < N; cc += 16 * kColGroups) {
      uint32_t r[16];
      const uint32_t taddr = tmem + ((uint32_t)(lg * 32) << 16) + (uint32_t)cc;
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,"
          "%14,%15}, [%16];\n"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
            "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
            "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
          : "r"(taddr));
      asm volatile("tcgen05.wait::ld.sync.aligned;\n");
      float v[16];
#pragma unroll
      for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
      store_f32x16(out + cc, v);
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"(NCOLS));
  }
}

// Of each group: out[q] = sum over splits s of part[s][q], and, for the
// layer's bias gradient, bout[c] = sum over p of bpart[p][c].  A block takes 64
// outputs side by side; its four groups of 64 threads each sum a quarter of
// the partials in order, and the quarters are added in order (fixed order, so
// the result does not depend on timing).  Four quarters instead of one chain:
// the loads of up to 152 partials are the time here.
constexpr int kRedOut = 64;
__global__ void __launch_bounds__(256) splitk_reduce_kernel(const __grid_constant__ SplitGroups args) {
  __shared__ float sh[4][kRedOut];
  int gi = 0;
  while (gi + 1 < args.n && (int)blockIdx.x >= args.g[gi + 1].rblock) ++gi;
  const SplitGroup &G = args.g[gi];
  const int lane = threadIdx.x & (kRedOut - 1), quarter = threadIdx.x / kRedOut;
  const int blk = (int)blockIdx.x - G.rblock, wblocks = G.Mrows * G.N / kRedOut;
  const bool bias = blk >= wblocks;
  const float *src = bias ? G.bpart : G.part;
  const int q = (bias ? blk - wblocks : blk) * kRedOut + lane;
  const int n = bias ? G.nparts : args.splits;
  const size_t step = bias ? (size_t)G.Mrows : (size_t)G.mtiles * TM * G.N;
  const int per = (n + 3) / 4, s1 = min(n, (quarter + 1) * per);
  float acc = 0.f;
#pragma unroll 8
  for (int s = quarter * per; s < s1; ++s) acc += src[(size_t)s * step + q];
  sh[quarter][lane] = acc;
  __syncthreads();
  if (quarter == 0) {
    const float v = (sh[0][lane] + sh[1][lane]) + (sh[2][lane] + sh[3][lane]);
    if (bias) G.bout[q] = v;
    else G.out[q] = v;
  }
}

}  // namespace

// Weight and bias gradients of `ng` layers on tcgen05, one launch and one of
// sums: for each, out[Mrows x N] (FP32, row-major) = A^T B with A [K x Mrows]
// and B [K x N] BF16 row-major (row strides lda, ldb, multiples of 8), K (the
// batch) any number of rows, N 64 or 256, Mrows 64 or 256; bout[Mrows] = the
// sum of the nparts rows of bpart (column-sum partials of A's FP32 values).
// The K range is split over CTAs; each writes an FP32 partial to `scratch`
// and a fixed-order sum reduces them (deterministic).  The operands are read
// MN-major, so the batch needs no transposed copies (16384 rows: ten
// transposes were 100 us of a pass).  *err (device) is set to 1 if a CTA gave
// up waiting for its products.
cudaError_t gemm_tn_splitk_tc(const WeightGrad *w, int ng, int64_t K, float *scratch,
                              size_t scratch_bytes, cudaStream_t st, int *err) {
  if (K == 0 || ng == 0) return cudaSuccess;
  if (ng < 0 || ng > kMaxGroups || !err || ((uintptr_t)scratch % 32)) return cudaErrorInvalidValue;
  SplitGroups a;
  a.n = ng; a.K = K; a.err = err;
  int mtiles = 0, rblocks = 0;
  size_t per_split = 0;
  for (int i = 0; i < ng; ++i) {
    if (w[i].lda % 8 || w[i].ldb % 8 || (w[i].Mrows != 64 && w[i].Mrows != 256) ||
        (w[i].N != 64 && w[i].N != 256) || !w[i].bpart || !w[i].bout ||
        (((uintptr_t)w[i].A | (uintptr_t)w[i].B) % 16))
      return cudaErrorInvalidValue;
    SplitGroup &g = a.g[i];
    g.A = w[i].A; g.B = w[i].B; g.lda = w[i].lda; g.ldb = w[i].ldb;
    g.Mrows = w[i].Mrows; g.N = w[i].N;
    g.mtiles = (w[i].Mrows + TM - 1) / TM;
    g.out = w[i].out; g.bpart = w[i].bpart; g.nparts = w[i].nparts; g.bout = w[i].bout;
    g.rblock = rblocks;
    rblocks += (g.Mrows * g.N + g.Mrows) / kRedOut;
    mtiles += g.mtiles;
    per_split += (size_t)g.mtiles * TM * g.N;
  }
  constexpr size_t smem = kStages * ((size_t)TM * KC * 2 + (size_t)256 * KC * 2 + 8) + 16;
  cudaError_t e = cudaFuncSetAttribute(gemm_splitk_tc_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  // as many splits as give every multiprocessor a CTA
  const int64_t nchunks = (K + KC - 1) / KC;
  int64_t want = std::max<int64_t>(1, std::min<int64_t>(nchunks, (int64_t)sms / mtiles));
  want = std::min<int64_t>(want, (int64_t)(scratch_bytes / (per_split * sizeof(float))));
  if (want < 1) return cudaErrorInvalidValue;
  a.cps = (int)((nchunks + want - 1) / want);
  a.splits = (int)((nchunks + a.cps - 1) / a.cps);
  int first = 0;
  float *part = scratch;
  for (int i = 0; i < ng; ++i) {
    a.g[i].first = first;
    a.g[i].part = part;
    first += a.splits * a.g[i].mtiles;
    part += (size_t)a.splits * a.g[i].mtiles * TM * a.g[i].N;
  }
  gemm_splitk_tc_kernel<<<first, kTcThreads, smem, st>>>(a);
  splitk_reduce_kernel<<<rblocks, 256, 0, st>>>(a);
  note_launches(2);
  return cudaGetLastError();
}

}  // namespace pg
