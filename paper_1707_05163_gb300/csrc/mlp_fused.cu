// mlp_fused.cu -- the surrogate network's inference forward in one kernel on
// the 5th-generation tensor cores, activations kept on chip; and, in a
// second instance of the same kernel, a whole network step of the learned
// flow map (features gathered from the field, the network, the displacement
// applied to the particles), and, in a third, the forward pass of a training
// batch.
//
// Network: 64 (padded input) -> 256 -> 256 -> 256 -> 256 -> n_out (<= 16;
// the weights are padded to 64 outputs), GELU after the hidden layers (the
// shapes of the flow-map surrogate).  One persistent CTA per SM walks
// 128-row tiles, two at a time, with four kinds of warps:
//
//   * input warps put a tile's input where its activations will be (the last
//     layer of the tile before has read them): two convert FP32 feature rows
//     into BF16 in the operand layout of shared memory (zero-padded to 64
//     columns), the rows read ahead into registers; in the network step one
//     lane copies the tile the feature kernel packed (16 KB, one bulk copy);
//   * a copy warp streams, for every tile, fourteen weight pieces of up to
//     32 KB -- layer 0; layers 1-3 as four pieces of 64 K-columns each; the 16
//     rows of layer 4 -- into a ring of three slots, each copy completing on
//     the slot's "full" mbarrier;
//   * an MMA warp issues the tcgen05 products (128 x 256 x 16) into one of two
//     128 x 256 FP32 accumulators in tensor memory (512 columns) and commits
//     "accumulator ready", "slot free" and "input free" mbarriers;
//   * sixteen epilogue warps read an accumulator back (tcgen05.ld; a warp
//     reaches the 32 lanes -- rows -- of its lane group, four warps per group
//     share the columns), add the bias, apply GELU (two values per
//     instruction) and write BF16 activations into shared memory in the
//     operand layout of the next product; the last layer's 16 columns (plus
//     bias) go to global memory in FP32, or, in the network step, move the
//     particles (surrogate_apply).
//
// The epilogue stores 2 GELU(x) = x (1 + t), one multiply per element fewer
// than GELU(x) = h + h t with h = x / 2, and the packed weights of layers 1-4
// are halved; both scalings are by powers of two and exact in BF16 (for
// normal numbers), so every product and sum is the one of GELU(x) and W, bit
// for bit.
//
// What bounds it, and why two tiles: a layer is 2048 clocks of products and
// about as many of epilogue (tanh, issue), and within one tile they can only
// alternate -- the products need all activations, the epilogue all products
// -- plus the latency of every hand-over: 24.8k clocks per tile with one tile
// in flight (1M rows 617 us, tensor pipe 30 %).  With two, each with eight
// epilogue warps, one's products run while the other is read back: 16.5k
// clocks per tile, 1M rows in 445 us; what is left is the epilogue's latency
// of each layer, about 4k clocks of a tile.  Each tile has its own accumulator and its own
// 128 x 256 BF16 activation buffer; a CTA left with one tile alternates the
// accumulators instead.  The first two of a layer's four K-pieces need only the
// first half of the activations: of a tile alone they start when that is
// written; of a pair, whose accumulator they overwrite, once it has been read,
// with each warp's last 32 columns still to be written.
// An activation half is overwritten only after every product that reads it
// has completed (the commit that makes an accumulator ready covers all
// earlier products).
//
// Every wait is bounded; a warp that gives up raises a CTA-wide flag that
// the others poll, so all leave their loops; then the MMA warp waits
// (bounded) for its products in flight and the copy warp for its copies
// before the tensor memory is released, and *err is set.
//
// Shared-memory operand layout (K-major, no swizzle): 8-row x 16-byte core
// matrices; for a matrix KC 16-byte chunks wide, core (row group g, chunk c)
// sits at byte (g * KC + c) * 128 (descriptor: leading offset 128 bytes,
// stride offset KC * 128 bytes).
#include <cuda_bf16.h>

#include <algorithm>

#include "pg_host.h"
#include "surrogate_features.cuh"

namespace pg {

namespace {

constexpr int TMF = 128;                       // rows per tile
constexpr int kEpiWarps = 16;                  // epilogue warps (a multiple of 4)
constexpr int kCopyWarp = kEpiWarps;
constexpr int kMmaWarp = kEpiWarps + 1;
constexpr int kInWarp0 = kEpiWarps + 2;        // input warps follow the copy and MMA warps
constexpr int kInWarps = 2;
constexpr int kFThreads = 32 * (kEpiWarps + 2 + kInWarps);
static_assert(kEpiWarps == 16, "two groups of eight: four lane groups x two column groups");
constexpr long long kFSpin = 4000000;          // mbarrier polls before giving up
constexpr uint32_t kSuspendNs = 500;           // suspend-time hint of a poll
constexpr int kPieces = 14;                    // weight pieces per tile
constexpr uint32_t kPieceBytes = 32768;
constexpr uint32_t kLastBytes = 8192;          // the output layer's 16 rows
constexpr int kSlots = 3;
constexpr uint32_t kTileXBytes = 16384;        // 128 x 64 BF16 input tile
constexpr uint32_t kTileHBytes = 65536;        // 128 x 256 BF16 activations
constexpr float kGeluC0 = 0.7978845608028654f;     // sqrt(2 / pi)
constexpr float kGeluC1 = 0.035677408136300125f;   // sqrt(2 / pi) * 0.044715

// shared memory map (bytes)
constexpr uint32_t kOffH = 0;                              // two activation buffers
constexpr uint32_t kOffW = kOffH + 2 * kTileHBytes;        // weight ring
constexpr uint32_t kOffBar = kOffW + kSlots * kPieceBytes;
// mbarriers
constexpr int B_WFULL = 0;                  // [kSlots] weight slot landed
constexpr int B_WFREE = B_WFULL + kSlots;   // [kSlots] weight slot's products done
constexpr int B_XFULL = B_WFREE + kSlots;   // [tile] input landed
constexpr int B_XFREE = B_XFULL + 2;        // [tile] last layer's products done
constexpr int B_ACCFULL = B_XFREE + 2;      // [accumulator] products done
constexpr int B_ACCFREE = B_ACCFULL + 2;    // [accumulator] read back
constexpr int B_HFULL = B_ACCFREE + 2;      // [tile * 2 + half] activations written
constexpr int B_DRAIN = B_HFULL + 4;        // products in flight (failure path)
constexpr int kNumBars = B_DRAIN + 1;
constexpr uint32_t kOffMisc = kOffBar + kNumBars * 8;      // TMEM address, failure flag
constexpr uint32_t kSmem = kOffMisc + 16;
static_assert(kOffBar % 8 == 0, "mbarrier alignment");
static_assert(kSmem <= 232448, "shared memory per CTA");

__device__ __forceinline__ uint32_t su32f(const void *p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

__device__ __forceinline__ uint64_t desc_f(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  uint64_t d = 0;
  d |= (uint64_t)((addr & 0x3FFFF) >> 4);
  d |= (uint64_t)((lbo & 0x3FFFF) >> 4) << 16;
  d |= (uint64_t)((sbo & 0x3FFFF) >> 4) << 32;
  d |= (uint64_t)1 << 46;
  return d;
}

// kind::f16 instruction descriptor: FP32 accumulator, BF16 A and B, both
// K-major, N >> 3 at bit 17, M >> 4 at bit 24.
__host__ __device__ constexpr uint32_t idesc_f(int m, int n) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(n >> 3) << 17) |
         ((uint32_t)(m >> 4) << 24);
}

__device__ __forceinline__ float tanh_f(float x) {
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(x));
  return t;
}

// Twice GELU in its tanh form of two values, x (1 + tanh(sqrt(2/pi) (x +
// 0.044715 x^3))), as x + x t with the tanh argument x (c0 + c1 x^2); hardware
// tanh approximation.  Packed FP32 operations round each value as the scalar
// ones do, at half the instructions.  The layer-by-layer kernels (mlp_tc.cu,
// mlp.cu) form h + h t with h = x / 2 from the same t: exactly half of this
// value.
__device__ __forceinline__ float2 gelu2_f(float2 x) {
  const float2 p = __ffma2_rn(__fmul2_rn(x, x), make_float2(kGeluC1, kGeluC1),
                              make_float2(kGeluC0, kGeluC0));
  const float2 u = __fmul2_rn(x, p);
  return __ffma2_rn(x, make_float2(tanh_f(u.x), tanh_f(u.y)), x);
}

// Poll phase `parity` of an mbarrier: true once it has completed; false
// after `limit` polls, or (fail != nullptr) once *fail is set.  Each poll may
// suspend the thread for up to kSuspendNs until the phase completes, so a
// waiting warp takes few issue slots from the working ones.
__device__ __forceinline__ bool wait_bar(uint32_t bar, uint32_t parity, const volatile int *fail,
                                         long long limit = kFSpin) {
  for (long long spins = 0; spins < limit; ++spins) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n"
        " selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity), "r"(kSuspendNs)
        : "memory");
    if (done) return true;
    if (fail && (spins & 31) == 31 && *fail) return false;
  }
  return false;
}

__device__ __forceinline__ void bar_arrive(uint32_t bar, uint32_t count = 1) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}

// One lane of a converged warp.
__device__ __forceinline__ bool elect_one() {
  uint32_t p;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.u32 %0, 1, 0, p;\n}\n" : "=r"(p));
  return p != 0;
}

// wait_bar by a whole warp: the same answer in every lane.
__device__ __forceinline__ bool warp_wait(uint32_t bar, uint32_t parity, const volatile int *fail) {
  return __all_sync(0xffffffffu, wait_bar(bar, parity, fail));
}

__device__ __forceinline__ void bar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes)
               : "memory");
}

__device__ __forceinline__ void bulk_copy(uint32_t dst, const void *src, uint32_t bytes,
                                          uint32_t bar) {
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(
          dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void mma(uint32_t tacc, uint64_t da, uint64_t db, uint32_t idesc,
                                    uint32_t accumulate) {
  asm volatile(
      "{\n .reg .pred p;\n setp.ne.b32 p, %4, 0;\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tacc),
      "l"(da), "l"(db), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ void commit(uint32_t bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar)
      : "memory");
}

__device__ __forceinline__ void tmem_ld32(uint32_t taddr, uint32_t (&v)[32]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,%30,%31}, [%32];\n"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15]), "=r"(v[16]), "=r"(v[17]), "=r"(v[18]), "=r"(v[19]),
        "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]), "=r"(v[25]),
        "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(taddr));
}

// Wait for this thread's tensor-memory loads; the loaded registers pass
// through, so nothing that uses them can move ahead of the wait.
__device__ __forceinline__ void tmem_wait32(uint32_t (&v)[32]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;\n"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]),
                 "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]), "+r"(v[10]), "+r"(v[11]),
                 "+r"(v[12]), "+r"(v[13]), "+r"(v[14]), "+r"(v[15]), "+r"(v[16]), "+r"(v[17]),
                 "+r"(v[18]), "+r"(v[19]), "+r"(v[20]), "+r"(v[21]), "+r"(v[22]), "+r"(v[23]),
                 "+r"(v[24]), "+r"(v[25]), "+r"(v[26]), "+r"(v[27]), "+r"(v[28]), "+r"(v[29]),
                 "+r"(v[30]), "+r"(v[31])
               :
               : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, uint32_t (&v)[16]) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,"
      "%15}, [%16];\n"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]),
        "=r"(v[7]), "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]),
        "=r"(v[14]), "=r"(v[15])
      : "r"(taddr));
}

// Piece p of a tile: its layer, first K element, K length and N.
struct Piece {
  int layer, k0, kl, n;
};
__host__ __device__ __forceinline__ Piece piece_of(int p) {
  Piece q;
  if (p < 13) {
    q.layer = (p + 3) / 4; q.k0 = p == 0 ? 0 : ((p - 1) % 4) * 64; q.kl = 64; q.n = 256;
  } else {
    q.layer = 4; q.k0 = 0; q.kl = 256; q.n = 16;
  }
  return q;
}
__device__ __forceinline__ int layer_pieces(int L) { return L == 0 || L == 4 ? 1 : 4; }
__device__ __forceinline__ int layer_first(int L) { return L == 0 ? 0 : 1 + (L - 1) * 4; }

struct FusedArgs {
  const float *x;               // [M x n_in] FP32 features, row-major (inference)
  int n_in;                     // <= 64
  SurrogateStepIO io;           // the particles (network step)
  const uint8_t *xpk;           // [tiles x 16 KB] packed input tiles (network step)
  const uint8_t *wpk;           // packed weight pieces, 32 KB apart
  const float *bias[5];         // per layer, N floats
  float *y;                     // [M x n_out] FP32
  int64_t M;
  int n_out;
  int *err;
  // training: [M x 256] BF16 per hidden layer, before and after GELU
  __nv_bfloat16 *pre[4], *act[4];
};

// What an instance of the kernel does: inference, a network step of the flow
// map, or the forward pass of a training batch (inference that also keeps the
// hidden layers' values for the backward pass).
enum : int { FUSED_FORWARD = 0, FUSED_STEP = 1, FUSED_TRAIN = 2 };

__device__ __forceinline__ void store_row32(void *dst, const uint32_t (&w)[8]) {
  asm volatile("st.global.v8.b32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};\n" ::"l"(dst), "r"(w[0]),
               "r"(w[1]), "r"(w[2]), "r"(w[3]), "r"(w[4]), "r"(w[5]), "r"(w[6]), "r"(w[7])
               : "memory");
}

// Row m of the FP32 features as 64 BF16 columns, zero beyond n_in and for
// m >= M.  The loads of a half row are issued together, so one lane keeps 32
// in flight.
__device__ __forceinline__ void load_input_row(const FusedArgs &a, int64_t m, uint32_t (&w)[32]) {
  const bool in = m < a.M;
  const float *src = a.x + (in ? m * a.n_in : 0);
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    float f[32];
#pragma unroll
    for (int j = 0; j < 32; ++j) {
      const int col = h * 32 + j;
      f[j] = (in && col < a.n_in) ? __ldg(src + col) : 0.f;
    }
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const __nv_bfloat162 b = __floats2bfloat162_rn(f[2 * j], f[2 * j + 1]);
      w[h * 16 + j] = *reinterpret_cast<const uint32_t *>(&b);
    }
  }
}

// A row of 64 BF16 columns into row r of an input tile in the operand layout:
// core (r / 8, chunk) at ((r / 8) * 8 + chunk) * 128 + (r % 8) * 16.
__device__ __forceinline__ void store_input_row(uint8_t *dst, int r, const uint32_t (&w)[32]) {
  uint8_t *row = dst + (r >> 3) * 1024 + (r & 7) * 16;
#pragma unroll
  for (int c = 0; c < 8; ++c)
    *reinterpret_cast<uint4 *>(row + c * 128) =
        make_uint4(w[4 * c], w[4 * c + 1], w[4 * c + 2], w[4 * c + 3]);
}

// Network step: the features of every particle (zero for a deleted one and in
// the rows that fill the last tile), packed into 16 KB input tiles.  A kernel
// of its own, with the whole SM's threads to hide the chain of searches and
// the 64 scattered loads of a particle: gathered by four warps of the network
// kernel they took 46k clocks per 128-row tile, four times the network's.
__global__ void __launch_bounds__(128) pack_features_kernel(const __grid_constant__ SurrogateStepIO io,
                                                            int64_t rows, uint8_t *out) {
  // Particles of a set mostly share their time, and its interval costs some
  // fifty FP64 instructions of 16 clocks of the multiprocessor each: the first
  // warp finds that of the block's first particle for all that share it.
  __shared__ SurInterval first;
  const int64_t m0 = (int64_t)blockIdx.x * blockDim.x, m = m0 + threadIdx.x;
  const double t0 = m0 < io.n ? io.time[m0] : 0.0;
  if (threadIdx.x < 32) {
    const SurInterval v = surrogate_interval(io.f, t0);
    if (threadIdx.x == 0) first = v;
  }
  __syncthreads();
  if (m >= rows) return;
  float o[kSurFeat];
  bool ok = false;
  if (m < io.n && io.status[m] == 0) {
    const double t = io.time[m];
    const SurInterval iv = __double_as_longlong(t) == __double_as_longlong(t0)
                               ? first : surrogate_interval(io.f, t);
    const int e = surrogate_features(io.g, io.f, io.lon[m], io.lat[m], io.dep[m], iv, o);
    if (e) atomicCAS(io.ferr, 0, e);
    else ok = true;
  }
  uint32_t w[32];
#pragma unroll
  for (int j = 0; j < 32; ++j) {
    const int q = 2 * j;
    const float f0 = (ok && q < kSurFeat) ? o[q < kSurFeat ? q : 0] : 0.f;
    const float f1 = (ok && q + 1 < kSurFeat) ? o[q + 1 < kSurFeat ? q + 1 : 0] : 0.f;
    const __nv_bfloat162 h = __floats2bfloat162_rn(f0, f1);
    w[j] = *reinterpret_cast<const uint32_t *>(&h);
  }
  store_input_row(out + (m / TMF) * kTileXBytes, (int)(m % TMF), w);
}

// Bias, GELU and BF16 for 32 columns of a row: v (accumulator values) into
// four 16-byte chunks of the operand layout; KEEP: and the values before and
// after GELU to pre and act (32 columns of the row in global memory, null for
// a row beyond the batch).
template <bool KEEP>
__device__ __forceinline__ void gelu_store32(const uint32_t (&v)[32], const float *bias, uint8_t *dst,
                                             __nv_bfloat16 *pre, __nv_bfloat16 *act) {
  if constexpr (!KEEP) {
#pragma unroll
    for (int cc = 0; cc < 32; cc += 8) {
      const float4 b0 = __ldg(reinterpret_cast<const float4 *>(bias + cc));
      const float4 b1 = __ldg(reinterpret_cast<const float4 *>(bias + cc + 4));
      const float2 bb[4] = {make_float2(b0.x, b0.y), make_float2(b0.z, b0.w),
                            make_float2(b1.x, b1.y), make_float2(b1.z, b1.w)};
      uint32_t w[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float2 x = __fadd2_rn(make_float2(__uint_as_float(v[cc + 2 * j]),
                                                __uint_as_float(v[cc + 2 * j + 1])), bb[j]);
        const __nv_bfloat162 hv = __float22bfloat162_rn(gelu2_f(x));
        w[j] = *reinterpret_cast<const uint32_t *>(&hv);
      }
      *reinterpret_cast<uint4 *>(dst + (cc >> 3) * 128) = make_uint4(w[0], w[1], w[2], w[3]);
    }
    return;
  }
#pragma unroll
  for (int c16 = 0; c16 < 32; c16 += 16) {
    uint32_t pw[8], w[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int cc = c16 + 2 * j;
      const float4 b4 = __ldg(reinterpret_cast<const float4 *>(bias + (cc & ~3)));
      const float2 x = __fadd2_rn(make_float2(__uint_as_float(v[cc]), __uint_as_float(v[cc + 1])),
                                  (cc & 2) ? make_float2(b4.z, b4.w) : make_float2(b4.x, b4.y));
      const __nv_bfloat162 xv = __float22bfloat162_rn(x);
      pw[j] = *reinterpret_cast<const uint32_t *>(&xv);
      const __nv_bfloat162 hv = __float22bfloat162_rn(gelu2_f(x));
      w[j] = *reinterpret_cast<const uint32_t *>(&hv);
    }
    *reinterpret_cast<uint4 *>(dst + (c16 >> 3) * 128) = make_uint4(w[0], w[1], w[2], w[3]);
    *reinterpret_cast<uint4 *>(dst + ((c16 >> 3) + 1) * 128) = make_uint4(w[4], w[5], w[6], w[7]);
    if (pre) {
      store_row32(pre + c16, pw);
      // kept as GELU, not twice it
      const __nv_bfloat162 half = __floats2bfloat162_rn(0.5f, 0.5f);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const __nv_bfloat162 h = __hmul2(*reinterpret_cast<const __nv_bfloat162 *>(&w[j]), half);
        w[j] = *reinterpret_cast<const uint32_t *>(&h);
      }
      store_row32(act + c16, w);
    }
  }
}

// A hidden layer's epilogue of one warp: its lane group's 32 rows of 2 CPH
// pieces of 32 columns (CPH per 128-column half, from column c0 of each), a
// piece's values arriving while the one before is worked on.  Two arrivals
// per half for a warp of a group of eight (CPH 2), one for a warp of sixteen.
template <int CPH, bool KEEP>
__device__ __forceinline__ void epilogue_layer(uint32_t tacc, const float *bias, uint8_t *hrow,
                                               int c0, uint32_t accfree, uint32_t hfull, int lane,
                                               __nv_bfloat16 *pre, __nv_bfloat16 *act) {
  uint32_t v[2][32];
  tmem_ld32(tacc + (uint32_t)c0, v[0]);
#pragma unroll
  for (int q = 0; q < 2 * CPH; ++q) {
    const int col = c0 + (q / CPH) * 128 + (q % CPH) * 32;
    tmem_wait32(v[q & 1]);
    if (q + 1 < 2 * CPH) {
      const int cn = c0 + ((q + 1) / CPH) * 128 + ((q + 1) % CPH) * 32;
      tmem_ld32(tacc + (uint32_t)cn, v[(q + 1) & 1]);
    } else {
      // the accumulator has been read: the next products may overwrite it
      asm volatile("tcgen05.fence::before_thread_sync;\n");
      __syncwarp();
      if (lane == 0) bar_arrive(accfree, CPH);
    }
    gelu_store32<KEEP>(v[q & 1], bias + col, hrow + (col >> 3) * 128, KEEP && pre ? pre + col : nullptr,
                       KEEP && pre ? act + col : nullptr);
    if (q % CPH == CPH - 1) {
      // written by the generic proxy, read by the tensor cores
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) bar_arrive(hfull + 8u * (uint32_t)(q / CPH), CPH);
    }
  }
}

// FUSED_FORWARD, FUSED_TRAIN: y = the network on x.  FUSED_STEP: one network
// step of the learned flow map on the particles of a.io, from the packed
// features a.xpk.
template <int MODE>
__global__ void __launch_bounds__(kFThreads, 1) mlp_fused_kernel(const __grid_constant__ FusedArgs a) {
  constexpr bool STEP = MODE == FUSED_STEP, KEEP = MODE == FUSED_TRAIN;
  extern __shared__ __align__(1024) uint8_t smem[];
  uint32_t *tslot = reinterpret_cast<uint32_t *>(smem + kOffMisc);
  volatile int *fail = reinterpret_cast<volatile int *>(smem + kOffMisc + 4);
  const uint32_t sbase = su32f(smem);
  const uint32_t sH = sbase + kOffH, sW = sbase + kOffW;
  auto bar = [&](int i) -> uint32_t { return sbase + kOffBar + 8u * (uint32_t)i; };
  const int warp = __shfl_sync(0xffffffffu, (int)(threadIdx.x >> 5), 0), lane = threadIdx.x & 31;
  const int64_t ntiles = (a.M + TMF - 1) / TMF;

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     su32f(tslot)), "r"(512));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < kNumBars; ++i) {
      const uint32_t cnt = (i >= B_ACCFREE && i < B_DRAIN) ? (uint32_t)kEpiWarps
                           : (i >= B_XFULL && i < B_XFREE && !STEP) ? (uint32_t)kInWarps : 1u;
      asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar(i)), "r"(cnt));
    }
    *fail = 0;
    asm volatile("fence.mbarrier_init.release.cluster;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n");
  const uint32_t tmem = *tslot;
  long long pieces_issued = 0;   // copy warp: for the failure path
  long long inputs_issued = 0;   // input lane of the network step: likewise

  auto give_up = [&]() {
    *fail = 1;
    atomicCAS(a.err, 0, 1);
  };
  // The CTA's tiles are blockIdx.x + i gridDim.x, taken in pairs; the last
  // may be alone.  Every kind of warp walks them in the same order: for each
  // pair, layer by layer, the first tile then the second.
  const int64_t G = gridDim.x;

  if (warp == kCopyWarp) {
    // ------------------------------------------------------ weight copies
    // The whole warp walks the pieces (converged, so addresses and barriers
    // stay in uniform registers) and one lane issues.
    int s = 0;
    uint32_t lap = 0;          // completed rounds of the ring
    bool ok = true;
    for (int64_t t0 = blockIdx.x; t0 < ntiles && ok; t0 += 2 * G) {
      const int nt = t0 + G < ntiles ? 2 : 1;
      for (int L = 0; L < 5 && ok; ++L)
        for (int t = 0; t < nt && ok; ++t)
          for (int p = layer_first(L), e = p + layer_pieces(L); p < e; ++p) {
            if (lap > 0 && !warp_wait(bar(B_WFREE + s), (lap - 1) & 1u, fail)) {
              ok = false;
              break;
            }
            const uint32_t bytes = L < 4 ? kPieceBytes : kLastBytes;
            if (elect_one()) {
              bar_expect(bar(B_WFULL + s), bytes);
              bulk_copy(sW + (uint32_t)s * kPieceBytes, a.wpk + (size_t)p * kPieceBytes, bytes,
                        bar(B_WFULL + s));
            }
            __syncwarp();
            ++pieces_issued;
            if (++s == kSlots) { s = 0; ++lap; }
          }
    }
    if (!ok && lane == 0) give_up();
  } else if (warp >= kInWarp0) {
    // --------------------------------------------------------- input tiles
    // The i-th tile goes to buffer i & 1, once the last layer of the tile
    // before it there has been multiplied.
    const int wi = warp - kInWarp0;
    bool ok = true;
    int64_t i = 0;
    if constexpr (STEP) {
      if (wi == 0 && lane == 0) {
        for (int64_t tile = blockIdx.x; tile < ntiles; tile += G, ++i) {
          const int t = (int)(i & 1);
          if (i >= 2 && !wait_bar(bar(B_XFREE + t), (uint32_t)((i / 2 - 1) & 1), fail)) {
            ok = false;
            break;
          }
          bar_expect(bar(B_XFULL + t), kTileXBytes);
          bulk_copy(sH + (uint32_t)t * kTileHBytes, a.xpk + (size_t)tile * kTileXBytes, kTileXBytes,
                    bar(B_XFULL + t));
          ++inputs_issued;
        }
        if (!ok) give_up();
      }
    } else {
      for (int64_t tile = blockIdx.x; tile < ntiles; tile += G, ++i) {
        const int t = (int)(i & 1);
        uint32_t w0[32], w1[32];          // this lane's two rows, read before the wait
        load_input_row(a, tile * TMF + wi * 32 + lane, w0);
        load_input_row(a, tile * TMF + 64 + wi * 32 + lane, w1);
        if (i >= 2) {
          ok = warp_wait(bar(B_XFREE + t), (uint32_t)((i / 2 - 1) & 1), fail);
          if (!ok) break;
        }
        store_input_row(smem + kOffH + t * kTileHBytes, wi * 32 + lane, w0);
        store_input_row(smem + kOffH + t * kTileHBytes, 64 + wi * 32 + lane, w1);
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        __syncwarp();
        if (lane == 0) bar_arrive(bar(B_XFULL + t));
      }
      if (!ok && lane == 0) give_up();
    }
  } else if (warp == kMmaWarp) {
    // ---------------------------------------------------------- products
    // Converged like the copy warp: descriptors and addresses are uniform, so
    // a product costs the issuing warp a few instructions; and few waits, each
    // some hundred clocks of a warp that shares its scheduler with four busy
    // ones.  (Issued from a one-lane branch, 32 K-columns took 600 clocks of
    // that lane against 256 of the tensor cores.)
    int s = 0;
    uint32_t lap = 0;
    uint32_t use0 = 0u, use1 = 0u;   // uses of each accumulator so far
    uint32_t xpar = 0u;              // of the pair's inputs
    bool ok = true;
    const uint64_t dX = desc_f(sH, 128, 1024), dH = desc_f(sH, 128, 4096);
    const uint64_t dW = desc_f(sW, 128, 1024), dW4 = desc_f(sW, 128, 4096);
    // K-pieces [p0, p1) of a layer: A from descriptor `da` (16 columns every
    // 256 bytes), B in the ring (64 K-columns a piece)
    auto pieces = [&](uint32_t tacc, uint64_t da, int p0, int p1) -> bool {
      for (int p = p0; p < p1; ++p) {
        if (!warp_wait(bar(B_WFULL + s), lap & 1u, fail)) return false;
        const uint64_t db = dW + (uint64_t)((uint32_t)s * (kPieceBytes >> 4));
        const uint64_t dap = da + (uint64_t)((uint32_t)p * 64u);
        if (elect_one()) {
          mma(tacc, dap, db, idesc_f(128, 256), p > 0 ? 1u : 0u);
          mma(tacc, dap + 16, db + 16, idesc_f(128, 256), 1u);
          mma(tacc, dap + 32, db + 32, idesc_f(128, 256), 1u);
          mma(tacc, dap + 48, db + 48, idesc_f(128, 256), 1u);
          commit(bar(B_WFREE + s));
        }
        __syncwarp();
        if (++s == kSlots) { s = 0; ++lap; }
      }
      return true;
    };
    for (int64_t t0 = blockIdx.x; t0 < ntiles && ok; t0 += 2 * G) {
      const int nt = t0 + G < ntiles ? 2 : 1;
      for (int L = 0; L < 5 && ok; ++L)
        for (int t = 0; t < nt && ok; ++t) {
          const int acc = nt == 2 ? t : (L & 1);
          const uint32_t tacc = tmem + (uint32_t)acc * 256u;
          const uint64_t dt = (uint64_t)((uint32_t)t * (kTileHBytes >> 4));
          const uint64_t da = dH + dt;
          const uint32_t hp = (uint32_t)((L - 1) & 1);
          const uint32_t use = acc ? use1 : use0;
          // A warp of the epilogue arrives on "first half written", then
          // "accumulator read", then "second half written"; so of a tile of a
          // pair, whose accumulator is the one to be overwritten, the second
          // covers the first, and of a tile alone "first half written" of the
          // layer before covers the reading of the accumulator two layers ago.
          if (L == 0) {
            if (use >= 1) ok = warp_wait(bar(B_ACCFREE + acc), (use - 1) & 1u, fail);
            ok = ok && warp_wait(bar(B_XFULL + t), xpar, fail);
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            ok = ok && pieces(tacc, dX + dt, 0, 1);
            if (!ok) break;
          } else if (L < 4) {
            // the first two K-pieces read the first half of the activations
            ok = nt == 2 ? warp_wait(bar(B_ACCFREE + acc), (use - 1) & 1u, fail)
                         : warp_wait(bar(B_HFULL), hp, fail);
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            ok = ok && pieces(tacc, da, 0, 2) && warp_wait(bar(B_HFULL + 2 * t + 1), hp, fail);
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            ok = ok && pieces(tacc, da, 2, 4);
            if (!ok) break;
          } else {
            // output layer: N = 16 (the first 16 of the 64 padded rows of W4)
            ok = warp_wait(bar(B_HFULL + 2 * t + 1), hp, fail) &&
                 warp_wait(bar(B_WFULL + s), lap & 1u, fail);
            if (!ok) break;
            asm volatile("tcgen05.fence::after_thread_sync;\n");
            const uint64_t db = dW4 + (uint64_t)((uint32_t)s * (kPieceBytes >> 4));
            if (elect_one()) {
#pragma unroll
              for (int ks = 0; ks < 16; ++ks)
                mma(tacc, da + (uint64_t)(ks * 16), db + (uint64_t)(ks * 16), idesc_f(128, 16),
                    ks > 0 ? 1u : 0u);
              commit(bar(B_WFREE + s));
              commit(bar(B_XFREE + t));
            }
            if (++s == kSlots) { s = 0; ++lap; }
          }
          __syncwarp();
          if (elect_one()) commit(bar(B_ACCFULL + acc));
          __syncwarp();
          if (acc) ++use1; else ++use0;
        }
      xpar ^= 1u;
    }
    if (!ok && lane == 0) give_up();
    // every product (and every commit before it) has completed before the
    // CTA moves on: bounded, and without the flag so a failing CTA waits too
    __syncwarp();
    if (elect_one()) commit(bar(B_DRAIN));
    __syncwarp();
    if (!warp_wait(bar(B_DRAIN), 0u, nullptr) && lane == 0) atomicCAS(a.err, 0, 1);
  } else {
    // ---------------------------------------------------------- epilogue
    // Two groups of eight warps, one per tile of the pair, so that the two
    // tiles' epilogues run side by side and one's loads, tanh and fences hide
    // behind the other's; a tile alone is worked on by both.
    const int lg = warp & 3;
    const int r = lg * 32 + lane;
    const uint32_t lane_base = (uint32_t)(lg * 32) << 16;
    uint32_t use0 = 0u, use1 = 0u;
    bool ok = true;
    for (int64_t t0 = blockIdx.x; t0 < ntiles && ok; t0 += 2 * G) {
      const int nt = t0 + G < ntiles ? 2 : 1;
      const int t = nt == 2 ? warp >> 3 : 0;
      const int sub = nt == 2 ? (warp >> 2) & 1 : warp >> 2;
      for (int L = 0; L < 5; ++L) {
        const int acc = nt == 2 ? t : (L & 1);
        const uint32_t tacc = tmem + lane_base + (uint32_t)acc * 256u;
        const uint32_t par = (acc ? use1 : use0) & 1u;
        if (nt == 2) { ++use0; ++use1; }
        else if (acc) ++use1;
        else ++use0;
        ok = warp_wait(bar(B_ACCFULL + acc), par, fail);
        if (!ok) break;
        asm volatile("tcgen05.fence::after_thread_sync;\n");
        if (L < 4) {
          uint8_t *hrow = smem + kOffH + t * kTileHBytes + (r >> 3) * 32 * 128 + (r & 7) * 16;
          __nv_bfloat16 *pre = nullptr, *act = nullptr;
          if constexpr (KEEP) {
            const int64_t m = (t0 + t * G) * TMF + r;
            if (m < a.M) { pre = a.pre[L] + m * 256; act = a.act[L] + m * 256; }
          }
          if (nt == 2)
            epilogue_layer<2, KEEP>(tacc, a.bias[L], hrow, sub * 64, bar(B_ACCFREE + acc),
                                    bar(B_HFULL + 2 * t), lane, pre, act);
          else
            epilogue_layer<1, KEEP>(tacc, a.bias[L], hrow, sub * 32, bar(B_ACCFREE + acc),
                                    bar(B_HFULL + 2 * t), lane, pre, act);
        } else {
          const int64_t m0 = (t0 + t * G) * TMF;
          const int rows = (a.M - m0) < TMF ? (int)(a.M - m0) : TMF;
          uint32_t v[16];
          if (sub == 0) {        // one warp per lane group has the 16 columns
            tmem_ld16(tacc, v);
            asm volatile("tcgen05.wait::ld.sync.aligned;\n"
                         : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]),
                           "+r"(v[5]), "+r"(v[6]), "+r"(v[7]), "+r"(v[8]), "+r"(v[9]),
                           "+r"(v[10]), "+r"(v[11]), "+r"(v[12]), "+r"(v[13]), "+r"(v[14]),
                           "+r"(v[15])
                         :
                         : "memory");
          }
          asm volatile("tcgen05.fence::before_thread_sync;\n");
          __syncwarp();
          if (lane == 0) bar_arrive(bar(B_ACCFREE + acc), (uint32_t)nt);
          if (sub == 0 && r < rows) {
            const float *bias = a.bias[4];
            if constexpr (STEP) {
              // the displacement moves the particle (surrogate_apply)
              const int64_t m = m0 + r;
              if (a.io.status[m] == 0) {
                float l = a.io.lon[m], la = a.io.lat[m], d = a.io.dep[m];
                const uint8_t st = surrogate_apply(
                    a.io.g, l, la, d, __uint_as_float(v[0]) + __ldg(bias),
                    __uint_as_float(v[1]) + __ldg(bias + 1),
                    __uint_as_float(v[2]) + __ldg(bias + 2));
                if (st) {
                  a.io.status[m] = st;
                } else {
                  a.io.lon[m] = l; a.io.lat[m] = la; a.io.dep[m] = d;
                  a.io.time[m] += a.io.horizon;
                  a.io.step[m] += 1;
                }
              }
            } else {
              float *yr = a.y + (size_t)(m0 + r) * a.n_out;
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (j < a.n_out) yr[j] = __uint_as_float(v[j]) + __ldg(bias + j);
            }
          }
        }
      }
    }
    if (!ok && lane == 0) give_up();
  }

  __syncwarp();
  __syncthreads();
  if (*fail && lane == 0) {
    // the copies still in flight land before the CTA leaves
    if (warp == kCopyWarp)
      for (long long qq = pieces_issued - 1; qq >= 0 && qq >= pieces_issued - kSlots; --qq)
        wait_bar(bar(B_WFULL + (int)(qq % kSlots)), (uint32_t)((qq / kSlots) & 1), nullptr);
    if (STEP && warp == kInWarp0)
      for (long long qq = inputs_issued - 1; qq >= 0 && qq >= inputs_issued - 2; --qq)
        wait_bar(bar(B_XFULL + (int)(qq & 1)), (uint32_t)((qq / 2) & 1), nullptr);
  }
  __syncwarp();
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;\n");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(512));
  }
}

// A bounded wait on an mbarrier phase that nothing completes (no thread
// arrives on the barrier and no copy or product is in flight): the wait of
// the MLP kernels gives up after `polls` polls, and the block records it in
// *err as those kernels do, then leaves.
__global__ void wait_probe_kernel(long long polls, int *err) {
  __shared__ __align__(8) uint64_t bar;
  if (threadIdx.x == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(su32f(&bar)));
    asm volatile("fence.mbarrier_init.release.cluster;\n");
  }
  __syncthreads();
  const bool ok = wait_bar(su32f(&bar), 0u, nullptr, polls);
  if (__syncthreads_or(!ok) && threadIdx.x == 0) atomicCAS(err, 0, 1);
}

// Pack the BF16 weights of the five layers (W_l [dout x din] row-major, as
// mlp.cu keeps them) into the pieces of the operand layout; layers 1-4
// halved (their inputs are stored doubled).
__global__ void pack_weights_kernel(const __nv_bfloat16 *w0, const __nv_bfloat16 *w1,
                                    const __nv_bfloat16 *w2, const __nv_bfloat16 *w3,
                                    const __nv_bfloat16 *w4, uint8_t *out) {
  const __nv_bfloat16 *W[5] = {w0, w1, w2, w3, w4};
  for (int p = blockIdx.x; p < kPieces; p += gridDim.x) {
    const Piece q = piece_of(p);
    const int din = q.layer == 0 ? 64 : 256;
    const int kc = q.kl / 8;
    for (int idx = threadIdx.x; idx < q.n * kc; idx += blockDim.x) {
      const int n = idx / kc, c = idx - n * kc;
      uint4 v = *reinterpret_cast<const uint4 *>(W[q.layer] + (size_t)n * din + q.k0 + c * 8);
      if (q.layer > 0) {
        __nv_bfloat162 *h = reinterpret_cast<__nv_bfloat162 *>(&v);
#pragma unroll
        for (int j = 0; j < 4; ++j) h[j] = __hmul2(h[j], __floats2bfloat162_rn(0.5f, 0.5f));
      }
      *reinterpret_cast<uint4 *>(out + (size_t)p * kPieceBytes + ((n >> 3) * kc + c) * 128 +
                                 (n & 7) * 16) = v;
    }
  }
}

}  // namespace

// The bounded-wait probe: one block of 128 threads; *err (device) set to 1
// when the wait gave up.
cudaError_t mlp_wait_probe(long long polls, int *err, cudaStream_t st) {
  wait_probe_kernel<<<1, 128, 0, st>>>(polls, err);
  note_launches(1);
  return cudaGetLastError();
}

// Bytes of the packed weights of the fused forward.
size_t mlp_fused_packed_bytes() { return (size_t)kPieces * kPieceBytes; }

cudaError_t mlp_fused_pack(const __nv_bfloat16 *const w[5], uint8_t *out, cudaStream_t st) {
  pack_weights_kernel<<<kPieces, 256, 0, st>>>(w[0], w[1], w[2], w[3], w[4], out);
  note_launches(1);
  return cudaGetLastError();
}

namespace {

template <int MODE>
cudaError_t launch_fused(FusedArgs &a, const uint8_t *wpk, const float *const bias[5], int n_out,
                         cudaStream_t st, int *err) {
  // the attribute belongs to the current device's context: set it on every
  // launch (cheap), so a first launch on another device is configured too
  cudaError_t e = cudaFuncSetAttribute(mlp_fused_kernel<MODE>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kSmem);
  if (e != cudaSuccess) return e;
  int dev = 0, sms = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  a.wpk = wpk; a.n_out = n_out; a.err = err;
  for (int l = 0; l < 5; ++l) a.bias[l] = bias[l];
  const int64_t ntiles = (a.M + TMF - 1) / TMF;
  const int grid = (int)(ntiles < sms ? ntiles : sms);
  mlp_fused_kernel<MODE><<<grid, kFThreads, kSmem, st>>>(a);
  note_launches(1);
  return cudaGetLastError();
}

}  // namespace

// y [M x n_out] = the network on x [M x n_in] (FP32 features, n_in <= 64,
// zero-padded to 64 on chip); biases of the five layers (FP32, 256, 256,
// 256, 256, >= n_out entries); pre, act (both null, or four [M x 256] BF16
// arrays each, 32-byte aligned): the hidden layers' values before and after
// GELU, for a backward pass; *err (device) set to 1 if a CTA gave up waiting.
cudaError_t mlp_fused_forward(const float *x, int64_t M, int n_in, const uint8_t *wpk,
                              const float *const bias[5], float *y, int n_out, cudaStream_t st,
                              int *err, __nv_bfloat16 *const *pre, __nv_bfloat16 *const *act) {
  if (M == 0) return cudaSuccess;
  if (n_out < 1 || n_out > 16 || n_in < 1 || n_in > 64 || !err || ((uintptr_t)wpk % 16))
    return cudaErrorInvalidValue;
  FusedArgs a{};
  a.x = x; a.n_in = n_in; a.y = y; a.M = M;
  if (!pre) return launch_fused<FUSED_FORWARD>(a, wpk, bias, n_out, st, err);
  for (int l = 0; l < 4; ++l) {
    if (((uintptr_t)pre[l] | (uintptr_t)act[l]) % 32) return cudaErrorInvalidValue;
    a.pre[l] = pre[l]; a.act[l] = act[l];
  }
  return launch_fused<FUSED_TRAIN>(a, wpk, bias, n_out, st, err);
}

// Bytes of the packed input tiles of a network step on n particles.
size_t mlp_fused_step_scratch(int64_t n) {
  return (size_t)std::max<int64_t>((n + TMF - 1) / TMF, 1) * kTileXBytes;
}

// One network step of the learned flow map on io's particles (the network's
// shape: 37 features, 4 x 256, 3 outputs), the features packed into xpk
// (mlp_fused_step_scratch bytes); *err as for mlp_fused_forward, feature
// errors in *io.ferr.
cudaError_t mlp_fused_step_launch(const SurrogateStepIO &io, uint8_t *xpk, const uint8_t *wpk,
                                  const float *const bias[5], cudaStream_t st, int *err) {
  if (io.n == 0) return cudaSuccess;
  if (!err || !io.ferr || !xpk || (((uintptr_t)wpk | (uintptr_t)xpk) % 16))
    return cudaErrorInvalidValue;
  FusedArgs a{};
  a.n_in = kSurFeat; a.io = io; a.xpk = xpk; a.M = io.n;
  const int64_t ntiles = (io.n + TMF - 1) / TMF;
  pack_features_kernel<<<(unsigned)ntiles, TMF, 0, st>>>(io, ntiles * TMF, xpk);
  note_launches(1);
  return launch_fused<FUSED_STEP>(a, wpk, bias, 3, st, err);
}

}  // namespace pg
