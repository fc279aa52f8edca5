// rt_mlp.cu -- the multilayer perceptron of the PAH emission surrogate: forward
// pass, mean-squared-error gradients and Adam, on the 5th-generation tensor cores
// (tcgen05.mma, FP32 accumulators in tensor memory) in BF16 with FP32 accumulation.
// Inference runs the whole network per 128-row tile in one kernel; training runs a
// kernel per layer and direction, the element-wise work in the GEMMs' epilogues.
//
// Network: a_0 = x; z_l = a_{l-1} W_l^T + b_l; a_l = silu(z_l) for the hidden layers,
// linear output. Loss = mean over rows and outputs of (y - t)^2. Master weights,
// gradients and Adam moments are FP32; the GEMM operands are BF16 copies.
// Internally every dimension is padded to a multiple of 16 (zero weights, zero
// inputs); the exported parameter layout is the unpadded one: per layer W [out][in]
// row-major, then b [out].

#include "../../include/rt.h"
#include "rt_internal.h"

#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <new>
#include <vector>

typedef __nv_bfloat16 bf16;

namespace {

constexpr int kMaxLayers = 8;

inline int pad16(int x) { return (x + 15) / 16 * 16; }

struct Layer {
  int n_in, n_out;    // unpadded
  int in_p, out_p;    // padded to 16
  size_t w_off, b_off;  // offsets in the padded parameter arrays (floats)
};

}  // namespace

struct rt_mlp {
  int dev = 0;
  int n_layers_total = 0;
  Layer layer[kMaxLayers];
  int n_in = 0, n_out = 0;
  size_t n_padded = 0;     // padded parameter count
  int64_t n_params = 0;    // unpadded
  char* slab = nullptr;      // holds the arrays down to d_loss
  float* d_param = nullptr;  // padded FP32 master
  float* d_grad = nullptr;
  float* d_m = nullptr;
  float* d_v = nullptr;
  bf16* d_wbf = nullptr;     // padded BF16 weights
  // the same weights in the operand layouts of the two fused forward kernels (see
  // forward_tc), and whether each lags behind d_wbf
  bf16* d_wpk[2] = {nullptr, nullptr};
  bool pk_stale[2] = {true, true};
  unsigned* d_err = nullptr; // fused forward: nonzero after a wait ran out
  float* d_loss = nullptr;
  long long step = 0;
  long long wait_clocks = 4000000000ll;  // of the fused forward's waits (see kTcWaitClocks)
  float x_lo = -1e30f, x_hi = 1e30f;  // admissible range of the second-to-last input
  // activations for up to cap rows
  long long cap = 0;
  bf16* d_a[kMaxLayers] = {};   // the layers' inputs in BF16 [cap][in_p]
  float* d_z[kMaxLayers] = {};  // z_l of the hidden layers in FP32 [cap][out_p]
  bf16* d_dz[2] = {};           // dz of a layer and of the one below [cap][max_p]
  int max_p = 0;
};

namespace {

// ---------------------------------------------------------------- kernels
// logistic sigmoid as 1/2 + tanh(z/2)/2, with the hardware tanh approximation
// (relative error about 2^-11, below the BF16 rounding of the activations); both the
// layer-by-layer path and the fused forward use it, so their activations agree
__device__ __forceinline__ float sigmoid_fast(float z) {
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(0.5f * z));
  return fmaf(0.5f, t, 0.5f);
}

__device__ __forceinline__ float silu_fast(float z) {
  const float h = 0.5f * z;
  float t;
  asm("tanh.approx.f32 %0, %1;" : "=f"(t) : "f"(h));
  return fmaf(h, t, h);
}

__global__ void k_to_bf16(const float* p, bf16* q, size_t n) {
  size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i < n) q[i] = __float2bfloat16(p[i]);
}

// Adam, and the BF16 copy of the new weights. Four parameters a thread (the padded
// count is a multiple of 16).
__global__ void k_adam(float4* p, const float4* g, float4* m, float4* v, uint2* q, size_t n4,
                       float lr, float b1, float b2, float c1, float c2, float eps) {
  const size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  if (i >= n4) return;
  float4 pi = p[i], mi = m[i], vi = v[i];
  const float4 gi = g[i];
  auto step = [&](float& p1, float g1, float& m1, float& v1) {
    m1 = b1 * m1 + (1.0f - b1) * g1;
    v1 = b2 * v1 + (1.0f - b2) * g1 * g1;
    p1 -= lr * (m1 / c1) / (sqrtf(v1 / c2) + eps);
  };
  step(pi.x, gi.x, mi.x, vi.x);
  step(pi.y, gi.y, mi.y, vi.y);
  step(pi.z, gi.z, mi.z, vi.z);
  step(pi.w, gi.w, mi.w, vi.w);
  m[i] = mi;
  v[i] = vi;
  p[i] = pi;
  const __nv_bfloat162 lo = __floats2bfloat162_rn(pi.x, pi.y), hi = __floats2bfloat162_rn(pi.z, pi.w);
  q[i] = make_uint2(*reinterpret_cast<const uint32_t*>(&lo), *reinterpret_cast<const uint32_t*>(&hi));
}

// ---------------------------------------------------------------- fused forward
// The whole forward pass of 256 rows (two tiles of 128) in one CTA on the 5th-generation
// tensor cores: per layer, the activations (BF16, shared memory) times the layer's weights
// (BF16, streamed through shared memory) accumulate in FP32 in tensor memory, then 16 warps
// read the accumulators back, add the bias, apply silu and write the next layer's
// activations in place. Every padded input and hidden width must be at most 256; a wider
// output layer runs in chunks of 256 output columns.
//
// Two things bound a layer of 256 columns: its products (2048 SM clocks per 128 rows) and
// the activation function (one MUFU operation per element, 2048 clocks as well, with some
// seven other instructions around it). To run them at the same time a layer is cut in halves of
// 128 columns: while the second half's products run, the first half's activations are formed
// (in registers: the products still read the layer's input, which they will replace), and
// the next layer's products over its first 128 inputs run while the second half's
// activations are formed. Weights come in pieces of 128 x 128 (32 KB) through a ring of
// three, each piece used by both tiles; one warp issues the copies, one the products.
// With one tile per CTA, a whole layer's weights at a time and the steps one after another,
// 4.0e5 rows of 66 - 3x256 - 200 took 0.373 ms; now 0.262 ms (608 TFLOP/s of the 1863 that a
// dense product reaches; 65536 rows 83 -> 62 us). Half of that
// came from the halves and the ring (0.327 ms), half from one 32-column accumulator load per
// wait, biases from shared memory and input rows converted 8 columns at a time, before the
// previous step's last outputs are stored. What is left is the chain of a layer's products,
// read-back and activations: tensor pipe 38 % busy, issue slots 32 %.
//
// Operand layout in shared memory (no swizzle, K-major): 8-row x 16-byte core
// matrices; the core holding (row r, column k) starts at (r/8)*SBO + (k/8)*128 bytes;
// inside it row r%8 is 16 bytes at (r%8)*16. SBO is 4096 for the activations and
// (columns/8)*128 for a piece of weights.
constexpr int kTcRows = 128;
constexpr int kTcTiles = 2;
constexpr int kTcEpiWarps = 16;  // 4 lane quarters of the accumulators x 4 column groups
constexpr int kTcThreads = 32 * (kTcEpiWarps + 2);
constexpr int kTcMaxWidth = 256;
constexpr int kTcHalf = 128;
constexpr int kTcMaxOut = 4096;  // output layer: up to 16 chunks of 256 columns
constexpr uint32_t kTcActSbo = (kTcMaxWidth / 8) * 128;
constexpr uint32_t kTcActBytes = (kTcRows / 8) * kTcActSbo;  // 64 KB a tile
constexpr uint32_t kTcPieceBytes = kTcHalf * kTcHalf * 2;
constexpr int kTcRing = 3;
// give up a wait after 4e9 SM clocks: 2 s at full clock (the clock register is read in a
// few cycles, the global timer only slowly)
constexpr long long kTcWaitClocks = 4000000000ll;

__device__ __forceinline__ uint32_t smem_addr(const void* p) {
  return (uint32_t)__cvta_generic_to_shared(p);
}

// shared-memory matrix descriptor: start, LBO (K direction) and SBO (row direction)
// in 16-byte units, the fixed 0b001 at bits 46-48, no swizzle
__device__ __forceinline__ uint64_t tc_desc(uint32_t addr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((addr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | ((uint64_t)1 << 46);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both K-major
__device__ __forceinline__ uint32_t tc_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) |
         ((uint32_t)(M >> 4) << 24);
}

__device__ __forceinline__ void tc_mma(uint32_t d_tmem, uint64_t a, uint64_t b, uint32_t idesc,
                                       uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(a), "l"(b), "r"(idesc), "r"(accumulate));
}

__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity,
                                          long long limit = kTcWaitClocks) {
  if (limit <= 0) return false;
  const long long t0 = clock64();
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity));
    if (done) return true;
    if (clock64() - t0 > limit) return false;
  }
}

// one thread: the next phase of `bar` completes once `bytes` have arrived from the
// bulk copy of [src, src + bytes) into shared memory at dst (16-byte aligned, size a
// multiple of 16)
__device__ __forceinline__ void bulk_load(uint32_t dst, const void* src, uint32_t bytes,
                                          uint32_t bar) {
  asm volatile(
      "{\n\t.reg .b64 st;\n\tmbarrier.arrive.expect_tx.shared::cta.b64 st, [%0], %1;\n\t}\n" ::"r"(
          bar),
      "r"(bytes)
      : "memory");
  asm volatile(
      "cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, "
      "[%3];\n" ::"r"(dst),
      "l"(src), "r"(bytes), "r"(bar)
      : "memory");
}

__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t r[16];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15}, [%16];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
  for (int j = 0; j < 16; ++j) v[j] = __uint_as_float(r[j]);
}

// 32 columns of a lane quarter with one wait
__device__ __forceinline__ void tmem_ld32(uint32_t taddr, float* v) {
  uint32_t r[32];
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, "
      "%11, %12, %13, %14, %15, %16, %17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, "
      "%28, %29, %30, %31}, [%32];\n"
      : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]),
        "=r"(r[7]), "=r"(r[8]), "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]),
        "=r"(r[13]), "=r"(r[14]), "=r"(r[15]), "=r"(r[16]), "=r"(r[17]), "=r"(r[18]),
        "=r"(r[19]), "=r"(r[20]), "=r"(r[21]), "=r"(r[22]), "=r"(r[23]), "=r"(r[24]),
        "=r"(r[25]), "=r"(r[26]), "=r"(r[27]), "=r"(r[28]), "=r"(r[29]), "=r"(r[30]),
        "=r"(r[31])
      : "r"(taddr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
  for (int j = 0; j < 32; ++j) v[j] = __uint_as_float(r[j]);
}

// ---------------------------------------------------------------- layer kernels
// Training and the networks too wide for the fused forward run one kernel per layer and
// direction on the 5th-generation tensor cores (BF16 operands, FP32 accumulators in tensor
// memory). A minibatch of 1024 rows is a few megabytes in L2 and 0.1 GFLOP a layer, so a
// step is a chain of short kernels whose launches, first loads and epilogues are all there
// is: hence few kernels (a layer's bias, activation, loss, activation derivative and bias
// gradient in the epilogue of its GEMM; the weight gradient of a layer in one launch with
// the gradient passed down), small tiles (32 or more CTAs for 1024 rows) and all of a
// tile's loads in flight at once instead of a pipeline. 28 launches with GEMMs that packed
// column-major operands element by element took 307 us a step of 1024 rows (66 - 3x256 -
// 200), these nine and Adam 90 us (16384 rows: 797 and 295; the 66 - 3x512 - 200 network forward over
// 262144 rows: 4.3 and 3.1 ms). What bounds a step now is the latency within each kernel,
// 7 us from its first load to its last store.
//
// layer tile: C [128 rows][64 columns] = A [rows][K] . B^T, K in chunks of 256:
//   forward   A = the layer's input (or the FP32 input rows, converted), B = W
//   backward  A = dz, B = W transposed while it is packed into shared memory
// gradient tile: dW [128][128] += dz^T a over a range of rows, both operands transposed
// while packed, by vector reductions.
// A row-major operand with the contraction contiguous goes to its place in the core-matrix
// layout by 16-byte asynchronous copies (8 rows x 64 bytes per warp instruction: whole
// sectors, no bank conflicts). To transpose, a thread takes 8 columns of two rows and
// writes 8 pairs; LBO is 144 bytes there so that a warp's 4-byte stores hit 32 banks.
// Every wait is bounded: after 2 s the tile's outputs are left untouched and *err is set.
constexpr int kLayRows = 128, kLayCols = 64, kLayK = 256, kLayThreads = 256;
constexpr int kGradRows = 128;                       // rows of a gradient tile's chunk
constexpr uint32_t kSbo = (kLayK / 8) * 128;         // packed by copies: LBO 128
constexpr uint32_t kLboT = 144;                      // packed by transposing
constexpr uint32_t kSboT = (kLayK / 8) * kLboT;      // K = 256
constexpr uint32_t kSboG = (kGradRows / 8) * kLboT;  // K = 128
constexpr uint32_t kLaySmem = (kLayRows / 8) * kSbo + (kLayCols / 8) * kSboT;

enum Epilogue { kHidden, kLoss, kOutput, kBack };

struct LayerArgs {
  long long M;            // rows
  int N, K, n_valid;      // padded columns and contraction; valid columns
  int n_in;               // columns of x
  const float* x;         // [M][n_in] (first layer), else null
  const bf16* a;          // [M][K] input, or dz (backward)
  const bf16* w;          // forward W [N][K], backward W [K][N]
  const float* bias;
  float* z;               // hidden: [M][N] pre-activations (null: not kept); backward: read
  bf16* out;              // hidden: activations [M][N]; backward and loss: dz [M][N]
  bf16* a0;               // first layer: the converted input [M][K] (null: not kept)
  const float* target;    // loss: [M][n_valid]
  float* loss;
  float* y;               // output: [M][n_valid]
  float* db;              // loss, backward: [N] bias gradient, added to
  float* zero;            // first layer of a training step: buffer to clear
  long long n_zero;       // (a multiple of 4 floats) and the loss
  unsigned* err;
};

struct GradArgs {
  long long M;
  int out_p, in_p;
  const bf16* dz;   // [M][out_p]
  const bf16* a;    // [M][in_p]
  float* dw;        // [out_p][in_p], added to
  int tiles_n;      // column tiles
  int rows;         // rows of a CTA, a multiple of 64
};

__device__ __forceinline__ void copy16(uint32_t dst, const void* src, bool ok) {
  const int n = ok ? 16 : 0;  // the rest is zeroed
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;\n" ::"r"(dst), "l"(src), "r"(n)
               : "memory");
}

// [rows][kc] of src (row stride ld, rows below n_ok) -> core matrices, LBO 128, SBO kSbo
__device__ __forceinline__ void pack_rows(uint32_t dst, const bf16* src, size_t ld,
                                          long long n_ok, int rows, int kc) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int r = lane & 7, k8 = lane >> 3;  // 8 rows x 4 pieces of 8
  const int nk = (kc / 8 + 3) / 4;
  for (int u = warp; u < (rows / 8) * nk; u += kLayThreads / 32) {
    const int g = u / nk, c = (u % nk) * 4 + k8, row = g * 8 + r;
    if (c * 8 < kc)
      copy16(dst + g * kSbo + c * 128u + r * 16u,
             row < n_ok ? src + (size_t)row * ld + c * 8 : src, row < n_ok);
  }
}

// element (n, k) = src[k][n], n = 0 .. 8 kGroups - 1, k = 0 .. kc - 1 (a multiple of 16, at
// most kMaxK), zero where k >= k_ok or n >= n_ok (a multiple of 8) -> core matrices, LBO kLboT, SBO sbo
template <int kGroups, int kMaxK>
__device__ __forceinline__ void pack_transposed(unsigned char* dst, uint32_t sbo, const bf16* src,
                                                size_t ld, int n_ok, int kc, long long k_ok) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  constexpr int kUnits = kGroups * (kMaxK / 64) / (kLayThreads / 32);  // a warp's share
  uint4 v0[kUnits], v1[kUnits];  // all of a thread's loads in flight
#pragma unroll
  for (int i = 0; i < kUnits; ++i) {
    const int u = warp + i * (kLayThreads / 32), g = u % kGroups;
    const int k = (u / kGroups) * 64 + (lane >> 2) * 8 + (lane & 3) * 2;
    v0[i] = v1[i] = make_uint4(0, 0, 0, 0);
    if (g * 8 < n_ok && k < kc) {
      const bf16* p = src + (size_t)k * ld + g * 8;
      if (k < k_ok) v0[i] = *reinterpret_cast<const uint4*>(p);
      if (k + 1 < k_ok) v1[i] = *reinterpret_cast<const uint4*>(p + ld);
    }
  }
#pragma unroll
  for (int i = 0; i < kUnits; ++i) {
    const int u = warp + i * (kLayThreads / 32), g = u % kGroups;
    const int k = (u / kGroups) * 64 + (lane >> 2) * 8 + (lane & 3) * 2;
    if (k >= kc) continue;
    unsigned char* q = dst + g * sbo + (k >> 3) * kLboT + (k & 7) * 2;
    const uint32_t a[4] = {v0[i].x, v0[i].y, v0[i].z, v0[i].w};
    const uint32_t b[4] = {v1[i].x, v1[i].y, v1[i].z, v1[i].w};
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      *reinterpret_cast<uint32_t*>(q + (2 * j) * 16) = __byte_perm(a[j], b[j], 0x5410);
      *reinterpret_cast<uint32_t*>(q + (2 * j + 1) * 16) = __byte_perm(a[j], b[j], 0x7632);
    }
  }
}

// The tensor memory and barrier of a CTA's single accumulator, and one accumulation step:
// the packed chunk's MMAs, then the wait for them. All threads of the block.
struct Accumulator {
  uint32_t tmem, bar, parity;
  const uint32_t* slot;
  // no barrier: the first add() has one between the set-up and its use
  __device__ __forceinline__ void open(uint64_t* bar_mem, uint32_t* slot_mem, int cols) {
    slot = slot_mem;
    if (threadIdx.x < 32) {
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                       smem_addr(slot_mem)),
                   "r"(cols));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
    }
    bar = smem_addr(bar_mem);
    if (threadIdx.x == 0) {
      asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar));
      asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    }
    parity = 0;
  }
  // false when the wait ran out (the same in all threads)
  __device__ __forceinline__ bool add(uint32_t a, uint32_t lbo_a, uint32_t sbo_a, uint32_t b,
                                      uint32_t lbo_b, uint32_t sbo_b, uint32_t idesc, int kc,
                                      bool first, unsigned* err) {
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    tmem = *slot;
    if (threadIdx.x == 0) {
      for (int kk = 0; kk < kc / 16; ++kk)
        tc_mma(tmem, tc_desc(a + kk * 2 * lbo_a, lbo_a, sbo_a),
               tc_desc(b + kk * 2 * lbo_b, lbo_b, sbo_b), idesc, !first || kk > 0 ? 1u : 0u);
      asm volatile(
          "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
              bar)
          : "memory");
    }
    const bool got = mbar_wait(bar, parity);
    if (!__syncthreads_and(got)) {
      if (threadIdx.x == 0) atomicOr(err, 1u);
      mbar_wait(bar, parity);  // let the MMAs in flight land before the memory is released
      return false;
    }
    parity ^= 1u;
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    return true;
  }
  __device__ __forceinline__ void close(int cols) {
    asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
    __syncthreads();
    if (threadIdx.x < 32) {
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                   "r"(cols));
    }
  }
};

// Sums over the warp's lanes of v[0 .. 31]; lane c returns that of v[c] (v is used up).
__device__ __forceinline__ float transpose_sum(float* v) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const bool hi = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < o; ++i) {
      const float send = hi ? v[i] : v[i + o], keep = hi ? v[i + o] : v[i];
      v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
    }
  }
  return v[0];
}

__device__ __forceinline__ void store_bf16x16(bf16* dst, const float* v) {
  uint32_t h[8];
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    h[j] = *reinterpret_cast<const uint32_t*>(&p);
  }
  uint4* q = reinterpret_cast<uint4*>(dst);
  q[0] = make_uint4(h[0], h[1], h[2], h[3]);
  q[1] = make_uint4(h[4], h[5], h[6], h[7]);
}

// The layer kernels of a pass are launched as dependents of one another: the next one's
// blocks start, set up and fetch weights (which no kernel of a pass writes) while this one
// finishes, and wait here for all of its results.
__device__ __forceinline__ void after_previous_kernel() {
  asm volatile("griddepcontrol.wait;\n" ::: "memory");
  asm volatile("griddepcontrol.launch_dependents;\n" ::: "memory");
}

// One 128 x 64 tile of a layer. smem: kLaySmem bytes.
template <int kEpi>
__device__ void layer_tile(const LayerArgs& p, long long row_tile, int col_tile,
                           unsigned char* smem, Accumulator& acc) {
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const long long m0 = row_tile * kLayRows;
  const int n0 = col_tile * kLayCols;
  const int n_cols = min(kLayCols, p.N - n0);  // a multiple of 16
  const long long rows = p.M - m0 < kLayRows ? p.M - m0 : kLayRows;
  unsigned char* sB = smem + (kLayRows / 8) * kSbo;
  const uint32_t a_addr = smem_addr(smem), b_addr = smem_addr(sB);
  const uint32_t idesc = tc_idesc(kLayRows, kLayCols);
  constexpr bool kT = kEpi == kBack;
  // warp w reads rows 32 (w & 3) .. + 31, columns 32 (w >> 2) .. + 31 of the tile
  const int c0 = 32 * (warp >> 2);
  const long long row = m0 + 32 * (warp & 3) + lane;
  const bool live = row < p.M;
  float pre[32];  // the epilogue's own input, fetched while the product is under way
  __shared__ __align__(16) float s_bias[kLayCols];
  if (kEpi != kBack && tid < kLayCols)
    s_bias[tid] = n0 + tid < p.n_valid ? __ldg(&p.bias[n0 + tid]) : 0.0f;
  bool ok = true;
  for (int k0 = 0; k0 < p.K && ok; k0 += kLayK) {
    const int kc = min(kLayK, p.K - k0);
    if (!kT) pack_rows(b_addr, p.w + (size_t)n0 * p.K + k0, p.K, n_cols, kLayCols, kc);
    if (kT)
      pack_transposed<kLayCols / 8, kLayK>(sB, kSboT, p.w + (size_t)k0 * p.N + n0, p.N, n_cols,
                                           kc, p.K - k0);
    if (k0 == 0) after_previous_kernel();
    if (!p.x) pack_rows(a_addr, p.a + (size_t)m0 * p.K + k0, p.K, rows, kLayRows, kc);
    if (k0 == 0) {
      if constexpr (kEpi == kBack) {
#pragma unroll
        for (int j = 0; j < 32; j += 4) {
          float4 z = make_float4(0, 0, 0, 0);
          if (live && n0 + c0 + j < p.N)
            z = *reinterpret_cast<const float4*>(p.z + row * p.N + n0 + c0 + j);
          pre[j] = z.x;
          pre[j + 1] = z.y;
          pre[j + 2] = z.z;
          pre[j + 3] = z.w;
        }
      } else if constexpr (kEpi == kLoss) {
#pragma unroll
        for (int j = 0; j < 32; ++j)
          pre[j] = live && n0 + c0 + j < p.n_valid
                       ? __ldg(&p.target[row * p.n_valid + n0 + c0 + j]) : 0.0f;
      }
    }
    if (p.x) {  // the FP32 input rows: coalesced along a row, zero padding
      const int valid = min(kc, p.n_in - k0);
      for (int k = lane; k < kc; k += 32) {
        float v[kLayRows / 8];  // all of a thread's rows in flight
#pragma unroll
        for (int i = 0; i < kLayRows / 8; ++i) {
          const int r = warp + 8 * i;
          v[i] = r < rows && k < valid ? __ldg(&p.x[(m0 + r) * p.n_in + k0 + k]) : 0.0f;
        }
#pragma unroll
        for (int i = 0; i < kLayRows / 8; ++i) {
          const int r = warp + 8 * i;
          const bf16 h = __float2bfloat16(v[i]);
          *reinterpret_cast<bf16*>(smem + (r >> 3) * kSbo + (k >> 3) * 128 + (r & 7) * 16 +
                                   (k & 7) * 2) = h;
          if (p.a0 && col_tile == 0 && r < rows) p.a0[(m0 + r) * p.K + k0 + k] = h;
        }
      }
    }
    asm volatile("cp.async.wait_all;\n" ::: "memory");
    ok = acc.add(a_addr, 128, kSbo, b_addr, kT ? kLboT : 128, kT ? kSboT : kSbo, idesc, kc,
                 k0 == 0, p.err);
  }
  if (!ok) return;
  float v[32];
  tmem_ld16(acc.tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0, v);
  tmem_ld16(acc.tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c0 + 16, v + 16);
  float loss = 0.0f;
#pragma unroll
  for (int h = 0; h < 32; h += 16) {
    const int col = n0 + c0 + h;
    float* w = v + h;
    if (col >= p.N) {
#pragma unroll
      for (int j = 0; j < 16; ++j) w[j] = 0.0f;
      continue;
    }
    if constexpr (kEpi == kHidden || kEpi == kLoss || kEpi == kOutput) {
#pragma unroll
      for (int j = 0; j < 16; j += 4) {
        const float4 b = *reinterpret_cast<const float4*>(&s_bias[c0 + h + j]);
        w[j] = col + j < p.n_valid ? w[j] + b.x : 0.0f;
        w[j + 1] = col + j + 1 < p.n_valid ? w[j + 1] + b.y : 0.0f;
        w[j + 2] = col + j + 2 < p.n_valid ? w[j + 2] + b.z : 0.0f;
        w[j + 3] = col + j + 3 < p.n_valid ? w[j + 3] + b.w : 0.0f;
      }
    }
    if constexpr (kEpi == kHidden) {
      if (live && p.z) {
        float4* q = reinterpret_cast<float4*>(p.z + row * p.N + col);
#pragma unroll
        for (int j = 0; j < 4; ++j)
          q[j] = make_float4(w[4 * j], w[4 * j + 1], w[4 * j + 2], w[4 * j + 3]);
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) w[j] = silu_fast(w[j]);
    }
    if constexpr (kEpi == kLoss) {
      const float inv = (float)p.M * (float)p.n_valid;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float e = live && col + j < p.n_valid ? w[j] - pre[h + j] : 0.0f;
        loss += e * e;
        w[j] = 2.0f * e / inv;
      }
    }
    if constexpr (kEpi == kBack) {
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        const float zz = pre[h + j], s = sigmoid_fast(zz);
        w[j] = live && col + j < p.n_valid ? w[j] * s * (1.0f + zz * (1.0f - s)) : 0.0f;
      }
    }
    if constexpr (kEpi == kOutput) {
      if (live)
        for (int j = 0; j < 16; ++j)
          if (col + j < p.n_valid) p.y[row * p.n_valid + col + j] = w[j];
    } else {
      if (live) store_bf16x16(p.out + row * p.N + col, w);
    }
  }
  if constexpr (kEpi == kLoss) {
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (lane == 0 && loss != 0.0f)
      atomicAdd(p.loss, loss / ((float)p.M * (float)p.n_valid));
  }
  if constexpr (kEpi == kLoss || kEpi == kBack) {
    const float sum = transpose_sum(v);
    if (n0 + c0 + lane < p.n_valid) atomicAdd(&p.db[n0 + c0 + lane], sum);
  }
}

template <int kEpi>
__global__ void __launch_bounds__(kLayThreads) k_layer(const __grid_constant__ LayerArgs p) {
  extern __shared__ __align__(128) unsigned char lay_smem[];
  __shared__ uint64_t bar;
  __shared__ uint32_t slot;
  Accumulator acc;
  acc.open(&bar, &slot, kLayCols);
  if (p.zero) {  // the pass's first kernel, an ordinary launch
    const long long me = ((long long)blockIdx.y * gridDim.x + blockIdx.x) * kLayThreads + threadIdx.x;
    for (long long i = me; i < p.n_zero / 4; i += (long long)gridDim.x * gridDim.y * kLayThreads)
      reinterpret_cast<float4*>(p.zero)[i] = make_float4(0, 0, 0, 0);
    if (me == 0) *p.loss = 0.0f;
  }
  layer_tile<kEpi>(p, blockIdx.x, blockIdx.y, lay_smem, acc);
  acc.close(kLayCols);
}

// The backward kernel of a layer: the first n_layer blocks pass the gradient down (none
// for the first layer), the others form the weight gradient.
__global__ void __launch_bounds__(kLayThreads) k_layer_back(const __grid_constant__ LayerArgs p,
                                                            const __grid_constant__ GradArgs q,
                                                            int n_layer, int row_tiles) {
  extern __shared__ __align__(128) unsigned char lay_smem[];
  __shared__ uint64_t bar;
  __shared__ uint32_t slot;
  Accumulator acc;
  acc.open(&bar, &slot, 128);
  if ((int)blockIdx.x < n_layer) {
    layer_tile<kBack>(p, blockIdx.x % row_tiles, blockIdx.x / row_tiles, lay_smem, acc);
  } else {
    after_previous_kernel();
    const int i = blockIdx.x - n_layer;
    const int tiles = q.tiles_n * ((q.out_p + 127) / 128);
    const int t = i % tiles, m0 = (t / q.tiles_n) * 128, n0 = (t % q.tiles_n) * 128;
    const long long r0 = (long long)(i / tiles) * q.rows;
    const long long r1 = r0 + q.rows < q.M ? r0 + q.rows : q.M;
    unsigned char* sB = lay_smem + 16 * kSboG;
    bool ok = true;
    for (long long r = r0; r < r1 && ok; r += kGradRows) {
      const int kc = r1 - r < kGradRows ? ((int)(r1 - r) + 15) / 16 * 16 : kGradRows;
      pack_transposed<16, kGradRows>(lay_smem, kSboG, q.dz + r * q.out_p + m0, q.out_p,
                                     q.out_p - m0, kc, r1 - r);
      pack_transposed<16, kGradRows>(sB, kSboG, q.a + r * q.in_p + n0, q.in_p, q.in_p - n0, kc,
                                     r1 - r);
      ok = acc.add(smem_addr(lay_smem), kLboT, kSboG, smem_addr(sB), kLboT, kSboG,
                   tc_idesc(128, 128), kc, r == r0, p.err);
    }
    if (ok) {
      // warp w: rows 32 (w & 3) .., columns 64 (w >> 2) .. of the tile
      const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
      const int row = m0 + 32 * (warp & 3) + lane;
      for (int c = 64 * (warp >> 2); c < 64 * (warp >> 2) + 64; c += 16) {
        if (n0 + c >= q.in_p) break;
        float v[16];
        tmem_ld16(acc.tmem + ((uint32_t)(32 * (warp & 3)) << 16) + (uint32_t)c, v);
        if (row < q.out_p) {
          float* dst = q.dw + (size_t)row * q.in_p + n0 + c;
#pragma unroll
          for (int j = 0; j < 16; j += 4)
            asm volatile("red.global.add.v4.f32 [%0], {%1, %2, %3, %4};" ::"l"(
                             __cvta_generic_to_global(dst + j)),
                         "f"(v[j]), "f"(v[j + 1]), "f"(v[j + 2]), "f"(v[j + 3])
                         : "memory");
        }
      }
    }
  }
  acc.close(128);
}

struct TcNet {
  int n_layers, n_in, n_out;
  int in_p[kMaxLayers], out_p[kMaxLayers], n_valid[kMaxLayers];
  const bf16* w[kMaxLayers];    // packed weights of each layer
  const float* b[kMaxLayers];   // padded biases
  long long wait_clocks;        // limit of the waits for results; 0: give up without waiting
};

// A layer's weights [out_p][in_p] are packed piece by piece: rows in halves of 128, columns
// in halves of 128, the pieces of a half of rows one after the other (row halves of the
// wide output layer just go on). Elements before piece (rows from n0, columns from k0):
__host__ __device__ constexpr size_t piece_start(int n0, int k0, int out_p, int in_p) {
  return (size_t)n0 * in_p + (size_t)(out_p - n0 < kTcHalf ? out_p - n0 : kTcHalf) * k0;
}

__global__ void k_pack_weights(const bf16* w, int out_p, int in_p, bf16* out) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= (long long)out_p * in_p) return;
  const int n = (int)(i / in_p), k = (int)(i % in_p);
  const int n0 = n & ~(kTcHalf - 1), k0 = k & ~(kTcHalf - 1), r = n - n0, c = k - k0;
  const int kp = in_p - k0 < kTcHalf ? in_p - k0 : kTcHalf;
  out[piece_start(n0, k0, out_p, in_p) + (r >> 3) * (kp << 3) + (c >> 3) * 64 + (r & 7) * 8 +
      (c & 7)] = w[i];
}

// Barriers of the fused forward; each but the ring's completes once per stage (a layer, or
// a chunk of the output layer).
struct TcBars {
  uint64_t full[kTcRing], empty[kTcRing];  // weight pieces arrived / read by their products
  uint64_t acc[2];    // first half's products done; all of the stage's products done
  uint64_t ready[2];  // a half of the activations written (and its accumulators read)
  uint64_t drained;   // once: all products issued are done
  uint32_t tmem_slot, failed;
  alignas(16) float bias[2][kTcMaxWidth];  // of this stage and the next
};

__device__ __forceinline__ void mbar_init(uint64_t* bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(smem_addr(bar)), "r"(count));
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("{\n\t.reg .b64 st;\n\tmbarrier.arrive.shared::cta.b64 st, [%0];\n\t}\n" ::"r"(
                   smem_addr(bar))
               : "memory");
}

// A wait that also ends when another of the CTA's waits ran out.
__device__ __forceinline__ bool tc_wait(TcBars* bars, uint64_t* bar, uint32_t parity,
                                        long long limit = kTcWaitClocks) {
  if (limit <= 0) {
    *reinterpret_cast<volatile uint32_t*>(&bars->failed) = 1u;
    return false;
  }
  const long long t0 = clock64();
  const uint32_t addr = smem_addr(bar);
  for (;;) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
        "selp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(addr), "r"(parity)
        : "memory");
    if (done) return true;
    if (*reinterpret_cast<volatile uint32_t*>(&bars->failed)) return false;
    if (clock64() - t0 > limit) {
      *reinterpret_cast<volatile uint32_t*>(&bars->failed) = 1u;
      return false;
    }
  }
}

__device__ __forceinline__ void tc_commit(uint64_t* bar) {
  asm volatile(
      "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
          smem_addr(bar))
      : "memory");
}

// y[0 .. 31] of a row: whole sectors where rows lie on 32-byte boundaries, which is what this
// kernel is chosen for; else element by element. (Without that branch, or with a constant
// number of tiles, the compiler spills 92 bytes: 291 against 262 us for 4.0e5 rows.)
__device__ __forceinline__ void store_outputs(float* y, const float* v, int n, bool vec8) {
  if (!vec8) {
#pragma unroll
    for (int j = 0; j < 32; ++j)
      if (j < n) y[j] = v[j];
    return;
  }
#pragma unroll
  for (int j = 0; j < 32; j += 8)
    if (j < n)
      asm volatile("st.global.v8.f32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(
                       __cvta_generic_to_global(y + j)),
                   "f"(v[j]), "f"(v[j + 1]), "f"(v[j + 2]), "f"(v[j + 3]), "f"(v[j + 4]),
                   "f"(v[j + 5]), "f"(v[j + 6]), "f"(v[j + 7])
                   : "memory");
}

constexpr int kTcAhead = 3;  // input items (8 columns of a row) a thread has in flight

// tiles: of 128 rows per step of a CTA
__global__ void __launch_bounds__(kTcThreads, 1)
    k_mlp_forward_tc(const __grid_constant__ TcNet net, const float* x, long long M, float* y,
                     int tiles, unsigned* err) {
  extern __shared__ __align__(128) unsigned char tc_smem[];
  unsigned char* sW = tc_smem + kTcTiles * kTcActBytes;
  TcBars* bars = reinterpret_cast<TcBars*>(sW + kTcRing * kTcPieceBytes);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid == 0) {
    for (int i = 0; i < kTcRing; ++i) {
      mbar_init(&bars->full[i], 1);
      mbar_init(&bars->empty[i], 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(&bars->acc[i], 1);
      mbar_init(&bars->ready[i], kTcEpiWarps);
    }
    mbar_init(&bars->drained, 1);
    bars->failed = 0u;
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_addr(&bars->tmem_slot)),
                 "r"(kTcTiles * kTcMaxWidth));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = bars->tmem_slot;
  const int step_rows = tiles * kTcRows;
  const long long n_steps = (M + step_rows - 1) / step_rows;
  const int L = net.n_layers;

  if (warp == kTcEpiWarps) {
    // ---- weights: every step's pieces in the order of their products
    if (lane == 0) {
      uint32_t piece = 0;
      bool ok = true;
      for (long long step = blockIdx.x; step < n_steps && ok; step += gridDim.x)
        for (int l = 0; l < L && ok; ++l) {
          const int N = net.out_p[l], K = net.in_p[l];
          for (int n0 = 0; n0 < N && ok; n0 += kTcHalf)
            for (int k0 = 0; k0 < K; k0 += kTcHalf) {
              const uint32_t slot = piece % kTcRing, round = piece / kTcRing;
              if (round > 0) ok = tc_wait(bars, &bars->empty[slot], (round - 1) & 1u);
              if (!ok) break;  // this piece was not copied
              bulk_load(smem_addr(sW + slot * kTcPieceBytes),
                        net.w[l] + piece_start(n0, k0, N, K),
                        (uint32_t)(min(kTcHalf, N - n0) * min(kTcHalf, K - k0) * 2),
                        smem_addr(&bars->full[slot]));
              ++piece;
            }
        }
      // copies still in flight land before the memory is given up: the last of each slot
      for (uint32_t i = piece > kTcRing ? piece - kTcRing : 0; i < piece; ++i)
        mbar_wait(smem_addr(&bars->full[i % kTcRing]), (i / kTcRing) & 1u);
    }
  } else if (warp == kTcEpiWarps + 1) {
    // ---- products
    if (lane == 0) {
      uint32_t piece = 0, stage = 0;
      bool ok = true;
      for (long long step = blockIdx.x; step < n_steps && ok; step += gridDim.x)
        for (int l = 0; l < L && ok; ++l) {
          const int K = net.in_p[l];
          for (int col0 = 0; col0 < net.out_p[l] && ok; col0 += kTcMaxWidth, ++stage) {
            const int N = min(kTcMaxWidth, net.out_p[l] - col0);
            ok = tc_wait(bars, &bars->ready[0], stage & 1u);
            bool second = false;  // the second half's readiness waited for
            for (int h = 0; h * kTcHalf < N && ok; ++h) {
              const uint32_t idesc = tc_idesc(kTcRows, min(kTcHalf, N - h * kTcHalf));
              for (int k0 = 0; k0 < K && ok; k0 += kTcHalf, ++piece) {
                if (!second && (h > 0 || k0 > 0)) {
                  ok = tc_wait(bars, &bars->ready[1], stage & 1u);
                  second = true;
                }
                const uint32_t slot = piece % kTcRing;
                ok = ok && tc_wait(bars, &bars->full[slot], (piece / kTcRing) & 1u);
                if (!ok) break;
                asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
                const int kp = min(kTcHalf, K - k0);
                const uint32_t b0 = smem_addr(sW + slot * kTcPieceBytes);
                for (int t = 0; t < tiles; ++t) {
                  const uint32_t a0 = smem_addr(tc_smem + t * kTcActBytes) + (uint32_t)k0 * 16u;
                  for (int kk = 0; kk < kp / 16; ++kk)
                    tc_mma(tmem + (uint32_t)(t * kTcMaxWidth + h * kTcHalf),
                           tc_desc(a0 + kk * 256u, 128u, kTcActSbo),
                           tc_desc(b0 + kk * 256u, 128u, (uint32_t)kp * 16u), idesc,
                           k0 > 0 || kk > 0 ? 1u : 0u);
                }
                tc_commit(&bars->empty[slot]);
              }
              if (ok && h == 0) tc_commit(&bars->acc[0]);
            }
            if (ok && !second) ok = tc_wait(bars, &bars->ready[1], stage & 1u);
            if (ok) tc_commit(&bars->acc[1]);
          }
        }
      tc_commit(&bars->drained);
    }
  } else {
    // ---- input, activations and outputs
    const int quarter = warp & 3, row_in = quarter * 32 + lane, group = warp >> 2;
    const uint32_t lanes = (uint32_t)(quarter * 32) << 16;
    const int F = net.n_in, K0 = net.in_p[0];
    const bool vec8 = (net.n_out & 7) == 0 && (reinterpret_cast<uintptr_t>(y) & 31) == 0;
    const int total = step_rows * F;  // a step's rows are contiguous in x
    const bool pairs = (F & 1) == 0 && (reinterpret_cast<uintptr_t>(x) & 7) == 0;
    // an item is 8 columns of a row; the row of item i: (i + 1/2)/(K0/8) lies at least
    // 1/(2 * 32) from an integer and i < 2^13, so the FP32 product truncates to it exactly
    const int row_items = K0 >> 3;
    const float inv_items = 1.0f / (float)row_items;
    // the rows of a later step on their way to L2 meanwhile
    auto fetch = [&](long long step) {
      const char* xs = reinterpret_cast<const char*>(x + step * step_rows * F);
      const long long left = (M - step * step_rows) * F;
      const int bytes = 4 * (left < total ? (int)left : total);
      for (int o = 128 * tid; o < bytes; o += 128 * 32 * kTcEpiWarps)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(__cvta_generic_to_global(xs + o)));
    };
    // input rows -> BF16 activations, zero beyond the valid rows and in the padding columns:
    // 16 bytes of a core matrix at a time
    auto input = [&](long long step) {
      for (int i0 = tid; i0 < step_rows * row_items; i0 += kTcAhead * 32 * kTcEpiWarps) {
        float v[kTcAhead][8];  // loads in flight before the stores
#pragma unroll
        for (int u = 0; u < kTcAhead; ++u) {
          const int i = i0 + u * 32 * kTcEpiWarps;
          const int r = (int)(((float)i + 0.5f) * inv_items), k = (i - r * row_items) * 8;
          const bool in = r < step_rows && step * step_rows + r < M;
          const float* xr = x + (step * step_rows + r) * F + k;
#pragma unroll
          for (int j = 0; j < 8; j += 2) {
            float2 e = make_float2(0.0f, 0.0f);
            if (pairs) {
              if (in && k + j < F) e = __ldg(reinterpret_cast<const float2*>(xr + j));
            } else {
              if (in && k + j < F) e.x = __ldg(xr + j);
              if (in && k + j + 1 < F) e.y = __ldg(xr + j + 1);
            }
            v[u][j] = e.x;
            v[u][j + 1] = e.y;
          }
        }
#pragma unroll
        for (int u = 0; u < kTcAhead; ++u) {
          const int i = i0 + u * 32 * kTcEpiWarps;
          const int r = (int)(((float)i + 0.5f) * inv_items), k = (i - r * row_items) * 8;
          if (r >= step_rows) continue;
          uint32_t h[4];
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const __nv_bfloat162 p = __floats2bfloat162_rn(v[u][2 * j], v[u][2 * j + 1]);
            h[j] = *reinterpret_cast<const uint32_t*>(&p);
          }
          *reinterpret_cast<uint4*>(tc_smem + (r >> 7) * kTcActBytes +
                                    ((r & 127) >> 3) * kTcActSbo + (k >> 3) * 128 + (r & 7) * 16) =
              make_uint4(h[0], h[1], h[2], h[3]);
        }
      }
    };
    auto written = [&](int half) {  // this warp's part of a half is in place
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(&bars->ready[half]);
    };
    uint32_t stage = 0;
    bool ok = true;
    long long step = blockIdx.x;
    if (step < n_steps) {
      input(step);
      written(0);
      written(1);
    }
    for (; step < n_steps && ok; step += gridDim.x) {
      const bool more = step + gridDim.x < n_steps;
      for (int l = 0; l < L && ok; ++l) {
        const bool hidden = l + 1 < L;
        if (l == 0 && more) fetch(step + gridDim.x);
        for (int col0 = 0; col0 < net.out_p[l] && ok; col0 += kTcMaxWidth, ++stage) {
          const int N = min(kTcMaxWidth, net.out_p[l] - col0);
          const bool last = !hidden && col0 + kTcMaxWidth >= net.out_p[l];
          // this warp's 32 columns of half h: accumulators + bias (zero in the padding)
          auto columns = [&](int h, int t, float* v) {
            const int c = h * kTcHalf + group * 32;
            tmem_ld32(tmem + lanes + (uint32_t)(t * kTcMaxWidth + c), v);
#pragma unroll
            for (int j = 0; j < 32; j += 4) {
              const float4 b = *reinterpret_cast<const float4*>(&bars->bias[stage & 1][c + j]);
              v[j] += b.x;
              v[j + 1] += b.y;
              v[j + 2] += b.z;
              v[j + 3] += b.w;
            }
          };
          auto outputs = [&](int h) {
            const int c = col0 + h * kTcHalf + group * 32;
#pragma unroll 1
            for (int t = 0; t < tiles; ++t) {
              float v[32];
              columns(h, t, v);
              const long long row = step * step_rows + t * kTcRows + row_in;
              if (row < M) store_outputs(y + row * net.n_out + c, v, net.n_out - c, vec8);
            }
          };
          auto activations = [&](int h, uint32_t* q) {  // 16 pairs a tile
#pragma unroll
            for (int t = 0; t < kTcTiles; ++t) {
              if (t >= tiles) break;
              float v[32];
              columns(h, t, v);
#pragma unroll
              for (int j = 0; j < 16; ++j) {
                const __nv_bfloat162 p =
                    __floats2bfloat162_rn(silu_fast(v[2 * j]), silu_fast(v[2 * j + 1]));
                q[16 * t + j] = *reinterpret_cast<const uint32_t*>(&p);
              }
            }
          };
          auto place = [&](int h, const uint32_t* q) {
            const int c = h * kTcHalf + group * 32;
#pragma unroll
            for (int t = 0; t < kTcTiles; ++t) {
              if (t >= tiles) break;
              unsigned char* a = tc_smem + t * kTcActBytes + (row_in >> 3) * kTcActSbo +
                                 (row_in & 7) * 16 + (c >> 3) * 128;
#pragma unroll
              for (int j = 0; j < 4; ++j)
                if (c + 8 * j < N)
                  *reinterpret_cast<uint4*>(a + j * 128) =
                      make_uint4(q[16 * t + 4 * j], q[16 * t + 4 * j + 1], q[16 * t + 4 * j + 2],
                                 q[16 * t + 4 * j + 3]);
            }
          };
          const bool mine0 = group * 32 < N, mine1 = kTcHalf + group * 32 < N;
          uint32_t q[32];
          // the biases of this warp's columns (the four warps of a group write the same)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int c = h * kTcHalf + group * 32 + lane;
            bars->bias[stage & 1][c] =
                col0 + c < net.out_p[l] ? __ldg(&net.b[l][col0 + c]) : 0.0f;
          }
          __syncwarp();
          ok = __all_sync(0xffffffffu,
                          tc_wait(bars, &bars->acc[0], stage & 1u, net.wait_clocks));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
          if (hidden) {
            if (mine0) activations(0, q);
          } else {
            if (mine0) outputs(0);
            if (!last) written(0);
          }
          // the second half's products read the layer's input to their end
          ok = __all_sync(0xffffffffu,
                          tc_wait(bars, &bars->acc[1], stage & 1u, net.wait_clocks));
          if (!ok) break;
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
          if (hidden) {
            if (mine0) place(0, q);
            written(0);
            if (mine1) {
              activations(1, q);
              place(1, q);
            }
            written(1);
          } else {
            // every product that read the activations is done: the next step's input goes in
            // first, so that its products start while these outputs are stored
            if (last && more) {
              input(step + gridDim.x);
              written(0);
            }
            if (mine1) outputs(1);
            if (!last || more) written(1);
          }
        }
      }
    }
    // a wait ran out: the rows of that step (the loop has gone one past it) and the later ones
    // are not to be used. Every warp that gave up marks its rows: another may have found the
    // same barrier complete.
    if (!ok) {
      if (lane == 0) atomicOr(err, 1u);
      for (long long s = step - gridDim.x; s < n_steps; s += gridDim.x)
        for (int t = 0; t < tiles; ++t) {
          const long long row = s * step_rows + t * kTcRows + row_in;
          if (row < M)
            for (int c = 0; c < net.n_out; ++c)
              y[row * net.n_out + c] = __int_as_float(0x7fc00000);
        }
    }
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    // the products in flight land before the memory is given up, whichever warp's wait ran
    // out: a barrier of its own, whose one phase no other commit completes (long complete
    // where none did)
    mbar_wait(smem_addr(&bars->drained), 0u);
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"(kTcTiles * kTcMaxWidth));
  }
}

size_t tc_smem_bytes() {
  return kTcTiles * kTcActBytes + kTcRing * kTcPieceBytes + sizeof(TcBars);
}

// ---------------------------------------------------------------- few rows, or ragged outputs
// One 128-row tile at a time, a layer's weights in one copy, 32 warps on one epilogue, the
// outputs staged in shared memory and written coalesced. forward_tc says when it is taken.
constexpr int kTileThreads = 1024;

// element offset of (r, k) in a [rows][K] operand in the core-matrix layout
__device__ __forceinline__ int core_off(int r, int k, int K) {
  return (r >> 3) * (K << 3) + (k >> 3) * 64 + (r & 7) * 8 + (k & 7);
}

// weights [out_p][in_p] row-major -> the core-matrix layout (one thread per element)
__global__ void k_pack_layer(const bf16* w, int out_p, int in_p, bf16* out) {
  const long long i = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (i >= (long long)out_p * in_p) return;
  const int r = (int)(i / in_p), k = (int)(i % in_p);
  out[core_off(r, k, in_p)] = w[i];
}

__global__ void __launch_bounds__(kTileThreads, 1) k_mlp_forward_tile(const __grid_constant__ TcNet net,
                                                           const float* x, long long M,
                                                           float* y, unsigned* err) {
  extern __shared__ __align__(128) unsigned char tc_smem[];
  bf16* sA = reinterpret_cast<bf16*>(tc_smem);                       // [128][256]
  bf16* sB = sA + kTcRows * kTcMaxWidth;                             // [256][256]
  float* sBias = reinterpret_cast<float*>(sB + kTcMaxWidth * kTcMaxWidth);  // [layers][256]
  uint64_t* bar = reinterpret_cast<uint64_t*>(sBias + kMaxLayers * kTcMaxWidth);  // [2]
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(bar + 2);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  // biases of every layer, zero in the padding columns
  for (int i = tid; i < net.n_layers * kTcMaxWidth; i += kTileThreads) {
    const int l = i / kTcMaxWidth, c = i % kTcMaxWidth;
    sBias[i] = c < net.n_valid[l] ? net.b[l][c] : 0.0f;
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(
                     smem_addr(tmem_slot)),
                 "r"(kTcMaxWidth));
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_addr(bar)));
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(smem_addr(bar + 1)));
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = *tmem_slot;
  const uint32_t bar_a = smem_addr(bar);      // MMAs done
  const uint32_t bar_w = smem_addr(bar + 1);  // weights arrived
  uint32_t parity = 0, wparity = 0;
  bool ok = true;
  uint32_t pend = 0;  // after a wait ran out: the barrier still owed a completion
  const long long n_tiles = (M + kTcRows - 1) / kTcRows;
  long long tile = blockIdx.x;
  for (; tile < n_tiles && ok; tile += gridDim.x) {
    const long long r0 = tile * kTcRows;
    // the first layer's weights stream in while the input is converted
    asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
    __syncthreads();
    if (tid == 0) {
      const int n0 = net.out_p[0] < kTcMaxWidth ? net.out_p[0] : kTcMaxWidth;
      bulk_load(smem_addr(sB), net.w[0], (uint32_t)(n0 * net.in_p[0] * 2), bar_w);
    }
    // input rows -> BF16 activations: the tile's rows are contiguous in x, read
    // coalesced; zero beyond the valid rows and in the padding columns
    {
      const int K = net.in_p[0], F = net.n_in;
      const long long valid = M - r0 < kTcRows ? M - r0 : kTcRows;
      const float* xt = x + r0 * F;
      const int total = kTcRows * F, n_ok = (int)valid * F;
      // row of element i: (i + 1/2)/F lies at least 1/(2F) >= 2^-9 from an integer
      // and i < 2^15, so the FP32 product truncates to floor(i/F) exactly
      const float inv_f = 1.0f / (float)F;
      for (int i0 = tid; i0 < total; i0 += 4 * kTileThreads) {
        float v[4];  // four loads in flight before the stores
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * kTileThreads;
          v[u] = i < n_ok ? __ldg(&xt[i]) : 0.0f;
        }
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int i = i0 + u * kTileThreads;
          if (i < total) {
            const int r = (int)(((float)i + 0.5f) * inv_f), k = i - r * F;
            sA[core_off(r, k, K)] = __float2bfloat16(v[u]);
          }
        }
      }
      if (tid < kTcRows)
        for (int k = F; k < K; ++k) sA[core_off(tid, k, K)] = __float2bfloat16(0.0f);
    }
    // stages: (layer, chunk of at most 256 output columns); only the output layer
    // may have more than one chunk (its packed weight rows are contiguous per chunk)
    for (int l = 0; l < net.n_layers && ok; ++l) {
      const int K = net.in_p[l], Np = net.out_p[l];
      const bool hidden = l < net.n_layers - 1;
      const int n_chunks = (Np + kTcMaxWidth - 1) / kTcMaxWidth;
      for (int ch = 0; ch < n_chunks && ok; ++ch) {
        const int col0 = ch * kTcMaxWidth;                    // first output column
        const int N = Np - col0 < kTcMaxWidth ? Np - col0 : kTcMaxWidth;
        // this stage's weights (bulk copy issued earlier)
        const bool got_w = mbar_wait(bar_w, wparity, net.wait_clocks);
        if (!__syncthreads_and(got_w)) {
          if (tid == 0) atomicOr(err, 1u);
          ok = false;
          pend = bar_w;
          break;
        }
        wparity ^= 1u;
        asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncthreads();
        if (tid == 0) {
          asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
          const uint32_t idesc = tc_idesc(kTcRows, N);
          const uint32_t a0 = smem_addr(sA), b0 = smem_addr(sB);
          const uint32_t sbo = (uint32_t)K * 16u;  // (K/8) cores of 128 bytes
          for (int kk = 0; kk < K / 16; ++kk)
            tc_mma(tmem, tc_desc(a0 + kk * 256u, 128u, sbo), tc_desc(b0 + kk * 256u, 128u, sbo),
                   idesc, kk > 0 ? 1u : 0u);
          asm volatile(
              "tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(
                  bar_a)
              : "memory");
        }
        const bool waited = mbar_wait(bar_a, parity, net.wait_clocks);
        if (!__syncthreads_and(waited)) {  // the MMAs never signalled completion
          if (tid == 0) atomicOr(err, 1u);
          ok = false;
          pend = bar_a;
          break;
        }
        parity ^= 1u;
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        // the weight buffer is free: the next stage's weights stream in meanwhile
        // (after a single-chunk output layer the buffer stages the outputs instead)
        if (tid == 0) {
          if (ch + 1 < n_chunks) {
            const int n1 = Np - col0 - kTcMaxWidth < kTcMaxWidth ? Np - col0 - kTcMaxWidth
                                                                : kTcMaxWidth;
            bulk_load(smem_addr(sB), net.w[l] + (size_t)(col0 + kTcMaxWidth) * K,
                      (uint32_t)(n1 * K * 2), bar_w);
          } else if (hidden) {
            const int n1 = net.out_p[l + 1] < kTcMaxWidth ? net.out_p[l + 1] : kTcMaxWidth;
            bulk_load(smem_addr(sB), net.w[l + 1], (uint32_t)(n1 * net.in_p[l + 1] * 2), bar_w);
          }
        }
        // accumulators of this warp's 32 rows: bias, activation, next operand or output
        const int quarter = warp & 3;                 // lanes 32 quarter .. of the accumulators
        const int row = quarter * 32 + lane;
        const int group = warp >> 2, n_groups = kTileThreads / 128;
        const float* bias = sBias + l * kTcMaxWidth;
        // a single-chunk output layer is staged over both operand buffers (the last MMA
        // is done) with an odd row stride, so that the 32 rows a warp stores hit 32
        // different banks; wider output layers are stored from registers per chunk
        const int o_stride = net.n_out | 1;
        float* so = reinterpret_cast<float*>(sA);
        const long long grow = r0 + row;
        const bool vec4 = (net.n_out & 3) == 0 && (reinterpret_cast<uintptr_t>(y) & 15) == 0;
        for (int c0 = 16 * group; c0 < N; c0 += 16 * n_groups) {
          float v[16];
          tmem_ld16(tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)c0, v);
          float bv[16];
          if (n_chunks == 1) {
#pragma unroll
            for (int j = 0; j < 16; j += 4) *reinterpret_cast<float4*>(&bv[j]) =
                *reinterpret_cast<const float4*>(&bias[c0 + j]);
          } else {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const int c = col0 + c0 + j;
              bv[j] = c < net.n_valid[l] ? __ldg(&net.b[l][c]) : 0.0f;
            }
          }
          if (hidden) {
            uint32_t h[8];
#pragma unroll
            for (int j = 0; j < 8; ++j) {
              const __nv_bfloat162 p =
                  __floats2bfloat162_rn(silu_fast(v[2 * j] + bv[2 * j]),
                                        silu_fast(v[2 * j + 1] + bv[2 * j + 1]));
              h[j] = *reinterpret_cast<const uint32_t*>(&p);
            }
            // columns c0..c0+15 of this row: two 16-byte pieces of the next operand
            *reinterpret_cast<uint4*>(&sA[core_off(row, c0, N)]) = make_uint4(h[0], h[1], h[2], h[3]);
            *reinterpret_cast<uint4*>(&sA[core_off(row, c0 + 8, N)]) =
                make_uint4(h[4], h[5], h[6], h[7]);
          } else if (n_chunks == 1) {
#pragma unroll
            for (int j = 0; j < 16; ++j) {
              const int c = c0 + j;
              if (c < net.n_out) so[row * o_stride + c] = v[j] + bv[j];
            }
          } else if (grow < M) {
            float* yr = y + grow * net.n_out + col0 + c0;
            if (vec4 && col0 + c0 + 16 <= net.n_out) {
#pragma unroll
              for (int j = 0; j < 16; j += 4)
                *reinterpret_cast<float4*>(&yr[j]) =
                    make_float4(v[j] + bv[j], v[j + 1] + bv[j + 1], v[j + 2] + bv[j + 2],
                                v[j + 3] + bv[j + 3]);
            } else {
#pragma unroll
              for (int j = 0; j < 16; ++j)
                if (col0 + c0 + j < net.n_out) yr[j] = v[j] + bv[j];
            }
          }
        }
        asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
        __syncthreads();
        if (!hidden && n_chunks == 1) {  // the tile's output rows are contiguous in y
          const long long valid = M - r0 < kTcRows ? M - r0 : kTcRows;
          float* yt = y + r0 * net.n_out;
          for (int r = warp; r < (int)valid; r += kTileThreads / 32)
            for (int c = lane; c < net.n_out; c += 32)
              yt[(long long)r * net.n_out + c] = so[r * o_stride + c];
          __syncthreads();
        }
      }
    }
  }
  // after a wait that ran out: let the weight copy or the MMAs still in flight land
  // (again with a time limit) before the shared and tensor memory are released
  if (pend != 0 && warp == 0) mbar_wait(pend, pend == bar_w ? wparity : parity);
  // and the rows of that tile (the loop has gone one past it) and the later ones are not to
  // be used
  if (!ok)
    for (long long t = tile - gridDim.x; t < n_tiles; t += gridDim.x) {
      const long long gr = t * kTcRows + tid;
      if (tid < kTcRows && gr < M)
        for (int c = 0; c < net.n_out; ++c) y[gr * net.n_out + c] = __int_as_float(0x7fc00000);
    }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (warp == 0) {
    asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem),
                 "r"(kTcMaxWidth));
  }
}

size_t tile_smem_bytes() {
  return sizeof(bf16) * (size_t)(kTcRows + kTcMaxWidth) * kTcMaxWidth +
         sizeof(float) * kMaxLayers * kTcMaxWidth + 32;
}

inline unsigned nb(long long n, int t) { return (unsigned)((n + t - 1) / t); }

// ---------------------------------------------------------------- host helpers
// A kernel of a pass: `dependent` ones may start while the one before them finishes (they
// wait in after_previous_kernel for its results).
template <typename... P, typename... A>
cudaError_t launch_pass_kernel(void (*kernel)(P...), dim3 grid, bool dependent, cudaStream_t s,
                               A... args) {
  const cudaError_t e = cudaFuncSetAttribute(
      kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)kLaySmem);
  if (e != cudaSuccess) return e;
  cudaLaunchAttribute attr{};
  attr.id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr.val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t c{};
  c.gridDim = grid;
  c.blockDim = dim3(kLayThreads);
  c.dynamicSmemBytes = kLaySmem;
  c.stream = s;
  c.attrs = &attr;
  c.numAttrs = dependent ? 1 : 0;
  return cudaLaunchKernelEx(&c, kernel, args...);
}

template <int kEpi>
cudaError_t launch_layer(const LayerArgs& p, bool first, cudaStream_t s) {
  return launch_pass_kernel(k_layer<kEpi>, dim3(nb(p.M, kLayRows), nb(p.N, kLayCols)), !first, s,
                            p);
}

cudaError_t launch_layer_back(const LayerArgs& p, GradArgs q, bool down, cudaStream_t s) {
  const int row_tiles = (int)nb(p.M, kLayRows);
  const int n_layer = down ? row_tiles * (int)nb(p.N, kLayCols) : 0;
  // rows split so that the gradient tiles are about two per SM (two CTAs fit an SM), in
  // pieces of 64 rows at least
  q.tiles_n = (int)nb(q.in_p, 128);
  const long long tiles = (long long)q.tiles_n * nb(q.out_p, 128);
  const long long chunks = (q.M + 63) / 64;
  const long long splits = std::min(chunks, (304 + tiles - 1) / tiles);
  q.rows = (int)((chunks + splits - 1) / splits) * 64;
  const long long n_grad = tiles * ((q.M + q.rows - 1) / q.rows);
  return launch_pass_kernel(k_layer_back, dim3((unsigned)(n_layer + n_grad)), true, s, p, q,
                            n_layer, row_tiles);
}

uint64_t splitmix(uint64_t& x) {
  uint64_t z = (x += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

template <typename T>
rt_status alloc(T** p, size_t n) {
  *p = nullptr;
  cudaError_t e = cudaMalloc(reinterpret_cast<void**>(p), (n ? n : 1) * sizeof(T));
  if (e == cudaErrorMemoryAllocation) {
    cudaGetLastError();
    return RT_ERR_OOM;
  }
  return e == cudaSuccess ? RT_OK : RT_ERR_CUDA;
}

template <typename T>
void release(T*& p) {
  if (p) cudaFree(p);
  p = nullptr;
}

void free_acts(rt_mlp* m) {
  for (int l = 0; l < kMaxLayers; ++l) release(m->d_a[l]);
  for (int l = 0; l < kMaxLayers; ++l) release(m->d_z[l]);
  for (int i = 0; i < 2; ++i) release(m->d_dz[i]);
  m->cap = 0;
}

// Work arrays for `rows` rows: the layers' inputs, and for training the pre-activations
// and two layers' dz.
rt_status ensure_rows(rt_mlp* m, long long rows, bool train) {
  if (rows <= m->cap && (!train || m->d_dz[0])) return RT_OK;
  if (rows < m->cap) rows = m->cap;
  free_acts(m);
  rt_status st;
  for (int l = 0; l < m->n_layers_total; ++l) {
    if ((st = alloc(&m->d_a[l], (size_t)rows * m->layer[l].in_p)) != RT_OK) return st;
    if (train && l + 1 < m->n_layers_total &&
        (st = alloc(&m->d_z[l], (size_t)rows * m->layer[l].out_p)) != RT_OK)
      return st;
  }
  for (int i = 0; train && i < 2; ++i)
    if ((st = alloc(&m->d_dz[i], (size_t)rows * m->max_p)) != RT_OK) return st;
  m->cap = rows;
  return RT_OK;
}

rt_status refresh_bf16(rt_mlp* m, cudaStream_t s) {
  k_to_bf16<<<nb((long long)m->n_padded, 256), 256, 0, s>>>(m->d_param, m->d_wbf, m->n_padded);
  m->pk_stale[0] = m->pk_stale[1] = true;
  return cudaGetLastError() == cudaSuccess ? RT_OK : RT_ERR_CUDA;
}

// Every padded width fits one tensor-core MMA (N <= 256): the fused forward applies.
bool tc_eligible(const rt_mlp* m) {
  const int L = m->n_layers_total;
  for (int l = 0; l < L; ++l) {
    if (m->layer[l].in_p > kTcMaxWidth) return false;
    // hidden widths are one MMA; the output layer runs in chunks of 256 columns
    if (m->layer[l].out_p > (l + 1 < L ? kTcMaxWidth : kTcMaxOut)) return false;
  }
  return true;
}

// forward of M rows with a fused tensor-core kernel (weights repacked when stale): the
// pieces' kernel where there are more tiles than SMs, so that a CTA has two to overlap, and
// whole 32-byte sectors to write; else one tile at a time. 49 to 66 inputs, 64 to 256 wide,
// pieces against tile, us: 4.0e5 rows with 200 outputs 262 against 374, 3.0e5 with 400 outputs
// 195 against 328, with 131 (whose rows it writes through a transpose) 292 against 274; 500
// rows 31 against 28.
rt_status forward_tc(rt_mlp* m, const float* x, float* y, long long M, cudaStream_t s) {
  int sms = 0;
  if (cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, m->dev) != cudaSuccess)
    return RT_ERR_CUDA;
  const long long n_tiles = (M + kTcRows - 1) / kTcRows;
  const int pieces = n_tiles > sms && m->n_out % 8 == 0 &&
                     (reinterpret_cast<uintptr_t>(y) & 31) == 0;
  if (m->pk_stale[pieces]) {
    for (int l = 0; l < m->n_layers_total; ++l) {
      const Layer& ly = m->layer[l];
      const auto pack = pieces ? k_pack_weights : k_pack_layer;
      pack<<<nb((long long)ly.out_p * ly.in_p, 256), 256, 0, s>>>(
          m->d_wbf + ly.w_off, ly.out_p, ly.in_p, m->d_wpk[pieces] + ly.w_off);
    }
    if (cudaGetLastError() != cudaSuccess) return RT_ERR_CUDA;
    m->pk_stale[pieces] = false;
  }
  TcNet net{};
  net.n_layers = m->n_layers_total;
  net.n_in = m->n_in;
  net.n_out = m->n_out;
  for (int l = 0; l < m->n_layers_total; ++l) {
    const Layer& ly = m->layer[l];
    net.in_p[l] = ly.in_p;
    net.out_p[l] = ly.out_p;
    net.n_valid[l] = ly.n_out;
    net.w[l] = m->d_wpk[pieces] + ly.w_off;
    net.b[l] = m->d_param + ly.b_off;
  }
  net.wait_clocks = m->wait_clocks;
  const size_t smem = pieces ? tc_smem_bytes() : tile_smem_bytes();
  if (cudaFuncSetAttribute(pieces ? reinterpret_cast<const void*>(k_mlp_forward_tc)
                                  : reinterpret_cast<const void*>(k_mlp_forward_tile),
                           cudaFuncAttributeMaxDynamicSharedMemorySize,
                           (int)smem) != cudaSuccess)
    return RT_ERR_CUDA;
  const long long steps = pieces ? (n_tiles + kTcTiles - 1) / kTcTiles : n_tiles;
  const unsigned grid = (unsigned)(steps < sms ? steps : sms);
  if (pieces)
    k_mlp_forward_tc<<<grid, kTcThreads, smem, s>>>(net, x, M, y, kTcTiles, m->d_err);
  else
    k_mlp_forward_tile<<<grid, kTileThreads, smem, s>>>(net, x, M, y, m->d_err);
  return cudaGetLastError() == cudaSuccess ? RT_OK : RT_ERR_CUDA;
}

// forward of M rows layer by layer: the last layer into y, or (t) its loss and dz
rt_status forward_rows(rt_mlp* m, const float* x, long long M, float* y, const float* t,
                       cudaStream_t s) {
  const int L = m->n_layers_total;
  for (int l = 0; l < L; ++l) {
    const Layer& ly = m->layer[l];
    LayerArgs p{};
    p.M = M;
    p.N = ly.out_p;
    p.K = ly.in_p;
    p.n_valid = ly.n_out;
    p.n_in = m->n_in;
    p.x = l == 0 ? x : nullptr;
    p.a0 = l == 0 && t ? m->d_a[0] : nullptr;
    p.a = m->d_a[l];
    p.w = m->d_wbf + ly.w_off;
    p.bias = m->d_param + ly.b_off;
    p.err = m->d_err;
    p.loss = m->d_loss;
    if (l == 0 && t) {
      p.zero = m->d_grad;
      p.n_zero = (long long)m->n_padded;
    }
    cudaError_t e;
    if (l + 1 < L) {
      p.z = t ? m->d_z[l] : nullptr;
      p.out = m->d_a[l + 1];
      e = launch_layer<kHidden>(p, l == 0, s);
    } else if (t) {
      p.target = t;
      p.out = m->d_dz[l & 1];
      p.db = m->d_grad + ly.b_off;
      e = launch_layer<kLoss>(p, l == 0, s);
    } else {
      p.y = y;
      e = launch_layer<kOutput>(p, l == 0, s);
    }
    if (e != cudaSuccess) return RT_ERR_CUDA;
  }
  return RT_OK;
}

}  // namespace

const unsigned* rt::mlp_error_word(const rt_mlp* m) { return m->d_err; }

extern "C" {

rt_status rt_mlp_create(int n_in, int n_hidden, int n_layers, int n_out, uint64_t seed,
                        rt_mlp** out) {
  if (!out || n_in < 1 || n_hidden < 1 || n_layers < 1 || n_layers > kMaxLayers - 1 ||
      n_out < 1 || n_in > 4096 || n_hidden > 4096 || n_out > 4096)
    return RT_ERR_ARG;
  *out = nullptr;
  rt_mlp* m = new (std::nothrow) rt_mlp();
  if (!m) return RT_ERR_OOM;
  if (cudaGetDevice(&m->dev) != cudaSuccess) {
    delete m;
    return RT_ERR_CUDA;
  }
  m->n_in = n_in;
  m->n_out = n_out;
  m->n_layers_total = n_layers + 1;
  size_t off = 0;
  int64_t np = 0;
  for (int l = 0; l <= n_layers; ++l) {
    Layer& ly = m->layer[l];
    ly.n_in = l == 0 ? n_in : n_hidden;
    ly.n_out = l == n_layers ? n_out : n_hidden;
    ly.in_p = pad16(ly.n_in);
    ly.out_p = pad16(ly.n_out);
    ly.w_off = off;
    off += (size_t)ly.in_p * ly.out_p;
    ly.b_off = off;
    off += (size_t)ly.out_p;
    np += (int64_t)ly.n_in * ly.n_out + ly.n_out;
    if (ly.in_p > m->max_p) m->max_p = ly.in_p;
    if (ly.out_p > m->max_p) m->max_p = ly.out_p;
  }
  // keep BF16 weight offsets 16-element aligned: offsets are sums of multiples of 16
  m->n_padded = off;
  m->n_params = np;
  // one allocation, as each takes some 30 us from 1 MB on: a network of 66 - 3x256 - 200 made and
  // closed in 569 us with eight, 380 with one. Four FP32 and three BF16 arrays of `off`, a
  // multiple of 16, the error word and the loss.
  rt_status st;
  if ((st = alloc(&m->slab, (4 * sizeof(float) + 3 * sizeof(bf16)) * off + 32)) != RT_OK) {
    rt_mlp_destroy(m);
    return st;
  }
  m->d_param = reinterpret_cast<float*>(m->slab);
  m->d_grad = m->d_param + off;
  m->d_m = m->d_grad + off;
  m->d_v = m->d_m + off;
  m->d_wbf = reinterpret_cast<bf16*>(m->d_v + off);
  m->d_wpk[0] = m->d_wbf + off;
  m->d_wpk[1] = m->d_wpk[0] + off;
  m->d_err = reinterpret_cast<unsigned*>(m->d_wpk[1] + off);
  m->d_loss = reinterpret_cast<float*>(m->d_err + 1);
  // He-uniform weights from a seeded splitmix64 stream, zero biases
  std::vector<float> h(off, 0.0f);
  uint64_t x = seed;
  for (int l = 0; l <= n_layers; ++l) {
    const Layer& ly = m->layer[l];
    float lim = std::sqrt(6.0f / (float)ly.n_in);
    for (int r = 0; r < ly.n_out; ++r)
      for (int c = 0; c < ly.n_in; ++c) {
        double u = (double)(splitmix(x) >> 11) * (1.0 / 9007199254740992.0);
        h[ly.w_off + (size_t)r * ly.in_p + c] = (float)((2.0 * u - 1.0) * lim);
      }
  }
  cudaError_t e = cudaMemcpy(m->d_param, h.data(), sizeof(float) * off, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(m->d_grad, 0, sizeof(float) * 3 * off);  // and moments
  if (e == cudaSuccess) e = cudaMemset(m->d_err, 0, sizeof(unsigned));
  if (e != cudaSuccess || refresh_bf16(m, nullptr) != RT_OK) {
    rt_mlp_destroy(m);
    return RT_ERR_CUDA;
  }
  *out = m;
  return RT_OK;
}

rt_status rt_mlp_destroy(rt_mlp* m) {
  if (!m) return RT_OK;
  cudaSetDevice(m->dev);
  free_acts(m);
  release(m->slab);
  delete m;
  return RT_OK;
}

rt_status rt_mlp_dims(const rt_mlp* m, int* n_in, int* n_out) {
  if (!m || !n_in || !n_out) return RT_ERR_ARG;
  *n_in = m->n_in;
  *n_out = m->n_out;
  return RT_OK;
}

rt_status rt_mlp_set_range(rt_mlp* m, float lo, float hi) {
  if (!m || !(hi >= lo)) return RT_ERR_ARG;
  m->x_lo = lo;
  m->x_hi = hi;
  return RT_OK;
}

rt_status rt_mlp_get_range(const rt_mlp* m, float* lo, float* hi) {
  if (!m || !lo || !hi) return RT_ERR_ARG;
  *lo = m->x_lo;
  *hi = m->x_hi;
  return RT_OK;
}

rt_status rt_mlp_set_wait_limit(rt_mlp* m, double seconds) {
  if (!m || !(seconds >= 0) || seconds > 60) return RT_ERR_ARG;
  m->wait_clocks = (long long)(seconds * 2e9);
  return RT_OK;
}

rt_status rt_mlp_n_params(const rt_mlp* m, int64_t* n) {
  if (!m || !n) return RT_ERR_ARG;
  *n = m->n_params;
  return RT_OK;
}

static rt_status copy_params(rt_mlp* m, float* host, const float* src_dev) {
  std::vector<float> h(m->n_padded);
  if (cudaMemcpy(h.data(), src_dev, sizeof(float) * m->n_padded, cudaMemcpyDeviceToHost) !=
      cudaSuccess)
    return RT_ERR_CUDA;
  size_t o = 0;
  for (int l = 0; l < m->n_layers_total; ++l) {
    const Layer& ly = m->layer[l];
    for (int r = 0; r < ly.n_out; ++r)
      for (int c = 0; c < ly.n_in; ++c) host[o++] = h[ly.w_off + (size_t)r * ly.in_p + c];
    for (int r = 0; r < ly.n_out; ++r) host[o++] = h[ly.b_off + r];
  }
  return RT_OK;
}

rt_status rt_mlp_get_params(rt_mlp* m, float* out) {
  if (!m || !out) return RT_ERR_ARG;
  if (cudaSetDevice(m->dev) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess)
    return RT_ERR_CUDA;
  unsigned err = 0;
  if (cudaMemcpy(&err, m->d_err, sizeof(err), cudaMemcpyDeviceToHost) != cudaSuccess)
    return RT_ERR_CUDA;
  rt_status st = copy_params(m, out, m->d_param);
  return st != RT_OK ? st : (err ? RT_ERR_TIMEOUT : RT_OK);
}

rt_status rt_mlp_set_params(rt_mlp* m, const float* in) {
  if (!m || !in) return RT_ERR_ARG;
  std::vector<float> h(m->n_padded, 0.0f);
  size_t o = 0;
  for (int l = 0; l < m->n_layers_total; ++l) {
    const Layer& ly = m->layer[l];
    for (int r = 0; r < ly.n_out; ++r)
      for (int c = 0; c < ly.n_in; ++c) h[ly.w_off + (size_t)r * ly.in_p + c] = in[o++];
    for (int r = 0; r < ly.n_out; ++r) h[ly.b_off + r] = in[o++];
  }
  if (cudaSetDevice(m->dev) != cudaSuccess) return RT_ERR_CUDA;
  if (cudaMemcpy(m->d_param, h.data(), sizeof(float) * m->n_padded, cudaMemcpyHostToDevice) !=
      cudaSuccess)
    return RT_ERR_CUDA;
  return refresh_bf16(m, nullptr);
}

rt_status rt_mlp_forward(rt_mlp* m, const float* x, float* y, int64_t M, void* stream) {
  if (!m || !x || !y || M < 0) return RT_ERR_ARG;
  if (M == 0) return RT_OK;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (cudaSetDevice(m->dev) != cudaSuccess) return RT_ERR_CUDA;
  if (tc_eligible(m)) return forward_tc(m, x, y, M, s);
  const long long chunk = 1ll << 18;
  for (long long r0 = 0; r0 < M; r0 += chunk) {
    const long long Mc = M - r0 < chunk ? M - r0 : chunk;
    rt_status st = ensure_rows(m, Mc, false);
    if (st == RT_OK) st = forward_rows(m, x + r0 * m->n_in, Mc, y + r0 * m->n_out, nullptr, s);
    if (st != RT_OK) return st;
  }
  return RT_OK;
}

rt_status rt_mlp_loss_grad(rt_mlp* m, const float* x, const float* t, int64_t M, float* loss_out,
                           float* grad_out, void* stream) {
  if (!m || !x || !t || M < 1 || M > (1ll << 24)) return RT_ERR_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (cudaSetDevice(m->dev) != cudaSuccess) return RT_ERR_CUDA;
  rt_status st = ensure_rows(m, M, true);
  if (st != RT_OK) return st;
  const int L = m->n_layers_total;
  if ((st = forward_rows(m, x, M, nullptr, t, s)) != RT_OK) return st;
  for (int l = L - 1; l >= 0; --l) {
    const Layer& ly = m->layer[l];
    GradArgs q{};
    q.M = M;
    q.out_p = ly.out_p;
    q.in_p = ly.in_p;
    q.dz = m->d_dz[l & 1];
    q.a = m->d_a[l];
    q.dw = m->d_grad + ly.w_off;
    LayerArgs p{};
    p.M = M;
    p.err = m->d_err;
    if (l > 0) {  // da_{l-1} = dz W_l, through silu'
      const Layer& lp = m->layer[l - 1];
      p.N = ly.in_p;
      p.K = ly.out_p;
      p.n_valid = lp.n_out;
      p.a = m->d_dz[l & 1];
      p.w = m->d_wbf + ly.w_off;
      p.z = m->d_z[l - 1];
      p.out = m->d_dz[(l - 1) & 1];
      p.db = m->d_grad + lp.b_off;
    }
    if (launch_layer_back(p, q, l > 0, s) != cudaSuccess) return RT_ERR_CUDA;
  }
  if (loss_out &&
      cudaMemcpyAsync(loss_out, m->d_loss, sizeof(float), cudaMemcpyDeviceToHost, s) != cudaSuccess)
    return RT_ERR_CUDA;
  if (grad_out || loss_out) {
    if (cudaStreamSynchronize(s) != cudaSuccess) return RT_ERR_CUDA;
  }
  if (grad_out) return copy_params(m, grad_out, m->d_grad);
  return RT_OK;
}

rt_status rt_mlp_adam_step(rt_mlp* m, float lr, void* stream) {
  if (!m || !(lr > 0)) return RT_ERR_ARG;
  cudaStream_t s = reinterpret_cast<cudaStream_t>(stream);
  if (cudaSetDevice(m->dev) != cudaSuccess) return RT_ERR_CUDA;
  m->step += 1;
  const float b1 = 0.9f, b2 = 0.999f;
  float c1 = 1.0f - std::pow(b1, (float)m->step), c2 = 1.0f - std::pow(b2, (float)m->step);
  const long long n4 = (long long)m->n_padded / 4;
  k_adam<<<nb(n4, 128), 128, 0, s>>>(
      reinterpret_cast<float4*>(m->d_param), reinterpret_cast<const float4*>(m->d_grad),
      reinterpret_cast<float4*>(m->d_m), reinterpret_cast<float4*>(m->d_v),
      reinterpret_cast<uint2*>(m->d_wbf), (size_t)n4, lr, b1, b2, c1, c2, 1e-8f);
  m->pk_stale[0] = m->pk_stale[1] = true;
  return cudaGetLastError() == cudaSuccess ? RT_OK : RT_ERR_CUDA;
}

}  // extern "C"
