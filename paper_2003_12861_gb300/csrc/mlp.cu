// Learned fit start: a multilayer perceptron from the 64-bin histogram of a
// toy dataset to a starting point for its fit (the paper has no learned part;
// this is the learned-start configuration: 64 -> 128 -> 128 -> 128 -> 6 with
// GELU, BF16 operands, FP32 accumulation, trained on the GPU).
//
// Kernels: a tensor-core GEMM on the fifth-generation tensor cores (tcgen05:
// BF16 x BF16 -> FP32 accumulated in tensor memory; the operands are rounded
// to BF16, nearest even, as they are staged into shared memory) with a fused
// bias / GELU / pre-activation epilogue, used for the forward pass and both
// backward products, with the loss gradient, GELU's derivative and the output
// map in its epilogue as well; bias gradients (column sums); the sums of the
// gradients' partial results; Adam (Kingma & Ba
// 2015) on FP32 master weights; a row gather for shuffled mini-batches; and
// target standardisation.  Every reduction has a fixed order, so training is
// bitwise reproducible.
//
// Parameter layout (flat FP32): for each layer W[n_in x n_out] row-major,
// then b[n_out].
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstdio>
#include <cstring>
#include <random>
#include <vector>

#include "api_internal.h"

namespace rf {

// Learned starts of bounded parameters stay this fraction of the range
// inside the bounds (rf_mlp_predict).
constexpr double kStartMargin = 0.05;

namespace {

struct GemmArgs {
  const float* A;  // M x K (or K x M when transA)
  const float* B;  // K x N (or N x K when transB)
  float* C;        // M x N
  const float* bias;  // N or null
  float* Z;        // pre-activation out (M x N, like C) or null
  const float* Zg; // or null: C is multiplied by GELU'(Zg) (M x N, like C)
  const float *scale, *shift;  // or null: C's columns are mapped by v scale + shift (after all else)
  // or null: the targets (M x N, like C) of a training pass's last layer; C is
  // then the loss gradient lscale (v - T) and loss[tile] the tile's sum of (v - T)^2
  const float* T;
  double* loss;
  float lscale;
  int M, N, K, lda, ldb, ldc;
  int transA, transB, gelu;
  int vecA, vecB, vecC, vecZ;  // 16-byte rows (leading dimension and pointers)
  int splits, kc;        // K rows [z kc, (z + 1) kc) are summed on their own, then added in order
  // null, or (weight gradients) split z's raw partial tile goes to part + z M N
  // (row-major) from a block of its own; else one block holds the splits'
  // accumulators side by side in tensor memory
  float* part;
};

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * __expf(-0.5f * z * z) * 0.3989422804014327f;
}

// Set when a GEMM's wait for its tensor-core work gave up (checked by the
// synchronous entry points).
__device__ int g_gemm_timeout;

// The GEMM's tile: 128 rows (the MMA's M, one TMEM lane per row) x 32
// columns (N; 32 FP32 accumulator columns of TMEM, the smallest allocation),
// K staged 128 at a time.  (64 columns measured 4-25 % slower on the
// network's shapes: half as many blocks for these small GEMMs.)
constexpr int TM = 128, TN = 32, TK = 128, kGemmThreads = 256;
constexpr int kSmemA = TM * TK * 2, kSmemB = TN * TK * 2;
constexpr int kGemmSmem = kSmemA + kSmemB + 128;

__device__ __forceinline__ uint32_t smem_u32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// A K-major operand tile without swizzle is stored as core matrices of 8
// rows x 8 BF16 (16 bytes per row, 128 contiguous bytes); rows 8g.., k
// 8j.. at byte (g * TK / 8 + j) * 128.  Its shared-memory descriptor: start
// address, the leading byte offset (next core matrix along K: 128), the
// stride byte offset (next 8 rows: TK / 8 * 128), descriptor version 1, no
// swizzle.
__device__ __forceinline__ uint64_t operand_desc(uint32_t saddr) {
  const uint64_t lbo = 128, sbo = (TK / 8) * 128;
  return (uint64_t)((saddr >> 4) & 0x3FFF) | ((lbo >> 4) & 0x3FFF) << 16 | ((sbo >> 4) & 0x3FFF) << 32 |
         (uint64_t)1 << 46;
}
// The instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B,
// both K-major, N >> 3 and M >> 4.
__host__ __device__ constexpr uint32_t mma_idesc(int M, int N) {
  return (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Waits for phase `parity` of the barrier; gives up (false) after 2^22 tries.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity) {
  for (int it = 0; it < (1 << 22); ++it) {
    uint32_t done;
    asm volatile(
        "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(bar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

__device__ __forceinline__ void store8(unsigned char* dst, const float* v) {
  uint32_t w[4];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    const __nv_bfloat162 h = __floats2bfloat162_rn(v[2 * j], v[2 * j + 1]);
    w[j] = *reinterpret_cast<const uint32_t*>(&h);
  }
  *reinterpret_cast<uint4*>(dst) = make_uint4(w[0], w[1], w[2], w[3]);
}
// Group q of an operand tile of ROWS rows is 8 consecutive k of one row: its
// row and 8-k group, and where it goes.  Along k in memory: a warp takes 8
// rows x 4 groups (32-byte pieces of 8 rows; the stores are then linear in q).
// Along the rows (trans): a warp takes 32 rows of one group, each of its 8
// loads contiguous.  Both store 16 bytes per thread without bank conflicts.
template <int ROWS, bool kTrans>
__device__ __forceinline__ void group_of(int q, int* r, int* kg, int* off) {
  if (kTrans) {
    *r = q % ROWS;
    *kg = q / ROWS;
    *off = ((*r >> 3) * (TK / 8) + *kg) * 128 + (*r & 7) * 16;
  } else {
    *r = (q >> 7) * 8 + (q & 7);
    *kg = (q >> 3) & 15;
    *off = q * 16;
  }
}
// Stages rows [r0, r0 + ROWS) x k [k0, k0 + kn) of an operand (element (row, k)
// at src[row ld + k], or src[k ld + row] when kTrans), rounded to BF16, zero in
// rows >= R and in k up to the next multiple of 16.  A tile whose rows are all
// there and whose k come in whole groups has four groups' loads in flight per
// thread; others go element by element.  The loops stay rolled: with
// everything unrolled the kernel waited for its instructions (14 of 24
// stalled warps).  The chained kernels below read through L2: a predecessor
// may still be writing when the kernel starts.
template <int ROWS, bool kTrans>
__device__ __forceinline__ void stage(unsigned char* dst, const float* src, int ld, bool vec, int r0, int R, int k0,
                                      int kn) {
  constexpr int kGroups = ROWS * TK / 8 / kGemmThreads, kIn = kGroups < 4 ? kGroups : 4;
  const int kg1 = (kn + 15) / 16 * 2;
  if (r0 + ROWS <= R && kn % 8 == 0 && (kTrans || vec)) {
#pragma unroll 1
    for (int h = 0; h < kGroups; h += kIn) {
      float v[kIn][8];
#pragma unroll
      for (int i = 0; i < kIn; ++i) {
        int r, kg, off;
        group_of<ROWS, kTrans>(threadIdx.x + (h + i) * kGemmThreads, &r, &kg, &off);
        if (8 * kg < kn) {
          if (kTrans) {
            const float* p = src + (size_t)(k0 + 8 * kg) * ld + r0 + r;
#pragma unroll
            for (int j = 0; j < 8; ++j) v[i][j] = __ldcg(p + j * ld);
          } else {
            const float4* p = reinterpret_cast<const float4*>(src + (size_t)(r0 + r) * ld + k0 + 8 * kg);
            const float4 a = __ldcg(p), b = __ldcg(p + 1);
            v[i][0] = a.x; v[i][1] = a.y; v[i][2] = a.z; v[i][3] = a.w;
            v[i][4] = b.x; v[i][5] = b.y; v[i][6] = b.z; v[i][7] = b.w;
          }
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j) v[i][j] = 0.f;
        }
      }
#pragma unroll
      for (int i = 0; i < kIn; ++i) {
        int r, kg, off;
        group_of<ROWS, kTrans>(threadIdx.x + (h + i) * kGemmThreads, &r, &kg, &off);
        if (kg < kg1) store8(dst + off, v[i]);
      }
    }
    return;
  }
#pragma unroll 1
  for (int h = 0; h < kGroups; ++h) {
    int r, kg, off;
    group_of<ROWS, kTrans>(threadIdx.x + h * kGemmThreads, &r, &kg, &off);
    if (kg >= kg1) continue;
    float v[8];
#pragma unroll
    for (int j = 0; j < 8; ++j) {
      const int k = k0 + 8 * kg + j;
      v[j] = r0 + r < R && 8 * kg + j < kn
                 ? __ldcg(src + (kTrans ? (size_t)k * ld + r0 + r : (size_t)(r0 + r) * ld + k))
                 : 0.f;
    }
    store8(dst + off, v);
  }
}

// One 128 x 32 tile of C = act(op(A) op(B) + bias) by a block of 8 warps.  Per
// K stage the block converts its A and B tiles to BF16 into shared memory (out
// of range: zero; these GEMMs are bound by the latency of their FP32
// operands), one thread issues the 128 x 32 x 16 MMAs accumulating in tensor
// memory and commits them to a barrier that every thread waits on; then warps
// w and w + 4 read half the columns each of 32 rows of the accumulator
// (tcgen05.ld) for the epilogue.  Warp 0 allocates and frees the TMEM columns.
// bz: the split of a block that holds one (g.part), else 0.
__device__ __forceinline__ void gemm_tile(const GemmArgs& g, int bx, int by, int bz, unsigned char* gsm) {
  unsigned char* As = gsm;
  unsigned char* Bs = gsm + kSmemA;
  uint64_t* bar = reinterpret_cast<uint64_t*>(gsm + kSmemA + kSmemB);
  uint32_t* tslot = reinterpret_cast<uint32_t*>(gsm + kSmemA + kSmemB + 8);
  double* red = reinterpret_cast<double*>(gsm + kSmemA + kSmemB + 16);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = by * TM, n0 = bx * TN;
  const int z0 = g.part ? bz : 0, z1 = g.part ? bz + 1 : g.splits;
  const uint32_t bar_a = smem_u32(bar);
  uint32_t cols = TN;
  while (cols < (uint32_t)(z1 - z0) * TN) cols *= 2;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(tslot)), "r"(cols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n" ::: "memory");
  }
  if (tid == 0) {
    asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;\n" ::"r"(bar_a) : "memory");
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
  const uint32_t tmem = *tslot;
  // what the epilogue multiplies by is loaded ahead of the operands
  const int row = m0 + (warp & 3) * 32 + lane, half = (warp >> 2) * 16;
  float zg[16];
  if (g.Zg && row < g.M) {
    const float* src = g.Zg + (size_t)row * g.ldc + n0 + half;
    if (g.vecZ && n0 + half + 16 <= g.N) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 q = __ldcg(reinterpret_cast<const float4*>(src) + j);
        zg[4 * j] = q.x; zg[4 * j + 1] = q.y; zg[4 * j + 2] = q.z; zg[4 * j + 3] = q.w;
      }
    } else {
#pragma unroll
      for (int j = 0; j < 16; ++j) zg[j] = n0 + half + j < g.N ? __ldcg(src + j) : 0.f;
    }
  }
  uint32_t parity = 0;
  bool ok = true;
  for (int z = z0; z < z1 && ok; ++z) {
    const int kb = z * g.kc, ke = min(g.K, kb + g.kc);
    for (int k0 = kb; k0 < ke && ok; k0 += TK) {
      const int kn = min(TK, ke - k0), steps = (kn + 15) / 16;
      if (g.transB) stage<TN, false>(Bs, g.B, g.ldb, g.vecB, n0, g.N, k0, kn);
      else stage<TN, true>(Bs, g.B, g.ldb, false, n0, g.N, k0, kn);
      if (g.transA) stage<TM, true>(As, g.A, g.lda, false, m0, g.M, k0, kn);
      else stage<TM, false>(As, g.A, g.lda, g.vecA, m0, g.M, k0, kn);
      // the tiles were written through the generic proxy; the MMAs read them
      // through the async proxy
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      __syncthreads();
      if (tid == 0) {
        asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
        const uint32_t sa = smem_u32(As), sb = smem_u32(Bs);
        for (int s = 0; s < steps; ++s) {
          const uint64_t da = operand_desc(sa + s * 256), db = operand_desc(sb + s * 256);
          const uint32_t accumulate = (k0 > kb || s > 0) ? 1u : 0u;
          asm volatile(
              "{\n .reg .pred p;\n setp.ne.u32 p, %4, 0;\n"
              " tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem + (uint32_t)(z - z0) * TN),
              "l"(da), "l"(db), "r"(mma_idesc(TM, TN)), "r"(accumulate)
              : "memory");
        }
        asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar_a)
                     : "memory");
      }
      ok = mbar_wait(bar_a, parity);
      parity ^= 1u;
      asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory");
      ok = __syncthreads_and(ok) != 0;  // block-uniform: every warp takes the same path
    }
  }
  double sq = 0.0;
  if (!ok) {
    if (tid == 0) atomicExch(&g_gemm_timeout, 1);
    mbar_wait(bar_a, parity ^ 1u);  // once more (bounded) for MMAs still in flight
  } else {
    // every lane reads the accumulator (the loads are warp-wide), then those
    // with a row of C go on
    float acc[16];
    for (int z = 0; z < z1 - z0; ++z) {
      uint32_t r[16];
      const uint32_t ta = tmem + ((uint32_t)((warp & 3) * 32) << 16) + (uint32_t)(z * TN + half);
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15}, [%16];\n"
          : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
            "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
          : "r"(ta)
          : "memory");
      asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
#pragma unroll
      for (int j = 0; j < 16; ++j) acc[j] = z == 0 ? __uint_as_float(r[j]) : acc[j] + __uint_as_float(r[j]);
    }
#pragma unroll
    for (int c = 0; c < 2; ++c) {
      const int col0 = n0 + half + c * 8;
      if (row >= g.M || col0 >= g.N) continue;
      float* v = acc + c * 8;
      const size_t at = g.part ? ((size_t)bz * g.M + row) * g.N + col0 : (size_t)row * g.ldc + col0;
      const bool whole = g.vecC && col0 + 8 <= g.N;  // (g.part has rows of N = ldc floats too)
      auto put = [&](float* dst, const float* x) {
        if (whole) {
          *reinterpret_cast<float4*>(dst) = make_float4(x[0], x[1], x[2], x[3]);
          *reinterpret_cast<float4*>(dst + 4) = make_float4(x[4], x[5], x[6], x[7]);
        } else {
#pragma unroll
          for (int j = 0; j < 8; ++j)
            if (col0 + j < g.N) dst[j] = x[j];
        }
      };
      if (g.part) {
        put(g.part + at, v);
        continue;
      }
      if (g.bias)
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] += col0 + j < g.N ? __ldcg(g.bias + col0 + j) : 0.f;
      if (g.Z) put(g.Z + at, v);
      if (g.gelu)
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] = gelu_f(v[j]);
      if (g.Zg)
#pragma unroll
        for (int j = 0; j < 8; ++j) v[j] *= gelu_grad_f(zg[c * 8 + j]);
      if (g.T)
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (col0 + j < g.N) {
            const float d = v[j] - __ldcg(g.T + at + j);
            sq += (double)d * d;
            v[j] = g.lscale * d;
          }
      if (g.scale)
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (col0 + j < g.N) v[j] = v[j] * __ldcg(g.scale + col0 + j) + __ldcg(g.shift + col0 + j);
      put(g.C + at, v);
    }
  }
  if (g.T) {  // the tile's squared errors: lanes by butterfly, then the warps in order
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
    if (lane == 0) red[warp] = sq;
  }
  asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory");
  __syncthreads();
  if (g.T && tid == 0) {
    double t = 0.0;
    for (int w = 0; w < kGemmThreads / 32; ++w) t += red[w];
    g.loss[(size_t)by * ((g.N + TN - 1) / TN) + bx] = t;
  }
  __syncwarp();  // the deallocation is warp-wide
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(cols) : "memory");
}

// The launches of a pass follow one another as programmatic dependents: a
// kernel is scheduled while its predecessor runs and waits here for it to be
// complete (and so, in turn, for all before it).  The wait comes before the
// tensor-memory allocation: a waiting block holding columns that a block of
// the predecessor needs would never be released.
__device__ __forceinline__ void chain_wait() {
  asm volatile("griddepcontrol.launch_dependents;");
  asm volatile("griddepcontrol.wait;" ::: "memory");
}

__global__ void __launch_bounds__(kGemmThreads) gemm_bf16_kernel(const __grid_constant__ GemmArgs g) {
  extern __shared__ __align__(128) unsigned char gsm[];
  chain_wait();
  gemm_tile(g, blockIdx.x, blockIdx.y, 0, gsm);
}

// One layer's backward pass, whose three products depend on the layer's dZ
// alone, as one launch: blocks [0, n_in) compute dZ of the layer below (dZ W^T
// with GELU' in the epilogue), [n_in, n_in + n_w) the weight gradient's tiles
// and splits, the rest column sums of dZ over `chunk` rows for the bias gradient.
struct BackArgs {
  GemmArgs in, w;
  int n_in, n_w;
  const float* dZ;
  float* db;  // per chunk: its column sums
  int rows, cols, chunk;
};
__global__ void __launch_bounds__(kGemmThreads) backward_kernel(const __grid_constant__ BackArgs b) {
  extern __shared__ __align__(128) unsigned char gsm[];
  chain_wait();
  int i = blockIdx.x;
  if (i < b.n_in + b.n_w) {  // one call for both products: the code is large
    const bool below = i < b.n_in;
    const GemmArgs& g = below ? b.in : b.w;
    if (!below) i -= b.n_in;
    const int nx = (g.N + TN - 1) / TN, ny = (g.M + TM - 1) / TM;
    gemm_tile(g, i % nx, i / nx % ny, i / (nx * ny), gsm);
    return;
  }
  i -= b.n_in + b.n_w;
  // 32 columns x 8 row lanes; the lanes' sums in order
  const int nx = (b.cols + 31) / 32, c = i % nx * 32 + (threadIdx.x & 31), rl = threadIdx.x >> 5;
  const int r0 = i / nx * b.chunk, r1 = min(b.rows, r0 + b.chunk);
  float s = 0.f;
  if (c < b.cols) {
#pragma unroll 8
    for (int r = r0 + rl; r < r1; r += kGemmThreads / 32) s += __ldcg(b.dZ + (size_t)r * b.cols + c);
  }
  float* red = reinterpret_cast<float*>(gsm);
  red[threadIdx.x] = s;
  __syncthreads();
  if (rl == 0 && c < b.cols) {
    for (int w = 1; w < kGemmThreads / 32; ++w) s += red[w * 32 + threadIdx.x];
    b.db[(size_t)(i / nx) * b.cols + c] = s;
  }
}

// The end of a backward pass: every layer's partial weight and bias gradients
// summed in order (item i: blocks [block0, next item's block0)), and by the
// last block the loss (the tiles' squared errors over n) beside the GEMMs'
// give-up flag.
constexpr int kMaxLayers = 17;
struct ReduceItem {
  const float* part;
  float* out;
  int n, splits, block0;
};
struct ReduceArgs {
  ReduceItem it[2 * kMaxLayers];
  int n_items;
  const double* loss;
  int n_loss;
  double n;      // targets: the loss is the sum over them divided by n
  float* out;    // loss, flag
};
__global__ void __launch_bounds__(256) reduce_kernel(const __grid_constant__ ReduceArgs a) {
  const int tid = threadIdx.x;
  chain_wait();
  if (blockIdx.x == gridDim.x - 1) {
    __shared__ double red[256];
    double s = 0.0;
    for (int i = tid; i < a.n_loss; i += 256) s += a.loss[i];
    red[tid] = s;
    __syncthreads();
    for (int o = 128; o > 0; o >>= 1) {
      if (tid < o) red[tid] += red[tid + o];
      __syncthreads();
    }
    if (tid == 0) {
      a.out[0] = (float)(red[0] / a.n);
      reinterpret_cast<int*>(a.out)[1] = g_gemm_timeout;
    }
    return;
  }
  int i = 0;
  while (i + 1 < a.n_items && (int)blockIdx.x >= a.it[i + 1].block0) ++i;
  const ReduceItem& it = a.it[i];
  const int e = ((int)blockIdx.x - it.block0) * 256 + tid;
  if (e >= it.n) return;
  float v = 0.f;
#pragma unroll 4
  for (int z = 0; z < it.splits; ++z) v += __ldcg(it.part + (size_t)z * it.n + e);
  it.out[e] = v;
}

__global__ void adam_kernel(float* p, const float* g, float* m, float* v, int64_t n, float lr, float b1, float b2,
                            float eps, float c1, float c2) {
  chain_wait();
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.f - b1) * gi;
  const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  p[i] -= lr * (mi / c1) / (sqrtf(vi / c2) + eps);
}

// The rows idx of x (ni columns) and t (no columns), by one launch.
__global__ void gather_rows_kernel(const float* x, const float* t, const int32_t* idx, int rows, int ni, int no,
                                   float* xb, float* tb) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)rows * (ni + no)) return;
  const int r = (int)(i / (ni + no)), c = (int)(i % (ni + no));
  if (c < ni) xb[(size_t)r * ni + c] = x[(size_t)idx[r] * ni + c];
  else tb[(size_t)r * no + c - ni] = t[(size_t)idx[r] * no + c - ni];
}

// Per-column mean and standard deviation of T (rows x cols), fixed order.
__global__ void col_stats_kernel(const float* T, int rows, int cols, float* mean, float* sd) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cols) return;
  double s = 0.0, s2 = 0.0;
  for (int r = 0; r < rows; ++r) {
    const double x = T[(size_t)r * cols + c];
    s += x;
    s2 += x * x;
  }
  const double mu = s / rows;
  const double var = s2 / rows - mu * mu;
  mean[c] = (float)mu;
  sd[c] = (float)(var > 1e-30 ? sqrt(var) : 1.0);
}

__global__ void standardise_kernel(const float* T, int rows, int cols, const float* mean, const float* sd, float* out) {
  const int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (int64_t)rows * cols) return;
  const int c = (int)(i % cols);
  out[i] = (T[i] - mean[c]) / sd[c];
}

unsigned blocks_for(int64_t n, int t) { return (unsigned)((n + t - 1) / t); }

}  // namespace

// A GEMM whose output tiles are few and whose K is long sums K in up to
// kMaxSplits pieces: the weight gradients (K = the batch) over as many blocks
// per tile, into partial tiles that reduce_kernel adds up; the others, whose K
// is a layer's width, side by side in one block's tensor memory.
constexpr int kMaxSplits = 16, kSplitK = 64;
int gemm_splits(int M, int N, int K) {
  const int tiles = ((N + TN - 1) / TN) * ((M + TM - 1) / TM);
  if (tiles >= 32 || K < 4 * kSplitK) return 1;
  return std::max(1, std::min(kMaxSplits, K / (2 * kSplitK)));
}
bool rows16(const void* p, int ld) { return ((uintptr_t)p & 15) == 0 && ld % 4 == 0; }
// The GEMM C = op(A) op(B) with its splits and vector widths; the caller adds the epilogue.
GemmArgs gemm_args(const float* A, int lda, bool tA, const float* B, int ldb, bool tB, float* C, int ldc, int M, int N,
                   int K) {
  GemmArgs g{};
  g.A = A; g.B = B; g.C = C;
  g.M = M; g.N = N; g.K = K;
  g.lda = lda; g.ldb = ldb; g.ldc = ldc;
  g.transA = tA; g.transB = tB;
  g.vecA = rows16(A, lda); g.vecB = rows16(B, ldb); g.vecC = rows16(C, ldc);
  g.splits = gemm_splits(M, N, K);
  g.kc = g.splits > 1 ? ((K + g.splits - 1) / g.splits + kSplitK - 1) / kSplitK * kSplitK : K;
  g.splits = (K + g.kc - 1) / g.kc;
  return g;
}
int gemm_tiles(const GemmArgs& g) { return ((g.N + TN - 1) / TN) * ((g.M + TM - 1) / TM); }

// After a synchronisation: RF_E_TIMEOUT (and the flag cleared) if a GEMM gave
// up waiting for its tensor-core work since the last check.
rf_status gemm_status(const char* what) {
  int flag = 0;
  if (!cuda_ok(cudaMemcpyFromSymbol(&flag, g_gemm_timeout, sizeof(int)), what)) return RF_E_CUDA;
  if (!flag) return RF_OK;
  const int zero = 0;
  cudaMemcpyToSymbol(g_gemm_timeout, &zero, sizeof(int));
  set_error(std::string(what) + ": a GEMM's wait for its tensor-core work gave up");
  return RF_E_TIMEOUT;
}

}  // namespace rf

using namespace rf;

struct rf_mlp {
  std::vector<int> dims;  // n_in, hidden..., n_out
  int64_t n_params = 0;
  std::vector<int64_t> w_off, b_off;
  DevBuf params, grads, m, v;
  DevBuf acts, zs, dbuf, dbuf2, y, loss, xb, tb, mean, sd, scale, shift;
  DevBuf pred_h, pred_y;  // rf_mlp_predict: histograms and outputs of the sets
  DevBuf partial;         // the weight and bias gradients' partial sums
  DevBuf sq;              // the last layer's tiles' squared errors
  HostBuf h_loss;
  int cap = 0;  // batch capacity of the activation buffers
  int64_t step = 0;
  bool has_affine = false;
};

namespace rf {
namespace {

// Rows per partial column sum of a batch: at most 16 of them.
int bias_chunk(int batch) { return std::max(128, (batch + 15) / 16); }

bool mlp_reserve(rf_mlp* n, int batch) {
  if (batch <= n->cap) return true;
  n->cap = 0;  // (a buffer that cannot grow is lost with what it had)
  int64_t act = 0, z = 0, part = 0;
  const int wmax = *std::max_element(n->dims.begin(), n->dims.end());
  const int nout = n->dims.back();
  for (size_t l = 0; l + 1 < n->dims.size(); ++l) {
    const int64_t ni = n->dims[l], no = n->dims[l + 1];
    if (l) act += batch * ni;
    z += batch * no;
    part += kMaxSplits * no;  // bias
    // the splits of a smaller batch are at most those of tiles below 32
    if (gemm_splits((int)ni, (int)no, 1 << 30) > 1) part += kMaxSplits * ni * no;
  }
  const int64_t sq = (int64_t)((batch + TM - 1) / TM) * ((nout + TN - 1) / TN);
  bool ok = n->acts.ensure(sizeof(float) * std::max<int64_t>(1, act)) && n->zs.ensure(sizeof(float) * z) &&
            n->dbuf.ensure(sizeof(float) * (size_t)batch * wmax) && n->dbuf2.ensure(sizeof(float) * (size_t)batch * wmax) &&
            n->y.ensure(sizeof(float) * (size_t)batch * nout) && n->loss.ensure(2 * sizeof(float)) &&
            n->h_loss.ensure(2 * sizeof(float)) && n->xb.ensure(sizeof(float) * (size_t)batch * n->dims[0]) &&
            n->tb.ensure(sizeof(float) * (size_t)batch * nout) && n->partial.ensure(sizeof(float) * part) &&
            n->sq.ensure(sizeof(double) * sq);
  if (!ok) return false;
  n->cap = batch;
  return true;
}

// Launches a kernel that begins with chain_wait().
template <class... Args>
void launch_chained(void (*kernel)(Args...), dim3 grid, int threads, size_t smem, cudaStream_t st, Args... args) {
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid;
  cfg.blockDim = dim3((unsigned)threads);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  note_launches(1, st);
  cudaLaunchKernelEx(&cfg, kernel, args...);
}

void launch_gemm(const GemmArgs& g, cudaStream_t st) {
  launch_chained(gemm_bf16_kernel, dim3((g.N + TN - 1) / TN, (g.M + TM - 1) / TM), kGemmThreads, kGemmSmem, st, g);
}

// Layer l's forward product from a_in: activation and (keep) pre-activation.
GemmArgs forward_args(rf_mlp* n, int l, const float* a_in, float* out, int batch, float* z) {
  const float* P = (const float*)n->params.p;
  const int ni = n->dims[l], no = n->dims[l + 1], L = (int)n->dims.size() - 1;
  GemmArgs g = gemm_args(a_in, ni, false, P + n->w_off[l], no, false, out, no, batch, no, ni);
  g.bias = P + n->b_off[l];
  g.Z = z;
  g.vecC = g.vecC && rows16(z, no);
  g.gelu = l < L - 1;
  return g;
}

// y = net(x): each layer's activations follow the one before in acts (the
// pre-activations are not kept); the last layer writes y.
void mlp_forward(rf_mlp* n, const float* x, int batch, float* y, cudaStream_t st) {
  const int L = (int)n->dims.size() - 1;
  const float* a_in = x;
  int64_t ao = 0;
  for (int l = 0; l < L; ++l) {
    float* out = l == L - 1 ? y : (float*)n->acts.p + ao;
    GemmArgs g = forward_args(n, l, a_in, out, batch, nullptr);
    if (l == L - 1 && n->has_affine) {
      g.scale = (const float*)n->scale.p;
      g.shift = (const float*)n->shift.p;
    }
    launch_gemm(g, st);
    a_in = out;
    ao += (int64_t)batch * n->dims[l + 1];
  }
}

// Mean-squared loss against t (batch x n_out, already standardised) and its
// gradient into n->grads; the loss and the GEMMs' give-up flag into out[0..1].
// One launch per layer forward (the last one also forms the loss gradient),
// one per layer backward, one to add up the partial sums: with Adam 10 for the
// 64-128-128-128-6 network, 26 when every product, GELU', column sum and
// split had its own.  At 1024 rows a step takes 91 us, 403 before (column sums
// on one block 40-60 us each, uncoalesced operand loads 15-37 us a product).
// What is left is latency: 8-10 us a launch (launch, two trips to L2, a chain
// of MMAs, the epilogue), the products themselves under 1 us.
rf_status mlp_loss_grad(rf_mlp* n, const float* x, const float* t, int batch, float* out, cudaStream_t st) {
  const int L = (int)n->dims.size() - 1, no_last = n->dims.back();
  float* G = (float*)n->grads.p;
  const float* P = (const float*)n->params.p;
  const int64_t cnt = (int64_t)batch * no_last;
  float* d = (float*)n->dbuf.p;
  float* d2 = (float*)n->dbuf2.p;
  std::vector<const float*> a(L);  // each layer's input
  std::vector<float*> z(L);
  int64_t ao = 0, zo = 0;
  a[0] = x;
  for (int l = 0; l < L; ++l) {
    z[l] = (float*)n->zs.p + zo;
    zo += (int64_t)batch * n->dims[l + 1];
    const bool last = l == L - 1;
    float* y = last ? d : (float*)n->acts.p + ao;
    GemmArgs g = forward_args(n, l, a[l], y, batch, last ? nullptr : z[l]);
    if (last) {
      g.T = t;
      g.loss = (double*)n->sq.p;
      g.lscale = 2.0f / (float)cnt;
    } else {
      a[l + 1] = y;
      ao += (int64_t)batch * n->dims[l + 1];
    }
    launch_gemm(g, st);
  }
  ReduceArgs r{};
  int block = 0;
  float* part = (float*)n->partial.p;
  const int chunk = bias_chunk(batch), n_chunks = (batch + chunk - 1) / chunk;
  auto add = [&](float* to, int cells, int splits) {
    r.it[r.n_items++] = ReduceItem{part, to, cells, splits, block};
    block += (cells + 255) / 256;
    part += (size_t)cells * splits;
  };
  for (int l = L - 1; l >= 0; --l) {
    const int ni = n->dims[l], no = n->dims[l + 1];
    BackArgs b{};
    b.w = gemm_args(a[l], ni, true, d, no, false, G + n->w_off[l], no, ni, no, batch);
    if (b.w.splits > 1) {
      b.w.part = part;
      b.w.vecC = rows16(part, no);
      add(G + n->w_off[l], ni * no, b.w.splits);
    }
    b.n_w = gemm_tiles(b.w) * (b.w.part ? b.w.splits : 1);
    if (l > 0) {  // dZ of the layer below: (dZ W^T) GELU'(Z)
      b.in = gemm_args(d, no, false, P + n->w_off[l], no, true, d2, ni, batch, ni, no);
      b.in.Zg = z[l - 1];
      b.in.vecZ = rows16(z[l - 1], ni);
      b.n_in = gemm_tiles(b.in);
    }
    b.dZ = d;
    b.db = part;
    b.rows = batch;
    b.cols = no;
    b.chunk = chunk;
    add(G + n->b_off[l], no, n_chunks);
    launch_chained(backward_kernel, dim3(b.n_in + b.n_w + (no + 31) / 32 * n_chunks), kGemmThreads, kGemmSmem, st, b);
    std::swap(d, d2);
  }
  r.loss = (const double*)n->sq.p;
  r.n_loss = ((batch + TM - 1) / TM) * ((no_last + TN - 1) / TN);
  r.n = (double)cnt;
  r.out = out;
  launch_chained(reduce_kernel, dim3(block + 1), 256, 0, st, r);
  return cuda_ok(cudaGetLastError(), "mlp launch") ? RF_OK : RF_E_CUDA;
}

void mlp_adam(rf_mlp* n, float lr, cudaStream_t st) {
  ++n->step;
  const float b1 = 0.9f, b2 = 0.999f;
  const float c1 = 1.f - powf(b1, (float)n->step), c2 = 1.f - powf(b2, (float)n->step);
  launch_chained(adam_kernel, dim3(blocks_for(n->n_params, 256)), 256, 0, st, (float*)n->params.p,
                 (const float*)n->grads.p, (float*)n->m.p, (float*)n->v.p, n->n_params, lr, b1, b2, 1e-8f, c1, c2);
}

}  // namespace
}  // namespace rf

extern "C" {

rf_status rf_mlp_create(int32_t n_in, int32_t n_hidden, int32_t n_hidden_layers, int32_t n_out, uint64_t seed,
                        rf_mlp** out) {
  if (!out || n_in < 1 || n_hidden < 1 || n_hidden_layers < 0 || n_out < 1 || n_in > 4096 || n_hidden > 4096 ||
      n_out > 4096 || n_hidden_layers > 16) {
    set_error("rf_mlp_create: bad dimensions");
    return RF_E_INVALID;
  }
  rf_mlp* n = new (std::nothrow) rf_mlp();
  if (!n) return RF_E_OOM;
  n->dims.push_back(n_in);
  for (int i = 0; i < n_hidden_layers; ++i) n->dims.push_back(n_hidden);
  n->dims.push_back(n_out);
  int64_t off = 0;
  for (size_t l = 0; l + 1 < n->dims.size(); ++l) {
    n->w_off.push_back(off);
    off += (int64_t)n->dims[l] * n->dims[l + 1];
    n->b_off.push_back(off);
    off += n->dims[l + 1];
  }
  n->n_params = off;
  // Uniform(-1/sqrt(fan_in), 1/sqrt(fan_in)) weights, zero biases, from a seeded mt19937_64.
  std::vector<float> h(off, 0.f);
  std::mt19937_64 rng(seed);
  std::uniform_real_distribution<double> U(-1.0, 1.0);
  for (size_t l = 0; l + 1 < n->dims.size(); ++l) {
    const double bound = 1.0 / std::sqrt((double)n->dims[l]);
    for (int64_t i = 0; i < (int64_t)n->dims[l] * n->dims[l + 1]; ++i) h[n->w_off[l] + i] = (float)(bound * U(rng));
  }
  std::vector<float> zeros(off, 0.f);
  if (!n->params.ensure(sizeof(float) * off) || !n->grads.ensure(sizeof(float) * off) ||
      !n->m.ensure(sizeof(float) * off) || !n->v.ensure(sizeof(float) * off) ||
      !n->scale.ensure(sizeof(float) * n_out) || !n->shift.ensure(sizeof(float) * n_out) ||
      !n->mean.ensure(sizeof(float) * n_out) || !n->sd.ensure(sizeof(float) * n_out)) {
    delete n;
    return RF_E_OOM;
  }
  if (!cuda_ok(cudaMemcpy(n->params.p, h.data(), sizeof(float) * off, cudaMemcpyHostToDevice), "mlp init") ||
      !cuda_ok(cudaMemcpy(n->m.p, zeros.data(), sizeof(float) * off, cudaMemcpyHostToDevice), "mlp init") ||
      !cuda_ok(cudaMemcpy(n->v.p, zeros.data(), sizeof(float) * off, cudaMemcpyHostToDevice), "mlp init") ||
      !cuda_ok(cudaMemcpy(n->grads.p, zeros.data(), sizeof(float) * off, cudaMemcpyHostToDevice), "mlp init")) {
    delete n;
    return RF_E_CUDA;
  }
  *out = n;
  return RF_OK;
}

void rf_mlp_destroy(rf_mlp* n) { delete n; }

int64_t rf_mlp_n_params(const rf_mlp* n) { return n ? n->n_params : 0; }

rf_status rf_mlp_get_params(const rf_mlp* n, float* host) {
  if (!n || !host) { set_error("rf_mlp_get_params: bad argument"); return RF_E_INVALID; }
  return cuda_ok(cudaMemcpy(host, n->params.p, sizeof(float) * n->n_params, cudaMemcpyDeviceToHost), "mlp params")
             ? RF_OK : RF_E_CUDA;
}

rf_status rf_mlp_set_params(rf_mlp* n, const float* host) {
  if (!n || !host) { set_error("rf_mlp_set_params: bad argument"); return RF_E_INVALID; }
  return cuda_ok(cudaMemcpy(n->params.p, host, sizeof(float) * n->n_params, cudaMemcpyHostToDevice), "mlp params")
             ? RF_OK : RF_E_CUDA;
}

rf_status rf_mlp_forward(rf_mlp* n, const float* d_x, int32_t batch, float* d_y, void* stream) {
  if (!n || !d_x || !d_y || batch < 0) { set_error("rf_mlp_forward: bad argument"); return RF_E_INVALID; }
  if (batch == 0) return RF_OK;
  if (!mlp_reserve(n, batch)) return RF_E_OOM;
  cudaStream_t st = (cudaStream_t)stream;
  if (n->dims.size() == 2) {  // one layer: y may be x itself, so not written while x is read
    mlp_forward(n, d_x, batch, (float*)n->y.p, st);
    cudaMemcpyAsync(d_y, n->y.p, sizeof(float) * (size_t)batch * n->dims.back(), cudaMemcpyDeviceToDevice, st);
  } else {
    mlp_forward(n, d_x, batch, d_y, st);
  }
  return cuda_ok(cudaGetLastError(), "rf_mlp_forward") ? RF_OK : RF_E_CUDA;
}

rf_status rf_mlp_grad(rf_mlp* n, const float* d_x, const float* d_t, int32_t batch, float* loss, float* d_grad,
                      void* stream) {
  if (!n || !d_x || !d_t || batch < 1) { set_error("rf_mlp_grad: bad argument"); return RF_E_INVALID; }
  if (!mlp_reserve(n, batch)) return RF_E_OOM;
  cudaStream_t st = (cudaStream_t)stream;
  rf_status s = mlp_loss_grad(n, d_x, d_t, batch, (float*)n->loss.p, st);
  if (s != RF_OK) return s;
  if (d_grad) cudaMemcpyAsync(d_grad, n->grads.p, sizeof(float) * n->n_params, cudaMemcpyDeviceToDevice, st);
  if (loss) {
    const float* h = (const float*)n->h_loss.p;
    if (!cuda_ok(cudaMemcpyAsync(n->h_loss.p, n->loss.p, 2 * sizeof(float), cudaMemcpyDeviceToHost, st), "loss") ||
        !cuda_ok(cudaStreamSynchronize(st), "loss"))
      return RF_E_CUDA;
    *loss = h[0];
    int flag;
    std::memcpy(&flag, h + 1, sizeof flag);
    if (flag) return gemm_status("rf_mlp_grad");
  }
  return RF_OK;
}

rf_status rf_mlp_adam(rf_mlp* n, float lr, void* stream) {
  if (!n || !(lr >= 0.f)) { set_error("rf_mlp_adam: bad argument"); return RF_E_INVALID; }
  mlp_adam(n, lr, (cudaStream_t)stream);
  return cuda_ok(cudaGetLastError(), "rf_mlp_adam") ? RF_OK : RF_E_CUDA;
}

rf_status rf_mlp_train(rf_mlp* n, const float* d_x, const float* d_t, int32_t rows, int32_t batch, int32_t epochs,
                       float lr, uint64_t seed, int32_t standardise, float* final_loss) {
  if (!n || !d_x || !d_t || rows < 1 || batch < 1 || epochs < 1 || !(lr > 0.f)) {
    set_error("rf_mlp_train: bad argument");
    return RF_E_INVALID;
  }
  batch = std::min(batch, rows);
  if (!mlp_reserve(n, batch)) return RF_E_OOM;
  const int ni = n->dims[0], no = n->dims.back();
  DevBuf tstd;
  const float* targets = d_t;
  if (standardise) {
    if (!tstd.ensure(sizeof(float) * (size_t)rows * no)) return RF_E_OOM;
    note_launches(1, nullptr);
    col_stats_kernel<<<1, 128>>>(d_t, rows, no, (float*)n->mean.p, (float*)n->sd.p);
    note_launches(1, nullptr);
    standardise_kernel<<<blocks_for((int64_t)rows * no, 256), 256>>>(d_t, rows, no, (const float*)n->mean.p,
                                                                    (const float*)n->sd.p, (float*)tstd.p);
    targets = (const float*)tstd.p;
    cudaMemcpy(n->scale.p, n->sd.p, sizeof(float) * no, cudaMemcpyDeviceToDevice);
    cudaMemcpy(n->shift.p, n->mean.p, sizeof(float) * no, cudaMemcpyDeviceToDevice);
    n->has_affine = true;
  }
  std::mt19937_64 rng(seed);
  std::vector<int32_t> perm(rows);
  for (int i = 0; i < rows; ++i) perm[i] = i;
  DevBuf dperm, dloss;
  const int steps_per_epoch = rows / batch;  // drop the ragged remainder
  const int64_t total = (int64_t)steps_per_epoch * epochs;
  int64_t it = 0;
  double last_epoch = 0.0;
  if (!dperm.ensure(sizeof(int32_t) * rows) || !dloss.ensure(2 * sizeof(float) * steps_per_epoch)) return RF_E_OOM;
  std::vector<float> losses(2 * steps_per_epoch);  // per step: loss, flag
  for (int e = 0; e < epochs; ++e) {
    std::shuffle(perm.begin(), perm.end(), rng);
    if (!cuda_ok(cudaMemcpy(dperm.p, perm.data(), sizeof(int32_t) * rows, cudaMemcpyHostToDevice), "perm"))
      return RF_E_CUDA;
    double sum = 0.0;
    for (int s = 0; s < steps_per_epoch; ++s, ++it) {
      const int32_t* ids = (const int32_t*)dperm.p + (size_t)s * batch;
      note_launches(1, nullptr);
      gather_rows_kernel<<<blocks_for((int64_t)batch * (ni + no), 256), 256>>>(d_x, targets, ids, batch, ni, no,
                                                                              (float*)n->xb.p, (float*)n->tb.p);
      rf_status st = mlp_loss_grad(n, (const float*)n->xb.p, (const float*)n->tb.p, batch, (float*)dloss.p + 2 * s, 0);
      if (st != RF_OK) return st;
      // cosine decay from lr to 0 over all steps
      const float lr_t = (float)(0.5 * lr * (1.0 + std::cos(M_PI * (double)it / (double)total)));
      mlp_adam(n, lr_t, 0);
    }
    if (!cuda_ok(cudaMemcpy(losses.data(), dloss.p, sizeof(float) * losses.size(), cudaMemcpyDeviceToHost), "rf_mlp_train"))
      return RF_E_CUDA;
    const rf_status gs = gemm_status("rf_mlp_train");
    if (gs != RF_OK) return gs;
    for (int s = 0; s < steps_per_epoch; ++s) sum += losses[2 * s];
    last_epoch = steps_per_epoch > 0 ? sum / steps_per_epoch : 0.0;
  }
  if (final_loss) *final_loss = (float)last_epoch;
  return RF_OK;
}

rf_status rf_mlp_save(const rf_mlp* n, const char* path) {
  if (!n || !path) { set_error("rf_mlp_save: bad argument"); return RF_E_INVALID; }
  const int no = n->dims.back();
  std::vector<float> p(n->n_params), m(n->n_params), v(n->n_params), sc(no), sh(no);
  cudaMemcpy(p.data(), n->params.p, sizeof(float) * n->n_params, cudaMemcpyDeviceToHost);
  cudaMemcpy(m.data(), n->m.p, sizeof(float) * n->n_params, cudaMemcpyDeviceToHost);
  cudaMemcpy(v.data(), n->v.p, sizeof(float) * n->n_params, cudaMemcpyDeviceToHost);
  cudaMemcpy(sc.data(), n->scale.p, sizeof(float) * no, cudaMemcpyDeviceToHost);
  cudaMemcpy(sh.data(), n->shift.p, sizeof(float) * no, cudaMemcpyDeviceToHost);
  if (!cuda_ok(cudaGetLastError(), "rf_mlp_save")) return RF_E_CUDA;
  FILE* f = std::fopen(path, "wb");
  if (!f) { set_error("rf_mlp_save: cannot open file"); return RF_E_INVALID; }
  const int32_t magic = 0x524d4c50, nd = (int32_t)n->dims.size(), aff = n->has_affine ? 1 : 0;
  std::fwrite(&magic, 4, 1, f);
  std::fwrite(&nd, 4, 1, f);
  std::fwrite(n->dims.data(), 4, nd, f);
  std::fwrite(&n->step, 8, 1, f);
  std::fwrite(&aff, 4, 1, f);
  std::fwrite(p.data(), 4, n->n_params, f);
  std::fwrite(m.data(), 4, n->n_params, f);
  std::fwrite(v.data(), 4, n->n_params, f);
  std::fwrite(sc.data(), 4, no, f);
  std::fwrite(sh.data(), 4, no, f);
  const bool ok = std::fclose(f) == 0;
  if (!ok) { set_error("rf_mlp_save: write failed"); return RF_E_INVALID; }
  return RF_OK;
}

rf_status rf_mlp_load(const char* path, rf_mlp** out) {
  if (!path || !out) { set_error("rf_mlp_load: bad argument"); return RF_E_INVALID; }
  *out = nullptr;
  FILE* f = std::fopen(path, "rb");
  if (!f) { set_error("rf_mlp_load: cannot open file"); return RF_E_INVALID; }
  int32_t magic = 0, nd = 0;
  bool ok = std::fread(&magic, 4, 1, f) == 1 && magic == 0x524d4c50 && std::fread(&nd, 4, 1, f) == 1 && nd >= 2 && nd <= 18;
  std::vector<int32_t> dims(ok ? nd : 0);
  ok = ok && std::fread(dims.data(), 4, nd, f) == (size_t)nd;
  if (!ok || dims[1] < 1) {
    std::fclose(f);
    set_error("rf_mlp_load: not a model file");
    return RF_E_INVALID;
  }
  rf_mlp* n = nullptr;
  rf_status s = rf_mlp_create(dims[0], nd > 2 ? dims[1] : 1, nd - 2, dims[nd - 1], 0, &n);
  if (s != RF_OK) {
    std::fclose(f);
    return s;
  }
  int32_t aff = 0;
  const int no = dims[nd - 1];
  std::vector<float> p(n->n_params), m(n->n_params), v(n->n_params), sc(no), sh(no);
  ok = std::fread(&n->step, 8, 1, f) == 1 && std::fread(&aff, 4, 1, f) == 1 &&
       std::fread(p.data(), 4, n->n_params, f) == (size_t)n->n_params &&
       std::fread(m.data(), 4, n->n_params, f) == (size_t)n->n_params &&
       std::fread(v.data(), 4, n->n_params, f) == (size_t)n->n_params && std::fread(sc.data(), 4, no, f) == (size_t)no &&
       std::fread(sh.data(), 4, no, f) == (size_t)no;
  std::fclose(f);
  if (!ok) {
    delete n;
    set_error("rf_mlp_load: truncated file");
    return RF_E_INVALID;
  }
  n->has_affine = aff != 0;
  cudaMemcpy(n->params.p, p.data(), sizeof(float) * n->n_params, cudaMemcpyHostToDevice);
  cudaMemcpy(n->m.p, m.data(), sizeof(float) * n->n_params, cudaMemcpyHostToDevice);
  cudaMemcpy(n->v.p, v.data(), sizeof(float) * n->n_params, cudaMemcpyHostToDevice);
  cudaMemcpy(n->scale.p, sc.data(), sizeof(float) * no, cudaMemcpyHostToDevice);
  cudaMemcpy(n->shift.p, sh.data(), sizeof(float) * no, cudaMemcpyHostToDevice);
  if (!cuda_ok(cudaGetLastError(), "rf_mlp_load")) {
    delete n;
    return RF_E_CUDA;
  }
  *out = n;
  return RF_OK;
}

}  // extern "C"

extern "C" rf_status rf_mlp_predict(rf_mlp* n, const rf_model* m, const rf_data* d, int32_t col, double* theta0) {
  if (!n || !m || !d || !theta0) {
    set_error("rf_mlp_predict: bad argument (NULL)");
    return RF_E_INVALID;
  }
  const int S = rf_data_n_sets(d), no = n->dims.back();
  if (n->dims.front() != 64 || no != rf_model_n_free(m)) {
    set_error("rf_mlp_predict: the network must map 64 histogram bins to the model's free parameters");
    return RF_E_INVALID;
  }
  if (S == 0) return RF_OK;
  if (!n->pred_h.ensure(sizeof(float) * (size_t)S * 64) || !n->pred_y.ensure(sizeof(float) * (size_t)S * no))
    return RF_E_OOM;
  rf_status st = rf_hist64(m, d, col, (float*)n->pred_h.p, nullptr);
  if (st != RF_OK) return st;
  st = rf_mlp_forward(n, (const float*)n->pred_h.p, S, (float*)n->pred_y.p, nullptr);
  if (st != RF_OK) return st;
  std::vector<float> y((size_t)S * no);
  if (!cuda_ok(cudaMemcpy(y.data(), n->pred_y.p, sizeof(float) * y.size(), cudaMemcpyDeviceToHost), "rf_mlp_predict"))
    return RF_E_CUDA;
  st = gemm_status("rf_mlp_predict");
  if (st != RF_OK) return st;
  // A start on (or beyond) a bound sits where the fit's bound transform is
  // stationary (d theta / d phi = 0): that parameter barely moves.  Bounded
  // predictions are kept kStartMargin of the range inside the bounds.
  const std::vector<double>& lo = m->m.lo;
  const std::vector<double>& hi = m->m.hi;
  for (int s = 0; s < S; ++s)
    for (int k = 0; k < no; ++k) {
      double t = (double)y[(size_t)s * no + k];
      if (lo[k] < hi[k] && std::isfinite(lo[k]) && std::isfinite(hi[k])) {
        const double a = lo[k] + kStartMargin * (hi[k] - lo[k]), b = hi[k] - kStartMargin * (hi[k] - lo[k]);
        t = t < a ? a : (t > b ? b : t);
      }
      theta0[(size_t)s * no + k] = t;
    }
  return RF_OK;
}
