// Learned surrogate for l(t): ensemble MLP trained and evaluated by hand-written
// kernels (include/lb_mlp.h).
//
// Contractions: C = A B on tensor cores, mma.sync m16n8k16 with BF16 operands
// and FP32 accumulation over K in steps of 16, from K = 0 upwards (every kernel
// below keeps this order, so all of them give the same bits).  A 64x64 tile per CTA
// (4 warps of 32x32); the operands come through a ring of cp.async stages of 64 K
// values in 128-byte swizzled rows and leave it by ldmatrix, transposed where the
// backward pass contracts over the rows of an array, so no operand is copied.
// The weight gradients contract over the batch (K up to max_batch rows) into
// small outputs: they split K over CTAs, and the kernel that uses the gradient
// adds the FP32 partials in a fixed order (split-K, deterministic).
// Epilogues fuse the bias and tanh (forward), the loss and its derivative, the
// tanh derivative (backward) and the BF16 rounding of activations.  Ensemble
// members run in the z dimension of every launch.  Sixteen training iterations
// (forward, loss, backward, AdamW) are captured once as a CUDA graph and replayed.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdarg.h>
#include <stdint.h>
#include <stdio.h>
#include <string.h>

#include <new>
#include <utility>
#include <vector>

#include "lb_host.h"
#include "lb_mlp.h"

namespace {

typedef __nv_bfloat16 bf16;

constexpr int TM = 64, TN = 64, TK = 64;  // CTA tile; K values per stage
constexpr int kGemmThreads = 128;
constexpr int kStages = 3;
constexpr int kTileBytes = TM * TK * 2;  // one operand of one stage (TM == TN)
constexpr int kGemmSmem = kStages * 2 * kTileBytes;  // 48 KB: no opt-in, four CTAs per SM
constexpr int kWgradStages = 6;     // the weight gradients' long K: 96 KB in flight, two CTAs per SM
constexpr int kWgradThreads = 128;  // four warps of 32x32 (eight of 32x16: 38 instead of 33 us)
constexpr int kWgradSmem = kWgradStages * 2 * kTileBytes;
constexpr int kGraphSteps = 16;  // training steps per captured graph: the gap between graphs is 3 us (88 -> 85 us a step)
constexpr int kParts = 4;  // of a large prediction
constexpr int kBiasGroups = 8;  // partial sums of a bias gradient (32 row classes each)

enum { EPI_BIAS_F32 = 0, EPI_BIAS_TANH = 1, EPI_LOSS = 2, EPI_DTANH = 3 };

// C (M x N) = A B over K rows [kb, ke).  Non-transposed operands hold K contiguous
// (A[m][k], B[n][k]), transposed ones hold the other index contiguous (A[k][m],
// B[k][n]); ld: elements per row, a multiple of 8, rows starting on 16 bytes.
struct GemmArgs {
  int M, N, K;
  const bf16* A;
  long lda, a_mem;
  const bf16* B;
  long ldb, b_mem;
  int b_cols;  // transposed B: stored columns (>= N, a multiple of 8)
  const float* bias;
  long bias_mem;
  float* Cf;   // FP32 output, if any
  long ldcf, cf_mem;
  bf16* Cb;    // BF16 output, if any
  long ldcb, cb_mem;
  const bf16* H;  // activation whose tanh derivative multiplies (EPI_DTANH)
  long ldh, h_mem;
  const float* T;  // targets (EPI_LOSS) and the loss of every member
  float* loss;
  float scale;     // EPI_LOSS: 1 / (n n_out)
};

__device__ __forceinline__ uint32_t pack2(bf16 lo, bf16 hi) {
  return (uint32_t)__bfloat16_as_ushort(lo) | ((uint32_t)__bfloat16_as_ushort(hi) << 16);
}

__device__ __forceinline__ uint32_t pack2f(float lo, float hi) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(lo, hi);
  return *reinterpret_cast<const uint32_t*>(&v);
}

__device__ __forceinline__ void mma_bf16(float c[4], const uint32_t a[4], const uint32_t b[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// The kernels of a training step and of a prediction follow one another with programmatic
// stream serialisation: the next one's CTAs may start while the last ones of this one
// drain, and wait here before they touch memory.
__device__ __forceinline__ void pdl_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void pdl_trigger() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

template <bool TRANS>
__device__ __forceinline__ void ldmatrix4(uint32_t r[4], uint32_t addr) {
  if constexpr (TRANS)
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
  else
    asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
                 : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
                 : "r"(addr)
                 : "memory");
}

// 16 bytes global -> shared, zeros when !ok (nothing is then read, wherever src points)
__device__ __forceinline__ void cp16(uint32_t dst, const void* src, bool ok) {
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(dst), "l"(src), "r"(ok ? 16 : 0) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}

// Byte offset of 16-byte chunk c of row r in a stage of 128-byte rows: the chunks
// of a row are permuted by its low three bits, so that the eight rows one ldmatrix
// phase reads lie in different banks.
__device__ __forceinline__ uint32_t swz(int r, int c) { return (uint32_t)(r * 128 + ((c ^ (r & 7)) << 4)); }

// One operand of the ring: 64 x 64 values a stage, 16-byte chunks of 128 threads (rows
// tid / 8 + 16 i, chunk tid % 8).  Not transposed: rows are the output index (from r0,
// below rmax), columns K (a multiple of 8 ends the array).  Transposed: rows K, columns
// the output index.  What a thread can know beforehand is kept here.
template <bool TRANS>
struct Operand {
  static constexpr int kRows = 16, kChunks = 64 / kRows;
  const bf16* p;   // this thread's first chunk of the next stage
  long step, row;  // elements to the next stage, and to the thread's next row
  uint32_t dst;    // its place in a stage
  int k;           // K index of the first chunk
  unsigned in;     // bit i: chunk i's output index is inside
  __device__ __forceinline__ Operand(const bf16* X, long ld, int r0, int rmax, int kb) {
    const int r = threadIdx.x >> 3, c = threadIdx.x & 7;
    dst = swz(r, c);
    row = kRows * ld;
    in = 0;
    if constexpr (TRANS) {
      k = kb + r;
      p = X + (long)k * ld + r0 + 8 * c;
      step = TK * ld;
      if (r0 + 8 * c < rmax) in = 15u;
    } else {
      k = kb + 8 * c;
      p = X + (long)(r0 + r) * ld + k;
      step = TK;
#pragma unroll
      for (int i = 0; i < kChunks; ++i) in |= r0 + r + kRows * i < rmax ? 1u << i : 0u;
    }
  }
  __device__ __forceinline__ void stage(uint32_t base, int ke) {
#pragma unroll
    for (int i = 0; i < kChunks; ++i) {
      cp16(base + dst + i * kRows * 128, p + i * row, (TRANS ? k + kRows * i < ke : k < ke) && (in >> i & 1u));
    }
    p += step;
    k += TK;
  }
};

// The 64x64 tile (m0, n0) of member mem, K rows [kb, ke), in the accumulators of four
// warps (warp w: rows from 32 (w / 2), columns from 32 (w % 2)).  SPLIT: every kc rows the
// accumulators are added to a running sum and start again from zero (kc a multiple of
// 16 unless it covers the range).
template <bool TA, bool TB, int ST = kStages, bool SPLIT = false>
__device__ __forceinline__ void gemm_tile(const bf16* A, long lda, int M, const bf16* B, long ldb, int bmax, int m0,
                                          int n0, int kb, int ke, unsigned char* smem, float acc[2][4][4],
                                          int kc = 0) {
  constexpr int NI = 4;  // fragments of 8 columns per warp
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wm = (warp / 2) * 32, wn = (warp % 2) * 32;
  const uint32_t sb = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < NI; ++j)
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[i][j][k] = 0.0f;
  const int nk = (ke - kb + TK - 1) / TK;
  Operand<TA> oa(A, lda, m0, M, kb);
  Operand<TB> ob(B, ldb, n0, bmax, kb);
  uint32_t wr = sb, rd = sb;  // the stages written and read next
  auto load = [&](int c) {
    if (c < nk) {
      oa.stage(wr, ke);
      ob.stage(wr + kTileBytes, ke);
      wr = wr == sb + (ST - 1) * 2 * kTileBytes ? sb : wr + 2 * kTileBytes;
    }
    cp_commit();
  };
#pragma unroll
  for (int c = 0; c < ST - (SPLIT ? 2 : 1); ++c) load(c);
  const int l8 = lane & 7, li = lane >> 3;
  [[maybe_unused]] float run[2][NI][4];
  [[maybe_unused]] int next = kc;  // rows after which the running sum takes the accumulators
  if constexpr (SPLIT) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < NI; ++j)
#pragma unroll
        for (int k = 0; k < 4; ++k) run[i][j][k] = 0.0f;
  }
  // chunks per barrier: two where the ring is deep (SPLIT)
  constexpr int PER = SPLIT ? 2 : 1;
  for (int c = 0; c < nk; ++c) {
    if (PER == 1 || c % PER == 0) {
      cp_wait<ST - 2 * PER>();
      __syncthreads();
#pragma unroll
      for (int p = 0; p < PER; ++p) load(c + ST - PER + p);
    }
    const uint32_t sa = rd, sbb = rd + kTileBytes;
    rd = rd == sb + (ST - 1) * 2 * kTileBytes ? sb : rd + 2 * kTileBytes;
    const int steps = min((ke - kb - c * TK + 15) / 16, TK / 16);
    uint32_t a[2][2][4], b[2][NI / 2][4];
    auto frags = [&](int ks, int u) {
#pragma unroll
      for (int mi = 0; mi < 2; ++mi) {
        if constexpr (TA)
          ldmatrix4<true>(a[u][mi], sa + swz(ks * 16 + (li >> 1) * 8 + l8, ((wm + mi * 16) >> 3) + (li & 1)));
        else
          ldmatrix4<false>(a[u][mi], sa + swz(wm + mi * 16 + (li & 1) * 8 + l8, ks * 2 + (li >> 1)));
      }
#pragma unroll
      for (int nj = 0; nj < NI / 2; ++nj) {
        if constexpr (TB)
          ldmatrix4<true>(b[u][nj], sbb + swz(ks * 16 + (li & 1) * 8 + l8, ((wn + nj * 16) >> 3) + (li >> 1)));
        else
          ldmatrix4<false>(b[u][nj], sbb + swz(wn + nj * 16 + (li >> 1) * 8 + l8, ks * 2 + (li & 1)));
      }
    };
    frags(0, 0);
#pragma unroll
    for (int ks = 0; ks < TK / 16; ++ks) {
      if (ks >= steps) break;
      if constexpr (SPLIT) {
        if (c * TK + ks * 16 == next) {
          next += kc;
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int j = 0; j < NI; ++j)
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                run[i][j][k] += acc[i][j][k];
                acc[i][j][k] = 0.0f;
              }
        }
      }
      if (ks + 1 < TK / 16) frags(ks + 1, (ks + 1) & 1);  // the next step's, while this one multiplies
#pragma unroll
      for (int mi = 0; mi < 2; ++mi)
#pragma unroll
        for (int ni = 0; ni < NI; ++ni)
          mma_bf16(acc[mi][ni], a[ks & 1][mi], &b[ks & 1][ni >> 1][(ni & 1) * 2]);
    }
  }
  cp_wait<0>();
  if constexpr (SPLIT) {
#pragma unroll
    for (int i = 0; i < 2; ++i)
#pragma unroll
      for (int j = 0; j < NI; ++j)
#pragma unroll
        for (int k = 0; k < 4; ++k) acc[i][j][k] = run[i][j][k] + acc[i][j][k];
  }
}

// Store of the accumulators: f(m, n, v0, v1) for every pair of neighbouring columns
// n, n + 1 inside the output (N is even, so a pair is inside as a whole).
template <class F>
__device__ __forceinline__ void for_pairs(const float acc[2][4][4], int m0, int n0, int M, int N, F f) {
  constexpr int NI = 4;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wm = (warp / 2) * 32, wn = (warp % 2) * 32;
  const int gq = lane >> 2, tq = lane & 3;
#pragma unroll
  for (int mi = 0; mi < 2; ++mi)
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int m = m0 + wm + mi * 16 + gq + h * 8;
      if (m >= M) continue;
#pragma unroll
      for (int ni = 0; ni < NI; ++ni) {
        const int n = n0 + wn + ni * 8 + 2 * tq;
        if (n < N) f(m, n, acc[mi][ni][2 * h], acc[mi][ni][2 * h + 1]);
      }
    }
}

// Block sum of one value per thread, added to *out by thread 0 (sh: shared memory
// that nothing else uses any more).
__device__ __forceinline__ void block_add(float v, float scale, float* out, float* sh) {
  __syncthreads();
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  if (threadIdx.x == 0) {
    float s = 0.0f;
    for (int w = 0; w < kGemmThreads / 32; ++w) s += sh[w];
    atomicAdd(out, s * scale);
  }
}

// Layers two and three and the backward products: grid (N tiles, M tiles, members).
template <int EPI, bool TB>
__global__ void __launch_bounds__(kGemmThreads) gemm_kernel(GemmArgs g) {
  extern __shared__ __align__(128) unsigned char smem[];
  const int mem = blockIdx.z, m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
  float acc[2][4][4];
  gemm_tile<false, TB>(g.A + mem * g.a_mem, g.lda, g.M, g.B + mem * g.b_mem, g.ldb, TB ? g.b_cols : g.N, m0, n0, 0,
                       g.K, smem, acc);
  float* Cf = g.Cf ? g.Cf + mem * g.cf_mem : nullptr;
  bf16* Cb = g.Cb ? g.Cb + mem * g.cb_mem : nullptr;
  float sum = 0.0f;
  for_pairs(acc, m0, n0, g.M, g.N, [&](int m, int n, float v0, float v1) {
    if constexpr (EPI == EPI_BIAS_F32 || EPI == EPI_BIAS_TANH || EPI == EPI_LOSS) {
      const float2 b = *reinterpret_cast<const float2*>(g.bias + mem * g.bias_mem + n);
      v0 += b.x;
      v1 += b.y;
    }
    if constexpr (EPI == EPI_BIAS_TANH) {
      v0 = tanhf(v0);
      v1 = tanhf(v1);
    }
    if constexpr (EPI == EPI_LOSS) {
      // dY = 2 (Y - T) / (n n_out), and this tile's share of the loss
      const float2 t = *reinterpret_cast<const float2*>(g.T + (long)m * g.N + n);
      const float d0 = v0 - t.x, d1 = v1 - t.y;
      sum += d0 * d0;
      sum += d1 * d1;
      v0 = 2.0f * d0 * g.scale;
      v1 = 2.0f * d1 * g.scale;
    }
    if constexpr (EPI == EPI_DTANH) {
      const __nv_bfloat162 h = *reinterpret_cast<const __nv_bfloat162*>(g.H + mem * g.h_mem + (long)m * g.ldh + n);
      const float h0 = __bfloat162float(h.x), h1 = __bfloat162float(h.y);
      v0 *= 1.0f - h0 * h0;
      v1 *= 1.0f - h1 * h1;
    }
    if (Cf) *reinterpret_cast<float2*>(Cf + (long)m * g.ldcf + n) = make_float2(v0, v1);
    if (Cb)
      *reinterpret_cast<uint32_t*>(Cb + (long)m * g.ldcb + n) = pack2f(v0, v1);
  });
  if constexpr (EPI == EPI_LOSS) block_add(sum, g.scale, g.loss + mem, reinterpret_cast<float*>(smem));
}

// Layer one: K = n_in <= 16 is one step of the tensor core, so the operands go
// straight from global memory to registers (x is padded to 16 columns).
__global__ void __launch_bounds__(kGemmThreads) layer1_kernel(const bf16* x, const bf16* w, long w_mem, const float* bias,
                                                             long bias_mem, int n, int nin, int nh, bf16* h1,
                                                             long h_mem) {
  const int mem = blockIdx.z, m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
  const int gq = lane >> 2, tq = lane & 3;
  const bf16 zero = __float2bfloat16(0.0f);
  const bf16* W = w + mem * w_mem;
  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int k = 0; k < 4; ++k) acc[i][j][k] = 0.0f;
  uint32_t a[2][4], b[4][2];
#pragma unroll
  for (int mi = 0; mi < 2; ++mi)
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      const int m = m0 + wm + mi * 16 + gq + (q & 1) * 8;
      a[mi][q] = m < n ? *reinterpret_cast<const uint32_t*>(x + (long)m * 16 + 2 * tq + (q >> 1) * 8) : 0u;
    }
#pragma unroll
  for (int ni = 0; ni < 4; ++ni)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int c = n0 + wn + ni * 8 + gq, k = 2 * tq + q * 8;
      b[ni][q] = pack2(k < nin ? W[(long)c * nin + k] : zero, k + 1 < nin ? W[(long)c * nin + k + 1] : zero);
    }
#pragma unroll
  for (int mi = 0; mi < 2; ++mi)
#pragma unroll
    for (int ni = 0; ni < 4; ++ni) mma_bf16(acc[mi][ni], a[mi], b[ni]);
  bf16* H = h1 + mem * h_mem;
  for_pairs(acc, m0, n0, n, nh, [&](int m, int c, float v0, float v1) {
    const float2 bb = *reinterpret_cast<const float2*>(bias + mem * bias_mem + c);
    v0 = tanhf(v0 + bb.x);
    v1 = tanhf(v1 + bb.y);
    *reinterpret_cast<uint32_t*>(H + (long)m * nh + c) = pack2f(v0, v1);
  });
}

// ------------------------------------------------------------ fused row tiles
//
// Networks whose second weight matrix fits in shared memory (n_hidden <= 256): one
// kernel takes a tile of 16 RT rows through all three layers and, when training,
// through the loss and the backward products down to dZ1.  W2 and W3 stay in shared
// memory while a CTA walks the tiles of a member (one CTA per SM, the tiles of all
// members cut into equal runs), activations and upstream gradients never leave it
// between layers, and what the weight gradients need goes to global memory as bulk
// copies of whole rows behind the tensor-core work.  Against one GEMM launch per
// product this saves the launches, the reloading of weights and activations per tile
// and most of the address arithmetic; the tensor-core instructions and their order
// along K are the same, so the results are too.  A warp takes all rows of the tile and
// n_hidden / 8 columns, so that a weight fragment read from shared memory (whose
// bandwidth is the bound) serves three products.  Rows of shared memory are padded by
// 16 bytes: the eight rows of one ldmatrix phase then lie in different banks.
// 4096 rows x 5 members, n_hidden 256, n_out 64: 42 us for the forward pass, the loss
// and the backward products, against 88 us as five launches of the GEMM kernel above
// (which takes the wider networks).  The tensor pipe is active a quarter of the time;
// the rest is the FP32 gradients' stores, the tanh and the barriers between layers.
struct RowsArgs {
  int n, nin, nout, members;
  const bf16* xb;    // packed inputs [n][16] (training)
  const float* xf;   // inputs [n][n_in] (prediction)
  const float* p;
  const bf16* pb;
  long P, ob1, ow2, ob2, ow3, ob3;
  long B;            // rows between members in the activations
  float* y;          // prediction
  bf16 *h1, *h2, *dyb, *dz2b, *dz1b;
  float *dyf, *dz2f, *dz1f;
  const float* T;
  float* loss;
  float scale;
};

constexpr int kRowThreads = 256;  // eight warps (sixteen of half the columns: 49 instead of 46 us)

// Shared memory of a row-tile CTA in bytes (o16: n_out rounded up to 16).
constexpr size_t rows_smem(int nh, int nout, int rt, bool train) {
  const size_t o16 = (nout + 15) / 16 * 16, ph = 2 * nh + 16;
  return (nh + o16) * ph + 2 * 16 * rt * ph + (train ? 16 * rt * (2 * o16 + 16) : 0) + 64;
}

__device__ __forceinline__ void ldmatrix2(uint32_t r[2], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.shared.b16 {%0,%1}, [%2];" : "=r"(r[0]), "=r"(r[1]) : "r"(addr) : "memory");
}
__device__ __forceinline__ void ldmatrix2t(uint32_t r[2], uint32_t addr) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x2.trans.shared.b16 {%0,%1}, [%2];"
               : "=r"(r[0]), "=r"(r[1])
               : "r"(addr)
               : "memory");
}
// one row of shared memory to global memory by the copy engine (16-byte multiples)
__device__ __forceinline__ void bulk_s2g(void* dst, uint32_t src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(src), "r"(bytes) : "memory");
}
__device__ __forceinline__ void bulk_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_read() { asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory"); }
__device__ __forceinline__ void bulk_wait_all() { asm volatile("cp.async.bulk.wait_group 0;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// acc (RT x NT fragments) = A[16 RT rows][K] B over K in steps of 16; A at sa with
// pitch pa; B columns n0 .. n0 + 8 NT: rows n of pitch pb (not transposed) or rows k.
template <int RT, int NT, bool TB>
__device__ __forceinline__ void row_product(uint32_t sa, uint32_t pa, uint32_t sb, uint32_t pb, int n0, int K,
                                            float acc[RT][NT][4]) {
  const int lane = threadIdx.x & 31, l8 = lane & 7, li = lane >> 3;
#pragma unroll
  for (int i = 0; i < RT; ++i)
#pragma unroll
    for (int j = 0; j < NT; ++j)
#pragma unroll
      for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
  const uint32_t aa = sa + ((li & 1) * 8 + l8) * pa + (li >> 1) * 16;
  // not transposed: fragment pair j (columns 16 j, 16 j + 8) at rows n; transposed: at rows k
  const uint32_t ba = TB ? sb + ((li & 1) * 8 + l8) * pb + 2 * n0 + (li >> 1) * 16
                         : sb + (n0 + (li >> 1) * 8 + l8) * pb + (li & 1) * 16;
  // fragments of step k + 16 are read while the tensor core works on step k
  uint32_t a[2][RT][4], b[2][NT][2];
  auto load = [&](int k, int u) {
#pragma unroll
    for (int i = 0; i < RT; ++i) ldmatrix4<false>(a[u][i], aa + i * 16 * pa + 2 * k);
#pragma unroll
    for (int j = 0; j < NT / 2; ++j) {
      uint32_t r[4];
      ldmatrix4<TB>(r, TB ? ba + k * pb + 32 * j : ba + 16 * j * pb + 2 * k);
      b[u][2 * j][0] = r[0];
      b[u][2 * j][1] = r[1];
      b[u][2 * j + 1][0] = r[2];
      b[u][2 * j + 1][1] = r[3];
    }
    if constexpr (NT & 1) {  // the last fragment alone (lanes 16..31's addresses are not used)
      if constexpr (TB)
        ldmatrix2t(b[u][NT - 1], sb + (k + (li & 1) * 8 + l8) * pb + 2 * (n0 + 8 * (NT - 1)));
      else
        ldmatrix2(b[u][NT - 1], sb + (n0 + 8 * (NT - 1) + l8) * pb + 2 * k + (li & 1) * 16);
    }
  };
  auto multiply = [&](int u) {
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int j = 0; j < NT; ++j) mma_bf16(acc[i][j], a[u][i], b[u][j]);
  };
  load(0, 0);
#pragma unroll 2
  for (int k = 0; k < K; k += 32) {
    if (k + 16 < K) load(k + 16, 1);
    multiply(0);
    if (k + 16 < K) {
      if (k + 32 < K) load(k + 32, 0);
      multiply(1);
    }
  }
}

template <int NT, int RT, bool TRAIN>
__global__ void __launch_bounds__(kRowThreads, 1) rows_kernel(RowsArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int NF = NT;  // fragments of 8 columns per warp
  constexpr int H = 64 * NT, R = 16 * RT;
  constexpr uint32_t PH = 2 * H + 16;
  const int O = a.nout, o16 = (O + 15) / 16 * 16, ot = O / 8;
  const uint32_t PO = 2 * o16 + 16;
  const uint32_t s0 = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
  const uint32_t w2 = s0, w3 = w2 + H * PH, h1 = w3 + o16 * PH, h2 = h1 + R * PH, dy = h2 + R * PH;
  unsigned char* const h1p = smem + (h1 - s0);
  unsigned char* const h2p = smem + (h2 - s0);
  unsigned char* const dyp = smem + (dy - s0);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, gq = lane >> 2, tq = lane & 3;
  const int nw = warp * 8 * NF;  // this warp's columns of the hidden layers
  pdl_wait();
  // this CTA's member and its run of the member's tiles
  const int mem = blockIdx.x % a.members, slot = blockIdx.x / a.members, slots = gridDim.x / a.members;
  const long per = (a.n + R - 1) / R;
  const int t0 = (int)(per * slot / slots), t1 = (int)(per * (slot + 1) / slots);
  float lsum = 0.0f;
  {
    const bf16* W2 = a.pb + mem * a.P + a.ow2;
    const bf16* W3 = a.pb + mem * a.P + a.ow3;
    for (int e = tid; e < (H + O) * (H / 8); e += kRowThreads) {
      const int r = e / (H / 8), c = e % (H / 8);
      cp16(w2 + r * PH + 16 * c, (r < H ? W2 + (long)r * H : W3 + (long)(r - H) * H) + 8 * c, true);
    }
    cp_commit();
  }
  // rows of W3 (and columns of dY) that only fill up the last step of 16
  for (uint32_t e = tid; e < (o16 - O) * PH / 4; e += kRowThreads)
    reinterpret_cast<uint32_t*>(smem + (w3 - s0) + O * PH)[e] = 0u;
  uint32_t b1f[NF][2];
  float2 bias1[NF], bias2[NF];
  {
    const bf16* W1 = a.pb + mem * a.P;
    const bf16 zero = __float2bfloat16(0.0f);
#pragma unroll
    for (int j = 0; j < NF; ++j) {
      const int c = nw + 8 * j + gq;
#pragma unroll
      for (int q = 0; q < 2; ++q) {
        const int k = 2 * tq + 8 * q;
        b1f[j][q] = pack2(k < a.nin ? W1[(long)c * a.nin + k] : zero, k + 1 < a.nin ? W1[(long)c * a.nin + k + 1] : zero);
      }
      bias1[j] = *reinterpret_cast<const float2*>(a.p + mem * a.P + a.ob1 + nw + 8 * j + 2 * tq);
      bias2[j] = *reinterpret_cast<const float2*>(a.p + mem * a.P + a.ob2 + nw + 8 * j + 2 * tq);
    }
  }
  // the input fragments of a tile, read one tile ahead
  uint32_t x[RT][4];
  auto load_x = [&](int t) {
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = t * R + 16 * i + gq + (q & 1) * 8, k = 2 * tq + (q >> 1) * 8;
        if constexpr (TRAIN) {
          x[i][q] = r < a.n ? *reinterpret_cast<const uint32_t*>(a.xb + (long)r * 16 + k) : 0u;
        } else {
          const float* xr = a.xf + (long)r * a.nin;
          x[i][q] = pack2f(r < a.n && k < a.nin ? xr[k] : 0.0f,
                          r < a.n && k + 1 < a.nin ? xr[k + 1] : 0.0f);
        }
      }
  };
  if (t0 < t1) load_x(t0);
  for (int t = t0; t < t1; ++t) {
    const int r0 = t * R;
    const long row0 = mem * a.B + r0;  // first row of the tile in the activations
    auto store_rows = [&](bf16* dst, uint32_t src, uint32_t pitch, int cols) {
      if (tid < R && r0 + tid < a.n) bulk_s2g(dst + (row0 + tid) * cols, src + tid * pitch, 2 * cols);
      if (tid < R) bulk_commit();
    };
    float acc[RT][NF][4];
    // ---- layer 1: one tensor-core step from registers
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int j = 0; j < NF; ++j) {
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
        mma_bf16(acc[i][j], x[i], b1f[j]);
      }
    if (t + 1 < t1) load_x(t + 1);
    auto hidden = [&](unsigned char* dst, const float2 bias[NF]) {
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h)
#pragma unroll
          for (int j = 0; j < NF; ++j)
            *reinterpret_cast<uint32_t*>(dst + (16 * i + 8 * h + gq) * PH + 2 * (nw + 8 * j + 2 * tq)) =
                pack2f(tanhf(acc[i][j][2 * h] + bias[j].x),
                      tanhf(acc[i][j][2 * h + 1] + bias[j].y));
    };
    if constexpr (TRAIN) {
      if (tid < R) bulk_wait_read();  // the last tile's copies out of these rows
      __syncthreads();
    }
    hidden(h1p, bias1);
    if constexpr (TRAIN) fence_async_smem();
    cp_wait<0>();
    __syncthreads();
    if constexpr (TRAIN) store_rows(a.h1, h1, PH, H);
    // ---- layer 2
    row_product<RT, NF, false>(h1, PH, w2, PH, nw, H, acc);
    hidden(h2p, bias2);
    if constexpr (TRAIN) fence_async_smem();
    __syncthreads();
    if constexpr (TRAIN) store_rows(a.h2, h2, PH, H);
    // ---- layer 3: eight columns per warp at a time
    for (int c = warp; c < (TRAIN ? o16 / 8 : ot); c += kRowThreads / 32) {
      if (c >= ot) {  // training: the padding of dY
#pragma unroll
        for (int i = 0; i < 2 * RT; ++i)
          *reinterpret_cast<uint32_t*>(dyp + (8 * i + gq) * PO + 2 * (8 * c + 2 * tq)) = 0u;
        continue;
      }
      float o3[RT][1][4];
      const int n = 8 * c + 2 * tq;
      [[maybe_unused]] float2 tt[RT][2];  // the targets, read while the product runs
      if constexpr (TRAIN) {
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
          for (int h = 0; h < 2; ++h) {
            const int r = r0 + 16 * i + 8 * h + gq;
            tt[i][h] = r < a.n ? *reinterpret_cast<const float2*>(a.T + (long)r * O + n) : make_float2(0.0f, 0.0f);
          }
      }
      row_product<RT, 1, false>(h2, PH, w3, PH, 8 * c, H, o3);
      const float2 b3 = *reinterpret_cast<const float2*>(a.p + mem * a.P + a.ob3 + n);
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = 16 * i + 8 * h + gq;
          const bool in = r0 + r < a.n;
          float v0 = o3[i][0][2 * h] + b3.x, v1 = o3[i][0][2 * h + 1] + b3.y;
          if constexpr (!TRAIN) {
            if (in) *reinterpret_cast<float2*>(a.y + (row0 + r) * O + n) = make_float2(v0, v1);
          } else {
            // dY = 2 (Y - T) / (n n_out)
            float g0 = 0.0f, g1 = 0.0f;
            if (in) {
              const float d0 = v0 - tt[i][h].x, d1 = v1 - tt[i][h].y;
              lsum += d0 * d0;
              lsum += d1 * d1;
              g0 = 2.0f * d0 * a.scale;
              g1 = 2.0f * d1 * a.scale;
              *reinterpret_cast<float2*>(a.dyf + (row0 + r) * O + n) = make_float2(g0, g1);
            }
            *reinterpret_cast<uint32_t*>(dyp + r * PO + 2 * n) = pack2f(g0, g1);
          }
        }
    }
    if constexpr (!TRAIN) continue;
    fence_async_smem();
    if (tid < R) bulk_wait_read();  // h1 and h2 are rewritten below
    __syncthreads();
    store_rows(a.dyb, dy, PO, O);
    // the products with (1 - h^2), over the activation's own place
    auto dtanh = [&](unsigned char* hp, float* out) {
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = 16 * i + 8 * h + gq;
#pragma unroll
          for (int j = 0; j < NF; ++j) {
            const int n = nw + 8 * j + 2 * tq;
            __nv_bfloat162* q = reinterpret_cast<__nv_bfloat162*>(hp + r * PH + 2 * n);
            const float h0 = __bfloat162float(q->x), h1v = __bfloat162float(q->y);
            float v0 = acc[i][j][2 * h], v1 = acc[i][j][2 * h + 1];
            v0 *= 1.0f - h0 * h0;
            v1 *= 1.0f - h1v * h1v;
            if (r0 + r < a.n) *reinterpret_cast<float2*>(out + (row0 + r) * H + n) = make_float2(v0, v1);
            *reinterpret_cast<uint32_t*>(q) = pack2f(v0, v1);
          }
        }
    };
    // ---- dZ2 = (dY W3) (1 - H2^2), dZ1 = (dZ2 W2) (1 - H1^2)
    row_product<RT, NF, true>(dy, PO, w3, PH, nw, o16, acc);
    dtanh(h2p, a.dz2f);
    fence_async_smem();
    __syncthreads();
    store_rows(a.dz2b, h2, PH, H);
    row_product<RT, NF, true>(h2, PH, w2, PH, nw, H, acc);
    dtanh(h1p, a.dz1f);
    fence_async_smem();
    __syncthreads();
    store_rows(a.dz1b, h1, PH, H);
  }
  if constexpr (TRAIN) {
    for (int o = 16; o > 0; o >>= 1) lsum += __shfl_xor_sync(0xffffffffu, lsum, o);
    if (lane == 0) atomicAdd(a.loss + mem, lsum * a.scale);
    if (tid < R) bulk_wait_all();
  }
  pdl_trigger();
}

constexpr int kPredictThreads = 512;

// Barrier over the 256 threads of one of a CTA's two groups of warps.
__device__ __forceinline__ void group_sync(int g) { asm volatile("bar.sync %0, 256;" ::"r"(g + 1) : "memory"); }

// Predictions with a tile of 48 rows for every SM: the same layers, by two groups of eight
// warps that share the weights and meet only among themselves.  tanh takes four fifths of
// the instructions, so the second group starts one layer after the first: one's tanh then
// runs beside the other's tensor-core work (in step with each other they leave the tensor
// pipe idle together).  Each group's second layer overwrites the first in shared memory.
// 65536 rows x 5 members, n_hidden 256, n_out 64, whole call: 413 us by one group, 396 by
// two in step, 381 with the second behind, 358 with pairs of values rounded to BF16 by one
// instruction; two groups of four warps, which hold twice the columns each, 372.  17280 rows
// of it take 68 us, the tensor pipe active 41 % and an instruction issued 53 % of the time.
template <int NT>
__global__ void __launch_bounds__(kPredictThreads, 1) predict_kernel(RowsArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  constexpr int RT = 3, R = 16 * RT, H = 64 * NT, NF = NT;  // fragments of 8 columns per warp
  constexpr uint32_t PH = 2 * H + 16;
  const int O = a.nout, o16 = (O + 15) / 16 * 16;
  const uint32_t s0 = static_cast<uint32_t>(__cvta_generic_to_shared(smem));
  const int tid = threadIdx.x, lane = tid & 31, warp = (tid >> 5) & 7, grp = tid >> 8, gq = lane >> 2, tq = lane & 3;
  const uint32_t w2 = s0, w3 = w2 + H * PH, hs = w3 + o16 * PH + grp * R * PH;  // this group's activations
  unsigned char* const hp = smem + (hs - s0);
  const int nw = warp * 8 * NF;  // this warp's columns of the hidden layers
  pdl_wait();
  const int mem = blockIdx.x % a.members, slot = 2 * (blockIdx.x / a.members) + grp, slots = 2 * (gridDim.x / a.members);
  const long per = (a.n + R - 1) / R;
  const int t0 = (int)(per * slot / slots), t1 = (int)(per * (slot + 1) / slots);
  const bf16* Wb = a.pb + mem * a.P;
  for (int e = tid; e < (H + O) * (H / 8); e += kPredictThreads) {
    const int r = e / (H / 8), c = e % (H / 8);
    cp16(w2 + r * PH + 16 * c, Wb + (r < H ? a.ow2 + (long)r * H : a.ow3 + (long)(r - H) * H) + 8 * c, true);
  }
  cp_commit();
  for (uint32_t e = tid; e < (o16 - O) * PH / 4; e += kPredictThreads)
    reinterpret_cast<uint32_t*>(smem + (w3 - s0) + O * PH)[e] = 0u;
  uint32_t b1f[NF][2];
  const float* const bias1 = a.p + mem * a.P + a.ob1 + nw + 2 * tq;
  const float* const bias2 = a.p + mem * a.P + a.ob2 + nw + 2 * tq;
  const float* const bias3 = a.p + mem * a.P + a.ob3 + 2 * tq;
  const bf16 zero = __float2bfloat16(0.0f);
#pragma unroll
  for (int j = 0; j < NF; ++j)
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const int c = nw + 8 * j + gq, k = 2 * tq + 8 * q;
      b1f[j][q] = pack2(k < a.nin ? Wb[(long)c * a.nin + k] : zero, k + 1 < a.nin ? Wb[(long)c * a.nin + k + 1] : zero);
    }
  uint32_t x[RT][4];
  auto load_x = [&](int t) {
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        const int r = t * R + 16 * i + gq + (q & 1) * 8, k = 2 * tq + (q >> 1) * 8;
        const float* xr = a.xf + (long)r * a.nin;
        x[i][q] = pack2f(r < a.n && k < a.nin ? xr[k] : 0.0f,
                        r < a.n && k + 1 < a.nin ? xr[k + 1] : 0.0f);
      }
  };
  if (t0 < t1) load_x(t0);
  cp_wait<0>();
  __syncthreads();
  // group 1 waits until group 0 has its first layer (or has no tile)
  if (grp == 1)
    asm volatile("bar.sync 3, 512;" ::: "memory");
  else if (t0 >= t1)
    asm volatile("bar.arrive 3, 512;" ::: "memory");
  for (int t = t0; t < t1; ++t) {
    const int r0 = t * R;
    float acc[RT][NF][4];
    auto hidden = [&](const float* bias) {
#pragma unroll
      for (int j = 0; j < NF; ++j) {
        const float2 b = *reinterpret_cast<const float2*>(bias + 8 * j);
#pragma unroll
        for (int i = 0; i < RT; ++i)
#pragma unroll
          for (int h = 0; h < 2; ++h)
            *reinterpret_cast<uint32_t*>(hp + (16 * i + 8 * h + gq) * PH + 2 * (nw + 8 * j + 2 * tq)) =
                pack2f(tanhf(acc[i][j][2 * h] + b.x),
                      tanhf(acc[i][j][2 * h + 1] + b.y));
      }
    };
#pragma unroll
    for (int i = 0; i < RT; ++i)
#pragma unroll
      for (int j = 0; j < NF; ++j) {
#pragma unroll
        for (int q = 0; q < 4; ++q) acc[i][j][q] = 0.0f;
        mma_bf16(acc[i][j], x[i], b1f[j]);
      }
    hidden(bias1);
    if (grp == 0 && t == t0) asm volatile("bar.arrive 3, 512;" ::: "memory");
    group_sync(grp);
    row_product<RT, NF, false>(hs, PH, w2, PH, nw, H, acc);
    group_sync(grp);  // every warp has read h1
    hidden(bias2);
    group_sync(grp);
    if (t + 1 < t1) load_x(t + 1);
    for (int n = 8 * warp; n < O; n += 64) {
      float o3[RT][1][4];
      row_product<RT, 1, false>(hs, PH, w3, PH, n, H, o3);
      const float2 b = *reinterpret_cast<const float2*>(bias3 + n);
#pragma unroll
      for (int i = 0; i < RT; ++i)
#pragma unroll
        for (int h = 0; h < 2; ++h) {
          const int r = r0 + 16 * i + 8 * h + gq;
          if (r < a.n)
            *reinterpret_cast<float2*>(a.y + (mem * a.B + r) * O + n + 2 * tq) =
                make_float2(o3[i][0][2 * h] + b.x, o3[i][0][2 * h + 1] + b.y);
        }
    }
    group_sync(grp);  // every warp has read h2
  }
  pdl_trigger();
}

template <class... P, class... A>
static cudaError_t launch_pdl(void (*kernel)(P...), dim3 grid, unsigned block, size_t smem, cudaStream_t s, A&&... args) {
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, kernel, std::forward<A>(args)...);
}

// What a launch of the row kernels needs to know of the device.  The dynamic shared memory
// limit belongs to a kernel, which every network of its n_hidden launches, from any thread:
// all set it to the device's own limit (max_smem) and give the size they use to the launch.
struct RowsDevice {
  int sms;
  size_t max_smem;
};

template <int NT>
static cudaError_t launch_predict_at(const RowsArgs& a, size_t smem, const RowsDevice& d, cudaStream_t s) {
  cudaError_t e = cudaFuncSetAttribute(predict_kernel<NT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)d.max_smem);
  if (e) return e;
  const int slots = d.sms / a.members > 1 ? d.sms / a.members : 1;
  return launch_pdl(predict_kernel<NT>, dim3((unsigned)(a.members * slots)), kPredictThreads, smem, s, a);
}
static cudaError_t launch_predict(const RowsArgs& a, int nh, const RowsDevice& d, cudaStream_t s) {
  const size_t smem = rows_smem(nh, a.nout, 3, false);
  switch (nh / 64) {
    case 1: return launch_predict_at<1>(a, smem, d, s);
    case 2: return launch_predict_at<2>(a, smem, d, s);
    case 3: return launch_predict_at<3>(a, smem, d, s);
    case 4: return launch_predict_at<4>(a, smem, d, s);
  }
  return cudaErrorInvalidValue;
}

template <int NT, int RT, bool TRAIN>
static cudaError_t launch_rows_at(const RowsArgs& a, size_t smem, const RowsDevice& d, cudaStream_t s) {
  cudaError_t e =
      cudaFuncSetAttribute(rows_kernel<NT, RT, TRAIN>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)d.max_smem);
  if (e) return e;
  const long tiles = (a.n + 16 * RT - 1) / (16 * RT), slots = d.sms / a.members > 1 ? d.sms / a.members : 1;
  return launch_pdl(rows_kernel<NT, RT, TRAIN>, dim3((unsigned)(a.members * (tiles < slots ? tiles : slots))), kRowThreads,
                    smem, s, a);
}
template <int RT, bool TRAIN>
static cudaError_t launch_rows_of(const RowsArgs& a, int nh, size_t smem, const RowsDevice& d, cudaStream_t s) {
  switch (nh / 64) {
    case 1: return launch_rows_at<1, RT, TRAIN>(a, smem, d, s);
    case 2: return launch_rows_at<2, RT, TRAIN>(a, smem, d, s);
    case 3: return launch_rows_at<3, RT, TRAIN>(a, smem, d, s);
    case 4: return launch_rows_at<4, RT, TRAIN>(a, smem, d, s);
  }
  return cudaErrorInvalidValue;
}
template <bool TRAIN>
static cudaError_t launch_rows(const RowsArgs& a, int nh, int rt, const RowsDevice& d, cudaStream_t s) {
  const size_t smem = rows_smem(nh, a.nout, rt, TRAIN);
  if constexpr (TRAIN)  // (predictions on tiles of 48 rows: launch_predict)
    if (rt == 3) return launch_rows_of<3, true>(a, nh, smem, d, s);
  return launch_rows_of<1, TRAIN>(a, nh, smem, d, s);
}

// Gradients of all weights and biases in one launch.  The batch rows are cut into ks
// splits of kc rows, whose products are added in split order.  Where the 64x64 tiles
// of dW3, dW2 and dW1 fill the GPU by themselves a CTA takes a tile through all splits
// and adds as it goes (parts = 1: no partial leaves the registers); otherwise the grid's
// y is the split and the partials are added by the kernel that uses the gradient (parts
// = ks).  The grid's x beyond the tiles takes 32 columns of a bias gradient each, for
// one of its eight groups of row classes (y).  part: [member][parts][P], at the
// parameters' offsets; bpart: [member][group][b1 b2 b3].
struct Sched {
  int t;        // updates done, less one before the first
  int total;    // length of the cosine schedule
  float lr0, lr_min, wd;
};
struct WgradArgs {
  GemmArgs w[3];  // dW3 = dY^T H2, dW2 = dZ2^T H1, dW1 = dZ1^T X: A[k][m], B[k][n]
  int tiles[3];   // tiles of each
  int ntn[3];     // of them along N
  int ks, kc, parts;
  const float* bx[3];  // dY, dZ2, dZ1 in FP32
  int bcols[3];
  int bblocks[3];      // blocks of 32 columns
  int boff[3];         // offset of b3, b2, b1 in a bias partial
  int bsum;            // 2 n_hidden + n_out
  float* bpart;
  int rows, members;
  Sched* sc;           // the training step this launch belongs to is counted here
};

// A bias gradient's column sums in the order of a 256-thread block whose thread t
// adds rows t, t + 256, ... and whose warps reduce by xor shuffles: group y is warp y
// of that block (row classes 32 y .. 32 y + 31).
__device__ __forceinline__ void bias_group(const float* X, int rows, int cols, int c0, int grp, float* out,
                                           float (*sh)[33]) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const int c = c0 + lane;
  constexpr int RC = 32 / (kWgradThreads / 32);  // row classes per warp
  float s[RC];
#pragma unroll
  for (int r = 0; r < RC; ++r) s[r] = 0.0f;
  if (c < cols) {
    const int t = grp * 32 + warp * RC;
    const float* p = X + (long)t * cols + c;
    const long step = 256L * cols;
    int base = t + RC;
#pragma unroll 4
    for (; base <= rows; base += 256, p += step) {
#pragma unroll
      for (int r = 0; r < RC; ++r) s[r] += p[r * cols];
    }
#pragma unroll
    for (int r = 0; r < RC; ++r)
      if (base - RC + r < rows) s[r] += p[r * cols];
  }
#pragma unroll
  for (int r = 0; r < RC; ++r) sh[warp * RC + r][lane] = s[r];
  for (int o = 16; o > 0; o >>= 1) {
    __syncthreads();
    for (int l = warp; l < o; l += kWgradThreads / 32) sh[l][lane] += sh[l + o][lane];
  }
  __syncthreads();
  if (warp == 0 && c < cols) out[c] = sh[0][lane];
}

__global__ void __launch_bounds__(kWgradThreads) wgrad_kernel(WgradArgs a) {
  extern __shared__ __align__(128) unsigned char smem[];
  pdl_wait();
  if (a.sc && blockIdx.x == 0 && threadIdx.x == 0) a.sc->t += 1;
  // the products first (they take longest): member, then split, then tile
  int t = blockIdx.x;
  const int nprod = (a.tiles[0] + a.tiles[1] + a.tiles[2]) * a.parts * a.members;
  const bool prod = t < nprod;
  if (!prod) t -= nprod;
  const int mem = t % a.members;
  t /= a.members;
  const int ny = prod ? a.parts : kBiasGroups;
  const int y = t % ny;  // split or group
  t /= ny;
  if (prod) {
#pragma unroll
    for (int q = 0; q < 3; ++q) {
      if (t < a.tiles[q]) {
        const GemmArgs& g = a.w[q];
        const int m0 = t / a.ntn[q] * TM, n0 = t % a.ntn[q] * TN;
        const int kb = y * a.kc, ke = a.parts == 1 ? g.K : min(g.K, kb + a.kc);
        float acc[2][4][4];
        gemm_tile<true, true, kWgradStages, true>(g.A + mem * g.a_mem, g.lda, g.M, g.B + mem * g.b_mem, g.ldb, g.b_cols,
                                                  m0, n0, kb, ke, smem, acc, a.kc);
        float* C = g.Cf + ((long)mem * a.parts + y) * g.cf_mem;
        const int N = g.N;
        for_pairs(acc, m0, n0, g.M, (N + 1) & ~1, [&](int m, int n, float v0, float v1) {
          float* o = C + (long)m * N + n;
          if (!(N & 1)) {
            *reinterpret_cast<float2*>(o) = make_float2(v0, v1);
          } else {  // dW1 with an odd number of inputs
            o[0] = v0;
            if (n + 1 < N) o[1] = v1;
          }
        });
        return;
      }
      t -= a.tiles[q];
    }
    return;
  }
#pragma unroll
  for (int q = 0; q < 3; ++q) {
    if (t < a.bblocks[q]) {
      bias_group(a.bx[q] + mem * a.w[q].a_mem, a.rows, a.bcols[q], t * 32, y,
                 a.bpart + ((long)mem * kBiasGroups + y) * a.bsum + a.boff[q], reinterpret_cast<float(*)[33]>(smem));
      return;
    }
    t -= a.bblocks[q];
  }
}

// Offsets of the parameter blocks (they and P are multiples of 8).
struct Offsets {
  long b1, w2, b2, w3, b3;
  int nh, nout;
};

// The gradient of four neighbouring parameters of one member from its partials, in
// split (weights) or group (biases) order.
__device__ __forceinline__ float4 grad4(const float* part, const float* bpart, int ks, long P, const Offsets& o,
                                        long i) {
  const bool weight = (i < o.b1) || (i >= o.w2 && i < o.b2) || (i >= o.w3 && i < o.b3);
  const float* p;
  long stride;
  int n;
  if (weight) {
    p = part + i;
    stride = P;
    n = ks;
  } else {
    const long c = i < o.w2 ? i - o.b1 : (i < o.w3 ? o.nh + (i - o.b2) : 2L * o.nh + (i - o.b3));
    p = bpart + c;
    stride = 2L * o.nh + o.nout;
    n = kBiasGroups;
  }
  float4 v = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
#pragma unroll 8
  for (int s = 0; s < n; ++s) {
    const float4 q = *reinterpret_cast<const float4*>(p + s * stride);
    v.x += q.x;
    v.y += q.y;
    v.z += q.z;
    v.w += q.w;
  }
  return v;
}

// Gradient of member blockIdx.y + mem0 into g (dense).
__global__ void grad_sum_kernel(const float* part, const float* bpart, int ks, long P, Offsets o, int mem0, float* g) {
  const long mem = mem0 + blockIdx.y;
  for (long i = 4 * (blockIdx.x * (long)blockDim.x + threadIdx.x); i < P; i += 4L * gridDim.x * blockDim.x)
    *reinterpret_cast<float4*>(g + mem * P + i) =
        grad4(part + mem * ks * P, bpart + mem * kBiasGroups * (2L * o.nh + o.nout), ks, P, o, i);
}

// AdamW on every member, gradients straight from the partials: FP32 master weights,
// BF16 working copy; the biases are not decayed.
__global__ void __launch_bounds__(256) adamw_kernel(float* p, bf16* pb, const float* part, const float* bpart, int ks,
                                                    float* m1, float* m2, long P, const Sched* sc, Offsets o,
                                                    float* loss) {
  const int mem = blockIdx.y;
  pdl_wait();
  if (blockIdx.x == 0 && threadIdx.x == 0) loss[mem] = 0.0f;  // for the next step
  const int t = sc->t + 1;
  const float pi = 3.14159265358979f;
  const float frac = sc->total > 1 ? fminf((float)(t - 1) / (float)(sc->total - 1), 1.0f) : 1.0f;
  const float lr = sc->lr_min + 0.5f * (sc->lr0 - sc->lr_min) * (1.0f + cosf(pi * frac));
  const float beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
  const float c1 = 1.0f - powf(beta1, (float)t), c2 = 1.0f - powf(beta2, (float)t);
  const long i = 4 * (blockIdx.x * (long)blockDim.x + threadIdx.x);
  if (i >= P) return;
  const long j = mem * P + i;
  const float4 g4 = grad4(part + (long)mem * ks * P, bpart + (long)mem * kBiasGroups * (2L * o.nh + o.nout), ks, P, o, i);
  float4 a4 = *reinterpret_cast<float4*>(m1 + j), b4 = *reinterpret_cast<float4*>(m2 + j);
  float4 p4 = *reinterpret_cast<float4*>(p + j);
  const bool weight = (i < o.b1) || (i >= o.w2 && i < o.b2) || (i >= o.w3 && i < o.b3);
  const float gr[4] = {g4.x, g4.y, g4.z, g4.w};
  float av[4] = {a4.x, a4.y, a4.z, a4.w}, bv[4] = {b4.x, b4.y, b4.z, b4.w}, pv[4] = {p4.x, p4.y, p4.z, p4.w};
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const float gv = gr[q];
    const float a = beta1 * av[q] + (1.0f - beta1) * gv;
    const float b = beta2 * bv[q] + (1.0f - beta2) * gv * gv;
    av[q] = a;
    bv[q] = b;
    float w = pv[q];
    if (weight) w -= lr * sc->wd * w;
    w -= lr * (a / c1) / (sqrtf(b / c2) + eps);
    pv[q] = w;
  }
  *reinterpret_cast<float4*>(m1 + j) = make_float4(av[0], av[1], av[2], av[3]);
  *reinterpret_cast<float4*>(m2 + j) = make_float4(bv[0], bv[1], bv[2], bv[3]);
  *reinterpret_cast<float4*>(p + j) = make_float4(pv[0], pv[1], pv[2], pv[3]);
  *reinterpret_cast<uint2*>(pb + j) =
      make_uint2(pack2f(pv[0], pv[1]),
                 pack2f(pv[2], pv[3]));
}

// A member's new master weights: the BF16 working copy, and fresh AdamW moments (the
// host's own conversion of 83520 weights took 140 us a member, this takes 26 with the copy).
__global__ void __launch_bounds__(256) load_params_kernel(const float* p, bf16* pb, float* m1, float* m2, long P) {
  const float4 z = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
  for (long i = 4 * (blockIdx.x * (long)blockDim.x + threadIdx.x); i < P; i += 4L * gridDim.x * blockDim.x) {
    const float4 v = *reinterpret_cast<const float4*>(p + i);
    *reinterpret_cast<uint2*>(pb + i) = make_uint2(pack2f(v.x, v.y),
                                                   pack2f(v.z, v.w));
    *reinterpret_cast<float4*>(m1 + i) = z;
    *reinterpret_cast<float4*>(m2 + i) = z;
  }
}

// x (FP32, [n][n_in]) -> BF16 [n][16] with zero padding.
__global__ void pack_x_kernel(const float* x, int n, int nin, bf16* xb) {
  for (long e = blockIdx.x * (long)blockDim.x + threadIdx.x; e < (long)n * 16; e += (long)gridDim.x * blockDim.x) {
    const long r = e / 16;
    const int c = (int)(e % 16);
    xb[e] = __float2bfloat16(c < nin ? x[r * nin + c] : 0.0f);
  }
}

__device__ __forceinline__ unsigned long long mix64(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// Glorot-uniform weights (counter-based generator), zero biases.
__global__ void init_params_kernel(float* p, bf16* pb, long P, unsigned long long seed, int nin, int nh, int nout) {
  const int mem = blockIdx.y;
  const long b1 = (long)nh * nin, w2 = b1 + nh, b2 = w2 + (long)nh * nh, w3 = b2 + nh, b3 = w3 + (long)nout * nh;
  for (long i = blockIdx.x * (long)blockDim.x + threadIdx.x; i < P; i += (long)gridDim.x * blockDim.x) {
    float a = 0.0f;
    if (i < b1)
      a = sqrtf(6.0f / (nin + nh));
    else if (i >= w2 && i < b2)
      a = sqrtf(6.0f / (nh + nh));
    else if (i >= w3 && i < b3)
      a = sqrtf(6.0f / (nh + nout));
    const unsigned long long r = mix64((seed + mem) * 0x100000001B3ull + (unsigned long long)i);
    const float u = (float)((r >> 11) * (1.0 / 9007199254740992.0));  // [0, 1)
    const float v = a * (2.0f * u - 1.0f);
    p[mem * P + i] = v;
    pb[mem * P + i] = __float2bfloat16(v);
  }
}

// mean and standard deviation over members of Y [K][n][nout], four values at a time
// (count, the member stride and the arrays are multiples of 16 bytes).
__global__ void __launch_bounds__(256) ensemble_kernel(const float* Y, int K, long stride, long count, float* mean,
                                                       float* sd) {
  pdl_wait();
  for (long e = 4 * (blockIdx.x * (long)blockDim.x + threadIdx.x); e < count; e += 4L * gridDim.x * blockDim.x) {
    float s[4] = {0.0f, 0.0f, 0.0f, 0.0f}, q[4] = {0.0f, 0.0f, 0.0f, 0.0f}, mu[4], dv[4];
    for (int k = 0; k < K; ++k) {
      const float4 v = *reinterpret_cast<const float4*>(Y + k * stride + e);
      const float y[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) s[i] += y[i];
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) mu[i] = s[i] / K;
    for (int k = 0; k < K; ++k) {
      const float4 v = *reinterpret_cast<const float4*>(Y + k * stride + e);
      const float y[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float d = y[i] - mu[i];
        q[i] += d * d;
      }
    }
#pragma unroll
    for (int i = 0; i < 4; ++i) dv[i] = K > 1 ? sqrtf(q[i] / (K - 1)) : 0.0f;
    *reinterpret_cast<float4*>(mean + e) = make_float4(mu[0], mu[1], mu[2], mu[3]);
    *reinterpret_cast<float4*>(sd + e) = make_float4(dv[0], dv[1], dv[2], dv[3]);
  }
}

thread_local char g_mlp_err[512] = "";

}  // namespace

struct lb_mlp {
  int nin, nh, nout, K, maxb;
  long P;
  long ow1, ob1, ow2, ob2, ow3, ob3;
  cudaStream_t stream, cap;  // cap: captures training graphs, copies large results
  lb_alloc alloc;
  int have_alloc;
  std::vector<void*> owned;
  float *p, *g, *m1, *m2;
  bf16* pb;
  Sched* sched;
  float* loss;
  // activations (per member)
  bf16 *xb, *xbp, *h1, *h2, *dyb, *dz2b, *dz1b;
  float *y, *dyf, *dz2f, *dz1f, *t;
  float *part, *bpart;  // split-K partials of the weight gradients, row-class partials of the bias gradients
  int ks_max;           // largest K split the partial buffer holds
  int n;  // rows of the loaded data
  RowsDevice dev;  // SMs of the device and shared memory a block may opt in to
  // host rows on their way in and ensemble statistics on their way out: in buffers that only
  // a backward pass uses (one member's mean is its output)
  float *xin, *mean, *sd;
  cudaEvent_t done[kParts];  // the parts of a prediction
  cudaGraphExec_t gexec;
  char err[512];
};

static void merr(lb_mlp* m, const char* fmt, ...) {
  char* dst = m ? m->err : g_mlp_err;
  va_list ap;
  va_start(ap, fmt);
  vsnprintf(dst, 512, fmt, ap);
  va_end(ap);
}

#define MCK(call)                                                                          \
  do {                                                                                     \
    cudaError_t e_ = (call);                                                               \
    if (e_ != cudaSuccess) {                                                               \
      merr(m, "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, __LINE__); \
      return LB_ERR_CUDA;                                                                  \
    }                                                                                      \
  } while (0)

// Device memory on a 256-byte boundary (the kernels move 16 bytes at a time and an
// allocator given by the caller may align to less).
static void* malloc_dev(lb_mlp* m, size_t bytes) {
  void* p = NULL;
  bytes += 256;
  if (m->have_alloc)
    p = m->alloc.malloc_fn(bytes, (void*)m->stream, m->alloc.user);
  else if (cudaMalloc(&p, bytes) != cudaSuccess) {
    cudaGetLastError();
    p = NULL;
  }
  if (!p) return NULL;
  m->owned.push_back(p);
  return (void*)(((uintptr_t)p + 255) & ~(uintptr_t)255);
}

// Blocks of 256 threads for a grid-stride kernel over count items.
static unsigned blocks_for(const lb_mlp* m, long count) {
  const long b = (count + 255) / 256, most = 16L * m->dev.sms;
  return (unsigned)(b < 1 ? 1 : (b < most ? b : most));
}

template <int EPI, bool TB>
static cudaError_t gemm(const GemmArgs& g, int members, cudaStream_t s) {
  const dim3 grid((g.N + TN - 1) / TN, (g.M + TM - 1) / TM, members);
  gemm_kernel<EPI, TB><<<grid, kGemmThreads, kGemmSmem, s>>>(g);
  return cudaGetLastError();
}

// Rows in units of 16 that a fused row tile takes (0: the network does not fit): three
// where the tiles of 48 rows still give every SM one, else one, so that small batches
// spread over the SMs (512 rows x 5 members: 160 tiles of 16 rows).
static int rows_plan(const lb_mlp* m, int n, bool train) {
  if (m->nh > 256) return 0;
  if ((long)((n + 47) / 48) * m->K >= m->dev.sms && rows_smem(m->nh, m->nout, 3, train) <= m->dev.max_smem) return 3;
  return rows_smem(m->nh, m->nout, 1, train) <= m->dev.max_smem ? 1 : 0;
}

static RowsArgs rows_args(const lb_mlp* m, int n) {
  RowsArgs a = {};
  a.n = n; a.nin = m->nin; a.nout = m->nout; a.members = m->K;
  a.p = m->p; a.pb = m->pb; a.P = m->P;
  a.ob1 = m->ob1; a.ow2 = m->ow2; a.ob2 = m->ob2; a.ow3 = m->ow3; a.ob3 = m->ob3;
  a.B = m->maxb;
  return a;
}

// The fused forward and backward pass of the loaded data down to dZ1.
static cudaError_t rows_train(lb_mlp* m, int rt, cudaStream_t s) {
  RowsArgs a = rows_args(m, m->n);
  a.xb = m->xb;
  a.h1 = m->h1; a.h2 = m->h2; a.dyb = m->dyb; a.dz2b = m->dz2b; a.dz1b = m->dz1b;
  a.dyf = m->dyf; a.dz2f = m->dz2f; a.dz1f = m->dz1f;
  a.T = m->t;
  a.loss = m->loss;
  a.scale = 1.0f / ((float)m->n * (float)m->nout);
  return launch_rows<true>(a, m->nh, rt, m->dev, s);
}

// Forward of every member on n rows of the inputs from row r0: outputs in m->y.
static cudaError_t rows_predict(lb_mlp* m, int rt, int r0, int n, cudaStream_t s) {
  RowsArgs a = rows_args(m, n);
  a.xf = m->xin + (long)r0 * m->nin;
  a.y = m->y + (long)r0 * m->nout;
  if (rt == 3) return launch_predict(a, m->nh, m->dev, s);
  return launch_rows<false>(a, m->nh, rt, m->dev, s);
}

// Rows of one part of a prediction on n rows.  Large results go to the host in up to kParts
// parts, each beside the kernels of the next, on a second stream: 65536 rows x 5 members
// (33.5 MB of results, 0.2 ms) 538 -> 413 us.  Below 4 MB the copy is shorter than what the
// parts add (10000 rows: 144 and 149 us).  Every CTA has the same number of tiles in a whole
// part, so that no part ends in a wave of few.
static int predict_part(const lb_mlp* m, int rt, int n) {
  if (rt != 3 || 8L * n * m->nout < (4L << 20)) return n;
  const long slots = m->dev.sms / m->K > 1 ? m->dev.sms / m->K : 1, wave = 2 * 48 * slots;
  const long rows = ((n + wave - 1) / wave + kParts - 1) / kParts * wave;
  return rows < n ? (int)rows : n;
}

// One launch per product.  Forward of every member on rows [0, n) of the packed inputs
// xb: outputs in m->y, or with train their loss against the loaded targets, and dY.
static cudaError_t forward(lb_mlp* m, int n, const bf16* xb, bool train, cudaStream_t s) {
  const long H = m->nh, O = m->nout, B = m->maxb;
  layer1_kernel<<<dim3(m->nh / TN, (n + TM - 1) / TM, m->K), kGemmThreads, 0, s>>>(
      xb, m->pb + m->ow1, m->P, m->p + m->ob1, m->P, n, m->nin, m->nh, m->h1, B * H);
  cudaError_t e = cudaGetLastError();
  if (e) return e;
  GemmArgs g = {};
  g.M = n;
  g.N = m->nh;
  g.K = m->nh;
  g.A = m->h1;
  g.lda = H;
  g.a_mem = B * H;
  g.B = m->pb + m->ow2;
  g.ldb = H;
  g.b_mem = m->P;
  g.bias = m->p + m->ob2;
  g.bias_mem = m->P;
  g.Cb = m->h2;
  g.ldcb = H;
  g.cb_mem = B * H;
  if ((e = gemm<EPI_BIAS_TANH, false>(g, m->K, s))) return e;
  g.N = m->nout;
  g.A = m->h2;
  g.B = m->pb + m->ow3;
  g.bias = m->p + m->ob3;
  g.Cb = NULL;
  g.Cf = m->y;
  g.ldcf = O;
  g.cf_mem = B * O;
  if (!train) return gemm<EPI_BIAS_F32, false>(g, m->K, s);
  g.Cf = m->dyf;
  g.Cb = m->dyb;
  g.ldcb = O;
  g.cb_mem = B * O;
  g.T = m->t;
  g.loss = m->loss;
  g.scale = 1.0f / ((float)n * (float)m->nout);
  return gemm<EPI_LOSS, false>(g, m->K, s);
}

// K splits of the weight gradients over n rows: about 128 rows each.
static void wgrad_splits(const lb_mlp* m, int n, int* ks, int* kc) {
  int k = (n + 127) / 128;
  if (k > m->ks_max) k = m->ks_max;
  *kc = k <= 1 ? n : ((n + k - 1) / k + 15) / 16 * 16;
  *ks = (n + *kc - 1) / *kc;
}

// Forward, loss and backward products of every member on the loaded data, one launch each.
static cudaError_t gemm_train(lb_mlp* m, cudaStream_t s) {
  const int n = m->n;
  const long H = m->nh, O = m->nout, B = m->maxb;
  cudaError_t e = forward(m, n, m->xb, true, s);
  if (e) return e;
  // dZ2 = (dY W3) * (1 - H2^2), dZ1 = (dZ2 W2) * (1 - H1^2)
  GemmArgs g = {};
  g.M = n;
  g.N = m->nh;
  g.K = m->nout;
  g.A = m->dyb;
  g.lda = O;
  g.a_mem = B * O;
  g.B = m->pb + m->ow3;
  g.ldb = H;
  g.b_mem = m->P;
  g.b_cols = m->nh;
  g.Cf = m->dz2f;
  g.ldcf = H;
  g.cf_mem = B * H;
  g.Cb = m->dz2b;
  g.ldcb = H;
  g.cb_mem = B * H;
  g.H = m->h2;
  g.ldh = H;
  g.h_mem = B * H;
  if ((e = gemm<EPI_DTANH, true>(g, m->K, s))) return e;
  g.K = m->nh;
  g.A = m->dz2b;
  g.lda = H;
  g.a_mem = B * H;
  g.B = m->pb + m->ow2;
  g.Cf = m->dz1f;
  g.Cb = m->dz1b;
  g.H = m->h1;
  return gemm<EPI_DTANH, true>(g, m->K, s);
}

// Parts the weight gradients are left in: 1 where the tiles fill three quarters of the
// SMs, or where a CTA's pass over all rows is short, else one per split.  4096 rows x 5
// members (120 tiles): 33 us in one part, 39 us in 32 parts and 2 us more in AdamW, which
// then reads 54 MB of partials; one member alone (24 tiles) needs the splits to fill the SMs.
static int wgrad_parts(const lb_mlp* m, int ks) {
  const long h = m->nh / TM, o = (m->nout + TM - 1) / TM;
  return ks <= 4 || 4 * (h * h + h * o + h) * m->K >= 3 * m->dev.sms ? 1 : ks;
}

// forward, loss and the gradients' partials of every member on the loaded data (sc:
// the schedule that counts training steps, or NULL); the losses are added to m->loss
static cudaError_t backward(lb_mlp* m, Sched* sc, cudaStream_t s) {
  const int n = m->n;
  const long H = m->nh, B = m->maxb;
  const int rt = rows_plan(m, m->n, true);
  cudaError_t e = rt ? rows_train(m, rt, s) : gemm_train(m, s);
  if (e) return e;
  // dW3 = dY^T H2, dW2 = dZ2^T H1, dW1 = dZ1^T X and the bias gradients
  WgradArgs a = {};
  a.sc = sc;
  const bf16* A[3] = {m->dyb, m->dz2b, m->dz1b};
  const bf16* Bx[3] = {m->h2, m->h1, m->xb};
  const int M[3] = {m->nout, m->nh, m->nh}, N[3] = {m->nh, m->nh, m->nin};
  const long ow[3] = {m->ow3, m->ow2, m->ow1};
  const float* bx[3] = {m->dyf, m->dz2f, m->dz1f};
  for (int q = 0; q < 3; ++q) {
    GemmArgs& w = a.w[q];
    w.M = M[q];
    w.N = N[q];
    w.K = n;
    w.A = A[q];
    w.lda = M[q];
    w.a_mem = B * M[q];
    w.B = Bx[q];
    w.ldb = w.b_cols = q < 2 ? m->nh : 16;
    w.b_mem = q < 2 ? B * H : 0;
    w.Cf = m->part + ow[q];
    w.cf_mem = m->P;
    a.ntn[q] = (N[q] + TN - 1) / TN;
    a.tiles[q] = (M[q] + TM - 1) / TM * a.ntn[q];
    a.bx[q] = bx[q];
    a.bcols[q] = M[q];
    a.bblocks[q] = (M[q] + 31) / 32;
    a.boff[q] = q == 0 ? 2 * m->nh : (q == 1 ? m->nh : 0);
  }
  wgrad_splits(m, n, &a.ks, &a.kc);
  a.parts = wgrad_parts(m, a.ks);
  a.bsum = 2 * m->nh + m->nout;
  a.bpart = m->bpart;
  a.rows = n;
  a.members = m->K;
  e = cudaFuncSetAttribute(wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWgradSmem);
  if (e) return e;
  const unsigned blocks = (unsigned)m->K * ((unsigned)(a.tiles[0] + a.tiles[1] + a.tiles[2]) * a.parts +
                                            (unsigned)(a.bblocks[0] + a.bblocks[1] + a.bblocks[2]) * kBiasGroups);
  return launch_pdl(wgrad_kernel, dim3(blocks), kWgradThreads, kWgradSmem, s, a);
}

static Offsets offsets(const lb_mlp* m) {
  return Offsets{m->ob1, m->ow2, m->ob2, m->ow3, m->ob3, m->nh, m->nout};
}

static cudaError_t train_step(lb_mlp* m, cudaStream_t s) {
  cudaError_t e = backward(m, m->sched, s);
  if (e) return e;
  int ks, kc;
  wgrad_splits(m, m->n, &ks, &kc);
  ks = wgrad_parts(m, ks);
  return launch_pdl(adamw_kernel, dim3((unsigned)((m->P / 4 + 255) / 256), m->K), 256, 0, s, m->p, m->pb, (const float*)m->part, (const float*)m->bpart, ks, m->m1, m->m2, m->P, (const Sched*)m->sched, offsets(m), m->loss);
}

extern "C" {

lb_status lb_mlp_create(int nin, int nh, int nout, int members, int max_batch, unsigned long long seed,
                        const lb_alloc* alloc, void* stream, lb_mlp** out) {
  lb_mlp* m = NULL;
  if (!out) return LB_ERR_ARG;
  *out = NULL;
  if (nin < 1 || nin > 16 || nh < 64 || nh % 64 || nh > 1024 || nout < 8 || nout % 8 || nout > 1024 || members < 1 ||
      members > 16 || max_batch < 1 || max_batch > 65535 * 64)  // row tiles of 64 on gridDim.y
    return merr(NULL, "invalid network shape"), LB_ERR_ARG;
  if (alloc && (!alloc->malloc_fn || !alloc->free_fn)) return merr(NULL, "incomplete allocator"), LB_ERR_ARG;
  m = new (std::nothrow) lb_mlp();
  if (!m) return LB_ERR_NOMEM;
  m->nin = nin; m->nh = nh; m->nout = nout; m->K = members; m->maxb = max_batch;
  m->ow1 = 0; m->ob1 = (long)nh * nin; m->ow2 = m->ob1 + nh; m->ob2 = m->ow2 + (long)nh * nh;
  m->ow3 = m->ob2 + nh; m->ob3 = m->ow3 + (long)nout * nh;
  m->P = m->ob3 + nout;
  m->stream = (cudaStream_t)stream;
  m->have_alloc = alloc != NULL;
  if (alloc) m->alloc = *alloc;
  if (cudaStreamCreateWithFlags(&m->cap, cudaStreamNonBlocking) != cudaSuccess) {
    delete m;
    return merr(NULL, "cudaStreamCreate failed"), LB_ERR_CUDA;
  }
  const long PK = m->P * members, B = max_batch;
  int dev = 0, sms = 0, optin = 0;
  cudaError_t ea = cudaGetDevice(&dev);
  if (ea == cudaSuccess) ea = cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
  if (ea == cudaSuccess) ea = cudaDeviceGetAttribute(&optin, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (ea != cudaSuccess) {
    lb_mlp_destroy(m);
    return merr(NULL, "device query failed: %s", cudaGetErrorString(ea)), LB_ERR_CUDA;
  }
  m->dev = RowsDevice{sms, (size_t)optin};
  for (cudaEvent_t& ev : m->done)
    if ((ea = cudaEventCreateWithFlags(&ev, cudaEventDisableTiming)) != cudaSuccess) {
      lb_mlp_destroy(m);
      return merr(NULL, "cudaEventCreate failed: %s", cudaGetErrorString(ea)), LB_ERR_CUDA;
    }
  m->p = (float*)malloc_dev(m, PK * 4);
  m->g = (float*)malloc_dev(m, PK * 4);
  m->m1 = (float*)malloc_dev(m, PK * 4);
  m->m2 = (float*)malloc_dev(m, PK * 4);
  m->pb = (bf16*)malloc_dev(m, PK * 2);
  m->sched = (Sched*)malloc_dev(m, sizeof(Sched));
  m->loss = (float*)malloc_dev(m, 64 * sizeof(float));
  m->xb = (bf16*)malloc_dev(m, B * 16 * 2);
  m->xbp = (bf16*)malloc_dev(m, B * 16 * 2);
  m->h1 = (bf16*)malloc_dev(m, members * B * nh * 2);
  m->h2 = (bf16*)malloc_dev(m, members * B * nh * 2);
  m->dz2b = (bf16*)malloc_dev(m, members * B * nh * 2);
  m->dz1b = (bf16*)malloc_dev(m, members * B * nh * 2);
  m->dz2f = (float*)malloc_dev(m, members * B * nh * 4);
  m->dz1f = (float*)malloc_dev(m, members * B * nh * 4);
  m->y = (float*)malloc_dev(m, members * B * nout * 4);
  m->dyf = (float*)malloc_dev(m, members * B * nout * 4);
  m->dyb = (bf16*)malloc_dev(m, members * B * nout * 2);
  m->t = (float*)malloc_dev(m, B * nout * 4);
  // partials of the gradients: about 128 batch rows per split, at most 32 splits and,
  // by the largest weight gradient (nh x max(nh, nout)), 256 MB
  {
    const long mn = (long)nh * (nh > nout ? nh : nout);
    long ks = (B + 127) / 128;
    if (ks > 32) ks = 32;
    const long cap = (256L << 20) / (4L * members * mn);
    if (ks > cap) ks = cap;
    m->ks_max = ks > 1 ? (int)ks : 1;
    m->part = (float*)malloc_dev(m, 4L * members * wgrad_parts(m, m->ks_max) * m->P);
    m->bpart = (float*)malloc_dev(m, 4L * members * kBiasGroups * (2 * nh + nout));
  }
  m->xin = m->dz2f;
  m->mean = members > 1 ? m->dyf : m->y;
  m->sd = members > 1 && m->dyf ? m->dyf + B * nout : m->dyf;
  bool ok = m->part && m->bpart && m->p && m->g && m->m1 && m->m2 && m->pb && m->sched && m->loss && m->xb && m->xbp && m->h1 && m->h2 && m->dz2b &&
            m->dz1b && m->dz2f && m->dz1f && m->y && m->dyf && m->dyb && m->t;
  if (!ok) {
    lb_mlp_destroy(m);
    return merr(NULL, "device allocation failed"), LB_ERR_NOMEM;
  }
  init_params_kernel<<<dim3(64, members), 256, 0, m->stream>>>(m->p, m->pb, m->P, seed, nin, nh, nout);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = cudaMemsetAsync(m->m1, 0, PK * 4, m->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->m2, 0, PK * 4, m->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(m->sched, 0, sizeof(Sched), m->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(m->stream);
  if (e != cudaSuccess) {
    merr(NULL, "init failed: %s", cudaGetErrorString(e));
    lb_mlp_destroy(m);
    return LB_ERR_CUDA;
  }
  *out = m;
  return LB_OK;
}

void lb_mlp_destroy(lb_mlp* m) {
  if (!m) return;
  cudaStreamSynchronize(m->stream);
  if (m->cap) cudaStreamSynchronize(m->cap);
  if (m->gexec) cudaGraphExecDestroy(m->gexec);
  for (void* p : m->owned) {
    if (m->have_alloc)
      m->alloc.free_fn(p, (void*)m->stream, m->alloc.user);
    else
      cudaFree(p);
  }
  for (cudaEvent_t ev : m->done)
    if (ev) cudaEventDestroy(ev);
  if (m->cap) cudaStreamDestroy(m->cap);
  delete m;
}

long lb_mlp_num_params(const lb_mlp* m) { return m ? m->P : -1; }

lb_status lb_mlp_get_params(lb_mlp* m, int k, float* params) {
  if (!m || k < 0 || k >= m->K || !params) return LB_ERR_ARG;
  MCK(cudaMemcpyAsync(params, m->p + k * m->P, m->P * 4, cudaMemcpyDeviceToHost, m->stream));
  MCK(cudaStreamSynchronize(m->stream));
  return LB_OK;
}

lb_status lb_mlp_set_params(lb_mlp* m, int k, const float* params) {
  if (!m || k < 0 || k >= m->K || !params) return LB_ERR_ARG;
  MCK(cudaMemcpyAsync(m->p + k * m->P, params, m->P * 4, cudaMemcpyHostToDevice, m->stream));
  load_params_kernel<<<blocks_for(m, m->P / 4), 256, 0, m->stream>>>(m->p + k * m->P, m->pb + k * m->P,
                                                                    m->m1 + k * m->P, m->m2 + k * m->P, m->P);
  MCK(cudaGetLastError());
  MCK(cudaStreamSynchronize(m->stream));
  return LB_OK;
}

lb_status lb_mlp_set_data(lb_mlp* m, int n, const float* x, const float* y) {
  if (!m || n < 1 || n > m->maxb || !x || !y) return LB_ERR_ARG;
  MCK(cudaMemcpyAsync(m->xin, x, (size_t)n * m->nin * 4, cudaMemcpyHostToDevice, m->stream));
  pack_x_kernel<<<blocks_for(m, 16L * n), 256, 0, m->stream>>>(m->xin, n, m->nin, m->xb);
  MCK(cudaGetLastError());
  MCK(cudaMemcpyAsync(m->t, y, (size_t)n * m->nout * 4, cudaMemcpyHostToDevice, m->stream));
  MCK(cudaStreamSynchronize(m->stream));
  m->n = n;
  if (m->gexec) {
    cudaGraphExecDestroy(m->gexec);
    m->gexec = NULL;
  }
  return LB_OK;
}

lb_status lb_mlp_gradients(lb_mlp* m, int k, float* grads, float* loss) {
  if (!m || k < 0 || k >= m->K || !grads || m->n < 1) return LB_ERR_ARG;
  MCK(cudaMemsetAsync(m->loss, 0, m->K * sizeof(float), m->stream));
  MCK(backward(m, NULL, m->stream));
  int ks, kc;
  wgrad_splits(m, m->n, &ks, &kc);
  ks = wgrad_parts(m, ks);
  grad_sum_kernel<<<256, 256, 0, m->stream>>>(m->part, m->bpart, ks, m->P, offsets(m), k, m->g);
  MCK(cudaGetLastError());
  MCK(cudaMemcpyAsync(grads, m->g + k * m->P, m->P * 4, cudaMemcpyDeviceToHost, m->stream));
  float hl[64];
  MCK(cudaMemcpyAsync(hl, m->loss, m->K * 4, cudaMemcpyDeviceToHost, m->stream));
  MCK(cudaStreamSynchronize(m->stream));
  if (loss) *loss = hl[k];
  return LB_OK;
}

lb_status lb_mlp_train(lb_mlp* m, int steps, float lr, float lr_min, float wd, float* losses) {
  if (!m || steps < 1 || m->n < 1 || !(lr > 0)) return LB_ERR_ARG;
  Sched sc = {-1, steps, lr, lr_min, wd};  // every step's gradient launch counts it
  MCK(cudaMemcpyAsync(m->sched, &sc, sizeof sc, cudaMemcpyHostToDevice, m->stream));
  if (!m->gexec && steps >= kGraphSteps) {
    MCK(cudaStreamBeginCapture(m->cap, cudaStreamCaptureModeThreadLocal));
    cudaError_t e = cudaSuccess;
    for (int k = 0; k < kGraphSteps && e == cudaSuccess; ++k) e = train_step(m, m->cap);
    cudaGraph_t g = NULL;
    cudaError_t e2 = cudaStreamEndCapture(m->cap, &g);
    if (e == cudaSuccess) e = e2;
    if (e == cudaSuccess) e = cudaGraphInstantiate(&m->gexec, g, 0);
    if (g) cudaGraphDestroy(g);
    if (e != cudaSuccess) return merr(m, "graph capture failed: %s", cudaGetErrorString(e)), LB_ERR_CUDA;
  }
  MCK(cudaMemsetAsync(m->loss, 0, m->K * sizeof(float), m->stream));
  for (int i = 0; i < steps / kGraphSteps; ++i) MCK(cudaGraphLaunch(m->gexec, m->stream));
  for (int i = 0; i < steps % kGraphSteps; ++i) MCK(train_step(m, m->stream));
  if (losses) {
    // loss of the final parameters (the last update cleared the sums)
    const int rt = rows_plan(m, m->n, true);
    MCK(rt ? rows_train(m, rt, m->stream) : forward(m, m->n, m->xb, true, m->stream));
    MCK(cudaMemcpyAsync(losses, m->loss, m->K * 4, cudaMemcpyDeviceToHost, m->stream));
  }
  MCK(cudaStreamSynchronize(m->stream));
  return LB_OK;
}

static lb_status predict(lb_mlp* m, int n, const float* x, float* mean, float* sd, float* members) {
  MCK(cudaMemcpyAsync(m->xin, x, (size_t)n * m->nin * 4, cudaMemcpyHostToDevice, m->stream));
  const int rt = rows_plan(m, n, false), part = predict_part(m, rt, n);
  const long O = m->nout;
  if (!rt) {
    pack_x_kernel<<<blocks_for(m, 16L * n), 256, 0, m->stream>>>(m->xin, n, m->nin, m->xbp);
    MCK(cudaGetLastError());
    MCK(forward(m, n, m->xbp, false, m->stream));
  }
  for (int r0 = 0, c = 0; r0 < n; r0 += part, ++c) {
    const int rows = n - r0 < part ? n - r0 : part;
    if (rt) MCK(rows_predict(m, rt, r0, rows, m->stream));
    MCK(launch_pdl(ensemble_kernel, dim3(blocks_for(m, rows * O / 4)), 256, 0, m->stream, (const float*)m->y + r0 * O,
                   m->K, m->maxb * O, rows * O, m->mean + r0 * O, m->sd + r0 * O));
    if (part < n) MCK(cudaEventRecord(m->done[c], m->stream));
  }
  const size_t out = (size_t)n * O * 4;
  const lbk::HostRange host[3] = {{mean, out}, {sd, out}, {members, out * m->K}};
  // beside the kernels; with pages to make, which takes longer than they do, parts no longer pay
  const int step = lbk::populate_host(host, 3) ? n : part;
  cudaStream_t s = step < n ? m->cap : m->stream;
  for (int r0 = 0, c = 0; r0 < n; r0 += step, ++c) {
    const size_t bytes = (n - r0 < step ? n - r0 : step) * O * 4;
    if (step < n) MCK(cudaStreamWaitEvent(s, m->done[c], 0));
    MCK(cudaMemcpyAsync(mean + r0 * O, m->mean + r0 * O, bytes, cudaMemcpyDeviceToHost, s));
    MCK(cudaMemcpyAsync(sd + r0 * O, m->sd + r0 * O, bytes, cudaMemcpyDeviceToHost, s));
    if (members)
      for (int k = 0; k < m->K; ++k)
        MCK(cudaMemcpyAsync(members + ((size_t)k * n + r0) * O, m->y + ((size_t)k * m->maxb + r0) * O, bytes,
                            cudaMemcpyDeviceToHost, s));
  }
  MCK(cudaStreamSynchronize(s));  // (the copies follow the last kernels)
  return LB_OK;
}

lb_status lb_mlp_predict(lb_mlp* m, int n, const float* x, float* mean, float* sd, float* members) {
  if (!m || n < 1 || !x || !mean || !sd) return LB_ERR_ARG;
  if (n > m->maxb) return merr(m, "batch larger than max_batch"), LB_ERR_ARG;
  const lb_status st = predict(m, n, x, mean, sd, members);
  if (st != LB_OK) {  // no copy into the caller's arrays outlives the call
    cudaStreamSynchronize(m->stream);
    cudaStreamSynchronize(m->cap);
  }
  return st;
}

const char* lb_mlp_last_error(const lb_mlp* m) { return m ? m->err : g_mlp_err; }

}  // extern "C"
