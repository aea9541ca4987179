// mlp_train.cuh -- training steps of the candidate-proposal MLP as one persistent cooperative kernel
// (included once, by mlp.cu).
//
// A minibatch of this network is little work -- 4096 rows are 0.17 GFLOP of GEMM -- and every step
// needs the weights of the one before it, so training is bound by the length of a step's serial
// chain, not by arithmetic.  As separate kernels per GEMM and elementwise pass a step is 26
// launches and clears in a row, 186 us at 4096 rows on GB300; here all steps of an epoch are one
// launch and a step takes 15 us (an epoch of 2^20 samples: 49 -> 3.8 ms with the loading of the parameters
// before it and their reading back).  A step:
//   1. forward and backward of the block's row tiles; what the gradients need goes to global memory (L2): the
//      activations and deltas as mma fragments, the deltas in FP32 as well; grid barrier;
//   2. partial gradients, one warp per 16 x 16 tile of a weight gradient and chunk of rows, and per two columns
//      and eighth of a bias gradient; grid barrier;
//   3. each block adds the partials of its share of the parameters and updates them (Adam); grid barrier;
//      reload of the weights' image (31 KB, from L2).
//
// The sums are those of the plain kernels (mlp.cu), operation by operation: a chunk has the rows that one K chunk of
// their GEMM has, multiplied 16 rows after the other from a zero accumulator; the chunks are added in ascending order,
// one of the orders in which the plain kernels' atomics may arrive; a bias gradient has k_colsum's threads, tree and
// warps.  BF16 rounding of the next operands makes 1e-3 of a last bit within 250 steps, so that another grouping of
// the sums would be another training.  Gradients of up to two chunks, and trainings on them, are the plain kernels' bit for
// bit.  The order is fixed: results do not vary from run to run.
//
// A tile is 32 rows by all 64 hidden columns on 8 warps (2 row halves x 4 column groups of 16), so
// that a minibatch of 4096 rows fills 128 SMs and a layer is a few mma.sync per warp.  Products are
// mma.sync m16n8k16 (BF16 in, FP32 accumulation), the K chunks of an output in ascending order from a
// zero accumulator, bias added afterwards.  tcgen05 tiles need 128 rows per CTA: a quarter of the SMs
// and four times the elementwise work (erf, exp) per SM, on a chain that waits for latency anyway, and
// its sums over K are not the ones above.  ldmatrix.trans transposes the operands of the weight gradients once, where
// they are written; phase 2 reads whole fragments, 512 bytes a warp.
#pragma once

#include <cuda_bf16.h>

#include <cstdint>

#include "mlp_device.cuh"

namespace g4n {
namespace mlp {

constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kIn * kHid, kOffW2 = kOffB1 + kHid, kOffB2 = kOffW2 + kHid * kHid,
              kOffW3 = kOffB2 + kHid, kOffB3 = kOffW3 + kHid * kOut;

constexpr int kTrRows = 32, kTrThreads = 256;
constexpr int kSOutB = 40;                       // padded row stride of 32 BF16 columns (16-byte rows for ldmatrix)
constexpr unsigned kBarrierPolls = 1u << 22;     // polls of a grid barrier before it gives up (seconds)

__device__ __forceinline__ float gelu_grad(float x, float e) {  // e = erf(x / sqrt 2)
  return 0.5f * (1.0f + e) + x * 0.39894228040143268f * expf(-0.5f * x * x);
}

// Device control block of the kernel.
struct TrainCtrl {
  unsigned int arrived;   // grid barrier: blocks arrived, over all barriers of the launch
  unsigned int failed;    // a barrier gave up
  unsigned int begun;     // every block has kept its share of the parameters and moments (TrainParams::kept), updates may have begun
  unsigned int pad;
  double loss;            // sum of the losses over the launch
};

// A 16-row step of a minibatch as the weight-gradient products read it: A fragments (16 columns) of H1, H2 and X, B
// fragments (2 x 8 columns) of the deltas, 32 lanes x 16 bytes each.
constexpr int kFragH1 = 0, kFragH2 = 4, kFragX = 8, kFragD2 = 9, kFragD1 = 13, kFragD3 = 17, kFrags = 19;
constexpr int kColZ3 = 0, kColZ2 = kOut, kColZ1 = kOut + kHid, kCols = kOut + 2 * kHid;   // columns of the FP32 deltas
constexpr int kChunkTiles = 28;                  // 16 x 16 tiles of the weight gradients: W2 16, W3 8, W1 4
constexpr int kColParts = 8;                     // partial sums of a bias gradient: k_colsum's warps
constexpr int kMaxChunks = 256;                  // K chunks of the plain kernels' GEMM

struct TrainParams {
  int64_t n;                        // samples
  const float *feat;
  const int32_t *label, *ncand;
  int steps;
  int64_t batch;                    // rows of a minibatch
  int64_t chunk;                    // rows of a partial weight gradient (a multiple of 16)
  int chunks;
  bool permuted;                    // row r of step s is sample ((s batch + r) mod n * stride + offset) mod n, else s batch + r
  uint64_t stride, offset;
  float inv_scale;
  float *P, *M, *V;                 // parameters and Adam moments; M null: gradients of one step into `grads` instead
  float *grads;
  float *kept;                      // P, M and V as the launch found them, for a caller whose launch fails
  uint4 *frag;                      // [16-row step][kFrags][32]
  float *delta;                     // [kCols][delta_ld]
  int64_t delta_ld;
  float *part;                      // chunks x kNParams partial weight gradients, then kColParts x kCols bias partials
  double *part_loss;                // gridDim.x
  const float2 *bias_corr;          // per step: Adam's 1 / (1 - beta^t)
  float lr, b1, b2, eps;
  TrainCtrl *ctrl;
  unsigned polls;                   // of a grid barrier before it gives up
  struct TrainWeights *img;
};

// The weights as the products read them.  The blocks keep one image in global memory, each writing its share of the
// parameters, and copy it to shared memory 16 bytes at a time.
struct alignas(16) TrainWeights {
  __nv_bfloat16 w1t[kHid * kSIn];    // [n][k]: B operands of the forward products (padding stays zero)
  __nv_bfloat16 w2t[kHid * kSHid];
  __nv_bfloat16 w3t[kOut * kSHid];
  __nv_bfloat16 w2[kHid * kSHid];    // [k][n]: B operands of the backward products
  __nv_bfloat16 w3[kHid * kSOutB];
  float b1[kHid], b2[kHid], b3[kOut];
};
static_assert(sizeof(TrainWeights) % 16 == 0, "copied in 16-byte pieces");

struct TrainSmem {
  TrainWeights w;
  __nv_bfloat16 x[kTrRows * kSIn], h1[kTrRows * kSHid], h2[kTrRows * kSHid];
  __nv_bfloat16 d3[kTrRows * kSOutB], d2[kTrRows * kSHid], d1[kTrRows * kSHid];
  float logits[kTrRows * kSOut];
  double lossw[kTrThreads / 32];
  int32_t label[kTrRows], ncand[kTrRows];
};

__device__ __forceinline__ void ldsm4t(uint32_t &r0, uint32_t &r1, uint32_t &r2, uint32_t &r3, const __nv_bfloat16 *p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r0), "=r"(r1), "=r"(r2), "=r"(r3) : "r"(a) : "memory");
}
// d[4] (+)= a row-major 16 x K tile of `in` (row stride SA, first row row0) times B from wt ([n][k], stride SB) at
// columns n0 .. n0 + 7.
template <int K, int SA, int SB>
__device__ __forceinline__ void tile_mma(float d[4], const __nv_bfloat16 *in, int row0, const __nv_bfloat16 *wt, int n0) {
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const __nv_bfloat16 *a_lo = in + (row0 + g) * SA + 2 * q, *a_hi = a_lo + 8 * SA;
  const __nv_bfloat16 *bp = wt + (n0 + g) * SB + 2 * q;
#pragma unroll
  for (int kt = 0; kt < K / 16; ++kt)
    mma_bf16(d[0], d[1], d[2], d[3], ld_pair(a_lo + kt * 16), ld_pair(a_hi + kt * 16), ld_pair(a_lo + kt * 16 + 8),
             ld_pair(a_hi + kt * 16 + 8), ld_pair(bp + kt * 16), ld_pair(bp + kt * 16 + 8));
}

// Fragment of 16 columns from c0 and 16 rows from k of a row-major tile, transposed, to `out`.  As an A operand the second
// 8 x 8 matrix holds the next columns, as two B operands the next rows.
template <bool AS_A, int STRIDE>
__device__ __forceinline__ void put_fragment(uint4 *out, const __nv_bfloat16 *t, int k, int c0) {
  const int lane = threadIdx.x & 31, r = lane & 7, mat = lane >> 3;
  const int dk = AS_A ? mat >> 1 : mat & 1, dc = AS_A ? mat & 1 : mat >> 1;
  uint4 f;
  ldsm4t(f.x, f.y, f.z, f.w, t + (k + dk * 8 + r) * STRIDE + c0 + dc * 8);
  __stcg(out + lane, f);
}

// Phase 2, one 16 x 16 tile of a chunk's weight gradients: dW2 = H1^T dZ2, dW3 = H2^T dZ3, dW1 = X^T dZ1.
__device__ __forceinline__ void chunk_gradient(const TrainParams &T, int z, int tile) {
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  int fa, fb, off, ld, m0, n0;
  if (tile < 16) {
    fa = kFragH1 + (tile >> 2), fb = kFragD2 + (tile & 3), off = kOffW2, ld = kHid, m0 = (tile >> 2) * 16, n0 = (tile & 3) * 16;
  } else if (tile < 24) {
    const int t = tile - 16;
    fa = kFragH2 + (t >> 1), fb = kFragD3 + (t & 1), off = kOffW3, ld = kOut, m0 = (t >> 1) * 16, n0 = (t & 1) * 16;
  } else {
    fa = kFragX, fb = kFragD1 + (tile - 24), off = kOffW1, ld = kHid, m0 = 0, n0 = (tile - 24) * 16;
  }
  const int64_t s0 = z * T.chunk / 16, s1 = min(T.batch, (z + 1) * T.chunk) / 16;
  const uint4 *A = T.frag + (s0 * kFrags + fa) * 32 + lane, *B = T.frag + (s0 * kFrags + fb) * 32 + lane;
  float d[2][4] = {};
#pragma unroll 8
  for (int64_t s = s0; s < s1; ++s, A += kFrags * 32, B += kFrags * 32) {
    const uint4 a = __ldcg(A), b = __ldcg(B);
    mma_bf16(d[0][0], d[0][1], d[0][2], d[0][3], a.x, a.y, a.z, a.w, b.x, b.y);
    mma_bf16(d[1][0], d[1][1], d[1][2], d[1][3], a.x, a.y, a.z, a.w, b.z, b.w);
  }
  float *G = T.part + (int64_t)z * kNParams + off + (m0 + g) * ld + n0 + 2 * q;
#pragma unroll
  for (int t = 0; t < 2; ++t) {
    __stcg(reinterpret_cast<float2 *>(G + t * 8), make_float2(d[t][0], d[t][1]));
    if (tile < 24 || g + 8 < kIn) __stcg(reinterpret_cast<float2 *>(G + t * 8 + 8 * ld), make_float2(d[t][2], d[t][3]));
  }
}

// Phase 2, columns c and c + 1 of the FP32 deltas: the sum that warp w of k_colsum has.
__device__ __forceinline__ void column_sums(const TrainParams &T, int c, int w) {
  const int lane = threadIdx.x & 31;
  const float *x = T.delta + c * T.delta_ld, *y = x + T.delta_ld;
  float a = 0.f, b = 0.f;
#pragma unroll 16
  for (int64_t r = w * 32 + lane; r < T.batch; r += 32 * kColParts) {
    a += __ldcg(x + r);
    b += __ldcg(y + r);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    b += __shfl_xor_sync(0xffffffffu, b, o);
  }
  if (lane == 0)
    __stcg(reinterpret_cast<float2 *>(T.part + (int64_t)T.chunks * kNParams + w * kCols + c), make_float2(a, b));
}

// Phase 3, the gradient of parameter p: its partials, in ascending order.
__device__ __forceinline__ float gradient_of(const TrainParams &T, int p) {
  int col = -1;
  if (p >= kOffB3) col = kColZ3 + p - kOffB3;
  else if (p >= kOffB2 && p < kOffW3) col = kColZ2 + p - kOffB2;
  else if (p >= kOffB1 && p < kOffW2) col = kColZ1 + p - kOffB1;
  const float *g = col < 0 ? T.part + p : T.part + (int64_t)T.chunks * kNParams + col;
  const int n = col < 0 ? T.chunks : kColParts, step = col < 0 ? kNParams : kCols;
  float s = 0.f;
#pragma unroll 16
  for (int i = 0; i < n; ++i) s += __ldcg(g + (int64_t)i * step);
  return s;
}

// Parameter p of value v into the image.
__device__ __forceinline__ void train_image(TrainWeights &W, int p, float v) {
  const __nv_bfloat16 w = __float2bfloat16_rn(v);
  if (p < kOffB1) {
    W.w1t[(p & 63) * kSIn + (p >> 6)] = w;
  } else if (p < kOffW2) {
    W.b1[p - kOffB1] = v;
  } else if (p < kOffB2) {
    const int k = (p - kOffW2) >> 6, n = (p - kOffW2) & 63;
    W.w2t[n * kSHid + k] = w;
    W.w2[k * kSHid + n] = w;
  } else if (p < kOffW3) {
    W.b2[p - kOffB2] = v;
  } else if (p < kOffB3) {
    const int k = (p - kOffW3) >> 5, n = (p - kOffW3) & 31;
    W.w3t[n * kSHid + k] = w;
    W.w3[k * kSOutB + n] = w;
  } else {
    W.b3[p - kOffB3] = v;
  }
}

// The image to shared memory (written by other blocks: read past the L1).
__device__ __forceinline__ void train_load_weights(TrainWeights &S, const TrainWeights *img) {
  const uint4 *src = reinterpret_cast<const uint4 *>(img);
  uint4 *dst = reinterpret_cast<uint4 *>(&S);
  constexpr int kVec = sizeof(TrainWeights) / 16;
#pragma unroll
  for (int i = 0; i < (kVec + kTrThreads - 1) / kTrThreads; ++i) {
    const int e = threadIdx.x + i * kTrThreads;
    if (e < kVec) dst[e] = __ldcg(src + e);
  }
}

// Barrier number `k` (1, 2, ...) of the grid (cooperative launch: every block is resident).  A block that has polled
// `cap` times sets `failed` and ends; the others see it at their next barrier (or while they poll) and end too.
__device__ __forceinline__ bool grid_barrier(TrainCtrl *C, unsigned k, unsigned cap) {
  __shared__ bool ok;
  __syncthreads();
  if (threadIdx.x == 0) {
    __threadfence();
    atomicAdd(&C->arrived, 1u);
    const unsigned target = k * gridDim.x;
    unsigned polls = 0, seen;
    for (;;) {
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(seen) : "l"(&C->arrived) : "memory");
      if ((int)(seen - target) >= 0 || ++polls >= cap) break;
      if ((polls & 1023u) == 0 && *(volatile unsigned int *)&C->failed) break;
    }
    if ((int)(seen - target) < 0) atomicExch(&C->failed, 1u);
    ok = *(volatile unsigned int *)&C->failed == 0u;
  }
  __syncthreads();
  return ok;
}

// One element of a tile's inputs: sample row r = e / 11, its nine features, label and candidate count.
struct TrainFetch {
  uint32_t bits[2];
};

__device__ __forceinline__ TrainFetch train_fetch(const TrainParams &T, int64_t step, int64_t tile) {
  TrainFetch f{{0u, 0u}};
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int e = threadIdx.x + j * kTrThreads;
    const int r = e / (kIn + 2), k = e % (kIn + 2);
    const int64_t row = tile * kTrRows + r;
    if (r >= kTrRows || row >= T.batch || step >= T.steps) continue;
    uint64_t at = (uint64_t)(step * T.batch + row);
    if (T.permuted) at = ((at % (uint64_t)T.n) * T.stride + T.offset) % (uint64_t)T.n;
    if (k < kIn) f.bits[j] = __float_as_uint(__ldg(T.feat + at * kIn + k));
    else f.bits[j] = (uint32_t)__ldg((k == kIn ? T.label : T.ncand) + at);
  }
  return f;
}

__device__ __forceinline__ void train_put(TrainSmem &S, const TrainFetch &f) {
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int e = threadIdx.x + j * kTrThreads;
    const int r = e / (kIn + 2), k = e % (kIn + 2);
    if (r >= kTrRows) continue;
    if (k < kIn) S.x[r * kSIn + k] = __float2bfloat16_rn(__uint_as_float(f.bits[j]));
    else (k == kIn ? S.label : S.ncand)[r] = (int32_t)f.bits[j];
  }
}

__global__ void __launch_bounds__(kTrThreads) k_mlp_train(const TrainParams T) {
  extern __shared__ __align__(16) unsigned char smem[];
  TrainSmem &S = *reinterpret_cast<TrainSmem *>(smem);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, g = lane >> 2, q = lane & 3;
  const int wm = (warp & 1) * 16, wn = (warp >> 1) * 16;   // the warp's rows and hidden columns of a tile
  const int64_t tiles = (T.batch + kTrRows - 1) / kTrRows;
  const int tasks = T.chunks * kChunkTiles, wide = (int)gridDim.x * (kTrThreads / 32);
  for (int e = tid; e < kTrRows * kSIn; e += kTrThreads) S.x[e] = __float2bfloat16_rn(0.f);   // columns 9 .. 15 stay zero
  // the share of the parameters that this block updates
  const int share = (kNParams + (int)gridDim.x - 1) / (int)gridDim.x;
  const int p0 = min(kNParams, (int)blockIdx.x * share), p1 = min(kNParams, p0 + share);
  unsigned barriers = 0;
  for (int p = p0 + tid; p < p1; p += kTrThreads) {
    const float v = T.P[p];
    train_image(*T.img, p, v);
    if (T.M) {
      T.kept[p] = v;
      T.kept[kNParams + p] = T.M[p];
      T.kept[2 * kNParams + p] = T.V[p];
    }
  }
  if (!grid_barrier(T.ctrl, ++barriers, T.polls)) return;
  if (blockIdx.x == 0 && tid == 0) T.ctrl->begun = 1u;
  TrainFetch next = train_fetch(T, 0, blockIdx.x);
#pragma unroll 1
  for (int64_t step = 0; step < T.steps; ++step) {
    __syncthreads();
    train_load_weights(S.w, T.img);
    double loss = 0.0;   // every row in FP64, as the plain kernel adds them
#pragma unroll 1
    for (int64_t tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
      train_put(S, next);
      // the next tile's inputs come while this one is worked on
      const bool more = tile + gridDim.x < tiles;
      next = train_fetch(T, more ? step : step + 1, more ? tile + gridDim.x : blockIdx.x);
      __syncthreads();
      // fragments of the warp: 16-row step fk of the tile, 16 columns from 16 fc
      const int fk = warp & 1, fc = warp >> 1;
      uint4 *frag = T.frag + (tile * 2 + fk) * (kFrags * 32);
      float *delta = T.delta + tile * kTrRows;
      // forward; the pre-activations and their erf stay in registers for the backward pass
      float z1[2][4], e1[2][4], z2[2][4], e2[2][4];
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const int col = wn + t * 8 + 2 * q;
        float d[4] = {0.f, 0.f, 0.f, 0.f}, h[4];
        tile_mma<kInPad, kSIn, kSIn>(d, S.x, wm, S.w.w1t, wn + t * 8);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          z1[t][i] = d[i] + S.w.b1[col + (i & 1)];
          e1[t][i] = erff(z1[t][i] * 0.70710678118654752f);
          h[i] = 0.5f * z1[t][i] * (1.0f + e1[t][i]);
        }
        *reinterpret_cast<__nv_bfloat162 *>(S.h1 + (wm + g) * kSHid + col) = __floats2bfloat162_rn(h[0], h[1]);
        *reinterpret_cast<__nv_bfloat162 *>(S.h1 + (wm + g + 8) * kSHid + col) = __floats2bfloat162_rn(h[2], h[3]);
      }
      __syncthreads();
      put_fragment<true, kSHid>(frag + (kFragH1 + fc) * 32, S.h1, fk * 16, fc * 16);
#pragma unroll
      for (int t = 0; t < 2; ++t) {
        const int col = wn + t * 8 + 2 * q;
        float d[4] = {0.f, 0.f, 0.f, 0.f}, h[4];
        tile_mma<kHid, kSHid, kSHid>(d, S.h1, wm, S.w.w2t, wn + t * 8);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          z2[t][i] = d[i] + S.w.b2[col + (i & 1)];
          e2[t][i] = erff(z2[t][i] * 0.70710678118654752f);
          h[i] = 0.5f * z2[t][i] * (1.0f + e2[t][i]);
        }
        *reinterpret_cast<__nv_bfloat162 *>(S.h2 + (wm + g) * kSHid + col) = __floats2bfloat162_rn(h[0], h[1]);
        *reinterpret_cast<__nv_bfloat162 *>(S.h2 + (wm + g + 8) * kSHid + col) = __floats2bfloat162_rn(h[2], h[3]);
      }
      __syncthreads();
      put_fragment<true, kSHid>(frag + (kFragH2 + fc) * 32, S.h2, fk * 16, fc * 16);
      {
        const int n0 = (warp >> 1) * 8, col = n0 + 2 * q;
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        tile_mma<kHid, kSHid, kSHid>(d, S.h2, wm, S.w.w3t, n0);
#pragma unroll
        for (int i = 0; i < 4; ++i)
          S.logits[(wm + g + 8 * (i >> 1)) * kSOut + col + (i & 1)] = d[i] + S.w.b3[col + (i & 1)];
      }
      __syncthreads();
      {  // masked softmax cross-entropy: 8 lanes a row, 4 columns a lane
        const int r = tid >> 3, sub = tid & 7;
        const bool valid = (int64_t)tile * kTrRows + r < T.batch;
        const int nc = max(1, min(kOut, S.ncand[r])), y = S.label[r];
        const float *z = S.logits + r * kSOut;
        float zz[4], mx = -INFINITY, s = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          zz[j] = z[sub + 8 * j];
          if (sub + 8 * j < nc) mx = fmaxf(mx, zz[j]);
        }
#pragma unroll
        for (int o = 4; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o));
#pragma unroll
        for (int j = 0; j < 4; ++j) {   // in the order of the columns, as the plain kernel sums them
          const float ex = sub + 8 * j < nc ? expf(zz[j] - mx) : 0.f;
#pragma unroll
          for (int o = 0; o < 8; ++o) s += __shfl_sync(0xffffffffu, ex, o, 8);
        }
        const float lse = mx + logf(s);
        float row_loss = 0.f;
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const int c = sub + 8 * j;
          const float p = c < nc ? expf(zz[j] - lse) : 0.f;
          const float dz = valid ? (p - (c == y ? 1.f : 0.f)) * T.inv_scale : 0.f;
          if (valid && c == y) row_loss = lse - zz[j];
          __stcg(delta + (kColZ3 + c) * T.delta_ld + r, dz);
          S.d3[r * kSOutB + c] = __float2bfloat16_rn(dz);
        }
        loss += (double)row_loss;
      }
      __syncthreads();
      if (fc < 2) put_fragment<false, kSOutB>(frag + (kFragD3 + fc) * 32, S.d3, fk * 16, fc * 16);
      else if (fc == 2) put_fragment<true, kSIn>(frag + kFragX * 32, S.x, fk * 16, 0);
#pragma unroll
      for (int t = 0; t < 2; ++t) {  // dZ2 = (dZ3 W3^T) gelu'(Z2)
        const int col = wn + t * 8 + 2 * q;
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        tile_mma<kOut, kSOutB, kSOutB>(d, S.d3, wm, S.w.w3, wn + t * 8);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          d[i] *= gelu_grad(z2[t][i], e2[t][i]);
          __stcg(delta + (kColZ2 + col + (i & 1)) * T.delta_ld + wm + g + 8 * (i >> 1), d[i]);
        }
        *reinterpret_cast<__nv_bfloat162 *>(S.d2 + (wm + g) * kSHid + col) = __floats2bfloat162_rn(d[0], d[1]);
        *reinterpret_cast<__nv_bfloat162 *>(S.d2 + (wm + g + 8) * kSHid + col) = __floats2bfloat162_rn(d[2], d[3]);
      }
      __syncthreads();
      put_fragment<false, kSHid>(frag + (kFragD2 + fc) * 32, S.d2, fk * 16, fc * 16);
#pragma unroll
      for (int t = 0; t < 2; ++t) {  // dZ1 = (dZ2 W2^T) gelu'(Z1)
        const int col = wn + t * 8 + 2 * q;
        float d[4] = {0.f, 0.f, 0.f, 0.f};
        tile_mma<kHid, kSHid, kSHid>(d, S.d2, wm, S.w.w2, wn + t * 8);
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          d[i] *= gelu_grad(z1[t][i], e1[t][i]);
          __stcg(delta + (kColZ1 + col + (i & 1)) * T.delta_ld + wm + g + 8 * (i >> 1), d[i]);
        }
        *reinterpret_cast<__nv_bfloat162 *>(S.d1 + (wm + g) * kSHid + col) = __floats2bfloat162_rn(d[0], d[1]);
        *reinterpret_cast<__nv_bfloat162 *>(S.d1 + (wm + g + 8) * kSHid + col) = __floats2bfloat162_rn(d[2], d[3]);
      }
      __syncthreads();
      put_fragment<false, kSHid>(frag + (kFragD1 + fc) * 32, S.d1, fk * 16, fc * 16);
      // S.x, S.label and S.ncand are rewritten for the next tile: their readers are past the barrier above
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) loss += __shfl_xor_sync(0xffffffffu, loss, o);
    if (lane == 0) S.lossw[warp] = loss;
    __syncthreads();
    if (tid == 0) {
      double l = 0.0;
#pragma unroll
      for (int w = 0; w < kTrThreads / 32; ++w) l += S.lossw[w];
      T.part_loss[blockIdx.x] = step == 0 ? l : T.part_loss[blockIdx.x] + l;
    }
    if (!grid_barrier(T.ctrl, ++barriers, T.polls)) return;
    for (int task = (int)blockIdx.x + (int)gridDim.x * warp; task < tasks + kCols / 2 * kColParts; task += wide) {
      if (task < tasks) chunk_gradient(T, task / kChunkTiles, task % kChunkTiles);
      else column_sums(T, (task - tasks) / kColParts * 2, (task - tasks) % kColParts);
    }
    // the first parameters of the share and their moments are on their way while the barrier is waited for
    const bool own = T.M && p0 + tid < p1;
    float pv = own ? T.P[p0 + tid] : 0.f, mv = own ? T.M[p0 + tid] : 0.f, vv = own ? T.V[p0 + tid] : 0.f;
    if (!grid_barrier(T.ctrl, ++barriers, T.polls)) return;
    const float2 corr = T.M ? T.bias_corr[step] : make_float2(0.f, 0.f);
#pragma unroll 1
    for (int p = p0 + tid; p < p1; p += kTrThreads) {
      const float gr = gradient_of(T, p);
      if (!T.M) {
        T.grads[p] = gr;
        continue;
      }
      if (p != p0 + tid) {
        pv = T.P[p];
        mv = T.M[p];
        vv = T.V[p];
      }
      const float m = T.b1 * mv + (1.f - T.b1) * gr;
      const float v = T.b2 * vv + (1.f - T.b2) * gr * gr;
      pv -= T.lr * (m * corr.x) / (sqrtf(v * corr.y) + T.eps);
      T.M[p] = m;
      T.V[p] = v;
      T.P[p] = pv;
      train_image(*T.img, p, pv);
    }
    if (!grid_barrier(T.ctrl, ++barriers, T.polls)) return;
  }
  if (blockIdx.x == 0 && tid == 0) {
    double l = 0.0;
    for (int b = 0; b < (int)gridDim.x; ++b) l += __ldcg(T.part_loss + b);
    T.ctrl->loss = l;
  }
}

}  // namespace mlp
}  // namespace g4n
