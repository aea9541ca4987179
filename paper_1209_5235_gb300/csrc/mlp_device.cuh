// mlp_device.cuh -- the candidate-proposal MLP on the tensor cores (sm_103a).
//
// Network: 9 -> 64 -> 64 -> 32, GELU (erf form) after the two hidden layers,
// softmax over the first n_cand of the 32 outputs.  Inputs: the point in the
// voxel node's own coordinates (3, each in [-1, 1]), the direction (3), log E
// scaled to ~[0, 1], n_cand / 32 and 1.  Output: the list slot of the daughter
// the ray most likely enters first.  The proposal only orders the exact
// candidate tests; it never changes a result.
//
// Inference is warp-level: the 32 lanes' feature rows form a 32 x 16 BF16 tile
// (K padded from 9), and each layer is a few mma.sync m16n8k16 (BF16 inputs,
// FP32 accumulation) against BF16 weights held in shared memory.  A warp-level
// MMA is the right tensor-core instruction here: the persistent transport
// kernel runs its warps independently, so CTA-wide tcgen05 tiles (128 rows,
// TMEM, one issuing thread per CTA) cannot be formed inside it.
#pragma once

#include <cuda_bf16.h>

#include <cstdint>

namespace g4n {
namespace mlp {

constexpr int kIn = 9, kInPad = 16, kHid = 64, kOut = 32;
// padded row strides (bf16 elements) to keep shared-memory fragment loads conflict free
constexpr int kSIn = 24, kSHid = 72, kSOut = 33;
constexpr int kNParams = kIn * kHid + kHid + kHid * kHid + kHid + kHid * kOut + kOut;  // 6880

// Shared-memory image of the weights: transposed (n-major) BF16 with padded rows, FP32 biases.
struct SmemWeights {
  __nv_bfloat16 w1t[kHid * kSIn];   // [n][k], k < 16 (rows 9..15 zero)
  __nv_bfloat16 w2t[kHid * kSHid];  // [n][k], k < 64
  __nv_bfloat16 w3t[kOut * kSHid];  // [n][k], k < 64
  float b1[kHid], b2[kHid], b3[kOut];
};

// Per-warp scratch: input tile and FP32 logits.
struct SmemWarp {
  __nv_bfloat16 x[32 * kSIn];
  float logits[32 * kSOut];
};
static_assert(sizeof(SmemWeights) % 16 == 0 && sizeof(SmemWarp) % 16 == 0, "16-byte rows for ldmatrix");

__device__ __forceinline__ uint32_t ld_pair(const __nv_bfloat16 *p) { return *reinterpret_cast<const uint32_t *>(p); }

__device__ __forceinline__ void mma_bf16(float &d0, float &d1, float &d2, float &d3, uint32_t a0, uint32_t a1,
                                         uint32_t a2, uint32_t a3, uint32_t b0, uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};\n"
      : "+f"(d0), "+f"(d1), "+f"(d2), "+f"(d3)
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }

// GELU for outputs that are rounded to BF16: max(x, 0) - |x| tail(|x|), the normal distribution's tail as 2^P with P of
// degree 10, fitted to its logarithm on [0, 13] (least squares, reweighted towards equal errors of y tail(y): 3e-10) and
// decreasing beyond.  No branches, 16 instructions, about half of the erf form's, and closer to 64 bits: largest error on
// [-10, 10] 2.4e-7, root mean square 4.6e-8 (erf form 4.9e-7, 6.4e-8), on [-1, 1] 5.9e-8, 1.2e-8 (8.2e-8, 1.3e-8).
// Stack of plates 13.25 -> 12.67 ms.
__device__ __forceinline__ float gelu16(float x) {
  const float y = fabsf(x);
  float p = -5.68980263e-08f;
  p = fmaf(p, y, 1.40031331e-06f);
  p = fmaf(p, y, -1.52829445e-05f);
  p = fmaf(p, y, 9.4810299e-05f);
  p = fmaf(p, y, -0.000324589254f);
  p = fmaf(p, y, 6.37534364e-05f);
  p = fmaf(p, y, 0.00689659362f);
  p = fmaf(p, y, -0.0524214247f);
  p = fmaf(p, y, -0.459223877f);
  p = fmaf(p, y, -1.15110412f);
  p = fmaf(p, y, -1.0f);
  asm("ex2.approx.ftz.f32 %0, %1;" : "=f"(p) : "f"(p));
  return fmaf(-fminf(y, 3e38f), p, fmaxf(x, 0.f));
}

// Four 8 x 8 BF16 matrices; lane i gives the address of row i & 7 of matrix i >> 3.
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const __nv_bfloat16 *p) {
  const uint32_t a = (uint32_t)__cvta_generic_to_shared(p);
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]) : "r"(a) : "memory");
}

__device__ __forceinline__ uint32_t gelu_pair(float x, float y) {
  const __nv_bfloat162 h = __floats2bfloat162_rn(gelu16(x), gelu16(y));
  return *reinterpret_cast<const uint32_t *>(&h);
}

// Columns 8 nt .. 8 nt + 7 of `in` W + b for 16 rows: `in` as K / 16 A fragments, wt [n][k] with row stride SB.
template <int K, int SB>
__device__ __forceinline__ void column_tile(float (&d)[4], const uint32_t (&in)[K / 16][4], const __nv_bfloat16 *wt,
                                            const float *bias, int nt) {
  const int lane = threadIdx.x & 31, col = nt * 8 + 2 * (lane & 3);
  d[0] = d[2] = bias[col];
  d[1] = d[3] = bias[col + 1];
#pragma unroll
  for (int k2 = 0; k2 < K / 32; ++k2) {
    uint32_t b[4];
    ldsm4(b, wt + (nt * 8 + (lane & 7)) * SB + k2 * 32 + (lane >> 3) * 8);
    mma_bf16(d[0], d[1], d[2], d[3], in[2 * k2][0], in[2 * k2][1], in[2 * k2][2], in[2 * k2][3], b[0], b[1]);
    mma_bf16(d[0], d[1], d[2], d[3], in[2 * k2 + 1][0], in[2 * k2 + 1][1], in[2 * k2 + 1][2], in[2 * k2 + 1][3], b[2],
             b[3]);
  }
  if (K == 16) {
    const uint32_t *b = reinterpret_cast<const uint32_t *>(wt + (nt * 8 + (lane >> 2)) * SB + 2 * (lane & 3));
    mma_bf16(d[0], d[1], d[2], d[3], in[0][0], in[0][1], in[0][2], in[0][3], b[0], b[4]);
  }
}

// GELU of a layer with 64 outputs, as the next layer's A fragments: the accumulator fragments of two column tiles are the
// A fragment of 16 columns.
template <int K, int SB>
__device__ __forceinline__ void hidden_layer(uint32_t (&out)[4][4], const uint32_t (&in)[K / 16][4],
                                             const __nv_bfloat16 *wt, const float *bias) {
#pragma unroll
  for (int nt = 0; nt < kHid / 8; ++nt) {
    float d[4];
    column_tile<K, SB>(d, in, wt, bias, nt);
    out[nt >> 1][2 * (nt & 1)] = gelu_pair(d[0], d[1]);
    out[nt >> 1][2 * (nt & 1) + 1] = gelu_pair(d[2], d[3]);
  }
}

// Warp-collective forward pass.  Every lane writes its feature row (zeros if it has none)
// before the call; afterwards lane i's logits are in W.logits[i * kSOut ...].
//
// 16 rows at a time; the hidden layers never leave the registers and weights come by ldmatrix.  (Handed on
// through shared memory they cost six loads a product, and a block of the staged step kernel took 60 KB, three blocks an SM;
// it takes 41 KB now and registers allow four.  10^6 tracks in the stack of plates 16.1 -> 13.3 ms.)
__device__ __forceinline__ void forward_warp(const SmemWeights &Wt, SmemWarp &W) {
  const int lane = threadIdx.x & 31;
  __syncwarp();
#pragma unroll 1
  for (int mt = 0; mt < 2; ++mt) {
    uint32_t x[1][4], h1[4][4], h2[4][4];
    ldsm4(x[0], W.x + (mt * 16 + (lane & 15)) * kSIn + (lane >> 4) * 8);
    hidden_layer<kInPad, kSIn>(h1, x, Wt.w1t, Wt.b1);
    hidden_layer<kHid, kSHid>(h2, h1, Wt.w2t, Wt.b2);
    float *o = W.logits + (mt * 16 + (lane >> 2)) * kSOut + 2 * (lane & 3);
#pragma unroll
    for (int nt = 0; nt < kOut / 8; ++nt) {
      float d[4];
      column_tile<kHid, kSHid>(d, h2, Wt.w3t, Wt.b3, nt);
      o[nt * 8] = d[0];
      o[nt * 8 + 1] = d[1];
      o[nt * 8 + 8 * kSOut] = d[2];
      o[nt * 8 + 8 * kSOut + 1] = d[3];
    }
  }
  __syncwarp();
}

// Lane's feature row into the warp's input tile.
__device__ __forceinline__ void put_features(SmemWarp &W, const float *f) {
  const int lane = threadIdx.x & 31;
#pragma unroll
  for (int k = 0; k < kInPad; k += 2)
    *reinterpret_cast<__nv_bfloat162 *>(W.x + lane * kSIn + k) =
        __floats2bfloat162_rn(k < kIn ? f[k] : 0.f, k + 1 < kIn ? f[k + 1] : 0.f);
}

// Masked argmax of the lane's logits over slots [0, n) (first slot wins ties).
__device__ __forceinline__ int argmax_row(const SmemWarp &W, int n) {
  const int lane = threadIdx.x & 31;
  int best = 0;
  float bv = W.logits[lane * kSOut];
  for (int s = 1; s < n; ++s) {
    const float x = W.logits[lane * kSOut + s];
    if (x > bv) {
      bv = x;
      best = s;
    }
  }
  return best;
}

// Fill the shared-memory weight image from the device copy (block-collective).
__device__ __forceinline__ void load_weights(SmemWeights &S, const SmemWeights *g) {
  const int n = sizeof(SmemWeights) / 16;
  const uint4 *src = reinterpret_cast<const uint4 *>(g);
  uint4 *dst = reinterpret_cast<uint4 *>(&S);
  for (int i = threadIdx.x; i < n; i += blockDim.x) dst[i] = src[i];
}

}  // namespace mlp
}  // namespace g4n
