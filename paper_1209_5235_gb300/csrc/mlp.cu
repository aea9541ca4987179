// mlp.cu -- training and inference entry points of the candidate-proposal MLP.
//
// Training (g4n_mlp_train) on large minibatches, and the BF16 gradients of
// g4n_mlp_grad on many rows, are the persistent kernel of mlp_train.cuh: BF16
// products on the tensor cores with FP32 accumulation, masked softmax
// cross-entropy, Adam on FP32 master weights.  Smaller minibatches and the FP32
// reference gradients take one kernel of this file per product and elementwise pass.
// The packed FP32 parameter layout used by the API is
//   W1[9][64], b1[64], W2[64][64], b2[64], W3[64][32], b3[32]   (6880 floats),
// W[k][n] mapping input k to output n.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <memory>
#include <new>
#include <numeric>
#include <string>

#include "g4n_internal.h"
#include "mlp_device.cuh"
#include "mlp_train.cuh"

using namespace g4n;
using namespace g4n::mlp;

namespace {

// Rows from which BF16 gradients (g4n_mlp_grad) take the persistent kernel: from three K chunks on the plain kernels'
// atomics leave the order of the partial sums open (of 400 pairs of calls on the same 768 rows 144 differed), the persistent
// kernel adds them in ascending order.  Below, one or two chunks have one sum.
constexpr int64_t kFusedRows = 768;
// Rows from which a training does.  In trainings of 768 to 1300 rows a step (three to five chunks) the atomics of the plain kernels mostly
// arrive in one order as long as a process keeps its buffers where they are, and its trainings repeat; another order ends
// 1e-4 to 5e-4 away in the weights after 200 steps, as another process with other allocations before it does.  Those
// keep the plain kernels (26 launches and clears, 170 us a step).  From eight chunks on no two runs agree (2048 rows, 200
// steps: 3e-4 to 9e-4 between any two; 4096: 1e-3), and the persistent kernel's ascending order is one of theirs.
constexpr int64_t kFusedTrainRows = 2048;

// ---------------------------------------------------------------- plain kernels
// C[M x N] += op(A)[M x K] op(B)[K x N]; A(m, k) = transA ? A[k * lda + m] : A[m * lda + k],
// B(k, n) = transB ? B[n * ldb + k] : B[k * ldb + n].  BF16: M, K multiples of 16, N a multiple of 8.

__device__ __forceinline__ float ldA(const float *A, int lda, bool tA, int m, int k) {
  return tA ? A[(int64_t)k * lda + m] : A[(int64_t)m * lda + k];
}
__device__ __forceinline__ float ldB(const float *B, int ldb, bool tB, int k, int n) {
  return tB ? B[(int64_t)n * ldb + k] : B[(int64_t)k * ldb + n];
}

__device__ __forceinline__ uint32_t pack_bf16(float a, float b) {
  const __nv_bfloat162 v = __floats2bfloat162_rn(a, b);
  return *reinterpret_cast<const uint32_t *>(&v);
}

// One warp per 16 x 8 output tile and K chunk (blockIdx.z); chunks add into C atomically.
__global__ void k_gemm_bf16(int M, int N, int K, int kchunk, const float *__restrict__ A, int lda, bool tA,
                            const float *__restrict__ B, int ldb, bool tB, float *__restrict__ C, int ldc) {
  const int lane = threadIdx.x & 31, g = lane >> 2, q = lane & 3;
  const int warp = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int tiles_n = N / 8;
  const int tm = warp / tiles_n, tn = warp % tiles_n;
  if (tm * 16 >= M) return;
  const int k0 = blockIdx.z * kchunk, k1 = min(K, k0 + kchunk);
  const int m0 = tm * 16, n0 = tn * 8;
  float d0 = 0.f, d1 = 0.f, d2 = 0.f, d3 = 0.f;
  for (int k = k0; k < k1; k += 16) {
    const int kc = k + 2 * q;
    const uint32_t a0 = pack_bf16(ldA(A, lda, tA, m0 + g, kc), ldA(A, lda, tA, m0 + g, kc + 1));
    const uint32_t a1 = pack_bf16(ldA(A, lda, tA, m0 + g + 8, kc), ldA(A, lda, tA, m0 + g + 8, kc + 1));
    const uint32_t a2 = pack_bf16(ldA(A, lda, tA, m0 + g, kc + 8), ldA(A, lda, tA, m0 + g, kc + 9));
    const uint32_t a3 = pack_bf16(ldA(A, lda, tA, m0 + g + 8, kc + 8), ldA(A, lda, tA, m0 + g + 8, kc + 9));
    const uint32_t b0 = pack_bf16(ldB(B, ldb, tB, kc, n0 + g), ldB(B, ldb, tB, kc + 1, n0 + g));
    const uint32_t b1 = pack_bf16(ldB(B, ldb, tB, kc + 8, n0 + g), ldB(B, ldb, tB, kc + 9, n0 + g));
    mma_bf16(d0, d1, d2, d3, a0, a1, a2, a3, b0, b1);
  }
  float *c0 = C + (int64_t)(m0 + g) * ldc + n0 + 2 * q;
  float *c1 = c0 + (int64_t)8 * ldc;
  atomicAdd(c0, d0);
  atomicAdd(c0 + 1, d1);
  atomicAdd(c1, d2);
  atomicAdd(c1 + 1, d3);
}

// One thread per output element and K chunk (blockIdx.z); chunks add into C atomically.
__global__ void k_gemm_fp32(int M, int N, int K, int kchunk, const float *__restrict__ A, int lda, bool tA,
                            const float *__restrict__ B, int ldb, bool tB, float *__restrict__ C, int ldc) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= (int64_t)M * N) return;
  const int m = (int)(e / N), n = (int)(e % N);
  const int k0 = blockIdx.z * kchunk, k1 = min(K, k0 + kchunk);
  float acc = 0.f;
  for (int k = k0; k < k1; ++k) acc = fmaf(ldA(A, lda, tA, m, k), ldB(B, ldb, tB, k, n), acc);
  atomicAdd(&C[(int64_t)m * ldc + n], acc);
}

// Z += b (per column); H = GELU(Z).
__global__ void k_bias_gelu(int64_t rows, int cols, float *__restrict__ Z, const float *__restrict__ b,
                            float *__restrict__ H) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= rows * cols) return;
  const float z = Z[e] + b[e % cols];
  Z[e] = z;
  H[e] = gelu(z);
}

// Logits += b3; masked softmax over the first ncand[r] columns; loss (sum) and dZ3 = (p - onehot) / scale.
__global__ void k_softmax_ce(int64_t rows, float *__restrict__ Z3, const float *__restrict__ b3,
                             const int32_t *__restrict__ label, const int32_t *__restrict__ ncand,
                             const int64_t *__restrict__ idx, float inv_scale, float *__restrict__ dZ3,
                             double *__restrict__ loss) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= rows) return;
  const int64_t src = idx ? idx[r] : r;
  const int n = max(1, min(kOut, ncand[src]));
  const int y = label[src];
  float *z = Z3 + r * kOut;
  float mx = -INFINITY;
  for (int c = 0; c < kOut; ++c) {
    z[c] += b3[c];
    if (c < n) mx = fmaxf(mx, z[c]);
  }
  float s = 0.f;
  for (int c = 0; c < n; ++c) s += expf(z[c] - mx);
  const float lse = mx + logf(s);
  atomicAdd(loss, (double)(lse - z[y]));
  for (int c = 0; c < kOut; ++c) {
    const float p = c < n ? expf(z[c] - lse) : 0.f;
    dZ3[r * kOut + c] = (p - (c == y ? 1.f : 0.f)) * inv_scale;
  }
}

__global__ void k_gelu_bwd(int64_t n, float *__restrict__ dH, const float *__restrict__ Z) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e < n) dH[e] *= gelu_grad(Z[e], erff(Z[e] * 0.70710678118654752f));
}

__global__ void k_colsum(int64_t rows, int cols, const float *__restrict__ X, float *__restrict__ out) {
  const int c = blockIdx.x;
  float acc = 0.f;
  for (int64_t r = threadIdx.x; r < rows; r += blockDim.x) acc += X[r * cols + c];
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(0xffffffffu, acc, o);
  __shared__ float red[32];
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.f;
    for (int w = 0; w < (int)(blockDim.x >> 5); ++w) t += red[w];
    out[c] = t;
  }
}

// Gather a minibatch of padded feature rows (16 columns, zeros beyond 9).
__global__ void k_gather(int64_t rows, const float *__restrict__ feat, const int64_t *__restrict__ idx,
                         float *__restrict__ X) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= rows * kInPad) return;
  const int64_t r = e / kInPad;
  const int k = (int)(e % kInPad);
  const int64_t src = idx ? idx[r] : r;
  X[e] = k < kIn ? feat[src * kIn + k] : 0.f;
}

// Minibatch index: a fixed-stride walk through a random rotation, a permutation of [0, n).
__global__ void k_batch_index(int64_t rows, int64_t n, int64_t start, int64_t stride, int64_t offset,
                              int64_t *__restrict__ idx) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r < rows) idx[r] = (int64_t)((((uint64_t)(start + r) % (uint64_t)n) * (uint64_t)stride + (uint64_t)offset) % (uint64_t)n);
}

__global__ void k_add_double(double *dst, const double *src) { *dst += *src; }

__global__ void k_adam(int n, float *__restrict__ p, const float *__restrict__ g, float *__restrict__ m,
                       float *__restrict__ v, float lr, float b1, float b2, float c1, float c2, float eps) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  m[i] = b1 * m[i] + (1.f - b1) * g[i];
  v[i] = b2 * v[i] + (1.f - b2) * g[i] * g[i];
  p[i] -= lr * (m[i] * c1) / (sqrtf(v[i] * c2) + eps);
}

// Shared-memory image (transposed BF16, padded) from the packed FP32 parameters.
__global__ void k_pack_image(const float *__restrict__ P, SmemWeights *__restrict__ S) {
  const int t = blockIdx.x * blockDim.x + threadIdx.x;
  for (int e = t; e < kHid * kSIn; e += gridDim.x * blockDim.x) {
    const int n = e / kSIn, k = e % kSIn;
    S->w1t[e] = __float2bfloat16_rn(k < kIn ? P[kOffW1 + k * kHid + n] : 0.f);
  }
  for (int e = t; e < kHid * kSHid; e += gridDim.x * blockDim.x) {
    const int n = e / kSHid, k = e % kSHid;
    S->w2t[e] = __float2bfloat16_rn(k < kHid ? P[kOffW2 + k * kHid + n] : 0.f);
  }
  for (int e = t; e < kOut * kSHid; e += gridDim.x * blockDim.x) {
    const int n = e / kSHid, k = e % kSHid;
    S->w3t[e] = __float2bfloat16_rn(k < kHid ? P[kOffW3 + k * kOut + n] : 0.f);
  }
  for (int e = t; e < kHid; e += gridDim.x * blockDim.x) {
    S->b1[e] = P[kOffB1 + e];
    S->b2[e] = P[kOffB2 + e];
  }
  for (int e = t; e < kOut; e += gridDim.x * blockDim.x) S->b3[e] = P[kOffB3 + e];
}

// Padded copy of W1 (16 x 64; rows 9..15 zero) for the training GEMMs.
__global__ void k_pad_w1(const float *__restrict__ P, float *__restrict__ W1p) {
  const int e = blockIdx.x * blockDim.x + threadIdx.x;
  if (e < kInPad * kHid) W1p[e] = (e / kHid) < kIn ? P[kOffW1 + e] : 0.f;
}

// Inference through the fused device code path: one warp per 32 feature rows.
__global__ void __launch_bounds__(128) k_predict(int64_t n, const float *__restrict__ feat,
                                                 const SmemWeights *__restrict__ gw, float *__restrict__ logits) {
  extern __shared__ __align__(16) unsigned char smem[];
  SmemWeights &sw = *reinterpret_cast<SmemWeights *>(smem);
  load_weights(sw, gw);
  __syncthreads();
  SmemWarp &W = reinterpret_cast<SmemWarp *>(smem + sizeof(SmemWeights))[threadIdx.x >> 5];
  const int lane = threadIdx.x & 31;
  for (int64_t base = (blockIdx.x * (int64_t)blockDim.x) + (threadIdx.x & ~31); base < n;
       base += (int64_t)gridDim.x * blockDim.x) {
    const int64_t r = base + lane;
    float f[kIn];
    for (int k = 0; k < kIn; ++k) f[k] = r < n ? feat[r * kIn + k] : 0.f;
    put_features(W, f);
    forward_warp(sw, W);
    if (r < n)
      for (int c = 0; c < kOut; ++c) logits[r * kOut + c] = W.logits[lane * kSOut + c];
    __syncwarp();
  }
}

struct MlpState {
  float *P = nullptr, *G = nullptr, *M = nullptr, *V = nullptr;  // kNParams each
  SmemWeights *img = nullptr;
  float *W1p = nullptr;
  int64_t step = 0;
  // scratch of the plain kernels for `cap` rows
  int64_t cap = 0;
  float *X = nullptr, *Z1 = nullptr, *H1 = nullptr, *Z2 = nullptr, *H2 = nullptr, *Z3 = nullptr, *dZ3 = nullptr,
        *dH2 = nullptr, *dH1 = nullptr, *dW1p = nullptr;
  int64_t *idx = nullptr;
  double *loss = nullptr;
  // k_mlp_train: fragments and FP32 deltas of `train_rows` rows, partial gradients, losses per block, control block, Adam's
  // corrections per step
  uint4 *frag = nullptr;
  float *delta = nullptr;
  int64_t train_rows = 0;
  float *part = nullptr;
  double *part_loss = nullptr;
  TrainCtrl *ctrl = nullptr;
  TrainWeights *timg = nullptr;
  float2 *corr = nullptr;
  int64_t corr_cap = 0;
  float *kept = nullptr;
  unsigned polls = kBarrierPolls;
};

MlpState *state(g4n_ctx *ctx) { return reinterpret_cast<MlpState *>(ctx->mlp); }

void free_scratch(MlpState *s) {
  cudaFree(s->X); cudaFree(s->Z1); cudaFree(s->H1); cudaFree(s->Z2); cudaFree(s->H2); cudaFree(s->Z3);
  cudaFree(s->dZ3); cudaFree(s->dH2); cudaFree(s->dH1); cudaFree(s->dW1p); cudaFree(s->idx); cudaFree(s->loss);
  s->X = s->Z1 = s->H1 = s->Z2 = s->H2 = s->Z3 = s->dZ3 = s->dH2 = s->dH1 = s->dW1p = nullptr;
  s->idx = nullptr;
  s->loss = nullptr;
  s->cap = 0;
}

int ensure_scratch(g4n_ctx *ctx, MlpState *s, int64_t rows) {
  if (s->cap >= rows) return G4N_OK;
  cudaDeviceSynchronize();
  free_scratch(s);
  bool ok = cudaMalloc(&s->X, rows * kInPad * 4) == cudaSuccess && cudaMalloc(&s->Z1, rows * kHid * 4) == cudaSuccess &&
            cudaMalloc(&s->H1, rows * kHid * 4) == cudaSuccess && cudaMalloc(&s->Z2, rows * kHid * 4) == cudaSuccess &&
            cudaMalloc(&s->H2, rows * kHid * 4) == cudaSuccess && cudaMalloc(&s->Z3, rows * kOut * 4) == cudaSuccess &&
            cudaMalloc(&s->dZ3, rows * kOut * 4) == cudaSuccess && cudaMalloc(&s->dH2, rows * kHid * 4) == cudaSuccess &&
            cudaMalloc(&s->dH1, rows * kHid * 4) == cudaSuccess && cudaMalloc(&s->dW1p, kInPad * kHid * 4) == cudaSuccess &&
            cudaMalloc(&s->idx, rows * 8) == cudaSuccess && cudaMalloc(&s->loss, 8) == cudaSuccess;
  if (!ok) {
    free_scratch(s);
    return g4n_fail(ctx, G4N_ERR_OOM, "mlp: scratch allocation failed");
  }
  s->cap = rows;
  return G4N_OK;
}

// Length of a product's K chunks: one block column each, and one partial sum of every output.
int64_t chunk_rows(int64_t K) {
  const int64_t ksplit = std::max<int64_t>(1, std::min<int64_t>(kMaxChunks, K / 256));
  return ((K + ksplit - 1) / ksplit + 15) / 16 * 16;
}

void gemm(bool bf16, int M, int N, int K, const float *A, int lda, bool tA, const float *B, int ldb, bool tB, float *C,
          int ldc, cudaStream_t st) {
  const int kchunk = (int)chunk_rows(K);
  const int nz = (K + kchunk - 1) / kchunk;
  if (bf16) {
    const int warps = (M / 16) * (N / 8);
    dim3 grid((warps + 3) / 4, 1, nz);
    k_gemm_bf16<<<grid, 128, 0, st>>>(M, N, K, kchunk, A, lda, tA, B, ldb, tB, C, ldc);
  } else {
    dim3 grid((int)(((int64_t)M * N + 127) / 128), 1, nz);
    k_gemm_fp32<<<grid, 128, 0, st>>>(M, N, K, kchunk, A, lda, tA, B, ldb, tB, C, ldc);
  }
}

inline int blocks(int64_t n, int b = 256) { return (int)std::max<int64_t>(1, (n + b - 1) / b); }

// Forward + backward over `rows` samples (rows a multiple of 16; the caller pads with
// ncand = 1, label = 0 rows of zero weight via inv_scale).  Gradients into s->G.
void forward_backward(MlpState *s, bool bf16, int64_t rows, const float *feat, const int32_t *label,
                      const int32_t *ncand, const int64_t *idx, float inv_scale, cudaStream_t st) {
  const int R = (int)rows;
  float *P = s->P, *G = s->G;
  cudaMemsetAsync(s->loss, 0, 8, st);
  k_gather<<<blocks(rows * kInPad), 256, 0, st>>>(rows, feat, idx, s->X);
  k_pad_w1<<<blocks(kInPad * kHid), 256, 0, st>>>(P, s->W1p);
  cudaMemsetAsync(s->Z1, 0, rows * kHid * 4, st);
  gemm(bf16, R, kHid, kInPad, s->X, kInPad, false, s->W1p, kHid, false, s->Z1, kHid, st);
  k_bias_gelu<<<blocks(rows * kHid), 256, 0, st>>>(rows, kHid, s->Z1, P + kOffB1, s->H1);
  cudaMemsetAsync(s->Z2, 0, rows * kHid * 4, st);
  gemm(bf16, R, kHid, kHid, s->H1, kHid, false, P + kOffW2, kHid, false, s->Z2, kHid, st);
  k_bias_gelu<<<blocks(rows * kHid), 256, 0, st>>>(rows, kHid, s->Z2, P + kOffB2, s->H2);
  cudaMemsetAsync(s->Z3, 0, rows * kOut * 4, st);
  gemm(bf16, R, kOut, kHid, s->H2, kHid, false, P + kOffW3, kOut, false, s->Z3, kOut, st);
  k_softmax_ce<<<blocks(rows), 256, 0, st>>>(rows, s->Z3, P + kOffB3, label, ncand, idx, inv_scale, s->dZ3, s->loss);
  // backward
  cudaMemsetAsync(G, 0, kNParams * 4, st);
  gemm(bf16, kHid, kOut, R, s->H2, kHid, true, s->dZ3, kOut, false, G + kOffW3, kOut, st);    // dW3 = H2^T dZ3
  k_colsum<<<kOut, 256, 0, st>>>(rows, kOut, s->dZ3, G + kOffB3);
  cudaMemsetAsync(s->dH2, 0, rows * kHid * 4, st);
  gemm(bf16, R, kHid, kOut, s->dZ3, kOut, false, P + kOffW3, kOut, true, s->dH2, kHid, st);   // dH2 = dZ3 W3^T
  k_gelu_bwd<<<blocks(rows * kHid), 256, 0, st>>>(rows * kHid, s->dH2, s->Z2);
  gemm(bf16, kHid, kHid, R, s->H1, kHid, true, s->dH2, kHid, false, G + kOffW2, kHid, st);    // dW2 = H1^T dZ2
  k_colsum<<<kHid, 256, 0, st>>>(rows, kHid, s->dH2, G + kOffB2);
  cudaMemsetAsync(s->dH1, 0, rows * kHid * 4, st);
  gemm(bf16, R, kHid, kHid, s->dH2, kHid, false, P + kOffW2, kHid, true, s->dH1, kHid, st);   // dH1 = dZ2 W2^T
  k_gelu_bwd<<<blocks(rows * kHid), 256, 0, st>>>(rows * kHid, s->dH1, s->Z1);
  cudaMemsetAsync(s->dW1p, 0, kInPad * kHid * 4, st);
  gemm(bf16, kInPad, kHid, R, s->X, kInPad, true, s->dH1, kHid, false, s->dW1p, kHid, st);   // dW1 = X^T dZ1
  cudaMemcpyAsync(G + kOffW1, s->dW1p, kIn * kHid * 4, cudaMemcpyDeviceToDevice, st);
  k_colsum<<<kHid, 256, 0, st>>>(rows, kHid, s->dH1, G + kOffB1);
}

void free_train(MlpState *s) {
  cudaFree(s->frag); cudaFree(s->delta); cudaFree(s->part); cudaFree(s->part_loss); cudaFree(s->ctrl); cudaFree(s->timg);
  cudaFree(s->corr); cudaFree(s->kept);
  s->frag = nullptr;
  s->delta = s->part = s->kept = nullptr;
  s->part_loss = nullptr;
  s->ctrl = nullptr;
  s->timg = nullptr;
  s->corr = nullptr;
  s->train_rows = s->corr_cap = 0;
}

// Buffers of k_mlp_train for `steps` minibatches of `rows` rows, to be used on `st` (every earlier use has ended: run_train waits
// for its kernel).  The image's padding is cleared on `st`: the default stream does not order a clear before the kernels of
// a non-blocking one.
int ensure_train(g4n_ctx *ctx, MlpState *s, int64_t rows, int64_t steps, cudaStream_t st) {
  const size_t ld = (size_t)(rows + kTrRows - 1) / kTrRows * kTrRows;
  bool ok = true;
  if (!s->ctrl)
    ok = cudaMalloc(&s->part, ((size_t)kMaxChunks * kNParams + kColParts * kCols) * 4) == cudaSuccess &&
         cudaMalloc(&s->part_loss, (size_t)ctx->sm_count * 8) == cudaSuccess &&
         cudaMalloc(&s->kept, 3 * kNParams * 4) == cudaSuccess &&
         cudaMalloc(&s->ctrl, sizeof(TrainCtrl)) == cudaSuccess &&
         cudaMalloc(&s->timg, sizeof(TrainWeights)) == cudaSuccess &&
         cudaMemsetAsync(s->timg, 0, sizeof(TrainWeights), st) == cudaSuccess;
  if (ok && s->train_rows < rows) {
    cudaFree(s->frag);
    cudaFree(s->delta);
    s->frag = nullptr;
    s->delta = nullptr;
    s->train_rows = 0;
    ok = cudaMalloc(&s->frag, ld / 16 * kFrags * 32 * sizeof(uint4)) == cudaSuccess &&
         cudaMalloc(&s->delta, ld * kCols * 4) == cudaSuccess;
    if (ok) s->train_rows = rows;
  }
  if (ok && s->corr_cap < steps) {
    cudaFree(s->corr);
    s->corr = nullptr;
    s->corr_cap = 0;
    ok = cudaMalloc(&s->corr, (size_t)steps * sizeof(float2)) == cudaSuccess;
    if (ok) s->corr_cap = steps;
  }
  if (!ok) {
    cudaGetLastError();
    free_train(s);
    return g4n_fail(ctx, G4N_ERR_OOM, "mlp: scratch allocation failed");
  }
  return G4N_OK;
}

// Run k_mlp_train on `st` and wait for it: a block per tile of 32 rows, or a warp per task of the gradients where those are
// more (4096 rows: 128 tiles, 136 blocks for 1088 tasks), at most a block per SM.  *loss = sum of the losses.
// A launch whose barrier gave up leaves the parameters and moments as it found them.
int run_train(g4n_ctx *ctx, MlpState *s, TrainParams &T, double *loss, cudaStream_t st) {
  T.P = s->P;
  T.b1 = 0.9f;
  T.b2 = 0.999f;
  T.eps = 1e-8f;
  T.chunk = chunk_rows(T.batch);
  T.chunks = (int)((T.batch + T.chunk - 1) / T.chunk);
  T.frag = s->frag;
  T.delta = s->delta;
  T.delta_ld = (T.batch + kTrRows - 1) / kTrRows * kTrRows;
  T.part = s->part;
  T.part_loss = s->part_loss;
  T.bias_corr = s->corr;
  T.ctrl = s->ctrl;
  T.polls = s->polls;
  T.kept = s->kept;
  T.img = s->timg;
  const int64_t tasks = (int64_t)T.chunks * kChunkTiles + kCols / 2 * kColParts;
  const int grid = (int)std::min<int64_t>(std::max(T.delta_ld / kTrRows, (tasks + 7) / 8), ctx->sm_count);
  void *args[] = {&T};
  TrainCtrl end{};
  cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem));
  if (cudaMemsetAsync(s->ctrl, 0, sizeof(TrainCtrl), st) != cudaSuccess ||
      cudaLaunchCooperativeKernel((const void *)k_mlp_train, dim3(grid), dim3(kTrThreads), args, sizeof(TrainSmem), st) !=
          cudaSuccess ||
      cudaMemcpyAsync(&end, s->ctrl, sizeof(end), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return g4n_fail(ctx, G4N_ERR_CUDA, std::string("mlp training: ") + cudaGetErrorString(cudaGetLastError()));
  if (end.failed) {
    // before every block has kept its share none has updated it
    if (T.M && end.begun &&
        (cudaMemcpyAsync(s->P, s->kept, kNParams * 4, cudaMemcpyDeviceToDevice, st) != cudaSuccess ||
         cudaMemcpyAsync(s->M, s->kept + kNParams, kNParams * 4, cudaMemcpyDeviceToDevice, st) != cudaSuccess ||
         cudaMemcpyAsync(s->V, s->kept + 2 * kNParams, kNParams * 4, cudaMemcpyDeviceToDevice, st) != cudaSuccess ||
         cudaStreamSynchronize(st) != cudaSuccess))
      return g4n_fail(ctx, G4N_ERR_CUDA, std::string("mlp training: ") + cudaGetErrorString(cudaGetLastError()));
    return g4n_fail(ctx, G4N_ERR_TIMEOUT, "mlp training: a grid barrier reached its iteration cap");
  }
  *loss = end.loss;
  return G4N_OK;
}

// One epoch of `nb` minibatches by the plain kernels.  *loss = sum of the losses.
int train_plain(g4n_ctx *ctx, MlpState *s, int64_t n, const float *feat, const int32_t *label, const int32_t *ncand,
                int32_t batch, int64_t nb, uint64_t stride, uint64_t offset, float lr, const float2 *corr, double *loss,
                cudaStream_t st) {
  double *sum = nullptr;
  if (cudaMalloc(&sum, 8) != cudaSuccess) {
    cudaGetLastError();
    return g4n_fail(ctx, G4N_ERR_OOM, "mlp_train: allocation failed");
  }
  cudaMemsetAsync(sum, 0, 8, st);
  for (int64_t b = 0; b < nb; ++b) {
    k_batch_index<<<blocks(batch), 256, 0, st>>>(batch, n, b * batch, (int64_t)stride, (int64_t)offset, s->idx);
    forward_backward(s, true, batch, feat, label, ncand, s->idx, 1.0f / (float)batch, st);
    k_adam<<<blocks(kNParams), 256, 0, st>>>(kNParams, s->P, s->G, s->M, s->V, lr, 0.9f, 0.999f, corr[b].x, corr[b].y,
                                             1e-8f);
    k_add_double<<<1, 1, 0, st>>>(sum, s->loss);  // epoch loss accumulates on the device
  }
  k_pack_image<<<8, 256, 0, st>>>(s->P, s->img);
  cudaMemcpyAsync(loss, sum, 8, cudaMemcpyDeviceToHost, st);
  cudaStreamSynchronize(st);
  cudaFree(sum);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return g4n_fail(ctx, G4N_ERR_CUDA, std::string("mlp_train: ") + cudaGetErrorString(e));
  return G4N_OK;
}

int check_data(g4n_ctx *ctx, int64_t n, const void *feat, const void *label, const void *ncand) {
  if (!ctx) return G4N_ERR_ARG;
  if (ctx->device < 0) return g4n_fail(ctx, G4N_ERR_STATE, "host-only context: no device work");
  if (!state(ctx)) return g4n_fail(ctx, G4N_ERR_STATE, "mlp: no parameters loaded (g4n_mlp_load)");
  if (n < 1 || !feat || !label || !ncand) return g4n_fail(ctx, G4N_ERR_ARG, "mlp: empty or null training data");
  return G4N_OK;
}

}  // namespace

// Device image of the loaded weights (for the fused inference in the transport kernel); null if none.
const SmemWeights *g4n_mlp_image(g4n_ctx *ctx) {
  MlpState *s = state(ctx);
  return s ? s->img : nullptr;
}

void g4n_mlp_free(g4n_ctx *ctx) {
  MlpState *s = state(ctx);
  if (!s) return;
  free_scratch(s);
  cudaFree(s->P); cudaFree(s->G); cudaFree(s->M); cudaFree(s->V); cudaFree(s->img); cudaFree(s->W1p);
  free_train(s);
  delete s;
  ctx->mlp = nullptr;
}

extern "C" {

int g4n_mlp_load(g4n_ctx *ctx, const float *params) {
  if (!ctx || !params) return g4n_fail(ctx, G4N_ERR_ARG, "mlp_load: null argument");
  if (ctx->device < 0) return g4n_fail(ctx, G4N_ERR_STATE, "host-only context: no device work");
  for (int i = 0; i < kNParams; ++i)
    if (!std::isfinite(params[i])) return g4n_fail(ctx, G4N_ERR_ARG, "mlp_load: non-finite parameter");
  cudaSetDevice(ctx->device);
  MlpState *s = state(ctx);
  if (!s) {
    s = new MlpState();
    bool ok = cudaMalloc(&s->P, kNParams * 4) == cudaSuccess && cudaMalloc(&s->G, kNParams * 4) == cudaSuccess &&
              cudaMalloc(&s->M, kNParams * 4) == cudaSuccess && cudaMalloc(&s->V, kNParams * 4) == cudaSuccess &&
              cudaMalloc(&s->img, sizeof(SmemWeights)) == cudaSuccess &&
              cudaMalloc(&s->W1p, kInPad * kHid * 4) == cudaSuccess;
    ctx->mlp = s;
    if (!ok) {
      g4n_mlp_free(ctx);
      return g4n_fail(ctx, G4N_ERR_OOM, "mlp_load: allocation failed");
    }
  }
  if (cudaMemcpy(s->P, params, kNParams * 4, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemset(s->M, 0, kNParams * 4) != cudaSuccess || cudaMemset(s->V, 0, kNParams * 4) != cudaSuccess)
    return g4n_fail(ctx, G4N_ERR_CUDA, "mlp_load: upload failed");
  s->step = 0;
  k_pack_image<<<8, 256>>>(s->P, s->img);
  if (cudaDeviceSynchronize() != cudaSuccess) return g4n_fail(ctx, G4N_ERR_CUDA, "mlp_load: packing failed");
  return G4N_OK;
}

void g4n_mlp_barrier_cap(g4n_ctx *ctx, uint32_t polls) {
  if (MlpState *s = state(ctx)) s->polls = polls ? polls : kBarrierPolls;
}

int g4n_mlp_get(g4n_ctx *ctx, float *params) {
  if (!ctx || !params) return g4n_fail(ctx, G4N_ERR_ARG, "mlp_get: null argument");
  MlpState *s = state(ctx);
  if (!s) return g4n_fail(ctx, G4N_ERR_STATE, "mlp_get: no parameters loaded");
  cudaSetDevice(ctx->device);
  if (cudaMemcpy(params, s->P, kNParams * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
    return g4n_fail(ctx, G4N_ERR_CUDA, "mlp_get: copy failed");
  return G4N_OK;
}

int g4n_mlp_predict(g4n_ctx *ctx, int64_t n, const float *feat, float *out_logits, g4n_stream stream) {
  if (!ctx) return G4N_ERR_ARG;
  if (!state(ctx)) return g4n_fail(ctx, G4N_ERR_STATE, "mlp_predict: no parameters loaded");
  if (n < 0) return g4n_fail(ctx, G4N_ERR_ARG, "mlp_predict: n < 0");
  if (n == 0) return G4N_OK;
  if (!feat || !out_logits) return g4n_fail(ctx, G4N_ERR_ARG, "mlp_predict: null array");
  cudaSetDevice(ctx->device);
  const int grid = (int)std::min<int64_t>((n + 127) / 128, (int64_t)ctx->sm_count * 8);
  const size_t smem = sizeof(SmemWeights) + 4 * sizeof(SmemWarp);
  cudaFuncSetAttribute(k_predict, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  k_predict<<<grid, 128, smem, (cudaStream_t)stream>>>(n, feat, state(ctx)->img, out_logits);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return g4n_fail(ctx, G4N_ERR_CUDA, std::string("mlp_predict launch: ") + cudaGetErrorString(e));
  return G4N_OK;
}

int g4n_mlp_grad(g4n_ctx *ctx, int64_t n, const float *feat, const int32_t *label, const int32_t *ncand,
                 int32_t precision, float *out_grads, double *out_loss) {
  int rc = check_data(ctx, n, feat, label, ncand);
  if (rc) return rc;
  if (!out_grads || !out_loss) return g4n_fail(ctx, G4N_ERR_ARG, "mlp_grad: null output");
  if (n % 16) return g4n_fail(ctx, G4N_ERR_ARG, "mlp_grad: n must be a multiple of 16");
  cudaSetDevice(ctx->device);
  MlpState *s = state(ctx);
  double loss = 0.0;
  if (precision == 0 && n >= kFusedRows) {
    if ((rc = ensure_train(ctx, s, n, 0, 0))) return rc;
    TrainParams T{};
    T.n = n;
    T.feat = feat;
    T.label = label;
    T.ncand = ncand;
    T.steps = 1;
    T.batch = n;
    T.inv_scale = 1.0f / (float)n;
    T.grads = s->G;
    if ((rc = run_train(ctx, s, T, &loss, 0))) return rc;
  } else {
    if ((rc = ensure_scratch(ctx, s, n))) return rc;
    forward_backward(s, precision == 0, n, feat, label, ncand, nullptr, 1.0f / (float)n, 0);
    if (cudaMemcpy(&loss, s->loss, 8, cudaMemcpyDeviceToHost) != cudaSuccess)
      return g4n_fail(ctx, G4N_ERR_CUDA, "mlp_grad: failed");
  }
  if (cudaMemcpy(out_grads, s->G, kNParams * 4, cudaMemcpyDeviceToHost) != cudaSuccess)
    return g4n_fail(ctx, G4N_ERR_CUDA, "mlp_grad: failed");
  *out_loss = loss / (double)n;
  return G4N_OK;
}

int g4n_mlp_train(g4n_ctx *ctx, int64_t n, const float *feat, const int32_t *label, const int32_t *ncand,
                  int32_t epochs, int32_t batch, float lr, uint64_t seed, float *out_loss, g4n_stream stream) {
  int rc = check_data(ctx, n, feat, label, ncand);
  if (rc) return rc;
  if (epochs < 1 || batch < 16 || batch % 16 || !(lr > 0.f)) return g4n_fail(ctx, G4N_ERR_ARG, "mlp_train: bad settings");
  if (n < batch) return g4n_fail(ctx, G4N_ERR_ARG, "mlp_train: fewer samples than one batch");
  cudaSetDevice(ctx->device);
  cudaStream_t st = (cudaStream_t)stream;
  MlpState *s = state(ctx);
  const int64_t nb = n / batch;
  if (nb > INT32_MAX) return g4n_fail(ctx, G4N_ERR_ARG, "mlp_train: too many minibatches");
  const bool fused = batch >= kFusedTrainRows;
  if ((rc = fused ? ensure_train(ctx, s, batch, nb, st) : ensure_scratch(ctx, s, batch))) return rc;
  std::unique_ptr<float2[]> corr(new (std::nothrow) float2[(size_t)nb]);
  if (!corr) return g4n_fail(ctx, G4N_ERR_OOM, "mlp_train: allocation failed");
  for (int ep = 0; ep < epochs; ++ep) {
    // a random stride coprime with n and a random offset: a permutation of the samples per epoch
    uint64_t h = seed * 0x9E3779B97F4A7C15ull + (uint64_t)ep * 0xD1B54A32D192ED03ull + 1;
    h ^= h >> 31;
    h *= 0xBF58476D1CE4E5B9ull;
    h ^= h >> 27;
    uint64_t stride = (h % (uint64_t)n) | 1;
    while (std::gcd(stride, (uint64_t)n) != 1) stride += 2;
    double tot = 0.0;
    for (int64_t k = 0; k < nb; ++k) {
      const float step = (float)(s->step + k + 1);
      corr[k].x = 1.0f / (1.0f - std::pow(0.9f, step));
      corr[k].y = 1.0f / (1.0f - std::pow(0.999f, step));
    }
    const uint64_t offset = (h >> 17) % (uint64_t)n;
    if (!fused) {
      if ((rc = train_plain(ctx, s, n, feat, label, ncand, batch, nb, stride, offset, lr, corr.get(), &tot, st))) return rc;
      s->step += nb;
      if (out_loss) out_loss[ep] = (float)(tot / ((double)nb * batch));
      continue;
    }
    // the kernels of the epoch before have ended (run_train waits for them)
    if (cudaMemcpyAsync(s->corr, corr.get(), (size_t)nb * sizeof(float2), cudaMemcpyHostToDevice, st) != cudaSuccess)
      return g4n_fail(ctx, G4N_ERR_CUDA, "mlp_train: upload failed");
    TrainParams T{};
    T.n = n;
    T.feat = feat;
    T.label = label;
    T.ncand = ncand;
    T.steps = (int)nb;
    T.batch = batch;
    T.permuted = true;
    T.stride = stride;
    T.offset = offset;
    T.inv_scale = 1.0f / (float)batch;
    T.M = s->M;
    T.V = s->V;
    T.lr = lr;
    if ((rc = run_train(ctx, s, T, &tot, st))) return rc;
    s->step += nb;
    k_pack_image<<<8, 256, 0, st>>>(s->P, s->img);
    if (out_loss) out_loss[ep] = (float)(tot / ((double)nb * batch));
  }
  cudaStreamSynchronize(st);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return g4n_fail(ctx, G4N_ERR_CUDA, std::string("mlp_train: ") + cudaGetErrorString(e));
  return G4N_OK;
}

}  // extern "C"
