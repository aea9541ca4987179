// mlp.cu -- training and inference entry points of the candidate-proposal MLP.
//
// Training (g4n_mlp_train, and the BF16 gradients of g4n_mlp_grad) is the
// persistent kernel of mlp_train.cuh: BF16 products on the tensor cores with
// FP32 accumulation, masked softmax cross-entropy, Adam on FP32 master
// weights.  The FP32 reference gradients are plain kernels of this file.
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

// ---------------------------------------------------------------- FP32 reference gradients
// The FP32 path of g4n_mlp_grad: plain kernels, one per product and elementwise pass.
// C[M x N] += op(A)[M x K] op(B)[K x N]; A(m, k) = transA ? A[k * lda + m] : A[m * lda + k],
// B(k, n) = transB ? B[n * ldb + k] : B[k * ldb + n].

__device__ __forceinline__ float ldA(const float *A, int lda, bool tA, int m, int k) {
  return tA ? A[(int64_t)k * lda + m] : A[(int64_t)m * lda + k];
}
__device__ __forceinline__ float ldB(const float *B, int ldb, bool tB, int k, int n) {
  return tB ? B[(int64_t)n * ldb + k] : B[(int64_t)k * ldb + n];
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
                             float inv_scale, float *__restrict__ dZ3, double *__restrict__ loss) {
  const int64_t r = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (r >= rows) return;
  const int n = max(1, min(kOut, ncand[r]));
  const int y = label[r];
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

// Feature rows padded to 16 columns (zeros beyond 9).
__global__ void k_pad_rows(int64_t rows, const float *__restrict__ feat, float *__restrict__ X) {
  const int64_t e = blockIdx.x * (int64_t)blockDim.x + threadIdx.x;
  if (e >= rows * kInPad) return;
  const int64_t r = e / kInPad;
  const int k = (int)(e % kInPad);
  X[e] = k < kIn ? feat[r * kIn + k] : 0.f;
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
  // FP32 gradient scratch for `cap` rows
  int64_t cap = 0;
  float *X = nullptr, *Z1 = nullptr, *H1 = nullptr, *Z2 = nullptr, *H2 = nullptr, *Z3 = nullptr, *dZ3 = nullptr,
        *dH2 = nullptr, *dH1 = nullptr, *dW1p = nullptr;
  double *loss = nullptr;
  // k_mlp_train: partial gradients and losses (one row per block), control block, Adam's corrections per step
  float *part = nullptr;
  double *part_loss = nullptr;
  TrainCtrl *ctrl = nullptr;
  TrainWeights *timg = nullptr;
  float2 *corr = nullptr;
  int64_t corr_cap = 0;
};

MlpState *state(g4n_ctx *ctx) { return reinterpret_cast<MlpState *>(ctx->mlp); }

void free_scratch(MlpState *s) {
  cudaFree(s->X); cudaFree(s->Z1); cudaFree(s->H1); cudaFree(s->Z2); cudaFree(s->H2); cudaFree(s->Z3);
  cudaFree(s->dZ3); cudaFree(s->dH2); cudaFree(s->dH1); cudaFree(s->dW1p); cudaFree(s->loss);
  s->X = s->Z1 = s->H1 = s->Z2 = s->H2 = s->Z3 = s->dZ3 = s->dH2 = s->dH1 = s->dW1p = nullptr;
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
            cudaMalloc(&s->loss, 8) == cudaSuccess;
  if (!ok) {
    free_scratch(s);
    return g4n_fail(ctx, G4N_ERR_OOM, "mlp: scratch allocation failed");
  }
  s->cap = rows;
  return G4N_OK;
}

void gemm(int M, int N, int K, const float *A, int lda, bool tA, const float *B, int ldb, bool tB, float *C, int ldc,
          cudaStream_t st) {
  const int ksplit = std::max(1, std::min(256, K / 256));
  const int kchunk = ((K + ksplit - 1) / ksplit + 15) / 16 * 16;
  const int nz = (K + kchunk - 1) / kchunk;
  dim3 grid((int)(((int64_t)M * N + 127) / 128), 1, nz);
  k_gemm_fp32<<<grid, 128, 0, st>>>(M, N, K, kchunk, A, lda, tA, B, ldb, tB, C, ldc);
}

inline int blocks(int64_t n, int b = 256) { return (int)std::max<int64_t>(1, (n + b - 1) / b); }

// FP32 forward + backward over `rows` samples.  Gradients into s->G, the sum of the losses into s->loss.
void forward_backward_fp32(MlpState *s, int64_t rows, const float *feat, const int32_t *label, const int32_t *ncand,
                           float inv_scale, cudaStream_t st) {
  const int R = (int)rows;
  float *P = s->P, *G = s->G;
  cudaMemsetAsync(s->loss, 0, 8, st);
  k_pad_rows<<<blocks(rows * kInPad), 256, 0, st>>>(rows, feat, s->X);
  k_pad_w1<<<blocks(kInPad * kHid), 256, 0, st>>>(P, s->W1p);
  cudaMemsetAsync(s->Z1, 0, rows * kHid * 4, st);
  gemm(R, kHid, kInPad, s->X, kInPad, false, s->W1p, kHid, false, s->Z1, kHid, st);
  k_bias_gelu<<<blocks(rows * kHid), 256, 0, st>>>(rows, kHid, s->Z1, P + kOffB1, s->H1);
  cudaMemsetAsync(s->Z2, 0, rows * kHid * 4, st);
  gemm(R, kHid, kHid, s->H1, kHid, false, P + kOffW2, kHid, false, s->Z2, kHid, st);
  k_bias_gelu<<<blocks(rows * kHid), 256, 0, st>>>(rows, kHid, s->Z2, P + kOffB2, s->H2);
  cudaMemsetAsync(s->Z3, 0, rows * kOut * 4, st);
  gemm(R, kOut, kHid, s->H2, kHid, false, P + kOffW3, kOut, false, s->Z3, kOut, st);
  k_softmax_ce<<<blocks(rows), 256, 0, st>>>(rows, s->Z3, P + kOffB3, label, ncand, inv_scale, s->dZ3, s->loss);
  // backward
  cudaMemsetAsync(G, 0, kNParams * 4, st);
  gemm(kHid, kOut, R, s->H2, kHid, true, s->dZ3, kOut, false, G + kOffW3, kOut, st);    // dW3 = H2^T dZ3
  k_colsum<<<kOut, 256, 0, st>>>(rows, kOut, s->dZ3, G + kOffB3);
  cudaMemsetAsync(s->dH2, 0, rows * kHid * 4, st);
  gemm(R, kHid, kOut, s->dZ3, kOut, false, P + kOffW3, kOut, true, s->dH2, kHid, st);   // dH2 = dZ3 W3^T
  k_gelu_bwd<<<blocks(rows * kHid), 256, 0, st>>>(rows * kHid, s->dH2, s->Z2);
  gemm(kHid, kHid, R, s->H1, kHid, true, s->dH2, kHid, false, G + kOffW2, kHid, st);    // dW2 = H1^T dZ2
  k_colsum<<<kHid, 256, 0, st>>>(rows, kHid, s->dH2, G + kOffB2);
  cudaMemsetAsync(s->dH1, 0, rows * kHid * 4, st);
  gemm(R, kHid, kHid, s->dH2, kHid, false, P + kOffW2, kHid, true, s->dH1, kHid, st);   // dH1 = dZ2 W2^T
  k_gelu_bwd<<<blocks(rows * kHid), 256, 0, st>>>(rows * kHid, s->dH1, s->Z1);
  cudaMemsetAsync(s->dW1p, 0, kInPad * kHid * 4, st);
  gemm(kInPad, kHid, R, s->X, kInPad, true, s->dH1, kHid, false, s->dW1p, kHid, st);   // dW1 = X^T dZ1
  cudaMemcpyAsync(G + kOffW1, s->dW1p, kIn * kHid * 4, cudaMemcpyDeviceToDevice, st);
  k_colsum<<<kHid, 256, 0, st>>>(rows, kHid, s->dH1, G + kOffB1);
}

// Buffers of k_mlp_train for `steps` minibatches.
int ensure_train(g4n_ctx *ctx, MlpState *s, int64_t steps) {
  bool ok = true;
  if (!s->ctrl)
    ok = cudaMalloc(&s->part, (size_t)ctx->sm_count * kNParams * 4) == cudaSuccess &&
         cudaMalloc(&s->part_loss, (size_t)ctx->sm_count * 8) == cudaSuccess &&
         cudaMalloc(&s->ctrl, sizeof(TrainCtrl)) == cudaSuccess &&
         cudaMalloc(&s->timg, sizeof(TrainWeights)) == cudaSuccess &&
         cudaMemset(s->timg, 0, sizeof(TrainWeights)) == cudaSuccess;
  if (ok && s->corr_cap < steps) {
    cudaFree(s->corr);
    s->corr = nullptr;
    s->corr_cap = 0;
    ok = cudaMalloc(&s->corr, (size_t)steps * sizeof(float2)) == cudaSuccess;
    if (ok) s->corr_cap = steps;
  }
  if (!ok) {
    cudaGetLastError();
    cudaFree(s->part); cudaFree(s->part_loss); cudaFree(s->ctrl); cudaFree(s->timg);
    s->part = nullptr;
    s->part_loss = nullptr;
    s->ctrl = nullptr;
    s->timg = nullptr;
    return g4n_fail(ctx, G4N_ERR_OOM, "mlp: scratch allocation failed");
  }
  return G4N_OK;
}

// Run k_mlp_train on `st` and wait for it: one block per tile of 32 rows, at most one per SM.  *loss = sum of the losses.
int run_train(g4n_ctx *ctx, MlpState *s, TrainParams &T, double *loss, cudaStream_t st) {
  T.P = s->P;
  T.b1 = 0.9f;
  T.b2 = 0.999f;
  T.eps = 1e-8f;
  T.part = s->part;
  T.part_loss = s->part_loss;
  T.bias_corr = s->corr;
  T.ctrl = s->ctrl;
  T.img = s->timg;
  const int grid = std::min((T.batch + kTrRows - 1) / kTrRows, ctx->sm_count);
  void *args[] = {&T};
  TrainCtrl end{};
  cudaFuncSetAttribute(k_mlp_train, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sizeof(TrainSmem));
  if (cudaMemsetAsync(s->ctrl, 0, sizeof(TrainCtrl), st) != cudaSuccess ||
      cudaLaunchCooperativeKernel((const void *)k_mlp_train, dim3(grid), dim3(kTrThreads), args, sizeof(TrainSmem), st) !=
          cudaSuccess ||
      cudaMemcpyAsync(&end, s->ctrl, sizeof(end), cudaMemcpyDeviceToHost, st) != cudaSuccess ||
      cudaStreamSynchronize(st) != cudaSuccess)
    return g4n_fail(ctx, G4N_ERR_CUDA, std::string("mlp training: ") + cudaGetErrorString(cudaGetLastError()));
  if (end.failed) return g4n_fail(ctx, G4N_ERR_TIMEOUT, "mlp training: a grid barrier reached its iteration cap");
  *loss = end.loss;
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
  cudaFree(s->part); cudaFree(s->part_loss); cudaFree(s->ctrl); cudaFree(s->timg); cudaFree(s->corr);
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
  if (precision == 0) {
    if (n > INT32_MAX - kTrRows) return g4n_fail(ctx, G4N_ERR_ARG, "mlp_grad: too many samples");
    if ((rc = ensure_train(ctx, s, 0))) return rc;
    TrainParams T{};
    T.n = n;
    T.feat = feat;
    T.label = label;
    T.ncand = ncand;
    T.steps = 1;
    T.batch = (int)n;
    T.inv_scale = 1.0f / (float)n;
    T.grads = s->G;
    if ((rc = run_train(ctx, s, T, &loss, 0))) return rc;
  } else {
    if ((rc = ensure_scratch(ctx, s, n))) return rc;
    forward_backward_fp32(s, n, feat, label, ncand, 1.0f / (float)n, 0);
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
  if ((rc = ensure_train(ctx, s, nb))) return rc;
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
    for (int64_t k = 0; k < nb; ++k) {
      ++s->step;
      corr[k].x = 1.0f / (1.0f - std::pow(0.9f, (float)s->step));
      corr[k].y = 1.0f / (1.0f - std::pow(0.999f, (float)s->step));
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
    T.offset = (h >> 17) % (uint64_t)n;
    T.inv_scale = 1.0f / (float)batch;
    T.M = s->M;
    T.V = s->V;
    T.lr = lr;
    double tot = 0.0;
    if ((rc = run_train(ctx, s, T, &tot, st))) return rc;
    k_pack_image<<<8, 256, 0, st>>>(s->P, s->img);
    if (out_loss) out_loss[ep] = (float)(tot / ((double)nb * batch));
  }
  cudaStreamSynchronize(st);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return g4n_fail(ctx, G4N_ERR_CUDA, std::string("mlp_train: ") + cudaGetErrorString(e));
  return G4N_OK;
}

}  // extern "C"
