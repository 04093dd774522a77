// Small MLP for the learned initial density (three linear layers, SiLU, width
// 256): forward, backward and Adam, all in this file's kernels.
//
//   z1 = x W1 + b1, h1 = silu(z1), z2 = h1 W2 + b2, h2 = silu(z2), y = h2 W3 + b3
//   loss = sum(mask (y - t)^2) / sum(mask)
// Weights are kept in FP32 (master, Adam state) with BF16 copies packed for the
// GEMMs, which run on the fifth-generation tensor cores with the element-wise
// steps as their epilogues (tcgen05.mma, BF16 x BF16 -> FP32 accumulation in
// tensor memory, tc_gemm.cuh): a BF16 forward pass is 4 launches, a gradient 8.
// A plain FP32 GEMM path (no BF16 rounding) serves the gradient check.
// silu(z) = z s(z), s = logistic; silu'(z) = s(z) (1 + z (1 - s(z))).
#include <cuda_bf16.h>

#include <algorithm>
#include <cstdint>

#include <cmath>
#include <cstdio>
#include <cstring>
#include <vector>

#include "fsim_internal.h"
#include "tc_gemm.cuh"

struct fsim_mlp {
  int nin = 0, width = 0, nout = 0;
  size_t np = 0;
  float* p = nullptr;  // W1 [nin x w] | b1 [w] | W2 [w x w] | b2 [w] | W3 [w x nout] | b3 [nout]
  float* g = nullptr;
  float* m = nullptr;
  float* v = nullptr;
  __nv_bfloat16* pb = nullptr;  // packed BF16 weights (Pack)
  int maxb = 0;                 // batch the FP32 path's buffers hold
  float *z1 = nullptr, *h1 = nullptr, *z2 = nullptr, *h2 = nullptr, *y = nullptr;
  float *dy = nullptr, *d1 = nullptr, *d2 = nullptr;
  // BF16 path: batch its buffers hold, BF16 rows padded to whole K chunks
  int maxbt = 0, maxbg = 0;
  __nv_bfloat16 *xb = nullptr, *h1b = nullptr, *h2b = nullptr, *dyb = nullptr, *d1b = nullptr, *d2b = nullptr;
  float *z1t = nullptr, *z2t = nullptr;
  float* part = nullptr;   // weight-gradient partial products [split][np]
  float* partb = nullptr;  // column sums [row tile][2 width + nout], then loss partials
  float* scal = nullptr;  // [0] loss numerator, [1] mask sum, [2] (int) set by a tensor-core GEMM whose MMAs did not complete
  int* tc_err = nullptr;  // scal + 2
  long step = 0;
};

namespace fsim {
namespace {

struct Off {
  size_t W1, b1, W2, b2, W3, b3, n;
};
Off offsets(int nin, int w, int nout) {
  Off o;
  o.W1 = 0;
  o.b1 = o.W1 + (size_t)nin * w;
  o.W2 = o.b1 + w;
  o.b2 = o.W2 + (size_t)w * w;
  o.W3 = o.b2 + w;
  o.b3 = o.W3 + (size_t)w * nout;
  o.n = o.b3 + nout;
  return o;
}

// C[M x N] = op(A) op(B) (+ bias[N]), op(A) M x K, op(B) K x N, all row-major
// FP32 in memory; tA: A stored K x M; tB: B stored N x K.  This kernel is the
// plain FP32 path (FMAs, no BF16 rounding) of the gradient check; BF16 GEMMs
// run on the tensor cores (tc_layer_kernel, tc_wgrad_kernel).
constexpr int TM = 64, TN = 64, TK = 16;

__device__ __forceinline__ float ldA(const float* A, int M, int K, bool tA, int r, int k) {
  if (r >= M || k >= K) return 0.0f;
  return tA ? A[(size_t)k * M + r] : A[(size_t)r * K + k];
}
__device__ __forceinline__ float ldB(const float* B, int K, int N, bool tB, int k, int c) {
  if (k >= K || c >= N) return 0.0f;
  return tB ? B[(size_t)c * K + k] : B[(size_t)k * N + c];
}

__global__ void __launch_bounds__(128) gemm_kernel(const float* __restrict__ A, const float* __restrict__ B,
                                                   float* __restrict__ C, const float* __restrict__ bias, int M,
                                                   int N, int K, int tA, int tB) {
  __shared__ float Af[TM][TK + 1];
  __shared__ float Bf[TK][TN + 1];
  const int m0 = blockIdx.y * TM, n0 = blockIdx.x * TN;
  const int tid = threadIdx.x;
  // thread owns rows (tid / 4) * 2 .. +1 and columns (tid % 4) * 16 .. +15 of the tile (32 outputs)
  const int rr = (tid >> 2) * 2, cc = (tid & 3) * 16;
  float accf[32];
#pragma unroll
  for (int r = 0; r < 32; ++r) accf[r] = 0.0f;
  for (int k0 = 0; k0 < K; k0 += TK) {
    for (int x = tid; x < TM * TK; x += 128) {
      const int r = x / TK, k = x % TK;
      Af[r][k] = ldA(A, M, K, tA, m0 + r, k0 + k);
    }
    for (int x = tid; x < TK * TN; x += 128) {
      const int k = x / TN, c = x % TN;
      Bf[k][c] = ldB(B, K, N, tB, k0 + k, n0 + c);
    }
    __syncthreads();
#pragma unroll
    for (int k = 0; k < TK; ++k)
#pragma unroll
      for (int i = 0; i < 2; ++i)
#pragma unroll
        for (int j = 0; j < 16; ++j) accf[i * 16 + j] = fmaf(Af[rr + i][k], Bf[k][cc + j], accf[i * 16 + j]);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int j = 0; j < 16; ++j) {
      const int r = m0 + rr + i, c = n0 + cc + j;
      if (r < M && c < N) C[(size_t)r * N + c] = accf[i * 16 + j] + (bias ? bias[c] : 0.0f);
    }
}

__device__ __forceinline__ float sig(float z) { return 1.0f / (1.0f + expf(-z)); }

__global__ void silu_kernel(const float* z, float* h, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x)
    h[i] = z[i] * sig(z[i]);
}
// d <- d * silu'(z)
__global__ void silu_back_kernel(const float* z, float* d, size_t n) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float s = sig(z[i]);
    d[i] *= s * (1.0f + z[i] * (1.0f - s));
  }
}
// loss numerator / mask sum; dy = 2 mask (y - t) (scaled by 1/sum(mask) afterwards)
__global__ void loss_kernel(const float* y, const float* t, const float* mask, float* dy, float* scal, size_t n) {
  float a = 0.0f, s = 0.0f;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float d = y[i] - t[i];
    a += mask[i] * d * d;
    s += mask[i];
    dy[i] = 2.0f * mask[i] * d;
  }
  for (int o = 16; o > 0; o >>= 1) {
    a += __shfl_xor_sync(0xffffffffu, a, o);
    s += __shfl_xor_sync(0xffffffffu, s, o);
  }
  if ((threadIdx.x & 31) == 0) {
    atomicAdd(scal, a);
    atomicAdd(scal + 1, s);
  }
}
__global__ void scale_kernel(float* x, const float* scal, size_t n) {
  const float inv = 1.0f / fmaxf(scal[1], 1.0f);
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) x[i] *= inv;
}
// column sums (bias gradients): out[c] = sum_r d[r, c]
__global__ void colsum_kernel(const float* d, float* out, int M, int N) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= N) return;
  float s = 0.0f;
  for (int r = 0; r < M; ++r) s += d[(size_t)r * N + c];
  out[c] = s;
}
__global__ void adam_kernel(float* p, const float* g, float* m, float* v, size_t n, float lr, float b1, float b2,
                            float eps, float c1, float c2) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < n; i += (size_t)gridDim.x * blockDim.x) {
    const float gi = g[i];
    m[i] = b1 * m[i] + (1.0f - b1) * gi;
    v[i] = b2 * v[i] + (1.0f - b2) * gi * gi;
    p[i] -= lr * (m[i] / c1) / (sqrtf(v[i] / c2) + eps);
  }
}

// BF16 weights as the tensor-core GEMMs read them, rows padded with zeros to
// whole K chunks: the transposes [out x in] for the forward pass, W2 and W3 as
// they are [in x out] for the data gradients.
struct Pack {
  size_t T1, T2, T3, N2, N3, n;
};
Pack packing(int nin, int w, int nout) {
  Pack k;
  k.T1 = 0;
  k.T2 = k.T1 + (size_t)w * tc_ld(nin);
  k.T3 = k.T2 + (size_t)w * tc_ld(w);
  k.N2 = k.T3 + (size_t)nout * tc_ld(w);
  k.N3 = k.N2 + (size_t)w * tc_ld(w);
  k.n = k.N3 + (size_t)w * tc_ld(nout);
  return k;
}
__global__ void pack_kernel(const float* __restrict__ p, Off o, Pack k, int nin, int w, int nout,
                            __nv_bfloat16* __restrict__ pb) {
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < k.n; i += (size_t)gridDim.x * blockDim.x) {
    float v = 0.0f;
    if (i < k.N2) {  // transposes: row = output, column = input
      const bool l1 = i < k.T2, l3 = i >= k.T3;
      const size_t j = i - (l1 ? k.T1 : (l3 ? k.T3 : k.T2));
      const int K = l1 ? nin : w, N = l3 ? nout : w;
      const int r = (int)(j / tc_ld(K)), c = (int)(j % tc_ld(K));
      if (c < K) v = p[(l1 ? o.W1 : (l3 ? o.W3 : o.W2)) + (size_t)c * N + r];
    } else {
      const bool l3 = i >= k.N3;
      const size_t j = i - (l3 ? k.N3 : k.N2);
      const int N = l3 ? nout : w;
      const int r = (int)(j / tc_ld(N)), c = (int)(j % tc_ld(N));
      if (c < N) v = p[(l3 ? o.W3 : o.W2) + (size_t)r * N + c];
    }
    pb[i] = __float2bfloat16(v);
  }
}
cudaError_t pack(const fsim_mlp* n, cudaStream_t s) {
  pack_kernel<<<256, 256, 0, s>>>(n->p, offsets(n->nin, n->width, n->nout), packing(n->nin, n->width, n->nout), n->nin,
                                  n->width, n->nout, n->pb);
  return cudaGetLastError();
}

// x to BF16 rows of whole K chunks; sum of the mask (when there is one)
__global__ void prep_kernel(const float* __restrict__ x, __nv_bfloat16* __restrict__ xb, int b, int nin,
                            const float* __restrict__ mask, size_t nmask, float* __restrict__ scal) {
  const int ld = tc_ld(nin);
  const size_t step = (size_t)gridDim.x * blockDim.x, i0 = blockIdx.x * (size_t)blockDim.x + threadIdx.x;
  // a warp per row and step
  for (size_t r = i0 / 32; r < (size_t)b; r += step / 32)
    for (int c = threadIdx.x & 31; c < ld; c += 32)
      xb[r * ld + c] = __float2bfloat16(c < nin ? x[r * nin + c] : 0.0f);
  if (!mask) return;
  float s = 0.0f;
#pragma unroll 4
  for (size_t i = i0; i < nmask; i += step) s += mask[i];
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) atomicAdd(scal + 1, s);
}

// gradient from its partial sums, in order: weights over the batch splits,
// biases over the row tiles; scal[0] = the loss numerator
__global__ void reduce_kernel(const float* __restrict__ part, int nsplit, const float* __restrict__ partb, int ntile,
                              int nloss, Off o, int w, int nout, float* __restrict__ g, float* __restrict__ scal) {
  const size_t nb = 2 * (size_t)w + nout;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < o.n; i += (size_t)gridDim.x * blockDim.x) {
    size_t bcol = nb;  // column of the bias sums, nb for a weight
    if (i >= o.b1 && i < o.W2) bcol = i - o.b1;
    else if (i >= o.b2 && i < o.W3) bcol = w + (i - o.b2);
    else if (i >= o.b3) bcol = 2 * (size_t)w + (i - o.b3);
    const float* src = bcol < nb ? partb + bcol : part + i;
    const size_t ld = bcol < nb ? nb : o.n;
    const int cnt = bcol < nb ? ntile : nsplit;
    float s = 0.0f;
#pragma unroll 8
    for (int r = 0; r < cnt; ++r) s += src[r * ld];
    g[i] = s;
  }
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    float s = 0.0f;
    for (int r = 0; r < nloss; ++r) s += partb[ntile * nb + r];
    scal[0] = s;
  }
}

cudaError_t gemm(const float* A, const float* B, float* C, const float* bias, int M, int N, int K, bool tA, bool tB,
                 cudaStream_t s) {
  dim3 grid((N + TN - 1) / TN, (M + TM - 1) / TM);
  gemm_kernel<<<grid, 128, 0, s>>>(A, B, C, bias, M, N, K, tA, tB);
  return cudaGetLastError();
}

template <int EPI>
cudaError_t layer(const __nv_bfloat16* A, const __nv_bfloat16* B, int M, int N, int K, const TcEpi& e, int* err,
                  cudaStream_t s) {
  constexpr int smem = tc_smem(kTcStages);
  const cudaError_t rc = cudaFuncSetAttribute(tc_layer_kernel<EPI>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
  if (rc != cudaSuccess) return rc;
  // an epilogue that writes padded BF16 rows covers the padding too
  const int cols = EPI == kTcOut ? N : tc_ld(N);
  dim3 grid((cols + kTcN - 1) / kTcN, (M + kTcM - 1) / kTcM);
  tc_layer_kernel<EPI><<<grid, kTcThreads, smem, s>>>(A, B, M, N, K, e, err);
  return cudaGetLastError();
}

// The loss numerator, mask sum and tensor-core flag in one copy; synchronises
// the stream.  FSIM_ECUDA when a tensor-core GEMM since the last check gave up
// waiting for its MMAs (the flag is cleared).
int finish(fsim_mlp* n, float* loss, cudaStream_t s) {
  float sc[3];
  FSIM_CK(cudaMemcpyAsync(sc, n->scal, sizeof(sc), cudaMemcpyDeviceToHost, s));
  FSIM_CK(cudaStreamSynchronize(s));
  if (loss) *loss = sc[0] / std::max(sc[1], 1.0f);
  int flag;
  std::memcpy(&flag, sc + 2, sizeof(flag));
  if (flag) {
    FSIM_CK(cudaMemset(n->tc_err, 0, sizeof(int)));
    set_error("MLP GEMM: tensor-core MMAs did not complete");
    return FSIM_ECUDA;
  }
  return FSIM_OK;
}

int ensure_batch(fsim_mlp* n, int b) {
  if (b <= n->maxb) return FSIM_OK;
  float** bufs[] = {&n->z1, &n->h1, &n->z2, &n->h2, &n->d1, &n->d2};
  for (float** q : bufs) {
    dev_free(*q);
    FSIM_TRY(dev_alloc(q, (size_t)b * n->width));
  }
  dev_free(n->y);
  dev_free(n->dy);
  FSIM_TRY(dev_alloc(&n->y, (size_t)b * n->nout));
  FSIM_TRY(dev_alloc(&n->dy, (size_t)b * n->nout));
  n->maxb = b;
  return FSIM_OK;
}

// ---- FP32 path (gradient checks)
int forward32(fsim_mlp* n, const float* x, float* y, int b, cudaStream_t s) {
  const Off o = offsets(n->nin, n->width, n->nout);
  const int w = n->width;
  const size_t bw = (size_t)b * w;
  const int th = 256, bl = (int)std::min<size_t>((bw + th - 1) / th, 1024);
  FSIM_CK(gemm(x, n->p + o.W1, n->z1, n->p + o.b1, b, w, n->nin, false, false, s));
  silu_kernel<<<bl, th, 0, s>>>(n->z1, n->h1, bw);
  FSIM_CK(gemm(n->h1, n->p + o.W2, n->z2, n->p + o.b2, b, w, w, false, false, s));
  silu_kernel<<<bl, th, 0, s>>>(n->z2, n->h2, bw);
  FSIM_CK(gemm(n->h2, n->p + o.W3, y, n->p + o.b3, b, n->nout, w, false, false, s));
  return FSIM_OK;
}

// loss and gradient (into n->g)
int backward32(fsim_mlp* n, const float* x, const float* t, const float* mask, int b, cudaStream_t s) {
  const Off o = offsets(n->nin, n->width, n->nout);
  const int w = n->width;
  const size_t bw = (size_t)b * w, bo = (size_t)b * n->nout;
  const int th = 256;
  auto blocks = [&](size_t k) { return (int)std::min<size_t>((k + th - 1) / th, 1024); };
  FSIM_CK(cudaMemsetAsync(n->scal, 0, 2 * sizeof(float), s));
  loss_kernel<<<blocks(bo), th, 0, s>>>(n->y, t, mask, n->dy, n->scal, bo);
  scale_kernel<<<blocks(bo), th, 0, s>>>(n->dy, n->scal, bo);
  // layer 3
  FSIM_CK(gemm(n->h2, n->dy, n->g + o.W3, nullptr, w, n->nout, b, true, false, s));
  colsum_kernel<<<(n->nout + 127) / 128, 128, 0, s>>>(n->dy, n->g + o.b3, b, n->nout);
  FSIM_CK(gemm(n->dy, n->p + o.W3, n->d2, nullptr, b, w, n->nout, false, true, s));
  silu_back_kernel<<<blocks(bw), th, 0, s>>>(n->z2, n->d2, bw);
  // layer 2
  FSIM_CK(gemm(n->h1, n->d2, n->g + o.W2, nullptr, w, w, b, true, false, s));
  colsum_kernel<<<(w + 127) / 128, 128, 0, s>>>(n->d2, n->g + o.b2, b, w);
  FSIM_CK(gemm(n->d2, n->p + o.W2, n->d1, nullptr, b, w, w, false, true, s));
  silu_back_kernel<<<blocks(bw), th, 0, s>>>(n->z1, n->d1, bw);
  // layer 1
  FSIM_CK(gemm(x, n->d1, n->g + o.W1, nullptr, n->nin, w, b, true, false, s));
  colsum_kernel<<<(w + 127) / 128, 128, 0, s>>>(n->d1, n->g + o.b1, b, w);
  return FSIM_OK;
}

// ---- BF16 path
inline int row_tiles(int b) { return (b + kTcM - 1) / kTcM; }
// Splits of the batch in the weight gradients: enough for four CTAs an SM, 32 at most
// (width 256: 10 tiles, 32 splits).  Each keeps a copy of the gradient, so a wide
// network, whose tiles fill the device by themselves, takes few.
int max_splits(const fsim_mlp* n) {
  const long long ti = row_tiles(n->nin), tw = row_tiles(n->width), to = row_tiles(n->nout);
  return (int)std::max(1LL, std::min(32LL, 4LL * device_sm_count() / (ti * tw + tw * tw + tw * to)));
}
int split_rows(const fsim_mlp* n, int b) {
  const int most = max_splits(n);
  return (row_tiles(b) + most - 1) / most * kTcM;
}

template <typename T>
int regrow(T** p, size_t n) {
  dev_free(*p);
  return dev_alloc(p, n);
}

int ensure_forward(fsim_mlp* n, int b) {
  if (b <= n->maxbt) return FSIM_OK;
  n->maxbt = n->maxbg = 0;
  const size_t bs = b, w = n->width, lw = tc_ld(n->width);
  FSIM_TRY(regrow(&n->xb, bs * tc_ld(n->nin)));
  FSIM_TRY(regrow(&n->h1b, bs * lw));
  FSIM_TRY(regrow(&n->h2b, bs * lw));
  FSIM_TRY(regrow(&n->z1t, bs * w));
  FSIM_TRY(regrow(&n->z2t, bs * w));
  n->maxbt = b;
  return FSIM_OK;
}

int ensure_backward(fsim_mlp* n, int b) {
  FSIM_TRY(ensure_forward(n, b));
  if (b <= n->maxbg) return FSIM_OK;
  n->maxbg = 0;
  const size_t bs = b, lw = tc_ld(n->width), nb = 2 * (size_t)n->width + n->nout;
  FSIM_TRY(regrow(&n->dyb, bs * tc_ld(n->nout)));
  FSIM_TRY(regrow(&n->d1b, bs * lw));
  FSIM_TRY(regrow(&n->d2b, bs * lw));
  FSIM_TRY(regrow(&n->part, (size_t)std::min(row_tiles(b), max_splits(n)) * n->np));
  FSIM_TRY(regrow(&n->partb, row_tiles(b) * (nb + (tc_ld(n->nout) + kTcN - 1) / kTcN)));
  n->maxbg = b;
  return FSIM_OK;
}

// hidden layers; mask != nullptr: also its sum, for a gradient
int hidden(fsim_mlp* n, const float* x, const float* mask, int b, cudaStream_t s) {
  const Off o = offsets(n->nin, n->width, n->nout);
  const Pack k = packing(n->nin, n->width, n->nout);
  const int w = n->width;
  FSIM_CK(cudaMemsetAsync(n->scal, 0, 2 * sizeof(float), s));
  const size_t work = std::max((size_t)b * tc_ld(n->nin), mask ? (size_t)b * n->nout : 0);
  prep_kernel<<<(int)std::min<size_t>((work + 1023) / 1024, 608), 256, 0, s>>>(x, n->xb, b, n->nin, mask,
                                                                              (size_t)b * n->nout, n->scal);
  FSIM_CK(cudaGetLastError());
  TcEpi e{};
  e.bias = n->p + o.b1; e.Z = n->z1t; e.O = n->h1b;
  FSIM_CK(layer<kTcHidden>(n->xb, n->pb + k.T1, b, w, n->nin, e, n->tc_err, s));
  e.bias = n->p + o.b2; e.Z = n->z2t; e.O = n->h2b;
  FSIM_CK(layer<kTcHidden>(n->h1b, n->pb + k.T2, b, w, w, e, n->tc_err, s));
  return FSIM_OK;
}

int forward16(fsim_mlp* n, const float* x, float* y, int b, cudaStream_t s) {
  FSIM_TRY(ensure_forward(n, b));
  FSIM_TRY(hidden(n, x, nullptr, b, s));
  const Off o = offsets(n->nin, n->width, n->nout);
  TcEpi e{};
  e.bias = n->p + o.b3; e.Y = y;
  FSIM_CK(layer<kTcOut>(n->h2b, n->pb + packing(n->nin, n->width, n->nout).T3, b, n->nout, n->width, e, n->tc_err, s));
  return FSIM_OK;
}

// loss (scal) and gradient (n->g)
int grad16(fsim_mlp* n, const float* x, const float* t, const float* mask, int b, cudaStream_t s) {
  FSIM_TRY(ensure_backward(n, b));
  FSIM_TRY(hidden(n, x, mask, b, s));
  const Off o = offsets(n->nin, n->width, n->nout);
  const Pack k = packing(n->nin, n->width, n->nout);
  const int w = n->width, nt = row_tiles(b), nb = 2 * w + n->nout;
  const int loss_cols = (tc_ld(n->nout) + kTcN - 1) / kTcN;
  TcEpi e{};
  e.bias = n->p + o.b3; e.O = n->dyb; e.t = t; e.mask = mask; e.scal = n->scal;
  e.colsum = n->partb + 2 * w; e.cs_ld = nb; e.lossp = n->partb + (size_t)nt * nb;
  FSIM_CK(layer<kTcLoss>(n->h2b, n->pb + k.T3, b, n->nout, w, e, n->tc_err, s));
  e = TcEpi{};
  e.cs_ld = nb;
  e.Z = n->z2t; e.O = n->d2b; e.colsum = n->partb + w;
  FSIM_CK(layer<kTcBack>(n->dyb, n->pb + k.N3, b, w, n->nout, e, n->tc_err, s));
  e.Z = n->z1t; e.O = n->d1b; e.colsum = n->partb;
  FSIM_CK(layer<kTcBack>(n->d2b, n->pb + k.N2, b, w, w, e, n->tc_err, s));
  TcWgrad g{};
  const int lw = tc_ld(w), tw = (w + kTcM - 1) / kTcM;
  auto tiles = [&](int i) { return (g.l[i].M + kTcM - 1) / kTcM * g.l[i].tn; };
  g.l[0] = TcWLayer{n->h2b, n->dyb, lw, tc_ld(n->nout), w, n->nout, (n->nout + kTcN - 1) / kTcN, 0, o.W3};
  g.l[1] = TcWLayer{n->h1b, n->d2b, lw, lw, w, w, tw, tiles(0), o.W2};
  g.l[2] = TcWLayer{n->xb, n->d1b, tc_ld(n->nin), lw, n->nin, w, tw, g.l[1].tile0 + tiles(1), o.W1};
  g.part = n->part;
  g.np = n->np;
  g.batch = b;
  g.rows = split_rows(n, b);
  const int nsplit = (b + g.rows - 1) / g.rows;
  constexpr int smem = tc_smem(kTcWStages);
  FSIM_CK(cudaFuncSetAttribute(tc_wgrad_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
  tc_wgrad_kernel<<<dim3(g.l[2].tile0 + tiles(2), nsplit), kTcThreads, smem, s>>>(g, n->tc_err);
  FSIM_CK(cudaGetLastError());
  reduce_kernel<<<(int)std::min<size_t>((n->np + 127) / 128, 2048), 128, 0, s>>>(n->part, nsplit, n->partb, nt,
                                                                                 nt * loss_cols, o, w, n->nout, n->g,
                                                                                 n->scal);
  FSIM_CK(cudaGetLastError());
  return FSIM_OK;
}

// loss and gradient in the precision asked for
int gradient(fsim_mlp* n, const float* x, const float* t, const float* mask, int b, bool bf16, cudaStream_t s) {
  if (bf16) return grad16(n, x, t, mask, b, s);
  FSIM_TRY(ensure_batch(n, b));
  FSIM_TRY(forward32(n, x, n->y, b, s));
  return backward32(n, x, t, mask, b, s);
}

int adam(fsim_mlp* n, float lr, cudaStream_t s) {
  ++n->step;
  const float b1 = 0.9f, b2 = 0.999f;
  adam_kernel<<<256, 256, 0, s>>>(n->p, n->g, n->m, n->v, n->np, lr, b1, b2, 1e-8f,
                                  1.0f - std::pow(b1, (float)n->step), 1.0f - std::pow(b2, (float)n->step));
  FSIM_CK(cudaGetLastError());
  FSIM_CK(pack(n, s));
  return FSIM_OK;
}

}  // namespace
}  // namespace fsim

void fsim::mlp_dims(const fsim_mlp* n, int* nin, int* width, int* nout) {
  *nin = n->nin;
  *width = n->width;
  *nout = n->nout;
}

using namespace fsim;

extern "C" {

int fsim_mlp_create(int nin, int width, int nout, const float* init_params, fsim_mlp** out) {
  if (!out || nin <= 0 || width <= 0 || nout <= 0 || !init_params) {
    set_error("fsim_mlp_create: bad arguments");
    return FSIM_EINVAL;
  }
  fsim_mlp* n = new fsim_mlp();
  n->nin = nin;
  n->width = width;
  n->nout = nout;
  n->np = offsets(nin, width, nout).n;
  int rc;
  auto fail = [&](int r) {
    fsim_mlp_destroy(n);
    return r;
  };
  float** bufs[] = {&n->p, &n->g, &n->m, &n->v};
  for (float** q : bufs)
    if ((rc = dev_alloc(q, n->np)) != FSIM_OK) return fail(rc);
  if ((rc = dev_alloc(&n->pb, packing(nin, width, nout).n)) != FSIM_OK || (rc = dev_alloc(&n->scal, 3)) != FSIM_OK)
    return fail(rc);
  n->tc_err = reinterpret_cast<int*>(n->scal + 2);
  if (cudaMemcpy(n->p, init_params, sizeof(float) * n->np, cudaMemcpyHostToDevice) != cudaSuccess ||
      cudaMemset(n->tc_err, 0, sizeof(int)) != cudaSuccess ||
      cudaMemset(n->m, 0, sizeof(float) * n->np) != cudaSuccess ||
      cudaMemset(n->v, 0, sizeof(float) * n->np) != cudaSuccess) {
    set_error("fsim_mlp_create: upload failed");
    return fail(FSIM_ECUDA);
  }
  if (pack(n, nullptr) != cudaSuccess || cudaDeviceSynchronize() != cudaSuccess) return fail(FSIM_ECUDA);
  *out = n;
  return FSIM_OK;
}

void fsim_mlp_destroy(fsim_mlp* n) {
  if (!n) return;
  float** bufs[] = {&n->p, &n->g, &n->m, &n->v, &n->z1, &n->h1, &n->z2, &n->h2, &n->y, &n->dy, &n->d1, &n->d2,
                    &n->scal, &n->z1t, &n->z2t, &n->part, &n->partb};
  for (float** q : bufs) dev_free(*q);
  __nv_bfloat16** bufb[] = {&n->pb, &n->xb, &n->h1b, &n->h2b, &n->dyb, &n->d1b, &n->d2b};
  for (__nv_bfloat16** q : bufb) dev_free(*q);
  delete n;
}

long long fsim_mlp_nparams(const fsim_mlp* n) { return n ? (long long)n->np : -1; }

int fsim_mlp_params(fsim_mlp* n, float* host_out, const float* host_in) {
  if (!n) return FSIM_EINVAL;
  if (host_out) FSIM_CK(cudaMemcpy(host_out, n->p, sizeof(float) * n->np, cudaMemcpyDeviceToHost));
  if (host_in) {
    FSIM_CK(cudaMemcpy(n->p, host_in, sizeof(float) * n->np, cudaMemcpyHostToDevice));
    FSIM_CK(pack(n, nullptr));
    FSIM_CK(cudaDeviceSynchronize());
  }
  return FSIM_OK;
}

int fsim_mlp_save(fsim_mlp* n, const char* path) {
  if (!n || !path) {
    set_error("fsim_mlp_save: null pointer");
    return FSIM_EINVAL;
  }
  std::vector<float> p(n->np);
  FSIM_CK(cudaMemcpy(p.data(), n->p, sizeof(float) * n->np, cudaMemcpyDeviceToHost));
  FILE* f = std::fopen(path, "wb");
  if (!f) {
    set_error("fsim_mlp_save: cannot open %s", path);
    return FSIM_EINVAL;
  }
  const int32_t dims[3] = {n->nin, n->width, n->nout};
  const bool ok = std::fwrite("FSIMMLP1", 1, 8, f) == 8 && std::fwrite(dims, sizeof(int32_t), 3, f) == 3 &&
                  std::fwrite(p.data(), sizeof(float), n->np, f) == n->np;
  if (std::fclose(f) != 0 || !ok) {
    set_error("fsim_mlp_save: write to %s failed", path);
    return FSIM_EINVAL;
  }
  return FSIM_OK;
}

int fsim_mlp_load(const char* path, fsim_mlp** out) {
  if (!path || !out) {
    set_error("fsim_mlp_load: null pointer");
    return FSIM_EINVAL;
  }
  *out = nullptr;
  FILE* f = std::fopen(path, "rb");
  if (!f) {
    set_error("fsim_mlp_load: cannot open %s", path);
    return FSIM_EINVAL;
  }
  char magic[8];
  int32_t dims[3];
  bool ok = std::fread(magic, 1, 8, f) == 8 && std::memcmp(magic, "FSIMMLP1", 8) == 0 &&
            std::fread(dims, sizeof(int32_t), 3, f) == 3 && dims[0] > 0 && dims[1] > 0 && dims[2] > 0 &&
            dims[0] <= 4096 && dims[1] <= 4096 && dims[2] <= 4096;
  std::vector<float> p;
  if (ok) {
    p.resize(offsets(dims[0], dims[1], dims[2]).n);
    ok = std::fread(p.data(), sizeof(float), p.size(), f) == p.size() && std::fgetc(f) == EOF;
  }
  std::fclose(f);
  if (!ok) {
    set_error("fsim_mlp_load: %s is not a weights file of fsim_mlp_save", path);
    return FSIM_EINVAL;
  }
  return fsim_mlp_create(dims[0], dims[1], dims[2], p.data(), out);
}

int fsim_mlp_forward(fsim_mlp* n, const float* x, float* y, int batch, int bf16, void* stream) {
  if (!n || !x || !y || batch <= 0) {
    set_error("fsim_mlp_forward: bad arguments");
    return FSIM_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  if (bf16) {
    FSIM_TRY(forward16(n, x, y, batch, s));
    return finish(n, nullptr, s);
  }
  FSIM_TRY(ensure_batch(n, batch));
  return forward32(n, x, y, batch, s);
}

int fsim_mlp_grad(fsim_mlp* n, const float* x, const float* t, const float* mask, int batch, int bf16, float* loss,
                  float* grad_host, void* stream) {
  if (!n || !x || !t || !mask || batch <= 0) {
    set_error("fsim_mlp_grad: bad arguments");
    return FSIM_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  FSIM_TRY(gradient(n, x, t, mask, batch, bf16 != 0, s));
  if (grad_host) FSIM_CK(cudaMemcpyAsync(grad_host, n->g, sizeof(float) * n->np, cudaMemcpyDeviceToHost, s));
  return finish(n, loss, s);
}

int fsim_mlp_adam_step(fsim_mlp* n, const float* grad_host, float lr, void* stream) {
  if (!n || !grad_host || !(lr > 0.0f)) {
    set_error("fsim_mlp_adam_step: bad arguments");
    return FSIM_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  FSIM_CK(cudaMemcpyAsync(n->g, grad_host, sizeof(float) * n->np, cudaMemcpyHostToDevice, s));
  FSIM_TRY(adam(n, lr, s));
  FSIM_CK(cudaStreamSynchronize(s));
  return FSIM_OK;
}

int fsim_mlp_train_step(fsim_mlp* n, const float* x, const float* t, const float* mask, int batch, float lr,
                        float* loss, void* stream) {
  if (!n || !x || !t || !mask || batch <= 0 || !(lr > 0.0f)) {
    set_error("fsim_mlp_train_step: bad arguments");
    return FSIM_EINVAL;
  }
  cudaStream_t s = (cudaStream_t)stream;
  FSIM_TRY(gradient(n, x, t, mask, batch, true, s));
  FSIM_TRY(adam(n, lr, s));
  return finish(n, loss, s);
}

}  // extern "C"
