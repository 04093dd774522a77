// BF16 x BF16 -> FP32 GEMMs on the fifth-generation tensor cores for the
// learned-guess network, with its element-wise steps as epilogues.
//
// One CTA of eight warps per 128 x 128 tile of the product.  The K dimension is
// walked in chunks of 64, each staged into shared memory in the canonical
// no-swizzle K-major layout (core matrices of 8 rows x 16 bytes, 128 contiguous
// bytes each); one thread issues four tcgen05.mma (M 128, N 128, K 16 each)
// that accumulate in tensor memory (128 lanes x 128 FP32 columns) and commits
// them to the chunk's mbarrier.  Then the accumulator goes through shared
// memory (tcgen05.ld gives a thread one row; the epilogue wants a column) and
// threads t and t + 128 run the epilogue on the halves of column t of the tile,
// eight rows' inputs in flight: global accesses coalesce and a column sum is
// one register.  A wait that runs out sets *err and the CTA frees its tensor
// memory and returns.
//
//  * tc_layer_kernel: forward layers and the data gradients.  Both operands lie
//    in memory K-contiguous, BF16, zero-padded to whole chunks (activations as
//    the previous epilogue left them, weights packed once per update), so a
//    chunk is 8 cp.async of 16 bytes per thread, kTcStages chunks in flight:
//    at K <= 256 every load is issued before the first MMA.
//  * tc_wgrad_kernel: weight gradients, K = the batch.  256 x 256 outputs are
//    only four tiles, so the batch is split over CTAs (partial products in a
//    workspace, summed in order by the caller: repeated calls give the same
//    bits), all layers in one launch; operands are batch-major and transposed
//    while they are staged (eight coalesced row loads per 16-byte unit).
// What bounds them is latency, not the tensor pipe (1.6 GFLOP in all): at batch
// 4096, width 256, a gradient took 4.4 ms when every GEMM staged 2-byte elements
// through FP32 loads and the weight gradients ran on 2-4 CTAs (1.1 ms each); it takes
// 0.16 ms now, the copy of its 0.54 MB to the host included.
#pragma once
#include <cuda_bf16.h>

#include <cstdint>

namespace fsim {

constexpr int kTcM = 128, kTcN = 128, kTcK = 64;
constexpr int kTcThreads = 256;
constexpr uint32_t kTcStage = (uint32_t)kTcM * kTcK * 2;  // bytes of one operand chunk
constexpr int kTcStages = 4;                      // chunks in flight, layers
constexpr int kTcWStages = 2;                     // chunks in flight, weight gradients
constexpr int kTcTileLd = kTcN + 1;               // accumulator tile in shared memory, padded against conflicts
constexpr uint32_t kTcTile = (uint32_t)kTcM * kTcTileLd * 4;
// dynamic shared memory per CTA: the larger of the operand ring and the
// accumulator tile (which reuses it), alignment slack and the barriers; at most
// three CTAs then share an SM and their tensor-memory allocations (3 x 128
// columns) fit the SM's 512 columns
__host__ __device__ constexpr uint32_t tc_ring(int stages) {
  return 2 * kTcStage * (uint32_t)stages > kTcTile ? 2 * kTcStage * (uint32_t)stages : (kTcTile + 63) / 64 * 64;
}
__host__ __device__ constexpr int tc_smem(int stages) { return (int)tc_ring(stages) + 1024 + 128; }
static_assert(4 * tc_smem(kTcWStages) > 227 * 1024, "four CTAs per SM would oversubscribe tensor memory");

// byte offset of element (row, k) of a 128 x 64 BF16 chunk: core matrix
// (row / 8, k / 8) at ((row / 8) * 8 + k / 8) * 128, row % 8 at 16-byte steps,
// k % 8 at 2-byte steps.  K-adjacent core matrices are 128 B apart, row groups
// 1024 B apart.
__host__ __device__ __forceinline__ uint32_t tc_off(int row, int k) {
  return ((uint32_t)(((row >> 3) * (kTcK / 8) + (k >> 3)) << 7)) + ((uint32_t)(row & 7) << 4) +
         ((uint32_t)(k & 7) << 1);
}

constexpr uint32_t kTcLbo = 128, kTcSbo = 1024;  // K-adjacent core matrices, 8-row groups

// shared-memory matrix descriptor: start address, leading-dimension byte offset
// (between K-adjacent core matrices), stride-dimension byte offset (between
// 8-row groups), descriptor version 1, no swizzle
__host__ __device__ __forceinline__ uint64_t tc_desc(uint32_t saddr, uint32_t lbo, uint32_t sbo) {
  return (uint64_t)((saddr >> 4) & 0x3FFFu) | ((uint64_t)((lbo >> 4) & 0x3FFFu) << 16) |
         ((uint64_t)((sbo >> 4) & 0x3FFFu) << 32) | (1ull << 46);
}

// instruction descriptor of kind::f16: FP32 accumulator, BF16 A and B, both
// K-major, N / 8 and M / 16
constexpr uint32_t kTcIdesc = (1u << 4) | (1u << 7) | (1u << 10) | ((uint32_t)(kTcN >> 3) << 17) |
                              ((uint32_t)(kTcM >> 4) << 24);

// bounded wait for the mbarrier phase of the given parity to complete
__device__ __forceinline__ bool tc_wait(uint32_t mbar, uint32_t parity) {
  for (int i = 0; i < (1 << 22); ++i) {
    uint32_t done;
    asm volatile(
        "{\n.reg .pred p;\nmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\nselp.u32 %0, 1, 0, p;\n}\n"
        : "=r"(done)
        : "r"(mbar), "r"(parity)
        : "memory");
    if (done) return true;
  }
  return false;
}

// One CTA's tensor memory (128 columns), ring of operand chunks and mbarriers
// (one per chunk slot).
struct TcCta {
  unsigned char* ring;
  uint32_t ringS, mS, tmem;
  int stages;

  __device__ __forceinline__ void init(unsigned char* raw_ptr, int nstages) {
    stages = nstages;
    const uint32_t raw = (uint32_t)__cvta_generic_to_shared(raw_ptr);
    const uint32_t pad = (1024u - (raw & 1023u)) & 1023u;
    ring = raw_ptr + pad;
    ringS = raw + pad;
    mS = ringS + tc_ring(nstages);
    const uint32_t tS = mS + 64;
    if (threadIdx.x < 32) {  // whole warp: 128 columns of tensor memory, address written to tS
      asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(tS), "r"(kTcN));
      asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;");
    }
    if (threadIdx.x == 0) {
      for (int i = 0; i < nstages; ++i) asm volatile("mbarrier.init.shared::cta.b64 [%0], 1;" ::"r"(mS + 8 * i));
      asm volatile("fence.mbarrier_init.release.cluster;");
    }
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    asm volatile("tcgen05.fence::after_thread_sync;");
    tmem = *reinterpret_cast<const uint32_t*>(ring + tc_ring(nstages) + 64);
  }
  __device__ __forceinline__ uint32_t chunk(int c) const { return (uint32_t)(c % stages) * 2 * kTcStage; }

  // one thread: the MMAs of chunk c (k0 = 64 c; the zero padding past K needs none)
  __device__ __forceinline__ void mma(int c, int K) const {
    asm volatile("tcgen05.fence::after_thread_sync;");
    const uint32_t aS = ringS + chunk(c), bS = aS + kTcStage;
#pragma unroll
    for (int kk = 0; kk < kTcK / 16; ++kk) {
      if (c * kTcK + kk * 16 >= K) break;
      const uint64_t ad = tc_desc(aS + (uint32_t)kk * 256u, kTcLbo, kTcSbo);
      const uint64_t bd = tc_desc(bS + (uint32_t)kk * 256u, kTcLbo, kTcSbo);
      const uint32_t accum = (c > 0 || kk > 0) ? 1u : 0u;
      asm volatile(
          "{\n.reg .pred p;\nsetp.ne.b32 p, %4, 0;\n"
          "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n}\n" ::"r"(tmem),
          "l"(ad), "l"(bd), "r"(kTcIdesc), "r"(accum));
    }
    asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(
                     mS + 8 * (c % stages))
                 : "memory");
  }
  // chunk c's MMAs (and all before them) are done
  __device__ __forceinline__ bool wait(int c) const {
    const bool ok = tc_wait(mS + 8 * (c % stages), (uint32_t)((c / stages) & 1));
    asm volatile("tcgen05.fence::after_thread_sync;");
    return ok;
  }
  // the accumulator as a row-major FP32 tile in the ring; every thread, all MMAs done
  __device__ __forceinline__ float* tile() const {
    float* t = reinterpret_cast<float*>(ring);
    const int warp = (threadIdx.x >> 5) & 3, half = threadIdx.x >> 7;  // warps w and w + 4: rows 32w .. 32w + 31
    const int row = threadIdx.x & 127;
#pragma unroll 1
    for (int c0 = half * (kTcN / 2); c0 < (half + 1) * (kTcN / 2); c0 += 16) {
      uint32_t v[16];
      asm volatile(
          "tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, "
          "%15}, [%16];\n"
          : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]),
            "=r"(v[8]), "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15])
          : "r"(tmem + ((uint32_t)(warp * 32) << 16) + (uint32_t)c0));
      asm volatile("tcgen05.wait::ld.sync.aligned;" ::: "memory");
#pragma unroll
      for (int j = 0; j < 16; ++j) t[row * kTcTileLd + c0 + j] = __uint_as_float(v[j]);
    }
    __syncthreads();
    return t;
  }
  __device__ __forceinline__ void release() const {
    asm volatile("tcgen05.fence::before_thread_sync;");
    __syncthreads();
    if (threadIdx.x < 32)
      asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kTcN));
  }
  // a chunk's MMAs did not complete in time: one more bounded wait before the
  // tensor memory they write is released
  __device__ __forceinline__ void give_up(int c, int* err) const {
    wait(c);
    if (threadIdx.x == 0) atomicExch(err, 1);
  }
};

__device__ __forceinline__ float tc_sig(float z) { return 1.0f / (1.0f + expf(-z)); }

// rows of the next GEMM's operands: whole 64-element chunks
__host__ __device__ constexpr int tc_ld(int k) { return (k + kTcK - 1) / kTcK * kTcK; }

// Epilogue of a layer.  M rows (batch), N columns; ldo = tc_ld(N).
struct TcEpi {
  const float* bias;    // kTcHidden, kTcOut, kTcLoss: [N]
  float* Z;             // kTcHidden out, kTcBack in: pre-activations [M x N]
  __nv_bfloat16* O;     // kTcHidden: silu(z); kTcLoss, kTcBack: the gradient; [M x ldo], padding written as zero
  float* Y;             // kTcOut: [M x N]
  const float *t, *mask;  // kTcLoss: [M x N]
  const float* scal;    // kTcLoss: [1] = sum of the mask
  float* colsum;        // kTcLoss, kTcBack: this row tile's column sums of the gradient, [row tile][cs_ld]
  int cs_ld;
  float* lossp;         // kTcLoss: this CTA's part of the loss numerator
};
enum { kTcHidden, kTcOut, kTcLoss, kTcBack };

// C[M x N] = A[M x K] B[N x K]^T: A, B BF16, K-contiguous, row strides tc_ld(K).
template <int EPI>
__global__ void __launch_bounds__(kTcThreads) tc_layer_kernel(const __nv_bfloat16* __restrict__ A,
                                                              const __nv_bfloat16* __restrict__ B, int M, int N,
                                                              int K, TcEpi e, int* __restrict__ err) {
  extern __shared__ unsigned char tc_smem_raw[];
  TcCta T;
  T.init(tc_smem_raw, kTcStages);
  const int tid = threadIdx.x;
  const int m0 = blockIdx.y * kTcM, n0 = blockIdx.x * kTcN;
  const int ld = tc_ld(K), nchunk = ld / kTcK;
  auto load = [&](int c) {  // 16-byte units of chunk c, rows past M or N zero-filled
    if (c < nchunk) {
      const uint32_t base = T.ringS + T.chunk(c);
#pragma unroll
      for (int i = 0; i < kTcM * kTcK / 8 / kTcThreads; ++i) {
        const int x = tid + i * kTcThreads, r = x >> 3, u = (x & 7) * 8;
        const bool va = m0 + r < M, vb = n0 + r < N;
        const __nv_bfloat16* pa = A + (size_t)(va ? m0 + r : 0) * ld + c * kTcK + u;
        const __nv_bfloat16* pb = B + (size_t)(vb ? n0 + r : 0) * ld + c * kTcK + u;
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(base + tc_off(r, u)), "l"(pa),
                     "r"(va ? 16 : 0)
                     : "memory");
        asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(base + kTcStage + tc_off(r, u)), "l"(pb),
                     "r"(vb ? 16 : 0)
                     : "memory");
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  for (int c = 0; c < kTcStages - 1; ++c) load(c);
  bool ok = true;
  int cfail = 0;
  for (int c = 0; c < nchunk; ++c) {
    // the slot of chunk c + kTcStages - 1 held chunk c - 1
    if (c > 0 && c + kTcStages - 1 < nchunk) ok = T.wait(c - 1);
    if (ok) load(c + kTcStages - 1);
    asm volatile("cp.async.wait_group %0;" ::"n"(kTcStages - 1) : "memory");
    // the copies become visible to the tensor cores' (async proxy) reads
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (__syncthreads_or(!ok)) {
      ok = false;
      cfail = c - 1;
      break;
    }
    if (tid == 0) T.mma(c, K);
  }
  if (ok) {
    ok = T.wait(nchunk - 1);
    cfail = nchunk - 1;
    ok = !__syncthreads_or(!ok);
  }
  asm volatile("cp.async.wait_all;" ::: "memory");
  if (ok) {
    float* tile = T.tile();
    const int tc = tid & 127, col = n0 + tc;
    const int r0 = (tid >> 7) * (kTcM / 2), r1 = min(r0 + kTcM / 2, M - m0);
    const int ldo = tc_ld(N);
    const bool in = col < N;
    const float b = (EPI != kTcBack && in) ? e.bias[col] : 0.0f;
    const float inv = EPI == kTcLoss ? 1.0f / fmaxf(e.scal[1], 1.0f) : 0.0f;
    float sum = 0.0f, num = 0.0f;
    if (in) {
      for (int r = r0; r < r1; r += 8) {
        float p[8], q[8];  // inputs of eight rows, all loads in flight
        if constexpr (EPI == kTcBack || EPI == kTcLoss) {
#pragma unroll
          for (int u = 0; u < 8; ++u) {
            const size_t at = (size_t)(m0 + min(r + u, r1 - 1)) * N + col;
            p[u] = EPI == kTcBack ? e.Z[at] : e.mask[at];
            if constexpr (EPI == kTcLoss) q[u] = e.t[at];
          }
        }
#pragma unroll
        for (int u = 0; u < 8; ++u) {
          if (r + u >= r1) break;
          const float acc = tile[(r + u) * kTcTileLd + tc];
          const size_t at = (size_t)(m0 + r + u) * N + col, ao = (size_t)(m0 + r + u) * ldo + col;
          if constexpr (EPI == kTcHidden) {
            const float z = acc + b;
            e.Z[at] = z;
            e.O[ao] = __float2bfloat16(z * tc_sig(z));
          } else if constexpr (EPI == kTcOut) {
            e.Y[at] = acc + b;
          } else if constexpr (EPI == kTcLoss) {
            // loss numerator, dy = 2 mask (y - t) / sum(mask)
            const float d = (acc + b) - q[u];
            num += p[u] * d * d;
            const float dy = 2.0f * p[u] * d * inv;
            sum += dy;
            e.O[ao] = __float2bfloat16(dy);
          } else {
            const float z = p[u], s = tc_sig(z);
            const float d = acc * (s * (1.0f + z * (1.0f - s)));
            sum += d;
            e.O[ao] = __float2bfloat16(d);
          }
        }
      }
    } else if (EPI != kTcOut && col < ldo) {
      for (int r = r0; r < r1; ++r) e.O[(size_t)(m0 + r) * ldo + col] = __float2bfloat16(0.0f);
    }
    if constexpr (EPI == kTcLoss || EPI == kTcBack) {
      __syncthreads();  // the tile has been read
      tile[tid] = sum;
      tile[kTcThreads + tid] = num;
      __syncthreads();
      if (tid < kTcN && in) e.colsum[(size_t)blockIdx.y * e.cs_ld + col] = tile[tid] + tile[tid + kTcN];
      if constexpr (EPI == kTcLoss) {
        for (int o = kTcThreads / 2; o > 0; o >>= 1) {
          if (tid < o) tile[kTcThreads + tid] += tile[kTcThreads + tid + o];
          __syncthreads();
        }
        if (tid == 0) e.lossp[blockIdx.y * gridDim.x + blockIdx.x] = tile[kTcThreads];
      }
    }
  } else {
    T.give_up(cfail < 0 ? 0 : cfail, err);
  }
  T.release();
}

// One layer's weight gradient G[M x N] = A^T B over the batch: A [batch x lda],
// B [batch x ldb] BF16; tiles of the launch from tile0 on, tn of them per row
// of tiles; the product lands at off in a workspace slice.
struct TcWLayer {
  const __nv_bfloat16 *A, *B;
  int lda, ldb, M, N, tn, tile0;
  size_t off;
};
struct TcWgrad {
  TcWLayer l[3];
  float* part;   // [split][np]
  size_t np;
  int batch, rows;  // batch rows per split (a multiple of 64)
};

__global__ void __launch_bounds__(kTcThreads) tc_wgrad_kernel(TcWgrad P, int* __restrict__ err) {
  extern __shared__ unsigned char tc_smem_raw[];
  TcCta T;
  T.init(tc_smem_raw, kTcWStages);
  const int tid = threadIdx.x;
  int li = 0;
  while (li < 2 && (int)blockIdx.x >= P.l[li + 1].tile0) ++li;
  const TcWLayer L = P.l[li];
  const int tile = blockIdx.x - L.tile0, m0 = tile / L.tn * kTcM, n0 = tile % L.tn * kTcN;
  const int k_lo = blockIdx.y * P.rows, k_hi = min(k_lo + P.rows, P.batch), K = k_hi - k_lo;
  const int nchunk = (K + kTcK - 1) / kTcK;
  // 16-byte units (8 batch rows) of two adjacent columns per thread and step
  auto stage = [&](const __nv_bfloat16* src, int ld, int c0, int k0, unsigned char* dst) {
#pragma unroll
    for (int i = 0; i < kTcM / 2 * (kTcK / 8) / kTcThreads; ++i) {
      const int x = tid + i * kTcThreads, m = (x & 63) * 2, u = (x >> 6) * 8;
      uint32_t w[8];
#pragma unroll
      for (int r = 0; r < 8; ++r) {
        const int k = k0 + u + r;
        w[r] = (k < k_hi && c0 + m < ld) ? *reinterpret_cast<const uint32_t*>(src + (size_t)k * ld + c0 + m) : 0u;
      }
      uint4 lo, hi;
      lo.x = __byte_perm(w[0], w[1], 0x5410); hi.x = __byte_perm(w[0], w[1], 0x7632);
      lo.y = __byte_perm(w[2], w[3], 0x5410); hi.y = __byte_perm(w[2], w[3], 0x7632);
      lo.z = __byte_perm(w[4], w[5], 0x5410); hi.z = __byte_perm(w[4], w[5], 0x7632);
      lo.w = __byte_perm(w[6], w[7], 0x5410); hi.w = __byte_perm(w[6], w[7], 0x7632);
      *reinterpret_cast<uint4*>(dst + tc_off(m, u)) = lo;
      *reinterpret_cast<uint4*>(dst + tc_off(m + 1, u)) = hi;
    }
  };
  bool ok = true;
  int cfail = 0;
  for (int c = 0; c < nchunk; ++c) {
    if (c >= kTcWStages) ok = T.wait(c - kTcWStages);
    if (ok) {
      unsigned char* s = T.ring + T.chunk(c);
      stage(L.A, L.lda, m0, k_lo + c * kTcK, s);
      stage(L.B, L.ldb, n0, k_lo + c * kTcK, s + kTcStage);
    }
    asm volatile("fence.proxy.async.shared::cta;" ::: "memory");
    if (__syncthreads_or(!ok)) {
      ok = false;
      cfail = c - kTcWStages;
      break;
    }
    if (tid == 0) T.mma(c, K);
  }
  if (ok) {
    ok = T.wait(nchunk - 1);
    cfail = nchunk - 1;
    ok = !__syncthreads_or(!ok);
  }
  if (ok) {
    const float* t = T.tile();
    float* out = P.part + (size_t)blockIdx.y * P.np + L.off;
    const int tc = tid & 127, r0 = (tid >> 7) * (kTcM / 2), r1 = min(r0 + kTcM / 2, L.M - m0);
    if (n0 + tc < L.N)
#pragma unroll 8
      for (int r = r0; r < r1; ++r) out[(size_t)(m0 + r) * L.N + n0 + tc] = t[r * kTcTileLd + tc];
  } else {
    T.give_up(cfail < 0 ? 0 : cfail, err);
  }
  T.release();
}

}  // namespace fsim
