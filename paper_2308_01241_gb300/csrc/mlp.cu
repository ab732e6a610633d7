// mlp.cu -- the learned surrogate's MLP: BF16 tensor-core GEMMs with FP32
// accumulation (mma.sync.m16n8k16), fused bias / GELU epilogues, backward
// pass and Adam, behind the C ABI of include/dtb_surrogate.h.
//
// The surrogate's layers are 256 wide: that case has kernels of its own, one
// launch per prediction and two per training step (chain_kernel, dw_kernel);
// gemm_kernel and its launches serve every other width.
// GELU(x) = 0.5 x (1 + erf(x / sqrt 2)) calls erff.
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <math.h>
#include <stdint.h>

#include <algorithm>
#include <string>
#include <vector>

#include "dtb.h"
#include "dtb_launch.h"
#include "dtb_surrogate.h"

namespace {

typedef __nv_bfloat16 bf16;

constexpr int kT = 64;   // block tile (rows and columns)
constexpr int kBK = 16;  // k step
constexpr int kPad = 8;  // shared-memory row padding (bank spread)

enum { EPI_GELU = 1, EPI_BIAS = 2, EPI_DGELU = 3, EPI_F32 = 4 };

struct Epi {
  const float* bias;  // [N]
  float* z;           // EPI_GELU: pre-activation out [M][N]
  bf16* a;            // EPI_GELU: activation out; EPI_DGELU: gradient out [M][N]
  float* y;           // EPI_BIAS / EPI_F32: fp32 out [M][N]
  const float* zin;   // EPI_DGELU: pre-activation of the layer below [M][N]
};

__device__ __forceinline__ float gelu(float x) { return 0.5f * x * (1.0f + erff(x * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float x) {
  return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * expf(-0.5f * x * x) * 0.39894228040143268f;
}

__device__ __forceinline__ void mma_bf16(float (&c)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k16.row.col.f32.bf16.bf16.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, {%8,%9}, "
      "{%0,%1,%2,%3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

// C[M][N] = sum_k A(m, k) B(k, n) with A(m, k) = TA ? a[k*lda + m] : a[m*lda + k]
// and B(k, n) = TB ? b[n*ldb + k] : b[k*ldb + n]; out-of-range elements read 0.
// 128 threads = 2 x 2 warps, each 32 x 32 = 2 x 4 mma tiles of 16 x 8.
template <bool TA, bool TB, int EPI>
__global__ void __launch_bounds__(128) gemm_kernel(const bf16* __restrict__ a, int lda, const bf16* __restrict__ b,
                                                   int ldb, int M, int N, int K, Epi ep) {
  __shared__ __align__(16) bf16 As[kT][kBK + kPad];  // [m][k]
  __shared__ __align__(16) bf16 Bs[kT][kBK + kPad];  // [n][k]
  const int m0 = blockIdx.y * kT, n0 = blockIdx.x * kT;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int wm = (warp >> 1) * 32, wn = (warp & 1) * 32;
  const int g = lane >> 2, t = lane & 3;
  const bf16 zero = __float2bfloat16(0.0f);
  float acc[2][4][4];
#pragma unroll
  for (int i = 0; i < 2; i++)
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
      for (int q = 0; q < 4; q++) acc[i][j][q] = 0.0f;

  for (int k0 = 0; k0 < K; k0 += kBK) {
    for (int idx = threadIdx.x; idx < kT * kBK; idx += 128) {
      int mm, kk;
      if (TA) { kk = idx / kT; mm = idx % kT; } else { mm = idx / kBK; kk = idx % kBK; }
      const int m = m0 + mm, k = k0 + kk;
      As[mm][kk] = (m < M && k < K) ? (TA ? a[(int64_t)k * lda + m] : a[(int64_t)m * lda + k]) : zero;
      int nn, kb;
      if (TB) { nn = idx / kBK; kb = idx % kBK; } else { kb = idx / kT; nn = idx % kT; }
      const int n = n0 + nn, kq = k0 + kb;
      Bs[nn][kb] = (n < N && kq < K) ? (TB ? b[(int64_t)n * ldb + kq] : b[(int64_t)kq * ldb + n]) : zero;
    }
    __syncthreads();
    uint32_t af[2][4], bfr[4][2];
#pragma unroll
    for (int i = 0; i < 2; i++) {
      const int r = wm + i * 16 + g;
      af[i][0] = *reinterpret_cast<const uint32_t*>(&As[r][2 * t]);
      af[i][1] = *reinterpret_cast<const uint32_t*>(&As[r + 8][2 * t]);
      af[i][2] = *reinterpret_cast<const uint32_t*>(&As[r][2 * t + 8]);
      af[i][3] = *reinterpret_cast<const uint32_t*>(&As[r + 8][2 * t + 8]);
    }
#pragma unroll
    for (int j = 0; j < 4; j++) {
      const int c = wn + j * 8 + g;
      bfr[j][0] = *reinterpret_cast<const uint32_t*>(&Bs[c][2 * t]);
      bfr[j][1] = *reinterpret_cast<const uint32_t*>(&Bs[c][2 * t + 8]);
    }
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
      for (int j = 0; j < 4; j++) mma_bf16(acc[i][j], af[i], bfr[j]);
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 2; i++)
#pragma unroll
    for (int j = 0; j < 4; j++)
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int m = m0 + wm + i * 16 + g + (q >= 2 ? 8 : 0);
        const int n = n0 + wn + j * 8 + 2 * t + (q & 1);
        if (m >= M || n >= N) continue;
        const int64_t o = (int64_t)m * N + n;
        const float v = acc[i][j][q];
        if (EPI == EPI_GELU) {
          const float z = v + ep.bias[n];
          ep.z[o] = z;
          ep.a[o] = __float2bfloat16(gelu(z));
        } else if (EPI == EPI_BIAS) {
          ep.y[o] = v + ep.bias[n];
        } else if (EPI == EPI_DGELU) {
          ep.a[o] = __float2bfloat16(v * gelu_grad(ep.zin[o]));
        } else {
          ep.y[o] = v;
        }
      }
}

__global__ void to_bf16_kernel(const float* x, bf16* y, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    y[i] = __float2bfloat16(x[i]);
}

// Mean-squared-error gradient dY = 2 (Y - T) / (B * n_out), stored in bf16 for
// the backward GEMMs; per-block sums of (Y - T)^2 for the loss.
__global__ void mse_grad_kernel(const float* y, const float* tgt, bf16* dy, int64_t n, float scale, float* part) {
  __shared__ float sh[8];
  float s = 0.0f;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    const float d = y[i] - tgt[i];
    s += d * d;
    dy[i] = __float2bfloat16(2.0f * d * scale);
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xFFFFFFFFu, s, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float tot = 0.0f;
    for (int w = 0; w < (int)(blockDim.x >> 5); w++) tot += sh[w];
    part[blockIdx.x] = tot;
  }
}

// db[n] = sum over rows of G[m][n] (bf16 gradient), fp32.
__global__ void colsum_kernel(const bf16* G, int M, int N, float* db) {
  const int n = blockIdx.x * blockDim.x + threadIdx.x;
  if (n >= N) return;
  float s = 0.0f;
  for (int m = 0; m < M; m++) s += __bfloat162float(G[(int64_t)m * N + n]);
  db[n] = s;
}

// ---- 256-wide networks: two launches per training step, one per prediction ----
//
// A prediction of a few thousand rows is about a GFLOP: separate launches per
// layer (each reloading its tiles element by element) took 99 us for 5,978 rows
// and 1.4 ms per training step of 4,096 rows, most of it in the serial column
// sums and in 16-block weight-gradient products.  Here
//   chain_kernel  carries R rows through all layers: activations stay in
//                 shared memory, weights stream through a ring of 64-row
//                 chunks (cp.async), and for training the loss gradient and
//                 the backward pass of the same rows follow in the same CTA;
//   dw_kernel     computes every layer's weight gradient in one launch, 32 x 32
//                 outputs per CTA over all rows, the bias gradients as serial
//                 column sums by a warp of their own, and Adam in the epilogue.
// Every output is accumulated over k in ascending steps of 16 by the same
// m16n8k16 product as gemm_kernel, and column sums add their rows in order, so
// the results are bit for bit those of the general path.  (The 5th-generation
// tensor cores accumulate in another order, which moves bfloat16 roundings of
// the activations.)
constexpr int kW = 256;          // width
constexpr int kMaxLayers = 8;    // hidden layers + 1
constexpr int kMaxOut = 16;
constexpr int kActLd = kW + 8;   // shared-memory row strides (elements), 16-byte aligned, spread over banks
constexpr int kFwdLd = kW + 8, kBwdLd = 64 + 8;
constexpr int kChunkBytes = kW * kBwdLd * 2;  // a 64-row forward chunk (64 x 264) fits as well
constexpr int kChunks = 4;
static_assert(64 * kFwdLd * 2 <= kChunkBytes, "chunk buffer");

struct ChainNet {
  int n_in, n_out, nl;               // nl = hidden layers + 1
  int xs, ys;                        // row strides of x16 and dy (multiples of 8)
  const bf16* w[kMaxLayers];         // bf16 weights [din][dout]
  const float* b[kMaxLayers];
  bf16* x16;                         // training: [B][xs]
  bf16* act[kMaxLayers];             // training: input of layer l >= 1, [B][kW]
  float* z[kMaxLayers];              // training: pre-activation of layer l - 1's output, [B][kW]
  bf16* g[kMaxLayers];               // training: gradient at the output of layer l < nl - 1, [B][kW]
  bf16* dy;                          // training: [B][ys]
  float* part;                       // training: [CTAs] sums of squared errors
};

__device__ __forceinline__ uint32_t smem32(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void cp_async16(void* dst, const void* src, bool in) {
  const int n = in ? 16 : 0;  // bytes read; the rest is filled with zeros
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem32(dst)), "l"(src), "r"(n) : "memory");
}
__device__ __forceinline__ void cp_commit() { asm volatile("cp.async.commit_group;" ::: "memory"); }
template <int N>
__device__ __forceinline__ void cp_wait() {
  asm volatile("cp.async.wait_group %0;" ::"n"(N) : "memory");
}
__device__ __forceinline__ void ldsm4(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem32(p)));
}
__device__ __forceinline__ void ldsm4t(uint32_t (&r)[4], const void* p) {
  asm volatile("ldmatrix.sync.aligned.m8n8.x4.trans.shared.b16 {%0,%1,%2,%3}, [%4];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3])
               : "r"(smem32(p)));
}

template <int R>
struct ChainSmem {
  static constexpr size_t kChunk = 0;
  static constexpr size_t kAct = kChunk + (size_t)kChunks * kChunkBytes;  // bf16 [R][kActLd]
  static constexpr size_t kWoT = kAct + (size_t)R * kActLd * 2;           // bf16 [kMaxOut][kActLd]: output weights by column
  static constexpr size_t kWo = kWoT + (size_t)kMaxOut * kActLd * 2;      // bf16 [kW][kMaxOut + 8]: by row
  static constexpr size_t kDy = kWo + (size_t)kW * (kMaxOut + 8) * 2;     // bf16 [R][kMaxOut + 8]
  static constexpr size_t kBytes = kDy + (size_t)R * (kMaxOut + 8) * 2;
};

// R rows per CTA, 8 warps: R / 32 along the rows (32 each) by 256 R / 32 / 8
// columns... the warp's tile is 32 x (R == 64 ? 64 : 32).
template <int R, bool TRAIN>
__global__ void __launch_bounds__(256) chain_kernel(ChainNet n, const float* __restrict__ x, const float* __restrict__ tgt,
                                                    float* __restrict__ y, int B, float scale) {
  using L = ChainSmem<R>;
  constexpr int kNT = R == 64 ? 8 : 4;  // 8-column tiles per warp
  extern __shared__ __align__(16) unsigned char sm[];
  bf16* act = reinterpret_cast<bf16*>(sm + L::kAct);
  bf16* woT = reinterpret_cast<bf16*>(sm + L::kWoT);
  bf16* wo = reinterpret_cast<bf16*>(sm + L::kWo);
  bf16* dys = reinterpret_cast<bf16*>(sm + L::kDy);
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int wm = R == 64 ? (warp >> 2) * 32 : 0, wn = R == 64 ? (warp & 3) * 64 : warp * 32;
  const int gq = lane >> 2, tq = lane & 3;
  const int m0 = blockIdx.x * R;
  const bf16 zero = __float2bfloat16(0.0f);

  // The weight chunks in the order they are used: layer 0 .. nl - 2 forward
  // (64 input rows each), then, training, layer nl - 2 .. 1 backward (64
  // output columns each: rows of the transposed weights).
  const int c0 = (n.n_in + 63) / 64;                // chunks of layer 0
  const int hid = n.nl - 2;                         // further hidden layers, 4 chunks each
  const int fwd_chunks = c0 + 4 * hid;
  const int all_chunks = fwd_chunks + (TRAIN ? 4 * hid : 0);
  auto fetch = [&](int c) {
    if (c < all_chunks) {
      unsigned char* buf = sm + L::kChunk + (size_t)(c % kChunks) * kChunkBytes;
      if (c < fwd_chunks) {
        const int l = c < c0 ? 0 : 1 + (c - c0) / 4, k0 = c < c0 ? c * 64 : ((c - c0) & 3) * 64;
        const int din = l == 0 ? n.n_in : kW;
        bf16* d = reinterpret_cast<bf16*>(buf);
#pragma unroll
        for (int q = 0; q < 8; q++) {  // 64 rows x 32 pieces of 16 bytes
          const int i = tid + 256 * q, r = i >> 5, s = i & 31;
          const bool in = k0 + r < din;
          cp_async16(d + r * kFwdLd + s * 8, n.w[l] + (int64_t)(in ? k0 + r : 0) * kW + s * 8, in);
        }
      } else {
        const int l = n.nl - 2 - (c - fwd_chunks) / 4, k0 = ((c - fwd_chunks) & 3) * 64;
        bf16* d = reinterpret_cast<bf16*>(buf);
#pragma unroll
        for (int q = 0; q < 8; q++) {  // 256 rows x 8 pieces
          const int i = tid + 256 * q, r = i >> 3, s = i & 7;
          cp_async16(d + r * kBwdLd + s * 8, n.w[l] + (int64_t)r * kW + k0 + s * 8, true);
        }
      }
    }
    cp_commit();  // one group per chunk, empty or not: the wait counts stay the same
  };
#pragma unroll
  for (int c = 0; c < kChunks - 1; c++) fetch(c);

  // inputs, and the output layer's weights both ways round, zero padded
  const int kin = (n.n_in + 15) & ~15;
  for (int i = tid; i < R * kin; i += 256) {
    const int r = i / kin, k = i - r * kin;
    const bf16 v = m0 + r < B && k < n.n_in ? __float2bfloat16(x[(int64_t)(m0 + r) * n.n_in + k]) : zero;
    act[r * kActLd + k] = v;
    if (TRAIN && m0 + r < B && k < n.xs) n.x16[(int64_t)(m0 + r) * n.xs + k] = v;
  }
  const bf16* wl = n.w[n.nl - 1];
  for (int i = tid; i < kW * kMaxOut; i += 256) {
    const int k = i / kMaxOut, o = i % kMaxOut;
    const bf16 v = o < n.n_out ? wl[(int64_t)k * n.n_out + o] : zero;
    woT[o * kActLd + k] = v;
    wo[k * (kMaxOut + 8) + o] = v;
  }

  float acc[2][kNT][4];
  auto clear = [&]() {
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
      for (int j = 0; j < kNT; j++)
#pragma unroll
        for (int q = 0; q < 4; q++) acc[i][j][q] = 0.0f;
  };
  auto load_a = [&](uint32_t (&a)[2][4], const bf16* base, int ld, int k) {
#pragma unroll
    for (int i = 0; i < 2; i++) ldsm4(a[i], base + (wm + i * 16 + (lane & 15)) * ld + k + (lane >> 4) * 8);
  };
  auto mma_all = [&](const uint32_t (&a)[2][4], const uint32_t (&b)[kNT][2]) {
#pragma unroll
    for (int i = 0; i < 2; i++)
#pragma unroll
      for (int j = 0; j < kNT; j++) mma_bf16(acc[i][j], a[i], b[j]);
  };
  int c = 0;
  // the next chunk: every warp is past the buffer that the fetch overwrites
  auto next_chunk = [&]() -> const bf16* {
    cp_wait<kChunks - 2>();
    __syncthreads();
    fetch(c + kChunks - 1);
    const bf16* p = reinterpret_cast<const bf16*>(sm + L::kChunk + (size_t)(c % kChunks) * kChunkBytes);
    c++;
    return p;
  };

  for (int l = 0; l < n.nl - 1; l++) {
    clear();
    const int din = l == 0 ? n.n_in : kW;
    for (int k0 = 0; k0 < din; k0 += 64) {
      const bf16* wc = next_chunk();
      const int steps = (min(64, din - k0) + 15) >> 4;
#pragma unroll 4
      for (int s = 0; s < steps; s++) {
        uint32_t a[2][4], b[kNT][2];
        load_a(a, act, kActLd, k0 + s * 16);
#pragma unroll
        for (int j = 0; j < kNT; j += 2) {  // two 8-column tiles per load, transposed
          uint32_t r[4];
          ldsm4t(r, wc + (s * 16 + (lane & 15)) * kFwdLd + wn + j * 8 + (lane >> 4) * 8);
          b[j][0] = r[0]; b[j][1] = r[1]; b[j + 1][0] = r[2]; b[j + 1][1] = r[3];
        }
        mma_all(a, b);
      }
    }
    __syncthreads();  // every warp has read its rows of act
#pragma unroll
    for (int j = 0; j < kNT; j++) {
      const int col = wn + j * 8 + 2 * tq;
      const float b0 = n.b[l][col], b1 = n.b[l][col + 1];
#pragma unroll
      for (int i = 0; i < 2; i++)
#pragma unroll
        for (int h = 0; h < 2; h++) {
          const int r = wm + i * 16 + gq + 8 * h;
          const float z0 = acc[i][j][2 * h] + b0, z1 = acc[i][j][2 * h + 1] + b1;
          __nv_bfloat162 v;
          v.x = __float2bfloat16(gelu(z0));
          v.y = __float2bfloat16(gelu(z1));
          *reinterpret_cast<__nv_bfloat162*>(act + r * kActLd + col) = v;
          if (TRAIN && m0 + r < B) {
            const int64_t o = (int64_t)(m0 + r) * kW + col;
            *reinterpret_cast<float2*>(n.z[l + 1] + o) = make_float2(z0, z1);
            *reinterpret_cast<__nv_bfloat162*>(n.act[l + 1] + o) = v;
          }
        }
    }
    __syncthreads();
  }

  // output layer: 16 rows per warp, both 8-column tiles
  float sq = 0.0f;
  if (warp < R / 16) {
    float o[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll 4
    for (int k = 0; k < kW; k += 16) {
      uint32_t a[4];
      ldsm4(a, act + (warp * 16 + (lane & 15)) * kActLd + k + (lane >> 4) * 8);
#pragma unroll
      for (int j = 0; j < 2; j++) {
        const uint32_t b[2] = {*reinterpret_cast<const uint32_t*>(woT + (j * 8 + gq) * kActLd + k + 2 * tq),
                               *reinterpret_cast<const uint32_t*>(woT + (j * 8 + gq) * kActLd + k + 2 * tq + 8)};
        mma_bf16(o[j], a, b);
      }
    }
#pragma unroll
    for (int j = 0; j < 2; j++)
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int r = warp * 16 + gq + (q >= 2 ? 8 : 0), col = j * 8 + 2 * tq + (q & 1);
        const bool in = m0 + r < B && col < n.n_out;
        float v = 0.0f;
        if (in) v = o[j][q] + n.b[n.nl - 1][col];
        if (!TRAIN) {
          if (in) y[(int64_t)(m0 + r) * n.n_out + col] = v;
        } else {
          bf16 d16 = zero;
          if (in) {
            const float d = v - tgt[(int64_t)(m0 + r) * n.n_out + col];
            sq += d * d;
            d16 = __float2bfloat16(2.0f * d * scale);
          }
          dys[r * (kMaxOut + 8) + col] = d16;
          if (m0 + r < B && col < n.ys) n.dy[(int64_t)(m0 + r) * n.ys + col] = d16;
        }
      }
  }
  if (!TRAIN) return;

  // loss: one partial sum per CTA
  __shared__ float s_sq[8];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sq += __shfl_xor_sync(0xFFFFFFFFu, sq, o);
  if (lane == 0) s_sq[warp] = sq;
  __syncthreads();  // also publishes dys
  if (tid == 0) {
    float t = 0.0f;
    for (int w = 0; w < R / 16; w++) t += s_sq[w];
    n.part[blockIdx.x] = t;
  }

  // backward: gradient at the output of layer l, from the layer above
  for (int l = n.nl - 2; l >= 0; l--) {
    clear();
    if (l == n.nl - 2) {  // from the output gradient: one step over its columns
      uint32_t a[2][4], b[kNT][2];
      load_a(a, dys, kMaxOut + 8, 0);
#pragma unroll
      for (int j = 0; j < kNT; j += 2) {
        uint32_t r[4];
        ldsm4(r, wo + (wn + j * 8 + (lane & 7) + (lane >> 4) * 8) * (kMaxOut + 8) + ((lane >> 3) & 1) * 8);
        b[j][0] = r[0]; b[j][1] = r[1]; b[j + 1][0] = r[2]; b[j + 1][1] = r[3];
      }
      mma_all(a, b);
    } else {
      for (int k0 = 0; k0 < kW; k0 += 64) {
        const bf16* wc = next_chunk();
#pragma unroll
        for (int s = 0; s < 4; s++) {
          uint32_t a[2][4], b[kNT][2];
          load_a(a, act, kActLd, k0 + s * 16);
#pragma unroll
          for (int j = 0; j < kNT; j += 2) {
            uint32_t r[4];
            ldsm4(r, wc + (wn + j * 8 + (lane & 7) + (lane >> 4) * 8) * kBwdLd + s * 16 + ((lane >> 3) & 1) * 8);
            b[j][0] = r[0]; b[j][1] = r[1]; b[j + 1][0] = r[2]; b[j + 1][1] = r[3];
          }
          mma_all(a, b);
        }
      }
      __syncthreads();  // every warp has read its rows of act
    }
#pragma unroll
    for (int j = 0; j < kNT; j++) {
      const int col = wn + j * 8 + 2 * tq;
#pragma unroll
      for (int i = 0; i < 2; i++)
#pragma unroll
        for (int h = 0; h < 2; h++) {
          const int r = wm + i * 16 + gq + 8 * h;
          __nv_bfloat162 v;
          v.x = v.y = zero;
          if (m0 + r < B) {
            const int64_t o = (int64_t)(m0 + r) * kW + col;
            // this thread stored these two pre-activations on the way forward
            const float2 z = *reinterpret_cast<const float2*>(n.z[l + 1] + o);
            v.x = __float2bfloat16(acc[i][j][2 * h] * gelu_grad(z.x));
            v.y = __float2bfloat16(acc[i][j][2 * h + 1] * gelu_grad(z.y));
            *reinterpret_cast<__nv_bfloat162*>(n.g[l] + o) = v;
          }
          *reinterpret_cast<__nv_bfloat162*>(act + r * kActLd + col) = v;
        }
    }
    __syncthreads();
  }
  cp_wait<0>();
}

// Adam (Kingma & Ba 2015) on an fp32 master parameter; refreshes the bf16 copy.
struct Adam {
  float *p, *m, *v;
  bf16* p16;
  float lr, b1, b2, eps, c1, c2;
};
__device__ __forceinline__ void adam_update(const Adam& a, int64_t i, float gi) {
  const float mi = a.b1 * a.m[i] + (1.0f - a.b1) * gi;
  const float vi = a.b2 * a.v[i] + (1.0f - a.b2) * gi * gi;
  a.m[i] = mi;
  a.v[i] = vi;
  const float upd = a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
  const float np_ = a.p[i] - upd;
  a.p[i] = np_;
  a.p16[i] = __float2bfloat16(np_);
}

// Weight gradients dW = A^T G of every layer: a CTA per 32 x 32 outputs, over
// all B rows in chunks of 64 (a ring of cp.async buffers); four warps of 16 x 16
// outputs each.  A fifth warp of the CTAs of a layer's first 32 inputs sums
// the columns of G, row after row, for the bias gradient.
constexpr int kDwRows = 64, kDwLd = 32 + 8, kDwStages = 6;
struct DwLayer {
  const bf16* a;   // [B][lda]
  const bf16* g;   // [B][ldg]
  int lda, ldg;    // row strides, multiples of 8, zero padded
  int din, dout;
  int first;       // first CTA of the layer
  int64_t woff, boff;
};
struct DwNet {
  int nl;
  DwLayer l[kMaxLayers];
  float* grad;     // NULL: not wanted
};

template <bool STEP>
__global__ void __launch_bounds__(160) dw_kernel(DwNet n, Adam ad, int B) {
  extern __shared__ __align__(16) unsigned char sm[];
  constexpr int kBuf = kDwRows * kDwLd;  // elements of one operand's chunk
  int li = 0;
  while (li + 1 < n.nl && (int)blockIdx.x >= n.l[li + 1].first) li++;
  const DwLayer& L = n.l[li];
  const int nt = (L.dout + 31) / 32, idx = (int)blockIdx.x - L.first;
  const int m0 = (idx / nt) * 32, n0 = (idx % nt) * 32;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int chunks = (B + kDwRows - 1) / kDwRows;
  auto fetch = [&](int c) {
    if (c < chunks) {
      bf16* as = reinterpret_cast<bf16*>(sm) + (size_t)(c % kDwStages) * 2 * kBuf;
      bf16* gs = as + kBuf;
      for (int i = tid; i < 2 * kDwRows * 4; i += 160) {  // 64 rows x 4 pieces of 16 bytes, both operands
        const int r = (i >> 2) & (kDwRows - 1), s = (i & 3) * 8, row = c * kDwRows + r;
        if (i < kDwRows * 4) {
          const bool in = row < B && m0 + s < L.lda;
          cp_async16(as + r * kDwLd + s, in ? L.a + (int64_t)row * L.lda + m0 + s : L.a, in);
        } else {
          const bool in = row < B && n0 + s < L.ldg;
          cp_async16(gs + r * kDwLd + s, in ? L.g + (int64_t)row * L.ldg + n0 + s : L.g, in);
        }
      }
    }
    cp_commit();
  };
  for (int c = 0; c < kDwStages - 1; c++) fetch(c);
  float acc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
  float bsum = 0.0f;
  const int wm = (warp >> 1) * 16, wn = (warp & 1) * 16;
  for (int c = 0; c < chunks; c++) {
    cp_wait<kDwStages - 2>();
    __syncthreads();
    fetch(c + kDwStages - 1);
    const bf16* as = reinterpret_cast<const bf16*>(sm) + (size_t)(c % kDwStages) * 2 * kBuf;
    const bf16* gs = as + kBuf;
    if (warp < 4) {
      const int steps = (min(kDwRows, B - c * kDwRows) + 15) >> 4;
#pragma unroll 4
      for (int s = 0; s < steps; s++) {
        uint32_t a[4], b[4];
        // A(m, k) = as[k][m]: transposed 8 x 8 blocks in the order of the fragment (m low, m high; then k high)
        ldsm4t(a, as + (s * 16 + (lane & 7) + (lane >> 4) * 8) * kDwLd + wm + ((lane >> 3) & 1) * 8);
        ldsm4t(b, gs + (s * 16 + (lane & 15)) * kDwLd + wn + (lane >> 4) * 8);
        const uint32_t b0[2] = {b[0], b[1]}, b1[2] = {b[2], b[3]};
        mma_bf16(acc[0], a, b0);
        mma_bf16(acc[1], a, b1);
      }
    } else if (m0 == 0) {
      const int rows = min(kDwRows, B - c * kDwRows);
#pragma unroll 16
      for (int r = 0; r < rows; r++) bsum += __bfloat162float(gs[r * kDwLd + lane]);
    }
  }
  cp_wait<0>();
  auto emit = [&](int64_t o, float v) {
    if (n.grad) n.grad[o] = v;
    if (STEP) adam_update(ad, o, v);
  };
  if (warp < 4) {
#pragma unroll
    for (int j = 0; j < 2; j++)
#pragma unroll
      for (int q = 0; q < 4; q++) {
        const int m = m0 + wm + (lane >> 2) + (q >= 2 ? 8 : 0), k = n0 + wn + j * 8 + 2 * (lane & 3) + (q & 1);
        if (m < L.din && k < L.dout) emit(L.woff + (int64_t)m * L.dout + k, acc[j][q]);
      }
  } else if (m0 == 0 && n0 + lane < L.dout) {
    emit(L.boff + n0 + lane, bsum);
  }
}

__global__ void adam_kernel(Adam a, const float* gr, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x)
    adam_update(a, i, gr[i]);
}

// The loss: the CTAs' partial sums added in double, in a fixed order, into host memory.
__global__ void __launch_bounds__(256) loss_kernel(const float* part, int n, double* out) {
  __shared__ double sh[256];
  double s = 0.0;
  for (int i = threadIdx.x; i < n; i += 256) s += (double)part[i];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) *out = sh[0];
}

template <bool TA, bool TB, int EPI>
cudaError_t gemm(const bf16* a, int lda, const bf16* b, int ldb, int M, int N, int K, const Epi& ep, cudaStream_t st) {
  dim3 grid((N + kT - 1) / kT, (M + kT - 1) / kT);
  gemm_kernel<TA, TB, EPI><<<grid, 128, 0, st>>>(a, lda, b, ldb, M, N, K, ep);
  return cudaGetLastError();
}

}  // namespace

struct dtb_mlp {
  int n_in, width, depth, n_out;
  int64_t max_batch;
  int nl;                         // layers = depth + 1
  std::vector<int> din, dout;     // per layer
  std::vector<int64_t> woff, boff;  // offsets in the flat parameter vector
  int64_t n_params = 0;
  float* p = nullptr;             // fp32 master parameters (flat)
  bf16* p16 = nullptr;            // bf16 copy of the weights (same offsets)
  float* m = nullptr;             // Adam moments
  float* v = nullptr;
  float* grad = nullptr;          // fp32 gradients (flat)
  bool fused = false;             // 256 wide: chain_kernel and dw_kernel
  int xs = 0, ys = 0;             // row strides of x16 and dy
  int sms = 1;
  bf16* x16 = nullptr;            // [B][xs]
  std::vector<bf16*> g;           // fused: g[l], gradient at the output of hidden layer l
  std::vector<bf16*> act;         // act[l]: input of layer l (bf16), l = 1..depth
  std::vector<float*> z;          // z[l]: pre-activation of hidden layer l
  float* y = nullptr;             // [B][n_out]
  bf16* g0 = nullptr;             // gradient ping-pong buffers [B][width]
  bf16* g1 = nullptr;
  bf16* dy = nullptr;             // [B][ys]
  float* part = nullptr;          // loss partial sums
  double* loss = nullptr;         // their sum, pinned host memory
  int adam_t = 0;
  std::vector<void*> mem;
  void* alloc(size_t bytes) {
    void* q = nullptr;
    if (cudaMalloc(&q, bytes ? bytes : 16) != cudaSuccess) {
      cudaGetLastError();
      return nullptr;
    }
    mem.push_back(q);
    return q;
  }
  void free_all() {
    for (void* q : mem) cudaFree(q);
    mem.clear();
  }
  ~dtb_mlp() {
    free_all();
    if (loss) cudaFreeHost(loss);
  }
};

namespace {

dtb_status cuda_err(cudaError_t e, const char* where) {
  return dtb::set_last_error(DTB_ECUDA, std::string(where) + ": " + cudaGetErrorString(e));
}

// Forward pass over B rows of x16 -> y (fp32), keeping z and activations.
cudaError_t forward(dtb_mlp* n, int64_t B, cudaStream_t st) {
  const bf16* in = n->x16;
  for (int l = 0; l < n->nl; l++) {
    Epi ep{};
    ep.bias = n->p + n->boff[l];
    const bf16* W = n->p16 + n->woff[l];
    cudaError_t e;
    if (l < n->nl - 1) {
      ep.z = n->z[l + 1];
      ep.a = n->act[l + 1];
      e = gemm<false, false, EPI_GELU>(in, n->din[l], W, n->dout[l], (int)B, n->dout[l], n->din[l], ep, st);
      in = n->act[l + 1];
    } else {
      ep.y = n->y;
      e = gemm<false, false, EPI_BIAS>(in, n->din[l], W, n->dout[l], (int)B, n->dout[l], n->din[l], ep, st);
    }
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

cudaError_t stage_input(dtb_mlp* n, const float* d_x, int64_t B, cudaStream_t st) {
  to_bf16_kernel<<<256, 256, 0, st>>>(d_x, n->x16, B * n->n_in);
  return cudaGetLastError();
}

// Loss gradient and backward pass: fills n->grad; partial sums of the loss in n->part.
cudaError_t backward(dtb_mlp* n, const float* d_t, int64_t B, cudaStream_t st, int* nparts) {
  const int64_t ny = B * n->n_out;
  const int parts = 256;
  mse_grad_kernel<<<parts, 256, 0, st>>>(n->y, d_t, n->dy, ny, 1.0f / (float)ny, n->part);
  *nparts = parts;
  const bf16* G = n->dy;
  bf16* bufs[2] = {n->g0, n->g1};
  int pb = 0;
  for (int l = n->nl - 1; l >= 0; l--) {
    const bf16* A = l == 0 ? n->x16 : n->act[l];
    Epi ew{};
    ew.y = n->grad + n->woff[l];
    // dW[l] = A^T G : [din][B] x [B][dout]
    cudaError_t e = gemm<true, false, EPI_F32>(A, n->din[l], G, n->dout[l], n->din[l], n->dout[l], (int)B, ew, st);
    if (e != cudaSuccess) return e;
    colsum_kernel<<<(n->dout[l] + 127) / 128, 128, 0, st>>>(G, (int)B, n->dout[l], n->grad + n->boff[l]);
    if (l > 0) {
      // G[l-1] = (G W^T) * gelu'(z[l])
      Epi ed{};
      ed.a = bufs[pb];
      ed.zin = n->z[l];
      e = gemm<false, true, EPI_DGELU>(G, n->dout[l], n->p16 + n->woff[l], n->dout[l], (int)B, n->din[l],
                                        n->dout[l], ed, st);
      if (e != cudaSuccess) return e;
      G = bufs[pb];
      pb ^= 1;
    }
  }
  return cudaGetLastError();
}

// ---- the 256-wide path ----
// Rows per CTA: 32 while one wave of them covers the batch (more CTAs at
// work), else 64 (half the passes over the weights).
int chain_rows(const dtb_mlp* n, int64_t B) { return (B + 31) / 32 <= n->sms ? 32 : 64; }

template <int R, bool TRAIN>
cudaError_t launch_chain(dtb_mlp* n, const float* x, const float* t, float* y, int64_t B, cudaStream_t st) {
  ChainNet c{};
  c.n_in = n->n_in; c.n_out = n->n_out; c.nl = n->nl; c.xs = n->xs; c.ys = n->ys;
  for (int l = 0; l < n->nl; l++) {
    c.w[l] = n->p16 + n->woff[l];
    c.b[l] = n->p + n->boff[l];
    c.act[l] = n->act[l];
    c.z[l] = n->z[l];
    c.g[l] = l < n->nl - 1 ? n->g[l] : nullptr;
  }
  c.x16 = n->x16; c.dy = n->dy; c.part = n->part;
  const float scale = 1.0f / (float)(B * n->n_out);
  chain_kernel<R, TRAIN><<<(unsigned)((B + R - 1) / R), 256, ChainSmem<R>::kBytes, st>>>(c, x, t, y, (int)B, scale);
  return cudaGetLastError();
}

cudaError_t fused_predict(dtb_mlp* n, const float* x, float* y, int64_t B, cudaStream_t st) {
  return chain_rows(n, B) == 32 ? launch_chain<32, false>(n, x, nullptr, y, B, st)
                                : launch_chain<64, false>(n, x, nullptr, y, B, st);
}

// Gradients of the batch: into n->grad (grads), or straight into an Adam step.
cudaError_t fused_gradients(dtb_mlp* n, const float* x, const float* t, int64_t B, const Adam* step, int* nparts,
                            cudaStream_t st) {
  const int R = chain_rows(n, B);
  cudaError_t e = R == 32 ? launch_chain<32, true>(n, x, t, nullptr, B, st) : launch_chain<64, true>(n, x, t, nullptr, B, st);
  if (e != cudaSuccess) return e;
  *nparts = (int)((B + R - 1) / R);
  DwNet d{};
  d.nl = n->nl;
  d.grad = step ? nullptr : n->grad;
  int ctas = 0;
  for (int l = 0; l < n->nl; l++) {
    DwLayer& L = d.l[l];
    L.a = l == 0 ? n->x16 : n->act[l];
    L.lda = l == 0 ? n->xs : kW;
    L.g = l == n->nl - 1 ? n->dy : n->g[l];
    L.ldg = l == n->nl - 1 ? n->ys : kW;
    L.din = n->din[l]; L.dout = n->dout[l];
    L.woff = n->woff[l]; L.boff = n->boff[l];
    L.first = ctas;
    ctas += ((L.din + 31) / 32) * ((L.dout + 31) / 32);
  }
  constexpr size_t smem = (size_t)kDwStages * 2 * kDwRows * kDwLd * 2;
  if (step) dw_kernel<true><<<ctas, 160, smem, st>>>(d, *step, (int)B);
  else dw_kernel<false><<<ctas, 160, smem, st>>>(d, Adam{}, (int)B);
  return cudaGetLastError();
}

// Dynamic shared-memory limits of the current device's kernels.
cudaError_t fused_setup() {
  cudaError_t e = cudaSuccess;
  auto set = [&](const void* f, size_t b) {
    if (e == cudaSuccess) e = cudaFuncSetAttribute(f, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)b);
  };
  set((const void*)chain_kernel<32, false>, ChainSmem<32>::kBytes);
  set((const void*)chain_kernel<64, false>, ChainSmem<64>::kBytes);
  set((const void*)chain_kernel<32, true>, ChainSmem<32>::kBytes);
  set((const void*)chain_kernel<64, true>, ChainSmem<64>::kBytes);
  constexpr size_t dw = (size_t)kDwStages * 2 * kDwRows * kDwLd * 2;
  set((const void*)dw_kernel<false>, dw);
  set((const void*)dw_kernel<true>, dw);
  return e;
}

// Loss and gradients of a batch queued on st (n->grad, or an Adam step when
// step is given); the loss sum lands in *n->loss when want_loss.
cudaError_t enqueue_gradients(dtb_mlp* n, const float* x, const float* t, int64_t B, const Adam* step, bool want_loss,
                              cudaStream_t st) {
  int parts = 0;
  cudaError_t e;
  if (n->fused) {
    e = fused_gradients(n, x, t, B, step, &parts, st);
  } else {
    e = stage_input(n, x, B, st);
    if (e == cudaSuccess) e = forward(n, B, st);
    if (e == cudaSuccess) e = backward(n, t, B, st, &parts);
    if (e == cudaSuccess && step) {
      adam_kernel<<<512, 256, 0, st>>>(*step, n->grad, n->n_params);
      e = cudaGetLastError();
    }
  }
  if (e == cudaSuccess && want_loss) {
    loss_kernel<<<1, 256, 0, st>>>(n->part, parts, n->loss);
    e = cudaGetLastError();
  }
  return e;
}

}  // namespace

extern "C" {

dtb_status dtb_mlp_create(int32_t n_in, int32_t width, int32_t depth, int32_t n_out, int64_t max_batch,
                          const float* params, dtb_mlp** out) {
  if (!out || !params) return dtb::set_last_error(DTB_EINVAL, "dtb_mlp_create: NULL argument");
  *out = nullptr;
  if (n_in < 1 || width < 1 || depth < 1 || n_out < 1 || max_batch < 1 || max_batch > (1 << 26))
    return dtb::set_last_error(DTB_EINVAL, "dtb_mlp_create: bad sizes");
  dtb_mlp* n = new dtb_mlp();
  n->n_in = n_in; n->width = width; n->depth = depth; n->n_out = n_out; n->max_batch = max_batch;
  n->nl = depth + 1;
  for (int l = 0; l < n->nl; l++) {
    n->din.push_back(l == 0 ? n_in : width);
    n->dout.push_back(l == n->nl - 1 ? n_out : width);
    n->woff.push_back(n->n_params);
    n->n_params += (int64_t)n->din[l] * n->dout[l];
    n->boff.push_back(n->n_params);
    n->n_params += n->dout[l];
  }
  const size_t P = (size_t)n->n_params;
  int dev = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&n->sms, cudaDevAttrMultiProcessorCount, dev);
  auto allocate = [&](bool fused) {
    bool ok = true;
    auto A = [&](size_t bytes) { void* q = n->alloc(bytes); if (!q) ok = false; return q; };
    n->fused = fused;
    n->xs = fused ? (n_in + 7) / 8 * 8 : n_in;
    n->ys = fused ? (n_out + 7) / 8 * 8 : n_out;
    n->p = (float*)A(4 * P);
    n->p16 = (bf16*)A(2 * P);
    n->m = (float*)A(4 * P);
    n->v = (float*)A(4 * P);
    n->grad = (float*)A(4 * P);
    n->x16 = (bf16*)A(2 * (size_t)max_batch * n->xs);
    n->act.assign(n->nl, nullptr);
    n->z.assign(n->nl, nullptr);
    for (int l = 1; l < n->nl; l++) {
      n->act[l] = (bf16*)A(2 * (size_t)max_batch * width);
      n->z[l] = (float*)A(4 * (size_t)max_batch * width);
    }
    n->y = (float*)A(4 * (size_t)max_batch * n_out);
    n->g.clear();
    if (fused) {
      for (int l = 0; l < n->nl - 1; l++) n->g.push_back((bf16*)A(2 * (size_t)max_batch * width));
    } else {
      n->g0 = (bf16*)A(2 * (size_t)max_batch * width);
      n->g1 = (bf16*)A(2 * (size_t)max_batch * width);
    }
    n->dy = (bf16*)A(2 * (size_t)max_batch * n->ys);
    n->part = (float*)A(4 * (size_t)std::max<int64_t>(256, fused ? max_batch / 32 + 1 : 0));
    return ok;
  };
  // The 256-wide path keeps the gradient of every hidden layer, the general one
  // of two: a batch size for which the former does not fit takes the latter,
  // with the same results.
  bool ok = width == kW && n_in <= kW && n_out <= kMaxOut && n->nl <= kMaxLayers && allocate(true);
  if (!ok) {
    n->free_all();
    ok = allocate(false);
  }
  if (cudaHostAlloc((void**)&n->loss, sizeof(double), cudaHostAllocDefault) != cudaSuccess) {
    cudaGetLastError();
    n->loss = nullptr;
    ok = false;
  }
  if (!ok) {
    delete n;
    return dtb::set_last_error(DTB_ENOMEM, "dtb_mlp_create: device allocation failed");
  }
  cudaError_t e = n->fused ? fused_setup() : cudaSuccess;
  if (e == cudaSuccess) e = cudaMemcpy(n->p, params, 4 * P, cudaMemcpyHostToDevice);
  if (e == cudaSuccess) e = cudaMemset(n->m, 0, 4 * P);
  if (e == cudaSuccess) e = cudaMemset(n->v, 0, 4 * P);
  if (e == cudaSuccess) {
    to_bf16_kernel<<<256, 256>>>(n->p, n->p16, (int64_t)P);
    e = cudaDeviceSynchronize();
  }
  if (e != cudaSuccess) {
    delete n;
    return cuda_err(e, "dtb_mlp_create");
  }
  *out = n;
  return DTB_OK;
}

dtb_status dtb_mlp_destroy(dtb_mlp* n) {
  if (!n) return dtb::set_last_error(DTB_EINVAL, "dtb_mlp_destroy: NULL");
  delete n;
  return DTB_OK;
}

dtb_status dtb_mlp_forward(dtb_mlp* n, const float* d_x, float* d_y, int64_t B, void* stream) {
  if (!n || !d_x || !d_y || B < 1 || B > n->max_batch) return dtb::set_last_error(DTB_EINVAL, "dtb_mlp_forward: NULL argument or batch outside 1..max_batch");
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e;
  if (n->fused) {
    // an output over its own input goes through a buffer: rows that a CTA has
    // still to read may lie where another one writes
    const bool over = (uintptr_t)d_y < (uintptr_t)(d_x + B * n->n_in) && (uintptr_t)d_x < (uintptr_t)(d_y + B * n->n_out);
    e = fused_predict(n, d_x, over ? n->y : d_y, B, st);
    if (e == cudaSuccess && over)
      e = cudaMemcpyAsync(d_y, n->y, 4 * (size_t)B * n->n_out, cudaMemcpyDeviceToDevice, st);
  } else {
    e = stage_input(n, d_x, B, st);
    if (e == cudaSuccess) e = forward(n, B, st);
    if (e == cudaSuccess) e = cudaMemcpyAsync(d_y, n->y, 4 * (size_t)B * n->n_out, cudaMemcpyDeviceToDevice, st);
  }
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  return e == cudaSuccess ? DTB_OK : cuda_err(e, "dtb_mlp_forward");
}

dtb_status dtb_mlp_gradients(dtb_mlp* n, const float* d_x, const float* d_t, int64_t B, float* grads, float* loss,
                             void* stream) {
  if (!n || !d_x || !d_t || B < 1 || B > n->max_batch) return dtb::set_last_error(DTB_EINVAL, "dtb_mlp_gradients: NULL argument or batch outside 1..max_batch");
  cudaStream_t st = (cudaStream_t)stream;
  cudaError_t e = enqueue_gradients(n, d_x, d_t, B, nullptr, loss != nullptr, st);
  if (e == cudaSuccess && grads) e = cudaMemcpyAsync(grads, n->grad, 4 * (size_t)n->n_params, cudaMemcpyDeviceToHost, st);
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_err(e, "dtb_mlp_gradients");
  if (loss) *loss = (float)(*n->loss / ((double)B * n->n_out));
  return DTB_OK;
}

dtb_status dtb_mlp_train_step(dtb_mlp* n, const float* d_x, const float* d_t, int64_t B, float lr, float* loss,
                              void* stream) {
  if (!n || !d_x || !d_t || B < 1 || B > n->max_batch) return dtb::set_last_error(DTB_EINVAL, "dtb_mlp_gradients: NULL argument or batch outside 1..max_batch");
  cudaStream_t st = (cudaStream_t)stream;
  const float b1 = 0.9f, b2 = 0.999f;
  const float at = (float)(n->adam_t + 1);
  const Adam ad{n->p, n->m, n->v, n->p16, lr, b1, b2, 1e-8f, 1.0f - powf(b1, at), 1.0f - powf(b2, at)};
  cudaError_t e = enqueue_gradients(n, d_x, d_t, B, &ad, loss != nullptr, st);
  if (e == cudaSuccess) n->adam_t++;
  if (e == cudaSuccess) e = cudaStreamSynchronize(st);
  if (e != cudaSuccess) return cuda_err(e, "dtb_mlp_train_step");
  if (loss) *loss = (float)(*n->loss / ((double)B * n->n_out));
  return DTB_OK;
}

dtb_status dtb_mlp_get_params(dtb_mlp* n, float* params) {
  if (!n || !params) return dtb::set_last_error(DTB_EINVAL, "dtb_mlp_get_params");
  cudaError_t e = cudaMemcpy(params, n->p, 4 * (size_t)n->n_params, cudaMemcpyDeviceToHost);
  return e == cudaSuccess ? DTB_OK : cuda_err(e, "dtb_mlp_get_params");
}

}  // extern "C"
