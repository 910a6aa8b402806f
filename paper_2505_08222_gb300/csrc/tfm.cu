// Transformer actor and critic in FP32 for the TransfMAPPO update (Sec. II-B,
// Sec. III-B.1, Fig. 3): the forward pass with stored activations, the PPO
// clipped-surrogate and value losses, the backward pass, Adam, and
// generalized advantage estimation.
//
// Layout: sample s of a call occupies token rows s*T .. s*T+T-1 (T = 1 +
// n_slots, row 0 its recurrent embedding); every activation is row-major
// [rows][width].  Rows past a sample's entity count are computed (from the
// embedding bias alone) but no row attends to them, so they receive exactly
// zero gradient and add nothing to the weight gradients.  The head reads the
// recurrent token alone, so of the last block only the keys and values are
// made for every token; its queries, attention output, feed-forward sub-block
// and their backward run on the n recurrent rows, stored densely ([n][width]).
//
// The dense contractions run on the tensor cores (tfm_tc.cuh; at d = 64 most of a
// block in four fused kernels, tfm_qkv.cuh and tfm_ffn.cuh) or, on the path chosen
// by tfm_set_gemm_path(0), on the CUDA cores in FP32 (the register-tiled GEMMs
// below).  The weight gradients are split along the token rows into partial slabs
// summed in a fixed order, so every result is deterministic.
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#include <cmath>
#include <cstring>
#include <initializer_list>
#include <string>
#include <vector>

#include "../../include/utrack.h"
#include "common.cuh"
#include "f32x2.cuh"
#include "tc.cuh"
#include "tfm.cuh"
#include "warp_sums.cuh"

namespace ut {
namespace tfm {

constexpr int kMaxT = 1 + UT_MAX_AGENTS + UT_MAX_TARGETS;  // tokens per sample
constexpr int kRowBlocks = 304;                             // blocks of the head / embedding-gradient kernels
constexpr int kLnBlocks = 1216;                             // blocks of the LayerNorm kernels
constexpr int kRowWarps = kRowBlocks * 8;                   // warps writing partial sums
constexpr int kTcSplitsMax = 3 * 152;                       // row splits of a tensor-core weight gradient (at most)

enum { EPI_STORE = 0, EPI_BIAS = 1, EPI_BIAS_RES = 2, EPI_BIAS_GELU = 3, EPI_GELU_GRAD = 4, EPI_PARTIAL = 5 };

// C = op(A) op(B) with an epilogue.  A(m, k) is A[m * lda + k] when AK (k
// contiguous), else A[k * lda + m]; B(k, n) is B[n * ldb + k] when BK, else
// B[k * ldb + n].  blockIdx.z takes K range [z * kchunk, (z + 1) * kchunk).
struct Gemm {
  const float* A;
  long long lda;
  const float* B;
  long long ldb;
  float* C;
  long long ldc;
  long long M, K, kchunk;
  int N, epi;
  const float* bias;   // [N] (EPI_BIAS*)
  const float* R;      // residual added (EPI_BIAS_RES), ld = ldr
  long long ldr;
  float* C2;           // GELU of the output (EPI_BIAS_GELU), ld = ldc
  const float* aux;    // pre-activation whose GELU derivative scales the output (EPI_GELU_GRAD), ld = ldc
  const uint16_t* bimg;  // BF16 image of B for the tensor-core path (kinds 0, 1), or NULL: CUDA cores
  int* status;           // device status word (a tensor-core wait that gave up)
};

__device__ __forceinline__ float gelu_f(float z) { return 0.5f * z * (1.0f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad_f(float z) {
  return 0.5f * (1.0f + erff(z * 0.70710678118654752f)) + z * expf(-0.5f * z * z) * 0.39894228040143268f;
}

// The epilogues of the GEMM kernels for output (m, n) with accumulator v.
__device__ __forceinline__ void epi_store(const Gemm& g, long long m, int n, float v) {
  const long long o = m * g.ldc + n;
  switch (g.epi) {
    case EPI_BIAS:
      g.C[o] = v + g.bias[n];
      break;
    case EPI_BIAS_RES:
      g.C[o] = v + g.bias[n] + g.R[m * g.ldr + n];
      break;
    case EPI_BIAS_GELU:
      v += g.bias[n];
      g.C[o] = v;
      g.C2[o] = gelu_f(v);
      break;
    case EPI_GELU_GRAD:
      g.C[o] = v * gelu_grad_f(g.aux[o]);
      break;
    case EPI_PARTIAL:
      g.C[((long long)blockIdx.z * g.M + m) * g.N + n] = v;
      break;
    default:
      g.C[o] = v;
  }
}

__device__ __forceinline__ float warp_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// 64 x 64 output tile per CTA of 256 threads, 4 x 4 outputs per thread,
// K staged 16 at a time through shared memory.
template <bool AK, bool BK>
__global__ void __launch_bounds__(256) sgemm_kernel(Gemm g) {
  __shared__ __align__(16) float As[16][68];
  __shared__ __align__(16) float Bs[16][68];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const long long m0 = (long long)blockIdx.x * 64;
  const int n0 = blockIdx.y * 64;
  const long long kb = (long long)blockIdx.z * g.kchunk;
  const long long ke = kb + g.kchunk < g.K ? kb + g.kchunk : g.K;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
  for (long long k0 = kb; k0 < ke; k0 += 16) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = tid + r * 256;
      const int mm = AK ? (i >> 4) : (i & 63), kk = AK ? (i & 15) : (i >> 6);
      const long long m = m0 + mm, k = k0 + kk;
      float v = 0.0f;
      if (m < g.M && k < ke) v = AK ? g.A[m * g.lda + k] : g.A[k * g.lda + m];
      As[kk][mm] = v;
    }
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = tid + r * 256;
      const int nn = BK ? (i >> 4) : (i & 63), kk = BK ? (i & 15) : (i >> 6);
      const long long k = k0 + kk;
      const int n = n0 + nn;
      float v = 0.0f;
      if (n < g.N && k < ke) v = BK ? g.B[(long long)n * g.ldb + k] : g.B[k * g.ldb + n];
      Bs[kk][nn] = v;
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < 16; ++kk) {
      const float4 a = *reinterpret_cast<const float4*>(&As[kk][ty * 4]);
      const float4 b = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
      const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const long long m = m0 + ty * 4 + i;
    if (m >= g.M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx * 4 + j;
      if (n >= g.N) continue;
      epi_store(g, m, n, acc[i][j]);
    }
  }
}

// The same product with a 128 x 64 tile, 8 x 4 outputs per thread, float4
// global loads, K staged 32 at a time, the next K slice prefetched into
// registers while the current one is multiplied.  Preconditions (checked on
// the host): the contiguous dimension of each operand is read in aligned
// float4 (leading dimensions and base addresses multiples of 4 floats; M, N
// multiples of 4 where they are contiguous), and with k-contiguous operands
// the K range is a multiple of 32.  by: the column tile.
template <bool AK, bool BK>
__device__ __forceinline__ void sgemm128_tile(const Gemm& g, int by) {
  __shared__ __align__(16) float As[32][132];
  __shared__ __align__(16) float Bs[32][68];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const long long m0 = (long long)blockIdx.x * 128;
  const int n0 = by * 64;
  const long long kb = (long long)blockIdx.z * g.kchunk;
  const long long ke = kb + g.kchunk < g.K ? kb + g.kchunk : g.K;
  float4 ra[4], rb[2];
  // A slice: 128 (m) x 32 (k) as 1024 float4, four per thread; B slice: 32 (k) x
  // 64 (n) as 512, two per thread.  Every load is made: past M or N from the last
  // row or column (what it feeds is not stored), past the range of k from its
  // last row, zeroed when it is staged.  (Behind bounds conditions each load of a
  // partial tile waited for the one before: a forward of 64 samples of 4 tokens at
  // d = 128, 2 blocks, 262 us, without them 221; with the addresses made once and
  // the last block's pair below 215.)
  const float *pa[4], *pb[2];
#pragma unroll
  for (int r = 0; r < 4; ++r) {
    const int i = tid + r * 256;
    pa[r] = g.A + (AK ? min(m0 + (i >> 3), g.M - 1) * g.lda + (i & 7) * 4 : min(m0 + (i & 31) * 4, g.M - 4));
  }
#pragma unroll
  for (int r = 0; r < 2; ++r) {
    const int i = tid + r * 256;
    pb[r] = g.B + (BK ? (long long)min(n0 + (i >> 3), g.N - 1) * g.ldb + (i & 7) * 4
                      : (long long)min(n0 + (i & 15) * 4, g.N - 4));
  }
  auto load_a = [&](long long k0) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const long long k = k0 + ((tid + r * 256) >> 5);
      ra[r] = *reinterpret_cast<const float4*>(pa[r] + (AK ? k0 : min(k, ke - 1) * g.lda));
    }
  };
  auto load_b = [&](long long k0) {
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const long long k = k0 + ((tid + r * 256) >> 4);
      rb[r] = *reinterpret_cast<const float4*>(pb[r] + (BK ? k0 : min(k, ke - 1) * g.ldb));
    }
  };
  auto store = [&](long long k0) {
#pragma unroll
    for (int r = 0; r < 4; ++r) {
      const int i = tid + r * 256;
      if (AK) {
        const int mm = i >> 3, kk = (i & 7) * 4;
        As[kk][mm] = ra[r].x;
        As[kk + 1][mm] = ra[r].y;
        As[kk + 2][mm] = ra[r].z;
        As[kk + 3][mm] = ra[r].w;
      } else {
        *reinterpret_cast<float4*>(&As[i >> 5][(i & 31) * 4]) =
            k0 + (i >> 5) < ke ? ra[r] : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
#pragma unroll
    for (int r = 0; r < 2; ++r) {
      const int i = tid + r * 256;
      if (BK) {
        const int nn = i >> 3, kk = (i & 7) * 4;
        Bs[kk][nn] = rb[r].x;
        Bs[kk + 1][nn] = rb[r].y;
        Bs[kk + 2][nn] = rb[r].z;
        Bs[kk + 3][nn] = rb[r].w;
      } else {
        *reinterpret_cast<float4*>(&Bs[i >> 4][(i & 15) * 4]) =
            k0 + (i >> 4) < ke ? rb[r] : make_float4(0.f, 0.f, 0.f, 0.f);
      }
    }
  };
  float acc[8][4];
#pragma unroll
  for (int i = 0; i < 8; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
  if (kb < ke) {
    load_a(kb);
    load_b(kb);
    store(kb);
  }
  __syncthreads();
  for (long long k0 = kb; k0 < ke; k0 += 32) {
    const bool more = k0 + 32 < ke;
    if (more) {
      load_a(k0 + 32);
      load_b(k0 + 32);
    }
#pragma unroll
    for (int kk = 0; kk < 32; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[kk][ty * 8]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[kk][ty * 8 + 4]);
      const float4 b = *reinterpret_cast<const float4*>(&Bs[kk][tx * 4]);
      const float av[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
    }
    __syncthreads();  // every thread is done with the slice before it is overwritten
    if (more) {
      store(k0 + 32);
      __syncthreads();
    }
  }
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const long long m = m0 + ty * 8 + i;
    if (m >= g.M) continue;
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int n = n0 + tx * 4 + j;
      if (n >= g.N) continue;
      epi_store(g, m, n, acc[i][j]);
    }
  }
}

template <bool AK, bool BK>
__global__ void __launch_bounds__(256) sgemm128_kernel(Gemm g) {
  sgemm128_tile<AK, BK>(g, blockIdx.y);
}
// Two products in one launch, column tiles 0 .. ny - 1 of a and then b's; the
// grid covers the larger of their rows and splits.
template <bool AK, bool BK>
__global__ void __launch_bounds__(256) sgemm128_pair_kernel(Gemm a, Gemm b, int ny) {
  const bool second = (int)blockIdx.y >= ny;
  const Gemm g = second ? b : a;
  if ((long long)blockIdx.x * 128 >= g.M || (long long)blockIdx.z * g.kchunk >= g.K) return;
  sgemm128_tile<AK, BK>(g, (int)blockIdx.y - (second ? ny : 0));
}

// The entity tokens of one sample, 4 slots per register: lane i of v[j] holds
// feature i % 8 of slot 4 j + i / 8 (one coalesced load for 4 tokens), zero for
// slots past the sample's ne entities.  A feature then comes by one shuffle.
constexpr int kTokRegs = (UT_MAX_AGENTS + UT_MAX_TARGETS + 3) / 4;
template <typename TokT>
__device__ __forceinline__ void load_tokens(const TokT* __restrict__ tok, long long bs, int NS, int ne, int lane,
                                            float (&v)[kTokRegs]) {
#pragma unroll
  for (int j = 0; j < kTokRegs; ++j)
    v[j] = 4 * j + (lane >> 3) < ne ? (float)tok[(bs * NS + 4 * j) * 8 + lane] : 0.0f;
}

// Embedding of the entity tokens; token 0 of each sample is its recurrent
// embedding.  Warps loop over samples (lane: outputs lane + 32 i, its rows of W
// and its biases held in registers).  Bound by its writes; a warp per token row,
// with a 64-bit division and eight scalar loads per row, took 265 us for
// 163,840 samples of 11 tokens, this 92.
template <typename TokT, int DJ>
__global__ void __launch_bounds__(256) embed_kernel(const TokT* __restrict__ tok, const int32_t* __restrict__ n_ent,
                                                    const float* __restrict__ h, const int32_t* __restrict__ sel,
                                                    const float* __restrict__ W, const float* __restrict__ b,
                                                    float* __restrict__ X, long long n, int T, int NS) {
  constexpr int d = 32 * DJ;
  const int lane = threadIdx.x & 31;
  const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  float wr[DJ][8], br[DJ];
#pragma unroll
  for (int i = 0; i < DJ; ++i) {
    br[i] = b[lane + 32 * i];
#pragma unroll
    for (int k = 0; k < 8; ++k) wr[i][k] = W[(lane + 32 * i) * 8 + k];
  }
  for (long long s = w0; s < n; s += nw) {
    const long long bs = sel ? (long long)sel[s] : s;
    int ne = n_ent[bs];
    ne = ne < 0 ? 0 : (ne > NS ? NS : ne);
    float v[kTokRegs];
    load_tokens(tok, bs, NS, ne, lane, v);
    float* x = X + s * T * d + lane;
#pragma unroll
    for (int i = 0; i < DJ; ++i) x[32 * i] = h[bs * d + lane + 32 * i];
#pragma unroll
    for (int t = 0; t < 4 * kTokRegs; ++t) {
      if (t >= NS) break;  // (warp-uniform)
      float q[8];
#pragma unroll
      for (int k = 0; k < 8; ++k) q[k] = __shfl_sync(0xffffffffu, v[t / 4], 8 * (t & 3) + k);
#pragma unroll
      for (int i = 0; i < DJ; ++i) {
        float acc = br[i];
#pragma unroll
        for (int k = 0; k < 8; ++k) acc = fmaf(wr[i][k], q[k], acc);
        x[(t + 1) * d + 32 * i] = acc;
      }
    }
  }
}

// LayerNorm forward, one warp per row: Y = (X - mean) rstd g + b and the row's
// (mean, rstd).
template <int DJ>
__global__ void ln_fwd_kernel(const float* __restrict__ X, const float* __restrict__ gam,
                              const float* __restrict__ bet, float* __restrict__ Y, float* __restrict__ stat,
                              long long rows) {
  constexpr int d = 32 * DJ;
  const int lane = threadIdx.x & 31;
  const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  float gj[DJ], bj[DJ], xn[DJ];
#pragma unroll
  for (int i = 0; i < DJ; ++i) {
    gj[i] = gam[lane + 32 * i];
    bj[i] = bet[lane + 32 * i];
    xn[i] = w0 < rows ? X[w0 * d + lane + 32 * i] : 0.0f;
  }
  for (long long r = w0; r < rows; r += nw) {
    float x[DJ], s = 0.0f;
#pragma unroll
    for (int i = 0; i < DJ; ++i) {
      x[i] = xn[i];
      s += x[i];
    }
    if (r + nw < rows) {  // the warp's next row: in flight during this one
#pragma unroll
      for (int i = 0; i < DJ; ++i) xn[i] = X[(r + nw) * d + lane + 32 * i];
    }
    const float mean = warp_sum(s) * (1.0f / d);
    float v = 0.0f;
#pragma unroll
    for (int i = 0; i < DJ; ++i) v += (x[i] - mean) * (x[i] - mean);
    const float rstd = 1.0f / sqrtf(warp_sum(v) * (1.0f / d) + 1e-5f);
#pragma unroll
    for (int i = 0; i < DJ; ++i) Y[r * d + lane + 32 * i] = (x[i] - mean) * rstd * gj[i] + bj[i];
    if (lane == 0) {
      stat[2 * r] = mean;
      stat[2 * r + 1] = rstd;
    }
  }
}

// LayerNorm backward, one warp per row: out = base + dL/dX from dY (the
// gradient at the LayerNorm output), and per-block partial sums of dL/dg
// (sum dY xh) and dL/db (sum dY) into part[block][2d] (blocks of 256
// threads).  out may equal base.  REC (the last block's first LayerNorm):
// row s T takes its gradient from dY0 at s instead of dY; base holds the
// recurrent rows alone in the same way and is zero elsewhere.
template <int DJ, bool REC>
__global__ void ln_bwd_kernel(const float* __restrict__ dY, const float* __restrict__ X,
                              const float* __restrict__ stat, const float* __restrict__ gam, const float* base,
                              float* out, float* __restrict__ part, long long rows, const float* __restrict__ dY0,
                              unsigned T) {
  constexpr int d = 32 * DJ;
  const int lane = threadIdx.x & 31;
  const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  float pg[DJ], pb[DJ], gj[DJ];
  // the warp's next row (dY, X, base, statistics): in flight during the
  // current one
  float dyn[DJ], xn[DJ], bn[DJ], mn = 0.0f, rn = 0.0f;
  auto fetch = [&](long long r) {
    const long long s0 = REC ? (long long)((unsigned)r / T) : 0;  // (rows < 2^32: max_batch <= 2^22)
    const bool rec = REC && r == s0 * T;
#pragma unroll
    for (int i = 0; i < DJ; ++i) {
      const long long o = r * d + lane + 32 * i;
      dyn[i] = dY[o];
      xn[i] = X[o];
      if (REC) {
        const long long c = s0 * d + lane + 32 * i;
        bn[i] = rec ? base[c] : 0.0f;
        if (rec) dyn[i] = dY0[c];
      } else {
        bn[i] = base[o];
      }
    }
    mn = stat[2 * r];
    rn = stat[2 * r + 1];
  };
#pragma unroll
  for (int i = 0; i < DJ; ++i) {
    pg[i] = pb[i] = 0.0f;
    gj[i] = gam[lane + 32 * i];
  }
  if (w0 < rows) fetch(w0);
  for (long long r = w0; r < rows; r += nw) {
    const float mean = mn, rstd = rn;
    float xh[DJ], dxh[DJ], bs[DJ], m1 = 0.0f, m2 = 0.0f;
#pragma unroll
    for (int i = 0; i < DJ; ++i) {
      const float dy = dyn[i];
      xh[i] = (xn[i] - mean) * rstd;
      bs[i] = bn[i];
      dxh[i] = dy * gj[i];
      pg[i] = fmaf(dy, xh[i], pg[i]);
      pb[i] += dy;
      m1 += dxh[i];
      m2 = fmaf(dxh[i], xh[i], m2);
    }
    if (r + nw < rows) fetch(r + nw);
    m1 = warp_sum(m1) * (1.0f / d);
    m2 = warp_sum(m2) * (1.0f / d);
#pragma unroll
    for (int i = 0; i < DJ; ++i) out[r * d + lane + 32 * i] = bs[i] + rstd * (dxh[i] - m1 - xh[i] * m2);
  }
  // the block's 8 warps combined in warp order: one partial per block
  __shared__ float red[8][2 * d];
  const int wl = threadIdx.x >> 5;
#pragma unroll
  for (int i = 0; i < DJ; ++i) {
    red[wl][lane + 32 * i] = pg[i];
    red[wl][d + lane + 32 * i] = pb[i];
  }
  __syncthreads();
  for (int j = threadIdx.x; j < 2 * d; j += blockDim.x) {
    float t = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) t += red[k][j];
    part[(long long)blockIdx.x * 2 * d + j] = t;
  }
}

// FP32 attention (the CUDA-core path, and on the tensor-core path heads other
// than 16 wide or samples of 17 tokens).  A block of 128 threads takes
// 128 / T consecutive (sample, head) items q = s * H + head, a thread per query
// token (119 of 128 threads busy at T = 17; a warp per item kept 17 of 32
// lanes).  Rows are staged in shared memory by 16-byte loads; P goes through
// it too, so that a block's P, one contiguous range, is read and written whole.
// The products run on packed FP32 pairs: two keys of a score at once (staged
// interleaved), two columns of an output at once, so each sum keeps its order.
// Bound by the latency of its shared-memory loads (issue 28 to 36 % active):
// 131,072 items of 17 x 16 forward 254 us, backward 500 (534 and 809 with a warp per item; 274 and 524 with the rows
// staged one load after the other and 64-bit divisions).
constexpr int kAttnThreads = 128;
__host__ __device__ __forceinline__ int attn_items(int T) { return kAttnThreads / T; }
constexpr size_t kAttnSmemMax = 112 * 1024;  // above attn_bwd_smem for every T and head width
// Shared-memory floats: rows staged as they are, and key pairs (T rounded up
// to even per item).
__host__ __device__ __forceinline__ int attn_rows(int T) { return attn_items(T) * T; }
__host__ __device__ __forceinline__ int attn_pair_rows(int T) { return attn_items(T) * ((T + 1) / 2 * 2); }
inline size_t attn_fwd_smem(int T, int DH) {
  const int kv = attn_rows(T) * DH + attn_pair_rows(T) * DH, p = attn_rows(T) * T;
  return (size_t)(kv > p ? kv : p) * 4;
}
inline size_t attn_bwd_smem(int T, int DH) {
  return ((size_t)3 * attn_rows(T) * DH + (size_t)attn_pair_rows(T) * DH + 2 * (size_t)attn_rows(T) * T + 4) * 4;
}

// (sample, head) of item w: a 32-bit division wherever it is enough.
struct AttItem {
  long long s;
  int hh;
};
__device__ __forceinline__ AttItem att_item(long long w, int H) {
  if ((w >> 32) == 0) {
    const uint32_t s = (uint32_t)w / (uint32_t)H;
    return {(long long)s, (int)((uint32_t)w - s * (uint32_t)H)};
  }
  const long long s = w / H;
  return {s, (int)(w - s * H)};
}

// Column j of key u in the interleaved layout of an item's rows.
template <int DH>
__device__ __forceinline__ int pair_pos(int u, int j) {
  return (u >> 1) * 2 * DH + 2 * j + (u & 1);
}

template <int DH>
__device__ __forceinline__ void attn_put_pair(float* item, int u, int j, float4 v) {
  item[pair_pos<DH>(u, j)] = v.x;
  item[pair_pos<DH>(u, j + 1)] = v.y;
  item[pair_pos<DH>(u, j + 2)] = v.z;
  item[pair_pos<DH>(u, j + 3)] = v.w;
}

// Where the rows of a block's items lie: row r (item r / T from q0 on, token
// r % T).  The divisions of r < 128 by T are products (exact: the error is below
// 128 / 65536 < 1 / T), those by H 32-bit.
struct AttnRows {
  AttItem first;
  int H, T, inv;
  __device__ __forceinline__ AttnRows(long long q0, int h, int t)
      : first(att_item(q0, h)), H(h), T(t), inv(65536 / t + 1) {}
  __device__ __forceinline__ int item(int r) const { return (r * inv) >> 16; }
  __device__ __forceinline__ void sample(int it, long long& s, int& hh) const {
    const unsigned h = (unsigned)(first.hh + it), ds = h / (unsigned)H;
    s = first.s + ds;
    hh = (int)(h - ds * (unsigned)H);
  }
  // float offset of its head's columns in an array of `ld` floats a token
  __device__ __forceinline__ long long offset(int r, int ld, int dh) const {
    const int it = item(r);
    long long s;
    int hh;
    sample(it, s, hh);
    return (s * T + r - it * T) * ld + hh * dh;
  }
};

// acc[u] = sum_j x[j] K[u][j] over the keys u < T of an item (pairs), j in
// order; two pairs at a time, two independent chains.
template <int DH>
__device__ __forceinline__ void attn_dots(const float (&x)[DH], const float* pairs, int T, float (&acc)[kMaxT + 1]) {
#pragma unroll
  for (int u = 0; u < kMaxT; u += 4) {
    constexpr int kLast = kMaxT - 1;
    acc[u] = acc[u + 1] = 0.0f;
    if (u + 2 <= kLast) acc[u + 2] = acc[u + 3] = 0.0f;
    if (u < T) {
      const float4* a4 = reinterpret_cast<const float4*>(pairs + (u >> 1) * 2 * DH);
      const float4* b4 = u + 2 < T ? a4 + DH / 2 : a4;  // (past the item: its sums are not used)
      unsigned long long sa = 0ull, sb = 0ull;
#pragma unroll
      for (int j = 0; j < DH; j += 2) {
        const float4 a = a4[j / 2];  // (u, j), (u + 1, j), (u, j + 1), (u + 1, j + 1)
        sa = f2fma(f2pk(x[j], x[j]), f2pk(a.x, a.y), sa);
        sa = f2fma(f2pk(x[j + 1], x[j + 1]), f2pk(a.z, a.w), sa);
        if (u + 2 <= kLast) {
          const float4 b = b4[j / 2];
          sb = f2fma(f2pk(x[j], x[j]), f2pk(b.x, b.y), sb);
          sb = f2fma(f2pk(x[j + 1], x[j + 1]), f2pk(b.z, b.w), sb);
        }
      }
      f2upk(sa, acc[u], acc[u + 1]);
      if (u + 2 <= kLast) f2upk(sb, acc[u + 2], acc[u + 3]);
    }
  }
}

// o[j] += p row[j] on pairs of columns.
template <int DH>
__device__ __forceinline__ void attn_axpy(float p, const float* row, unsigned long long (&o)[DH / 2]) {
  const float4* r4 = reinterpret_cast<const float4*>(row);
  const unsigned long long pp = f2pk(p, p);
#pragma unroll
  for (int j = 0; j < DH / 4; ++j) {
    const float4 v = r4[j];
    o[2 * j] = f2fma(pp, f2pk(v.x, v.y), o[2 * j]);
    o[2 * j + 1] = f2fma(pp, f2pk(v.z, v.w), o[2 * j + 1]);
  }
}

template <int DH>
__device__ __forceinline__ void attn_store(float* dst, const unsigned long long (&o)[DH / 2]) {
#pragma unroll
  for (int j = 0; j < DH / 4; ++j) {
    float4 v;
    f2upk(o[2 * j], v.x, v.y);
    f2upk(o[2 * j + 1], v.z, v.w);
    reinterpret_cast<float4*>(dst)[j] = v;
  }
}

// P[s][head][t][u] (zero for masked keys u > n_ent) and O = P V.
template <int DH>
__global__ void __launch_bounds__(kAttnThreads) attn_fwd_kernel(const float* __restrict__ QKV,
                                                                const int32_t* __restrict__ n_ent,
                                                                const int32_t* __restrict__ sel, float* __restrict__ P,
                                                                float* __restrict__ O, long long n, int T, int NS,
                                                                int H, float scale) {
  extern __shared__ __align__(16) float sm_attn[];
  const int tid = threadIdx.x, ipb = attn_items(T), Tp = (T + 1) / 2 * 2;
  float* sV = sm_attn;                       // [items][T][DH]
  float* sK = sV + attn_rows(T) * DH;        // [items][Tp / 2][DH][2]
  const long long q0 = (long long)blockIdx.x * ipb, nq = n * H;
  const int items = (int)(nq - q0 < ipb ? nq - q0 : ipb);
  const int d = DH * H, ld = 3 * d, rows = items * T;
  const AttnRows at(q0, H, T);
  const int it = at.item(tid), t = tid - it * T;
  const bool on = it < items;
  long long s;
  int hh;
  at.sample(on ? it : 0, s, hh);
  int ne = __ldg(n_ent + (sel ? (long long)__ldg(sel + s) : s));
  ne = ne < 0 ? 0 : (ne > NS ? NS : ne);
  float qv[DH];
#pragma unroll
  for (int j = 0; j < DH; j += 4) {
    const float4 v = __ldg(reinterpret_cast<const float4*>(QKV + (s * T + (on ? t : 0)) * ld + hh * DH + j));
    qv[j] = v.x; qv[j + 1] = v.y; qv[j + 2] = v.z; qv[j + 3] = v.w;
  }
  constexpr int C = DH / 4, KB = C < 4 ? C : 4;
#pragma unroll
  for (int k0 = 0; k0 < C; k0 += KB) {
    float4 kk[KB], vv[KB];
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      const int i = tid + kAttnThreads * (k0 + k);
      const float* src = QKV + d + at.offset(min(i / C, rows - 1), ld, DH) + 4 * (i % C);
      kk[k] = __ldg(reinterpret_cast<const float4*>(src));
      vv[k] = __ldg(reinterpret_cast<const float4*>(src + d));
    }
#pragma unroll
    for (int k = 0; k < KB; ++k) {
      const int i = tid + kAttnThreads * (k0 + k), r = i / C;
      if (r < rows) {
        attn_put_pair<DH>(sK + at.item(r) * Tp * DH, r - at.item(r) * T, 4 * (i % C), kk[k]);
        reinterpret_cast<float4*>(sV)[i] = vv[k];
      }
    }
  }
  __syncthreads();
  float sc[kMaxT + 1];
  if (on) {
    attn_dots<DH>(qv, sK + it * Tp * DH, T, sc);
    float mx = -INFINITY;
#pragma unroll
    for (int u = 0; u < kMaxT; ++u) {
      sc[u] = u < T && u <= ne ? sc[u] * scale : -INFINITY;
      mx = fmaxf(mx, sc[u]);
    }
    float z = 0.0f;
#pragma unroll
    for (int u = 0; u < kMaxT; ++u) {
      const float e = (u < T && u <= ne) ? expf(sc[u] - mx) : 0.0f;
      sc[u] = e;
      z += e;
    }
    const float iz = 1.0f / z;
    unsigned long long o[DH / 2];
#pragma unroll
    for (int j = 0; j < DH / 2; ++j) o[j] = 0ull;
#pragma unroll
    for (int u = 0; u < kMaxT; ++u) {
      sc[u] *= iz;
      if (u < T && u <= ne) attn_axpy<DH>(sc[u], sV + (it * T + u) * DH, o);
    }
    attn_store<DH>(O + (s * T + t) * d + hh * DH, o);
  }
  __syncthreads();
  if (on) {
#pragma unroll
    for (int u = 0; u < kMaxT; ++u)
      if (u < T) sm_attn[tid * T + u] = sc[u];
  }
  __syncthreads();
  float* Pb = P + q0 * T * T;
  for (int i = tid; i < items * T * T; i += kAttnThreads) Pb[i] = sm_attn[i];
}

// Attention backward: from dO and the stored P, dS = P (dP - rowsum(P dP))
// scale with dP = dO V^T; the thread of query t writes dQ_t, then the thread of
// key u writes dK_u = sum_t dS_tu Q_t and dV_u = sum_t P_tu dO_t.
template <int DH>
__global__ void __launch_bounds__(kAttnThreads) attn_bwd_kernel(const float* __restrict__ QKV,
                                                                const float* __restrict__ P,
                                                                const float* __restrict__ dO,
                                                                float* __restrict__ dQKV, long long n, int T, int H,
                                                                float scale) {
  extern __shared__ __align__(16) float sm_attn[];
  const int tid = threadIdx.x, ipb = attn_items(T), Tp = (T + 1) / 2 * 2, R = attn_rows(T);
  float* sQ = sm_attn;                     // [items][T][DH]
  float* sK = sQ + R * DH;
  float* sG = sK + R * DH;                 // dO
  float* sV = sG + R * DH;                 // [items][Tp / 2][DH][2]
  float* sP = sV + attn_pair_rows(T) * DH; // [items][T][T]
  float* sS = sP + R * T;                  // dS
  const long long q0 = (long long)blockIdx.x * ipb, nq = n * H;
  const int items = (int)(nq - q0 < ipb ? nq - q0 : ipb);
  const int d = DH * H, ld = 3 * d, rows = items * T, np = rows * T;
  const AttnRows at(q0, H, T);
  const float* const Pb = P + q0 * T * T;
  // two 16-byte columns of each row image and eight of P's elements per turn
  constexpr int C = DH / 4;
  for (int b = 0; b < C / 2 || 8 * b < T; ++b) {
    float4 x[2][4];
    float pe[8];
    if (b < C / 2) {
#pragma unroll
      for (int k = 0; k < 2; ++k) {
        const int i = tid + kAttnThreads * (2 * b + k), r = min(i / C, rows - 1);
        const float* src = QKV + at.offset(r, ld, DH) + 4 * (i % C);
        x[k][0] = __ldg(reinterpret_cast<const float4*>(src));
        x[k][1] = __ldg(reinterpret_cast<const float4*>(src + d));
        x[k][2] = __ldg(reinterpret_cast<const float4*>(dO + at.offset(r, d, DH) + 4 * (i % C)));
        x[k][3] = __ldg(reinterpret_cast<const float4*>(src + 2 * d));
      }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k) pe[k] = __ldg(Pb + min(tid + kAttnThreads * (8 * b + k), np - 1));
#pragma unroll
    for (int k = 0; k < 2; ++k) {
      const int i = tid + kAttnThreads * (2 * b + k), r = i / C;  // (from turn C / 2 on: past every row)
      if (r < rows) {
        reinterpret_cast<float4*>(sQ)[i] = x[k][0];
        reinterpret_cast<float4*>(sK)[i] = x[k][1];
        reinterpret_cast<float4*>(sG)[i] = x[k][2];
        attn_put_pair<DH>(sV + at.item(r) * Tp * DH, r - at.item(r) * T, 4 * (i % C), x[k][3]);
      }
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)
      if (tid + kAttnThreads * (8 * b + k) < np) sP[tid + kAttnThreads * (8 * b + k)] = pe[k];
  }
  __syncthreads();
  const int it = at.item(tid), t = tid - it * T;
  const bool on = it < items;
  long long s;
  int hh;
  at.sample(on ? it : 0, s, hh);
  float* out = dQKV + (s * T + t) * ld + hh * DH;
  unsigned long long o[DH / 2];
  if (on) {
    float g[DH], dp[kMaxT + 1];
#pragma unroll
    for (int j = 0; j < DH; j += 4) {
      const float4 v = *reinterpret_cast<const float4*>(sG + tid * DH + j);
      g[j] = v.x; g[j + 1] = v.y; g[j + 2] = v.z; g[j + 3] = v.w;
    }
    attn_dots<DH>(g, sV + it * Tp * DH, T, dp);
    float dot = 0.0f;
#pragma unroll
    for (int u = 0; u < kMaxT; ++u)
      if (u < T) dot = fmaf(sP[tid * T + u], dp[u], dot);
#pragma unroll
    for (int j = 0; j < DH / 2; ++j) o[j] = 0ull;
#pragma unroll
    for (int u = 0; u < kMaxT; ++u) {
      if (u < T) {
        const float ds = sP[tid * T + u] * (dp[u] - dot) * scale;
        sS[tid * T + u] = ds;
        attn_axpy<DH>(ds, sK + (it * T + u) * DH, o);
      }
    }
    attn_store<DH>(out, o);
  }
  __syncthreads();
  if (on) {
    unsigned long long dv[DH / 2];
#pragma unroll
    for (int j = 0; j < DH / 2; ++j) o[j] = dv[j] = 0ull;
    for (int r = it * T; r < it * T + T; ++r) {
      attn_axpy<DH>(sS[r * T + t], sQ + r * DH, o);
      attn_axpy<DH>(sP[r * T + t], sG + r * DH, dv);
    }
    attn_store<DH>(out + d, o);
    attn_store<DH>(out + 2 * d, dv);
  }
}

// m16n8k8 TF32 MMA on FP32 registers (operands rounded to TF32 first, FP32
// accumulation).  Fragments (g = lane / 4, t = lane % 4): A a0 (g, t),
// a1 (g + 8, t), a2 (g, t + 4), a3 (g + 8, t + 4); B b0 (k t, n g),
// b1 (k t + 4, n g); C c0 (g, 2t), c1 (g, 2t + 1), c2 (g + 8, 2t),
// c3 (g + 8, 2t + 1).
__device__ __forceinline__ uint32_t tf32r(float x) {
  uint32_t r;
  asm("cvt.rna.tf32.f32 %0, %1;" : "=r"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ void mma_tf32(float (&c)[4], uint32_t a0, uint32_t a1, uint32_t a2, uint32_t a3, uint32_t b0,
                                         uint32_t b1) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0, %1, %2, %3}, {%4, %5, %6, %7}, {%8, %9}, "
      "{%0, %1, %2, %3};"
      : "+f"(c[0]), "+f"(c[1]), "+f"(c[2]), "+f"(c[3])
      : "r"(a0), "r"(a1), "r"(a2), "r"(a3), "r"(b0), "r"(b1));
}
constexpr int kAttLd = 20;  // floats per staged 16-wide row (conflict-free fragment loads)

// C[16 x 16] (+)= A B over k = 16 from staged [16][kAttLd] tiles: A(r, k) =
// TA ? a[k][r] : a[r][k], B(k, n) = TB ? b[n][k] : b[k][n].  c[j] holds the
// n-tile of columns 8 j .. 8 j + 7.
template <bool TA, bool TB>
__device__ __forceinline__ void mma16x16(float (&c)[2][4], const float* a, const float* b, int g, int t) {
#pragma unroll
  for (int kk = 0; kk < 2; ++kk) {
    const int k0 = 8 * kk + t, k1 = k0 + 4;
    const uint32_t a0 = tf32r(TA ? a[k0 * kAttLd + g] : a[g * kAttLd + k0]);
    const uint32_t a1 = tf32r(TA ? a[k0 * kAttLd + g + 8] : a[(g + 8) * kAttLd + k0]);
    const uint32_t a2 = tf32r(TA ? a[k1 * kAttLd + g] : a[g * kAttLd + k1]);
    const uint32_t a3 = tf32r(TA ? a[k1 * kAttLd + g + 8] : a[(g + 8) * kAttLd + k1]);
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int nn = 8 * j + g;
      const uint32_t b0 = tf32r(TB ? b[nn * kAttLd + k0] : b[k0 * kAttLd + nn]);
      const uint32_t b1 = tf32r(TB ? b[nn * kAttLd + k1] : b[k1 * kAttLd + nn]);
      mma_tf32(c[j], a0, a1, a2, a3, b0, b1);
    }
  }
}

// Per-warp staging of one (sample, head) item: rows u = lane / 4 + 8 r
// (r = 0, 1) of the item's 16-wide Q, K, V slices (and dO in the backward),
// quarter lane % 4 of each row, as float4; rows u >= T are zero (and not
// loaded: loading a row that exists in their place was slower).  The warps are
// persistent: the next item's slices are loaded into registers while the
// current item is computed from shared memory.
struct AttRows {
  float4 q[2], k[2], v[2];
};
__device__ __forceinline__ void att_fetch(AttRows& r, const float* __restrict__ QKV, long long s, int hh, int T, int d,
                                          int lane) {
  const int u0 = lane >> 2, j4 = lane & 3;
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const int u = u0 + 8 * i;
    r.q[i] = r.k[i] = r.v[i] = make_float4(0.f, 0.f, 0.f, 0.f);
    if (u < T) {
      const float4* base = reinterpret_cast<const float4*>(QKV + (s * T + u) * 3 * d + hh * 16) + j4;
      r.q[i] = __ldg(base);
      r.k[i] = __ldg(base + d / 4);
      r.v[i] = __ldg(base + d / 2);
    }
  }
}
__device__ __forceinline__ void att_stage(const float4 (&x)[2], float* dst, int lane) {
  const int u0 = lane >> 2, j4 = lane & 3;
#pragma unroll
  for (int i = 0; i < 2; ++i) *reinterpret_cast<float4*>(dst + (u0 + 8 * i) * kAttLd + 4 * j4) = x[i];
}

// A row's two accumulator tiles to memory: lanes t and t ^ 1 of a quad trade, so
// that the even one has columns 2 t .. 2 t + 3 of the first tile and the odd one
// columns 8 + 2 (t - 1) .. of the second: half the stores, of whole sectors
// (655,360 items of 11 tokens: forward 504 -> 495 us, backward 872 -> 846).
// (Every lane of the warp calls it; `row` 16 floats, 16-byte aligned.)
__device__ __forceinline__ void att_store_row(float* row, float2 lo, float2 hi, int t, bool on) {
  const bool odd = t & 1;
  const float2 give = odd ? lo : hi;
  const float gx = __shfl_xor_sync(0xffffffffu, give.x, 1), gy = __shfl_xor_sync(0xffffffffu, give.y, 1);
  if (on)
    *reinterpret_cast<float4*>(row + (odd ? 6 + 2 * t : 2 * t)) =
        odd ? make_float4(gx, gy, hi.x, hi.y) : make_float4(lo.x, lo.y, gx, gy);
}

// Blocks of `threads` threads of `kernel` resident on the device at once (at
// least one per SM), for the persistent and grid-stride kernels.
template <typename K>
inline long long resident_blocks(K kernel, int threads) {
  int dev = 0, b = 0, m = 0;
  if (cudaGetDevice(&dev) != cudaSuccess ||
      cudaDeviceGetAttribute(&m, cudaDevAttrMultiProcessorCount, dev) != cudaSuccess ||
      cudaOccupancyMaxActiveBlocksPerMultiprocessor(&b, kernel, threads, 0) != cudaSuccess) {
    (void)cudaGetLastError();
    b = 1, m = 152;
  }
  return (long long)(b > 0 ? b : 1) * (m > 0 ? m : 152);
}

// Grid of a persistent attention kernel (4 items per block at a time): its
// resident blocks `cap`, or fewer when there are fewer items.
inline unsigned att_grid(long long cap, long long items) {
  const long long need = (items + 3) / 4;
  return (unsigned)(need < cap ? need : cap);
}

// Attention forward on the tensor cores (tensor-core path; T <= 16, head
// dimension 16), one (sample, head) item per warp at a time, persistent warps
// (4 per block) over the items: S = Q K^T as m16n8k8 TF32 MMAs over the
// tokens padded to 16, the masked softmax on the accumulator fragments (keys
// u <= n_ent of the sample, a row in the 4 lanes of a quad), P written out
// (zero at masked keys) and staged, then O = P V.
__global__ void __launch_bounds__(128, 8)
    attn_fwd_mma_kernel(const float* __restrict__ QKV, const int32_t* __restrict__ n_ent,
                        const int32_t* __restrict__ sel, float* __restrict__ P, float* __restrict__ O, long long n,
                        int T, int NS, int H, float scale) {
  __shared__ __align__(16) float sm[4][4][16 * kAttLd];  // Q, K, V, P of each warp
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int d = 16 * H;
  const long long items = n * H, stride = (long long)gridDim.x * 4;
  float *sQ = sm[wl][0], *sK = sm[wl][1], *sV = sm[wl][2], *sP = sm[wl][3];
  long long w = (long long)blockIdx.x * 4 + wl;
  AttRows r;
  int ne_next = 0;
  AttItem nx = {0, 0};
  auto fetch = [&](long long wi) {
    nx = att_item(wi, H);
    att_fetch(r, QKV, nx.s, nx.hh, T, d, lane);
    ne_next = __ldg(n_ent + (sel ? (long long)__ldg(sel + nx.s) : nx.s));
  };
  if (w < items) fetch(w);
  for (; w < items; w += stride) {
    const long long s = nx.s;
    const int hh = nx.hh;
    att_stage(r.q, sQ, lane);
    att_stage(r.k, sK, lane);
    att_stage(r.v, sV, lane);
    const int ne = ne_next < 0 ? 0 : (ne_next > NS ? NS : ne_next);
    if (w + stride < items) fetch(w + stride);  // in flight during this item
    __syncwarp();
    float sc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    mma16x16<false, true>(sc, sQ, sK, g, t);  // S = Q K^T
    float* Pb = P + (s * H + hh) * T * T;
#pragma unroll
    for (int hr = 0; hr < 2; ++hr) {
      const int row = g + 8 * hr;
      float mx = -INFINITY;
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int col = 8 * j + 2 * t + e;
          const float v = (col < T && col <= ne) ? sc[j][2 * hr + e] * scale : -INFINITY;
          sc[j][2 * hr + e] = v;
          mx = fmaxf(mx, v);
        }
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
      mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
      float z = 0.0f;
#pragma unroll
      for (int j = 0; j < 2; ++j)
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const float x = sc[j][2 * hr + e];
          const float ex = x == -INFINITY ? 0.0f : __expf(x - mx);
          sc[j][2 * hr + e] = ex;
          z += ex;
        }
      z += __shfl_xor_sync(0xffffffffu, z, 1);
      z += __shfl_xor_sync(0xffffffffu, z, 2);
      const float iz = 1.0f / z;
#pragma unroll
      for (int j = 0; j < 2; ++j) {
        const int col = 8 * j + 2 * t;
        const float p0 = sc[j][2 * hr] * iz, p1 = sc[j][2 * hr + 1] * iz;
        sP[row * kAttLd + col] = p0;
        sP[row * kAttLd + col + 1] = p1;
        if (row < T) {
          if (col < T) Pb[row * T + col] = p0;
          if (col + 1 < T) Pb[row * T + col + 1] = p1;
        }
      }
    }
    __syncwarp();
    float o[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    mma16x16<false, false>(o, sP, sV, g, t);  // O = P V
#pragma unroll
    for (int hr = 0; hr < 2; ++hr) {
      const int row = g + 8 * hr;
      att_store_row(O + (s * T + row) * d + hh * 16, make_float2(o[0][2 * hr], o[0][2 * hr + 1]),
                    make_float2(o[1][2 * hr], o[1][2 * hr + 1]), t, row < T);
    }
    __syncwarp();  // the staged tiles are read before the next item overwrites them
  }
}

// Attention backward on the tensor cores (tensor-core path; T <= 16, head
// dimension 16), one (sample, head) item per warp at a time, persistent warps
// (4 per block): the products of attn_bwd_kernel, dP = dO V^T, dQ = dS K,
// dK = dS^T Q, dV = P^T dO, as m16n8k8 TF32 MMAs over the tokens padded to
// 16 (padded rows and columns staged as zeros), and
// dS = P (dP - rowsum(P dP)) scale on the accumulator fragments (a row lives
// in the 4 lanes of a quad).  dS is staged over V (V is read only by dP).  PE:
// elements of P per lane, 32 PE >= T * T (att_p_per_lane).
constexpr int att_p_per_lane(int T) { return T * T <= 128 ? 4 : 8; }
template <int PE>
__global__ void __launch_bounds__(128, PE == 4 ? 6 : 5)
    attn_bwd_mma_kernel(const float* __restrict__ QKV, const float* __restrict__ P, const float* __restrict__ dO,
                        float* __restrict__ dQKV, long long n, int T, int H, float scale) {
  __shared__ __align__(16) float sm[4][5][16 * kAttLd];  // Q, K, V then dS, dO, P of each warp
  const int lane = threadIdx.x & 31, wl = threadIdx.x >> 5, g = lane >> 2, t = lane & 3;
  const int d = 16 * H, ld = 3 * d;
  const long long items = n * H, stride = (long long)gridDim.x * 4;
  float *sQ = sm[wl][0], *sK = sm[wl][1], *sV = sm[wl][2], *sS = sm[wl][2], *sG = sm[wl][3], *sP = sm[wl][4];
  // P of an item: T * T contiguous floats, element e = lane + 32 i at
  // (e / T, e % T) of the staged tile; the padding stays zero
  int pofs[PE];
#pragma unroll
  for (int i = 0; i < PE; ++i) {
    const int e = lane + 32 * i;
    pofs[i] = e < T * T ? (e / T) * kAttLd + e % T : -1;
  }
  for (int i = lane; i < 16 * kAttLd; i += 32) sP[i] = 0.0f;
  long long w = (long long)blockIdx.x * 4 + wl;
  AttRows r;
  float4 rg[2];
  float rp[PE];
  AttItem nx = {0, 0};
  auto fetch = [&](long long wi) {
    nx = att_item(wi, H);
    att_fetch(r, QKV, nx.s, nx.hh, T, d, lane);
    const int u0 = lane >> 2, j4 = lane & 3;
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int u = u0 + 8 * i;
      rg[i] = u < T ? __ldg(reinterpret_cast<const float4*>(dO + (nx.s * T + u) * d + nx.hh * 16) + j4)
                    : make_float4(0.f, 0.f, 0.f, 0.f);
    }
    const float* Pb = P + wi * T * T;
#pragma unroll
    for (int i = 0; i < PE; ++i) rp[i] = pofs[i] >= 0 ? __ldg(Pb + lane + 32 * i) : 0.0f;
  };
  if (w < items) fetch(w);
  for (; w < items; w += stride) {
    const long long s = nx.s;
    const int hh = nx.hh;
    att_stage(r.q, sQ, lane);
    att_stage(r.k, sK, lane);
    att_stage(r.v, sV, lane);
    att_stage(rg, sG, lane);
#pragma unroll
    for (int i = 0; i < PE; ++i)
      if (pofs[i] >= 0) sP[pofs[i]] = rp[i];
    if (w + stride < items) fetch(w + stride);  // in flight during this item
    __syncwarp();
    // dP = dO V^T
    float dp[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    mma16x16<false, true>(dp, sG, sV, g, t);
    // dS = P (dP - rowsum(P dP)) scale (rows g and g + 8 of this quad)
    float pv[2][4], r0 = 0.0f, r1 = 0.0f;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int c = 8 * j + 2 * t;
      pv[j][0] = sP[g * kAttLd + c];
      pv[j][1] = sP[g * kAttLd + c + 1];
      pv[j][2] = sP[(g + 8) * kAttLd + c];
      pv[j][3] = sP[(g + 8) * kAttLd + c + 1];
      r0 = fmaf(pv[j][0], dp[j][0], fmaf(pv[j][1], dp[j][1], r0));
      r1 = fmaf(pv[j][2], dp[j][2], fmaf(pv[j][3], dp[j][3], r1));
    }
    r0 += __shfl_xor_sync(0xffffffffu, r0, 1);
    r0 += __shfl_xor_sync(0xffffffffu, r0, 2);
    r1 += __shfl_xor_sync(0xffffffffu, r1, 1);
    r1 += __shfl_xor_sync(0xffffffffu, r1, 2);
    __syncwarp();  // every lane's V fragments are read: dS goes over V
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      const int c = 8 * j + 2 * t;
      sS[g * kAttLd + c] = pv[j][0] * (dp[j][0] - r0) * scale;
      sS[g * kAttLd + c + 1] = pv[j][1] * (dp[j][1] - r0) * scale;
      sS[(g + 8) * kAttLd + c] = pv[j][2] * (dp[j][2] - r1) * scale;
      sS[(g + 8) * kAttLd + c + 1] = pv[j][3] * (dp[j][3] - r1) * scale;
    }
    __syncwarp();
    float dq[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    float dk[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    float dv[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
    mma16x16<false, false>(dq, sS, sK, g, t);  // dQ = dS K
    mma16x16<true, false>(dk, sS, sQ, g, t);   // dK = dS^T Q
    mma16x16<true, false>(dv, sP, sG, g, t);   // dV = P^T dO
    float* out = dQKV + s * T * ld + hh * 16;
#pragma unroll
    for (int hr = 0; hr < 2; ++hr) {
      const int row = g + 8 * hr;
      auto store = [&](float* dst, const float (&c)[2][4]) {
        att_store_row(dst + row * ld, make_float2(c[0][2 * hr], c[0][2 * hr + 1]),
                      make_float2(c[1][2 * hr], c[1][2 * hr + 1]), t, row < T);
      };
      store(out, dq);
      store(out + d, dk);
      store(out + 2 * d, dv);
    }
    __syncwarp();  // the staged tiles are read before the next item overwrites them
  }
}

// ---- attention of the last block: the recurrent query alone ----------------
// The head reads nothing else, so the rest of the block (Wo, the feed-forward
// sub-block and their backward) runs on n rows instead of n T.  The actor's
// gradient step (163,840 samples, 11 tokens, d 64, 2 blocks) went from 19.5 to
// 14.3 ms, the critic's (32,768) from 4.40 to 3.24, d 128 with 17 tokens and 3
// blocks (16,384) from 14.1 to 11.6.
// One (sample, head) per warp.  Q0 [n][d] holds the recurrent queries, KV
// [rows][2d] the keys and values of every token; dKV [rows][2d] and D0 [n][3d]
// (dQ, dK, dV of the recurrent rows) are their gradients; P0 [n][H][T] and O0 [n][d]
// are row 0 of P and O above, by the same arithmetic.  The cost is one read
// of K and V (and in the backward one write of dK and dV).

// General form (lane u: key u of the scores; lane j: output column j).  Rows of V
// and K are loaded eight at a time, unconditionally: one by one behind their
// conditions 131,072 items of 17 x 16 took 155 us forward and 252 us backward,
// now 111 and 175.
template <int DH>
__global__ void __launch_bounds__(256) attn0_fwd_kernel(const float* __restrict__ Q0, const float* __restrict__ KV,
                                                        const int32_t* __restrict__ n_ent,
                                                        const int32_t* __restrict__ sel, float* __restrict__ P0,
                                                        float* __restrict__ O0, long long n, int T, int NS, int H,
                                                        float scale) {
  const int lane = threadIdx.x & 31;
  const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= n * H) return;  // whole warps leave together
  const AttItem it = att_item(w, H);
  const long long s = it.s;
  const int hh = it.hh, d = DH * H, ld = 2 * d;
  int ne = n_ent[sel ? (long long)sel[s] : s];
  ne = ne < 0 ? 0 : (ne > NS ? NS : ne);
  const float* K = KV + s * T * ld + hh * DH;
  const float* V = K + d;
  const bool on = lane < T && lane <= ne;
  float sc = -INFINITY;
  if (on) {
    const float4* q4 = reinterpret_cast<const float4*>(Q0 + s * d + hh * DH);
    const float4* k4 = reinterpret_cast<const float4*>(K + lane * ld);
    float acc = 0.0f;
#pragma unroll
    for (int j = 0; j < DH / 4; ++j) {
      const float4 q = __ldg(q4 + j), k = __ldg(k4 + j);
      acc = fmaf(q.x, k.x, acc);
      acc = fmaf(q.y, k.y, acc);
      acc = fmaf(q.z, k.z, acc);
      acc = fmaf(q.w, k.w, acc);
    }
    sc = acc * scale;
  }
  const float mx = warp_max(sc);
  const float e = on ? expf(sc - mx) : 0.0f;
  float z = 0.0f;
  for (int u = 0; u < T; ++u) z += __shfl_sync(0xffffffffu, e, u);  // (in key order, as attn_fwd_kernel)
  const float p = e * (1.0f / z);
  if (lane < T) P0[w * T + lane] = p;
  float o = 0.0f;
  const int j = lane < DH ? lane : 0;
  for (int u0 = 0; u0 <= ne && u0 < T; u0 += 8) {  // eight rows' loads at a time
    float v[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) v[i] = __ldg(V + min(u0 + i, T - 1) * ld + j);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const float pu = __shfl_sync(0xffffffffu, p, (u0 + i) & 31);
      if (u0 + i <= ne && u0 + i < T) o = fmaf(pu, v[i], o);
    }
  }
  if (lane < DH) O0[s * d + hh * DH + lane] = o;
}

template <int DH>
__global__ void __launch_bounds__(256) attn0_bwd_kernel(const float* __restrict__ Q0, const float* __restrict__ KV,
                                                        const float* __restrict__ P0, const float* __restrict__ dO0,
                                                        float* __restrict__ D0, float* __restrict__ dKV, long long n,
                                                        int T, int H, float scale) {
  const int lane = threadIdx.x & 31;
  const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= n * H) return;  // whole warps leave together
  const AttItem it = att_item(w, H);
  const long long s = it.s;
  const int hh = it.hh, d = DH * H, ld = 2 * d;
  const float* K = KV + s * T * ld + hh * DH;
  float* dK = dKV + s * T * ld + hh * DH;
  const float p = lane < T ? __ldg(P0 + w * T + lane) : 0.0f;
  float dp = 0.0f;
  if (lane < T) {
    const float4* g4 = reinterpret_cast<const float4*>(dO0 + s * d + hh * DH);
    const float4* v4 = reinterpret_cast<const float4*>(K + d + lane * ld);
#pragma unroll
    for (int j = 0; j < DH / 4; ++j) {
      const float4 g = __ldg(g4 + j), v = __ldg(v4 + j);
      dp = fmaf(g.x, v.x, dp);
      dp = fmaf(g.y, v.y, dp);
      dp = fmaf(g.z, v.z, dp);
      dp = fmaf(g.w, v.w, dp);
    }
  }
  float dot = 0.0f;
  for (int u = 0; u < T; ++u) dot = fmaf(__shfl_sync(0xffffffffu, p, u), __shfl_sync(0xffffffffu, dp, u), dot);
  const float ds = p * (dp - dot) * scale;
  const int j = lane < DH ? lane : 0;
  const float qj = __ldg(Q0 + s * d + hh * DH + j), gj = __ldg(dO0 + s * d + hh * DH + j);
  float dq = 0.0f;
  for (int u0 = 0; u0 < T; u0 += 8) {  // eight rows' loads at a time
    float k[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) k[i] = __ldg(K + min(u0 + i, T - 1) * ld + j);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const int u = u0 + i;
      const float su = __shfl_sync(0xffffffffu, ds, u & 31), pu = __shfl_sync(0xffffffffu, p, u & 31);
      if (u < T) {
        dq = fmaf(su, k[i], dq);
        if (lane < DH) {
          dK[u * ld + lane] = su * qj;
          dK[u * ld + d + lane] = pu * gj;
          if (u == 0) {
            D0[s * 3 * d + d + hh * DH + lane] = su * qj;
            D0[s * 3 * d + 2 * d + hh * DH + lane] = pu * gj;
          }
        }
      }
    }
  }
  if (lane < DH) D0[s * 3 * d + hh * DH + lane] = dq;
}

// The tensor-core path's form (T <= 16, head dimension 16): the products of
// attn_fwd_mma_kernel with the one query in row 0 of the A operand, every
// fragment straight from global memory (a row of K or V is two sectors that
// one load of the warp touches; no staging, so many warps' loads are in
// flight).  163,840 samples x 4 heads x 11 tokens: forward 283 us against 502
// for all queries, backward 426 against 870.
__device__ __forceinline__ float quad_pick(float lo, float hi, int t, int up) {
  // the quad lane that holds column t + up of an 8-wide accumulator tile
  const int src = (threadIdx.x & 28) | ((t + up) >> 1);
  const float a = __shfl_sync(0xffffffffu, lo, src), b = __shfl_sync(0xffffffffu, hi, src);
  return (t & 1) ? b : a;
}
__global__ void __launch_bounds__(256)
    attn0_fwd_mma_kernel(const float* __restrict__ Q0, const float* __restrict__ KV, const int32_t* __restrict__ n_ent,
                         const int32_t* __restrict__ sel, float* __restrict__ P0, float* __restrict__ O0, long long n,
                         int T, int NS, int H, float scale) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= n * H) return;  // whole warps leave together
  const long long s = w / H;
  const int hh = (int)(w - s * H), d = 16 * H, ld = 2 * d;
  const float* K = KV + s * T * ld + hh * 16;
  const float* V = K + d;
  float q[4], kf[2][4], vf[4][2];  // K rows g + 8 j, V rows t + 4 i (columns g, g + 8)
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    q[i] = g == 0 ? __ldg(Q0 + s * d + hh * 16 + t + 4 * i) : 0.0f;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      kf[j][i] = g + 8 * j < T ? __ldg(K + (g + 8 * j) * ld + t + 4 * i) : 0.0f;
      vf[i][j] = t + 4 * i < T ? __ldg(V + (t + 4 * i) * ld + g + 8 * j) : 0.0f;
    }
  }
  int ne = n_ent[sel ? (long long)__ldg(sel + s) : s];
  ne = ne < 0 ? 0 : (ne > NS ? NS : ne);
  float sc[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
  for (int kk = 0; kk < 2; ++kk)
#pragma unroll
    for (int j = 0; j < 2; ++j)
      mma_tf32(sc[j], tf32r(q[2 * kk]), 0u, tf32r(q[2 * kk + 1]), 0u, tf32r(kf[j][2 * kk]), tf32r(kf[j][2 * kk + 1]));
  float mx = -INFINITY;
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int col = 8 * j + 2 * t + e;
      const float v = (col < T && col <= ne) ? sc[j][e] * scale : -INFINITY;
      sc[j][e] = v;
      mx = fmaxf(mx, v);
    }
  mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
  mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
  float z = 0.0f;
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const float x = sc[j][e];
      const float ex = x == -INFINITY ? 0.0f : __expf(x - mx);
      sc[j][e] = ex;
      z += ex;
    }
  z += __shfl_xor_sync(0xffffffffu, z, 1);
  z += __shfl_xor_sync(0xffffffffu, z, 2);
  const float iz = 1.0f / z;
#pragma unroll
  for (int j = 0; j < 2; ++j) {
    const int col = 8 * j + 2 * t;
    sc[j][0] *= iz;
    sc[j][1] *= iz;
    if (g == 0 && col < T) P0[w * T + col] = sc[j][0];
    if (g == 0 && col + 1 < T) P0[w * T + col + 1] = sc[j][1];
  }
  float o[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
  for (int kk = 0; kk < 2; ++kk) {
    const float p0 = quad_pick(sc[kk][0], sc[kk][1], t, 0), p1 = quad_pick(sc[kk][0], sc[kk][1], t, 4);
    const uint32_t a0 = g == 0 ? tf32r(p0) : 0u, a2 = g == 0 ? tf32r(p1) : 0u;
#pragma unroll
    for (int j = 0; j < 2; ++j) mma_tf32(o[j], a0, 0u, a2, 0u, tf32r(vf[2 * kk][j]), tf32r(vf[2 * kk + 1][j]));
  }
  if (g == 0) {
#pragma unroll
    for (int j = 0; j < 2; ++j)
      *reinterpret_cast<float2*>(O0 + s * d + hh * 16 + 8 * j + 2 * t) = make_float2(o[j][0], o[j][1]);
  }
}

// Backward of the same: dP and dQ by MMAs; dK_u = dS_u q and dV_u = P_u dO
// are single products of TF32-rounded factors (exact in FP32), which is what
// the MMAs over the one query row give.
__global__ void __launch_bounds__(256)
    attn0_bwd_mma_kernel(const float* __restrict__ Q0, const float* __restrict__ KV, const float* __restrict__ P0,
                         const float* __restrict__ dO0, float* __restrict__ D0, float* __restrict__ dKV, long long n,
                         int T, int H, float scale) {
  const int lane = threadIdx.x & 31, g = lane >> 2, t = lane & 3;
  const long long w = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  if (w >= n * H) return;  // whole warps leave together
  const long long s = w / H;
  const int hh = (int)(w - s * H), d = 16 * H, ld = 2 * d;
  const float* K = KV + s * T * ld + hh * 16;
  const float* V = K + d;
  const float* dOb = dO0 + s * d + hh * 16;
  float gf[4], vf[2][4], kf[4][2], pv[2][2];  // V rows g + 8 j, K rows t + 4 i
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    gf[i] = g == 0 ? __ldg(dOb + t + 4 * i) : 0.0f;
#pragma unroll
    for (int j = 0; j < 2; ++j) {
      vf[j][i] = g + 8 * j < T ? __ldg(V + (g + 8 * j) * ld + t + 4 * i) : 0.0f;
      kf[i][j] = t + 4 * i < T ? __ldg(K + (t + 4 * i) * ld + g + 8 * j) : 0.0f;
    }
  }
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int e = 0; e < 2; ++e) {
      const int c = 8 * j + 2 * t + e;
      pv[j][e] = c < T ? __ldg(P0 + w * T + c) : 0.0f;
    }
  const float4 q4 = __ldg(reinterpret_cast<const float4*>(Q0 + s * d + hh * 16) + t);
  const float4 g4 = __ldg(reinterpret_cast<const float4*>(dOb) + t);
  float dp[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
  for (int kk = 0; kk < 2; ++kk)
#pragma unroll
    for (int j = 0; j < 2; ++j)
      mma_tf32(dp[j], tf32r(gf[2 * kk]), 0u, tf32r(gf[2 * kk + 1]), 0u, tf32r(vf[j][2 * kk]),
               tf32r(vf[j][2 * kk + 1]));
  float r0 = 0.0f;  // (row 0's sum: right in the lanes of the first quad)
#pragma unroll
  for (int j = 0; j < 2; ++j) r0 = fmaf(pv[j][0], dp[j][0], fmaf(pv[j][1], dp[j][1], r0));
  r0 += __shfl_xor_sync(0xffffffffu, r0, 1);
  r0 += __shfl_xor_sync(0xffffffffu, r0, 2);
  float ds[2][2];
#pragma unroll
  for (int j = 0; j < 2; ++j)
#pragma unroll
    for (int e = 0; e < 2; ++e) ds[j][e] = pv[j][e] * (dp[j][e] - r0) * scale;
  float dq[2][4] = {{0.f, 0.f, 0.f, 0.f}, {0.f, 0.f, 0.f, 0.f}};
#pragma unroll
  for (int kk = 0; kk < 2; ++kk) {
    const float s0 = quad_pick(ds[kk][0], ds[kk][1], t, 0), s1 = quad_pick(ds[kk][0], ds[kk][1], t, 4);
    const uint32_t a0 = g == 0 ? tf32r(s0) : 0u, a2 = g == 0 ? tf32r(s1) : 0u;
#pragma unroll
    for (int j = 0; j < 2; ++j) mma_tf32(dq[j], a0, 0u, a2, 0u, tf32r(kf[2 * kk][j]), tf32r(kf[2 * kk + 1][j]));
  }
  if (g == 0) {
#pragma unroll
    for (int j = 0; j < 2; ++j)
      *reinterpret_cast<float2*>(D0 + s * 3 * d + hh * 16 + 8 * j + 2 * t) = make_float2(dq[j][0], dq[j][1]);
  }
  const float qv[4] = {q4.x, q4.y, q4.z, q4.w}, gv[4] = {g4.x, g4.y, g4.z, g4.w};
#pragma unroll
  for (int j = 0; j < 2; ++j) {  // token u = g + 8 j, columns 4 t .. 4 t + 3
    const int src = g >> 1;      // (lane of the first quad holding column g of tile j)
    const float sa = __shfl_sync(0xffffffffu, ds[j][0], src), sb = __shfl_sync(0xffffffffu, ds[j][1], src);
    const float pa = __shfl_sync(0xffffffffu, pv[j][0], src), pb = __shfl_sync(0xffffffffu, pv[j][1], src);
    const float su = __uint_as_float(tf32r((g & 1) ? sb : sa)), pu = __uint_as_float(tf32r((g & 1) ? pb : pa));
    float a[4], b[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      a[i] = su * __uint_as_float(tf32r(qv[i]));
      b[i] = pu * __uint_as_float(tf32r(gv[i]));
    }
    if (g + 8 * j < T) {
      float* out = dKV + (s * T + g + 8 * j) * ld + hh * 16 + 4 * t;
      *reinterpret_cast<float4*>(out) = make_float4(a[0], a[1], a[2], a[3]);
      *reinterpret_cast<float4*>(out + d) = make_float4(b[0], b[1], b[2], b[3]);
    }
    if (g == 0 && j == 0) {
      float* out = D0 + s * 3 * d + d + hh * 16 + 4 * t;
      *reinterpret_cast<float4*>(out) = make_float4(a[0], a[1], a[2], a[3]);
      *reinterpret_cast<float4*>(out + d) = make_float4(b[0], b[1], b[2], b[3]);
    }
  }
}

struct HeadArgs {
  const float* XL;  // [n][d] residual stream of the recurrent tokens after the last block
  long long n;
  int n_out, mode;  // mode 0: forward, 1: PPO actor loss, 2: value loss
  const float *lnf_g, *lnf_b, *Wh, *bh;
  float* out;        // [n][n_out] (mode 0)
  float* h_out;      // [n][d] (mode 0, optional)
  const int32_t* sel;
  const int32_t* actions;
  const float *logp_old, *adv, *ret;
  float clip_eps, ent_coef, inv_n;
  float* dXL;        // [n][d] (modes 1, 2): gradient at XL
  float* part;       // [warps][2d + n_out d + n_out]: lnf_g, lnf_b, Wh, bh partial gradients
  double* spart;     // [warps][4] partial sums of the per-sample statistics
};

// Final LayerNorm and head on the recurrent token, one warp per sample; in the
// loss modes also the loss, dL/d(head output), the head's and final
// LayerNorm's backward, and per-warp partial sums of their parameter
// gradients.  NO: a compile-time bound of n_out, so that the outputs' dot
// products and exponentials are independent chains.  A sample's row, its index
// and then the values gathered by it are loaded during the previous sample.
// The statistics are summed in double: each lane keeps one sample's terms and
// all 32 are added at once (the FP64 pipe takes a warp instruction for 16
// cycles).  163,840 samples, 7 outputs: 146 us (583 with
// neither).
template <int DJ, int NO>
__global__ void __launch_bounds__(256) head_kernel(HeadArgs a) {
  constexpr int d = 32 * DJ;
  const int lane = threadIdx.x & 31;
  const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  const int no = a.n_out;
  float gW[NO][DJ], gB[NO], gg[DJ], gb[DJ], lg[DJ], lb[DJ];
#pragma unroll
  for (int o = 0; o < NO; ++o) {
    gB[o] = 0.0f;
#pragma unroll
    for (int i = 0; i < DJ; ++i) gW[o][i] = 0.0f;
  }
#pragma unroll
  for (int i = 0; i < DJ; ++i) {
    gg[i] = gb[i] = 0.0f;
    lg[i] = a.lnf_g[lane + 32 * i];
    lb[i] = a.lnf_b[lane + 32 * i];
  }
  double st[4] = {0.0, 0.0, 0.0, 0.0};
  float keep[4] = {0.0f, 0.0f, 0.0f, 0.0f};
  auto flush = [&]() {
    st[0] += a.mode == 2 ? (double)keep[0] * keep[0] : (double)keep[0];
#pragma unroll
    for (int k = 1; k < 4; ++k) st[k] += (double)keep[k];
#pragma unroll
    for (int k = 0; k < 4; ++k) keep[k] = 0.0f;
  };
  float xn[DJ], f0 = 0.0f, f1 = 0.0f;  // next sample: row; logp_old and advantage, or return
  int an = 0;                          // and its action
  long long bn = 0;                    // and its batch row
  auto fetch_row = [&](long long s) {
#pragma unroll
    for (int i = 0; i < DJ; ++i) xn[i] = a.XL[s * d + lane + 32 * i];
    bn = a.mode != 0 && a.sel ? (long long)a.sel[s] : s;
  };
  auto fetch_batch = [&]() {
    if (a.mode == 1) {
      an = a.actions[bn];
      f0 = a.logp_old[bn];
      f1 = a.adv[bn];
    } else if (a.mode == 2) {
      f0 = a.ret[bn];
    }
  };
  if (w0 < a.n) {
    fetch_row(w0);
    fetch_batch();
  }
  int it = 0;
  for (long long s = w0; s < a.n; s += nw, ++it) {
    const bool more = s + nw < a.n;
    const float lo = f0, A = f1;
    const int act = an;
    float x[DJ], xh[DJ], U[DJ], sum = 0.0f;
#pragma unroll
    for (int i = 0; i < DJ; ++i) {
      x[i] = xn[i];
      sum += x[i];
    }
    if (more) fetch_row(s + nw);
    const float mean = warp_sum(sum) * (1.0f / d);
    float v = 0.0f;
#pragma unroll
    for (int i = 0; i < DJ; ++i) v += (x[i] - mean) * (x[i] - mean);
    const float rstd = 1.0f / sqrtf(warp_sum(v) * (1.0f / d) + 1e-5f);
#pragma unroll
    for (int i = 0; i < DJ; ++i) {
      xh[i] = (x[i] - mean) * rstd;
      U[i] = xh[i] * lg[i] + lb[i];
    }
    float z[NO];
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      z[o] = 0.0f;
#pragma unroll
      for (int i = 0; i < DJ; ++i) z[o] = fmaf(o < no ? __ldg(a.Wh + o * d + lane + 32 * i) : 0.0f, U[i], z[o]);
    }
#pragma unroll
    for (int k = 16; k > 0; k >>= 1)
#pragma unroll
      for (int o = 0; o < NO; ++o) z[o] += __shfl_xor_sync(0xffffffffu, z[o], k);
#pragma unroll
    for (int o = 0; o < NO; ++o)
      if (o < no) z[o] += __ldg(a.bh + o);
    if (more) fetch_batch();
    if (a.mode == 0) {
      if (lane < no) {
#pragma unroll
        for (int o = 0; o < NO; ++o)
          if (o == lane) a.out[s * no + o] = z[o];
      }
      if (a.h_out)
#pragma unroll
        for (int i = 0; i < DJ; ++i) a.h_out[s * d + lane + 32 * i] = x[i];
      continue;
    }
    float dz[NO], stat[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    if (a.mode == 2) {
      const float e = z[0] - lo;
#pragma unroll
      for (int o = 0; o < NO; ++o) dz[o] = 0.0f;
      dz[0] = 2.0f * e * a.inv_n;
      stat[0] = e;
      stat[1] = z[0];
    } else {
      float mx = -INFINITY;
#pragma unroll
      for (int o = 0; o < NO; ++o)
        if (o < no) mx = fmaxf(mx, z[o]);
      float zs = 0.0f;
#pragma unroll
      for (int o = 0; o < NO; ++o)
        if (o < no) zs += expf(z[o] - mx);
      const float lse = mx + logf(zs);
      float ent = 0.0f, lpa = 0.0f, p[NO];
#pragma unroll
      for (int o = 0; o < NO; ++o) {
        p[o] = 0.0f;
        if (o < no) {
          const float lp = z[o] - lse;
          p[o] = expf(lp);
          ent -= p[o] * lp;
          if (o == act) lpa = lp;
        }
      }
      const float r = expf(lpa - lo);
      const float rc = fminf(fmaxf(r, 1.0f - a.clip_eps), 1.0f + a.clip_eps);
      const float s1 = r * A, s2 = rc * A;
      const float gl = s1 <= s2 ? -A * r : 0.0f;  // ties: the unclipped term carries the gradient
#pragma unroll
      for (int o = 0; o < NO; ++o) {
        dz[o] = 0.0f;
        if (o < no) {
          const float lp = z[o] - lse;
          dz[o] = (gl * ((o == act ? 1.0f : 0.0f) - p[o]) + a.ent_coef * p[o] * (lp + ent)) * a.inv_n;
        }
      }
      stat[0] = -fminf(s1, s2) - a.ent_coef * ent;
      stat[1] = ent;
      stat[2] = fabsf(r - 1.0f) > a.clip_eps ? 1.0f : 0.0f;
      stat[3] = lo - lpa;
    }
    if (lane == (it & 31)) {
#pragma unroll
      for (int k = 0; k < 4; ++k) keep[k] = stat[k];
    }
    if ((it & 31) == 31) flush();
    float dU[DJ];
#pragma unroll
    for (int i = 0; i < DJ; ++i) dU[i] = 0.0f;
#pragma unroll
    for (int o = 0; o < NO; ++o) {
      gB[o] += dz[o];
#pragma unroll
      for (int i = 0; i < DJ; ++i) {
        gW[o][i] = fmaf(dz[o], U[i], gW[o][i]);
        dU[i] = fmaf(o < no ? __ldg(a.Wh + o * d + lane + 32 * i) : 0.0f, dz[o], dU[i]);
      }
    }
    float dxh[DJ], m1 = 0.0f, m2 = 0.0f;
#pragma unroll
    for (int i = 0; i < DJ; ++i) {
      dxh[i] = dU[i] * lg[i];
      gg[i] = fmaf(dU[i], xh[i], gg[i]);
      gb[i] += dU[i];
      m1 += dxh[i];
      m2 = fmaf(dxh[i], xh[i], m2);
    }
    m1 = warp_sum(m1) * (1.0f / d);
    m2 = warp_sum(m2) * (1.0f / d);
    float* dx0 = a.dXL + s * d;
#pragma unroll
    for (int i = 0; i < DJ; ++i) dx0[lane + 32 * i] = rstd * (dxh[i] - m1 - xh[i] * m2);
  }
  if (a.mode == 0) return;
  flush();
#pragma unroll
  for (int k = 0; k < 4; ++k) st[k] = warp_sum_d(st[k]);
  const long long plen = 2 * d + (long long)no * d + no;
  float* pp = a.part + w0 * plen;
#pragma unroll
  for (int i = 0; i < DJ; ++i) {
    pp[lane + 32 * i] = gg[i];
    pp[d + lane + 32 * i] = gb[i];
  }
#pragma unroll
  for (int o = 0; o < NO; ++o)
    if (o < no) {
#pragma unroll
      for (int i = 0; i < DJ; ++i) pp[2 * d + o * d + lane + 32 * i] = gW[o][i];
      if (lane == 0) pp[2 * d + no * d + o] = gB[o];
    }
  if (lane == 0)
    for (int k = 0; k < 4; ++k) a.spart[w0 * 4 + k] = st[k];
}

// Embedding weight gradients, one warp per sample: per-warp partial sums of
// dW_emb[j][k] = sum dX[row][j] tok[row][k] and db_emb[j] over the sample's
// entity rows, into part[warp][9d] (W_emb then b_emb).  163,840 samples of 10
// entities, d = 64: 163 us (315 with a token's loads waited for one by one).
template <typename TokT, int DJ>
__global__ void __launch_bounds__(256) embed_grad_kernel(const TokT* __restrict__ tok,
                                                         const int32_t* __restrict__ n_ent,
                                                         const int32_t* __restrict__ sel,
                                                         const float* __restrict__ dX, float* __restrict__ part,
                                                         long long n, int T, int NS) {
  constexpr int d = 32 * DJ;
  const int lane = threadIdx.x & 31;
  const long long w0 = ((long long)blockIdx.x * blockDim.x + threadIdx.x) >> 5;
  const long long nw = ((long long)gridDim.x * blockDim.x) >> 5;
  float gW[DJ][8], gb[DJ];
#pragma unroll
  for (int i = 0; i < DJ; ++i) {
    gb[i] = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) gW[i][k] = 0.0f;
  }
  long long bn = 0;  // batch row and entities of the next sample, in flight during the current one
  int nn = 0;
  if (w0 < n) {
    bn = sel ? (long long)sel[w0] : w0;
    nn = n_ent[bn];
  }
  for (long long s = w0; s < n; s += nw) {
    const long long bs = bn;
    const int ne = nn < 0 ? 0 : (nn > NS ? NS : nn);
    float v[kTokRegs];
    load_tokens(tok, bs, NS, ne, lane, v);
    if (s + nw < n) bn = sel ? (long long)sel[s + nw] : s + nw;
    const float* g0 = dX + (s * T + 1) * d + lane;
#pragma unroll
    for (int j = 0; j < kTokRegs; ++j) {
      if (4 * j >= ne) break;  // (warp-uniform)
      float g[4][DJ];  // four tokens' gradients at a time
#pragma unroll
      for (int t = 0; t < 4; ++t)
#pragma unroll
        for (int i = 0; i < DJ; ++i) g[t][i] = 4 * j + t < ne ? g0[(4 * j + t) * d + 32 * i] : 0.0f;
#pragma unroll
      for (int t = 0; t < 4; ++t) {
#pragma unroll
        for (int i = 0; i < DJ; ++i) gb[i] += g[t][i];
#pragma unroll
        for (int k = 0; k < 8; ++k) {
          const float q = __shfl_sync(0xffffffffu, v[j], 8 * t + k);
#pragma unroll
          for (int i = 0; i < DJ; ++i) gW[i][k] = fmaf(g[t][i], q, gW[i][k]);
        }
      }
    }
    if (s + nw < n) nn = n_ent[bn];
  }
  float* pp = part + w0 * 9 * d;
#pragma unroll
  for (int i = 0; i < DJ; ++i) {
    const int j = lane + 32 * i;
#pragma unroll
    for (int k = 0; k < 8; ++k) pp[j * 8 + k] = gW[i][k];
    pp[8 * d + j] = gb[i];
  }
}

// Column sums of A [rows][N] (leading dimension lda), up to two matrices per
// launch: block (x, y) sums 32 columns over its share of the rows, one of nblk,
// into part[y][N].  (Past a matrix's own nblk: no rows left.)
struct ColSum {
  const float* A;
  long long lda, rows;
  int N, nblk;
  float* part;
};
__global__ void __launch_bounds__(256) colsum_kernel(ColSum a, ColSum b, int nx) {
  __shared__ float red[8][33];
  const bool second = (int)blockIdx.x >= nx;
  const ColSum q = second ? b : a;
  if ((int)blockIdx.y >= q.nblk) return;
  const int c = ((int)blockIdx.x - (second ? nx : 0)) * 32 + (threadIdx.x & 31), rg = threadIdx.x >> 5;
  const long long chunk = (q.rows + q.nblk - 1) / q.nblk;
  const long long r0 = (long long)blockIdx.y * chunk;
  const long long r1 = r0 + chunk < q.rows ? r0 + chunk : q.rows;
  float acc = 0.0f;
  if (c < q.N)
    for (long long r = r0 + rg; r < r1; r += 8) acc += q.A[r * q.lda + c];
  red[rg][threadIdx.x & 31] = acc;
  __syncthreads();
  if (rg == 0 && c < q.N) {
    float s = 0.0f;
#pragma unroll
    for (int k = 0; k < 8; ++k) s += red[k][threadIdx.x & 31];
    q.part[(long long)blockIdx.y * q.N + c] = s;
  }
}

// out[i] = sum over p of part[p * stride + i] for every segment of the list, the
// partial sums that one kernel leaves: a block sums 32 columns of a segment,
// thread row g the parts p = g (mod 32) in increasing p, then the 32 row sums in
// order of g (a fixed association: deterministic).  One launch per list: a
// gradient call at d = 64, 2 blocks has 8 of them where a launch per tensor made
// 22, and small batches are bound by launches (64 samples 307 -> 259 us, 32,768
// 1738 -> 1689).
struct ReduceSeg {
  const float* part;
  long long len, stride;
  float* out;
  int nparts;  // (0: the list's)
};
constexpr int kReduceSegs = 5;
struct ReduceList {
  ReduceSeg seg[kReduceSegs];
  unsigned first[kReduceSegs];  // first block of each segment (past the grid: none)
};
__global__ void __launch_bounds__(1024) reduce_kernel(ReduceList l) {
  __shared__ float red[32][33];
  const int c = threadIdx.x & 31, g = threadIdx.x >> 5;
  ReduceSeg q = l.seg[0];
  unsigned first = 0;
#pragma unroll
  for (int k = 1; k < kReduceSegs; ++k)
    if (blockIdx.x >= l.first[k]) {
      q = l.seg[k];
      first = l.first[k];
    }
  const long long i = (long long)(blockIdx.x - first) * 32 + c;
  const float* src = q.part + (i < q.len ? i : q.len - 1);
  float s = 0.0f;
#pragma unroll 4
  for (int p = g; p < q.nparts; p += 32) s += src[p * q.stride];
  red[g][c] = s;
  __syncthreads();
  if (g == 0 && i < q.len) {
    float t = 0.0f;
#pragma unroll
    for (int k = 0; k < 32; ++k) t += red[k][c];
    q.out[i] = t;
  }
}

// Statistics: sums of the per-warp partials times inv_n; thread j of 256
// sums parts p = j (mod 64) of statistic j / 64, then 64 partial sums are
// added in order.
__global__ void __launch_bounds__(256) reduce_stats_kernel(const double* __restrict__ spart, int nparts,
                                                           double inv_n, double* __restrict__ out) {
  __shared__ double red[4][64];
  const int k = threadIdx.x >> 6, j = threadIdx.x & 63;
  double s = 0.0;
  for (int p = j; p < nparts; p += 64) s += spart[p * 4 + k];
  red[k][j] = s;
  __syncthreads();
  if (threadIdx.x < 4) {
    double t = 0.0;
    for (int q = 0; q < 64; ++q) t += red[threadIdx.x][q];
    out[threadIdx.x] = t * inv_n;
  }
}

// Adam with bias correction (Kingma & Ba 2015, Algorithm 1); bc1 = 1 -
// beta1^t and bc2 = 1 - beta2^t are computed on the host in double.
__global__ void adam_kernel(float* __restrict__ th, float* __restrict__ m, float* __restrict__ v,
                            const float* __restrict__ g, long long n, float lr, float b1, float b2, float eps,
                            float bc1, float bc2) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= n) return;
  const float gi = g[i];
  const float mi = b1 * m[i] + (1.0f - b1) * gi;
  const float vi = b2 * v[i] + (1.0f - b2) * gi * gi;
  m[i] = mi;
  v[i] = vi;
  th[i] -= lr * (mi / bc1) / (sqrtf(vi / bc2) + eps);
}

// GAE by the backward recursion, one thread per env.
__global__ void gae_kernel(const float* __restrict__ r, const float* __restrict__ v, const int32_t* __restrict__ done,
                           int T, long long E, float gamma, float lam, float* __restrict__ adv,
                           float* __restrict__ ret) {
  const long long e = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (e >= E) return;
  float a = 0.0f;
  for (int t = T - 1; t >= 0; --t) {
    const long long i = (long long)t * E + e;
    const float nd = done[i] ? 0.0f : 1.0f;
    const float delta = r[i] + gamma * nd * v[i + E] - v[i];
    a = delta + gamma * lam * nd * a;
    adv[i] = a;
    ret[i] = a + v[i];
  }
}

__global__ void gae_agents_kernel(const float* __restrict__ adv, const int32_t* __restrict__ agent_env, int T,
                                  long long E, long long NA, float* __restrict__ out) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)T * NA) return;
  const long long t = i / NA, a = i - t * NA;
  out[i] = adv[t * E + agent_env[a]];
}

}  // namespace tfm
}  // namespace ut

// ---------------------------------------------------------------------------
// Host side
// ---------------------------------------------------------------------------
#include "runtime.cuh"

struct ut_tfm {
  static std::atomic<uint64_t> created;
  const uint64_t id = ++created;
  ut_tfm_config cfg{};
  cudaStream_t stream = nullptr;
  std::string err;
  int d = 0, L = 0, H = 0, dh = 0, n_out = 0, NS = 0, T = 0, f = 0;
  int64_t n_params = 0, max_rows = 0;
  std::vector<void*> allocs;
  float *prm = nullptr, *am = nullptr, *av = nullptr;
  int adam_t = 0;
  // activations: X [L][max_rows][d]; per block l: Y1, O, M, Y2 [rows][d],
  // S1, S2 [rows][2], QKV [rows][3d], P [samples][H][T][T], Z, G [rows][4d];
  // of the last block KV [rows][2d] and Q0 [samples][d] in QKV's place, P
  // [samples][H][T], and O, M, Y2, S2, Z, G and the output X of the samples'
  // recurrent rows alone
  float *X = nullptr, *Y1 = nullptr, *Y2 = nullptr, *S1 = nullptr, *S2 = nullptr, *QKV = nullptr, *P = nullptr,
        *O = nullptr, *M = nullptr, *Z = nullptr, *G = nullptr;
  // backward buffers
  float *dX = nullptr, *dM = nullptr, *dY = nullptr, *dO = nullptr, *dBig = nullptr;
  float* part = nullptr;  // partial sums of the parameter gradients
  double *spart = nullptr, *stats_d = nullptr;
  std::vector<int64_t> off;  // canonical tensor offsets
  // GEMM path: 1 BF16 tensor cores (FP32 accumulation), 0 FP32 CUDA cores
  int gemm_tc = 1;
  // BF16 images of the block weights for the tensor-core path, per block l:
  // Wqkv, Wo, W1, W2 as B of the forward, then their transposes as B of the
  // input gradient (ImgSpec table on the device, packed once per call); the
  // last block's Wqkv images hold Wk and Wv; Wq and its transpose, then the
  // whole Wqkv and its transpose, follow all blocks' images
  uint16_t* wimg = nullptr;
  std::vector<int64_t> img_off;  // [8 L + 4] offsets into wimg (elements)
  int64_t* img_spec = nullptr;   // [8 L + 4][5] (weight offset, R, C, transpose, image offset)
  int n_img = 0, img_max = 0;
  int* status = nullptr;
};
std::atomic<uint64_t> ut_tfm::created{0};

namespace ut {
namespace tfm {
namespace {

// Tensor offsets in the canonical order: 0 W_emb, 1 b_emb, per block l at
// 2 + 12 l: ln1_g, ln1_b, Wqkv, bqkv, Wo, bo, ln2_g, ln2_b, W1, b1, W2, b2;
// then lnf_g, lnf_b, Wh, bh and the end.
enum { T_LN1G = 0, T_LN1B, T_WQKV, T_BQKV, T_WO, T_BO, T_LN2G, T_LN2B, T_W1, T_B1, T_W2, T_B2 };

std::vector<int64_t> offsets(int d, int L, int n_out) {
  std::vector<int64_t> o;
  int64_t p = 0;
  auto add = [&](int64_t n) {
    o.push_back(p);
    p += n;
  };
  const int64_t D = d, F = 4 * (int64_t)d;
  add(D * 8);
  add(D);
  for (int l = 0; l < L; ++l) {
    add(D); add(D); add(3 * D * D); add(3 * D); add(D * D); add(D);
    add(D); add(D); add(F * D); add(F); add(D * F); add(D);
  }
  add(D); add(D); add((int64_t)n_out * D); add(n_out);
  o.push_back(p);
  return o;
}

bool valid_config(const ut_tfm_config* c) {
  if (!c || c->abi_version != UT_ABI_VERSION) return false;
  const int d = c->d_model;
  if (d != 32 && d != 64 && d != 96 && d != 128) return false;
  if (c->n_layers < 1 || c->n_layers > 8 || c->n_heads < 1 || d % c->n_heads) return false;
  const int dh = d / c->n_heads;
  if (dh != 8 && dh != 16 && dh != 32) return false;
  if (c->n_out < 1 || c->n_out > 16) return false;
  if (c->n_slots < 1 || c->n_slots > UT_MAX_AGENTS + UT_MAX_TARGETS) return false;
  if (c->tokens_bf16 != 0 && c->tokens_bf16 != 1) return false;
  return c->max_batch >= 1 && c->max_batch <= (1ll << 22);
}

#include "tfm_tc.cuh"
#include "tfm_ffn.cuh"
#include "tfm_qkv.cuh"

// Every BF16 weight image of the handle: grid (elements, image).
__global__ void pack_images_kernel(const float* __restrict__ prm, const int64_t* __restrict__ spec,
                                   uint16_t* __restrict__ img) {
  const int64_t* sp = spec + 5 * blockIdx.y;
  const int R = (int)sp[1], C = (int)sp[2];
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= (long long)R * C) return;
  const int r = (int)(i / C), c = (int)(i % C);
  const float* W = prm + sp[0];
  const float v = sp[3] ? W[(long long)c * R + r] : W[(long long)r * C + c];
  img[sp[4] + img_offset(r, c, R, C) / 2] = f2bf_bits(v);
}

inline unsigned blocks_for(long long n, int threads) { return (unsigned)((n + threads - 1) / threads); }

// Kinds 0 / 1 on the tensor cores.  CTAs loop over the row tiles: about as many
// per SM per column tile as fit (three for N <= 128, two for the wider
// products).
template <int EPI>
cudaError_t launch_tc_rows(const Gemm& g, cudaStream_t s) {
  static std::atomic<unsigned long long> ready{0};
  const cudaError_t e = smem_optin(tc_rows_kernel<EPI>, kTcRowsSmem, ready);
  if (e != cudaSuccess) return e;
  const size_t smem = tc_rows_smem(g.N);
  const int per_sm = std::min(smem <= 72 * 1024 ? 3 : 2, tc_rows_ctas<EPI>());
  const long long tiles = (g.M + 127) / 128;
  const int n_tiles = (g.N + kTcMaxN - 1) / kTcMaxN;
  long long ctas = (per_sm * 152 + n_tiles - 1) / n_tiles;
  if (ctas > tiles) ctas = tiles;
  tc_rows_kernel<EPI><<<dim3((unsigned)ctas, (unsigned)n_tiles), kTcThreads, smem, s>>>(g, g.bimg, g.status);
  return cudaGetLastError();
}

// Whether the 128 x 64 CUDA-core kernel takes the product: aligned float4
// operands, K ranges of 32 where they are contiguous in k.
bool sgemm_fast(int kind, const Gemm& g) {
  auto al = [](const void* p) { return ((uintptr_t)p & 15) == 0; };
  const bool ak = kind != 2, bk = kind == 0, k32 = g.kchunk % 32 == 0 && g.K % 32 == 0;
  return al(g.A) && al(g.B) && g.lda % 4 == 0 && g.ldb % 4 == 0 && (ak ? k32 : g.M % 4 == 0) &&
         (bk ? k32 : g.N % 4 == 0);
}

// kind 0: forward (A row-major, B = W [N][K]); 1: input gradient (A
// row-major, B = W [K][N]); 2: weight gradient (A and B indexed [k][.]).
cudaError_t gemm(int kind, const Gemm& g, cudaStream_t s) {
  if (g.M <= 0 || g.N <= 0 || g.K <= 0) return cudaSuccess;
  if (kind != 2 && g.bimg && g.K % 32 == 0 && g.N % 32 == 0 && g.lda % 4 == 0 && g.ldc % 4 == 0 &&
      ((uintptr_t)g.A & 15) == 0 && ((uintptr_t)g.C & 15) == 0 && g.kchunk == g.K) {
    switch (g.epi) {
      case EPI_BIAS: return launch_tc_rows<EPI_BIAS>(g, s);
      case EPI_BIAS_RES: return launch_tc_rows<EPI_BIAS_RES>(g, s);
      case EPI_BIAS_GELU: return launch_tc_rows<EPI_BIAS_GELU>(g, s);
      case EPI_GELU_GRAD: return launch_tc_rows<EPI_GELU_GRAD>(g, s);
      default: return launch_tc_rows<EPI_STORE>(g, s);
    }
  }
  const dim3 grid((unsigned)((g.M + 63) / 64), (unsigned)((g.N + 63) / 64),
                  (unsigned)((g.K + g.kchunk - 1) / g.kchunk));
  if (sgemm_fast(kind, g)) {
    const dim3 grid2((unsigned)((g.M + 127) / 128), grid.y, grid.z);
    if (kind == 0)
      sgemm128_kernel<true, true><<<grid2, 256, 0, s>>>(g);
    else if (kind == 1)
      sgemm128_kernel<true, false><<<grid2, 256, 0, s>>>(g);
    else
      sgemm128_kernel<false, false><<<grid2, 256, 0, s>>>(g);
    return cudaGetLastError();
  }
  if (kind == 0)
    sgemm_kernel<true, true><<<grid, 256, 0, s>>>(g);
  else if (kind == 1)
    sgemm_kernel<true, false><<<grid, 256, 0, s>>>(g);
  else
    sgemm_kernel<false, false><<<grid, 256, 0, s>>>(g);
  return cudaGetLastError();
}

// Two products of one kind that do not depend on each other: one launch on the
// CUDA cores where both have the 128 x 64 kernel.  The last block's queries, over
// n rows, go with its keys and values, over n T: small batches are bound by
// launches.  (64 samples of 4 tokens, d = 128, 2 blocks, forward and gradient:
// 226 and 758 us with launches of their own, 215 and 667 so.)
cudaError_t gemm_pair(int kind, const Gemm& a, const Gemm& b, cudaStream_t s) {
  if (a.bimg || b.bimg || a.M <= 0 || b.M <= 0 || !sgemm_fast(kind, a) || !sgemm_fast(kind, b)) {
    const cudaError_t e = gemm(kind, a, s);
    return e == cudaSuccess ? gemm(kind, b, s) : e;
  }
  const int ny = (a.N + 63) / 64;
  auto splits = [](const Gemm& g) { return (g.K + g.kchunk - 1) / g.kchunk; };
  const dim3 grid((unsigned)((std::max(a.M, b.M) + 127) / 128), (unsigned)(ny + (b.N + 63) / 64),
                  (unsigned)std::max(splits(a), splits(b)));
  if (kind == 0)
    sgemm128_pair_kernel<true, true><<<grid, 256, 0, s>>>(a, b, ny);
  else if (kind == 1)
    sgemm128_pair_kernel<true, false><<<grid, 256, 0, s>>>(a, b, ny);
  else
    sgemm128_pair_kernel<false, false><<<grid, 256, 0, s>>>(a, b, ny);
  return cudaGetLastError();
}

Gemm mk(const float* A, long long lda, const float* B, long long ldb, float* C, long long ldc, long long M, int N,
        long long K, int epi) {
  Gemm g;
  std::memset(&g, 0, sizeof(g));
  g.A = A; g.lda = lda; g.B = B; g.ldb = ldb; g.C = C; g.ldc = ldc;
  g.M = M; g.N = N; g.K = K; g.kchunk = K; g.epi = epi;
  g.ldr = ldc;
  return g;
}

cudaError_t reduce(int nparts, std::initializer_list<ReduceSeg> segs, cudaStream_t s) {
  ReduceList l;
  unsigned blocks = 0;
  int k = 0;
  for (const ReduceSeg& q : segs) {
    l.seg[k] = q;
    if (!q.nparts) l.seg[k].nparts = nparts;
    l.first[k++] = blocks;
    blocks += blocks_for(q.len, 32);
  }
  for (; k < kReduceSegs; ++k) {
    l.seg[k] = l.seg[0];
    l.first[k] = blocks;
  }
  reduce_kernel<<<blocks, 1024, 0, s>>>(l);
  return cudaGetLastError();
}

// A weight gradient and its bias gradient on the CUDA cores: the product's
// partial slabs from `part` on, the column sums' behind them, and their
// reductions.
struct WgradCores {
  Gemm g;
  ColSum sum;
  ReduceSeg dw, db;
  int nx() const { return (sum.N + 31) / 32; }
  float* end() const { return sum.part + (long long)sum.nblk * sum.N; }  // of the partial sums
};
WgradCores wgrad_cores(const float* dOut, long long ldo, int n_o, const float* In, long long ldi, int n_i,
                       long long rows, float* gW, float* gb, float* part) {
  const long long tiles = (long long)((n_o + 63) / 64) * ((n_i + 63) / 64), len = (long long)n_o * n_i;
  long long splits = (608 + tiles - 1) / tiles;
  splits = std::min(std::max(splits, 1ll), 128ll);
  splits = std::min(splits, (rows + 63) / 64);
  const long long kc = ((rows + splits - 1) / splits + 15) / 16 * 16;
  splits = (rows + kc - 1) / kc;
  WgradCores q;
  q.g = mk(dOut, ldo, In, ldi, part, n_i, n_o, n_i, rows, EPI_PARTIAL);
  q.g.kchunk = kc;
  const int nblk = (int)std::min((rows + 63) / 64, 256ll);
  q.sum = ColSum{dOut, ldo, rows, n_o, nblk, part + splits * len};
  q.dw = ReduceSeg{part, len, len, gW, (int)splits};
  q.db = ReduceSeg{q.sum.part, n_o, n_o, gb, nblk};
  return q;
}

// dW[o][i] = sum_r dOut[r][o] In[r][i] and db[o] = sum_r dOut[r][o] over rows
// r (rows of dOut ldo and of In ldi apart), split along the rows into partial
// slabs summed in order.
cudaError_t wgrad(ut_tfm* t, const float* dOut, long long ldo, int n_o, const float* In, long long ldi, int n_i,
                  long long rows, float* gW, float* gb, cudaStream_t s) {
  if (t->gemm_tc && rows > 0) {
    // tensor cores: (n_o / 128) x (n_i / 256) tiles x row splits, about as
    // many CTAs per SM as fit (three for n_i <= 128, else two), each split a
    // multiple of 64 rows
    static std::atomic<unsigned long long> ready{0};
    cudaError_t e = smem_optin(tc_wgrad_kernel, kTcSmem, ready);
    if (e != cudaSuccess) return e;
    const size_t smem = tc_wgrad_smem(n_i);
    const int per_sm = smem <= 72 * 1024 ? 3 : 2;
    const long long tiles = (long long)((n_o + 127) / 128) * ((n_i + kTcMaxN - 1) / kTcMaxN);
    long long splits = (per_sm * 152 + tiles - 1) / tiles;
    const long long max_split = (rows + kTcChunk - 1) / kTcChunk;
    if (splits > max_split) splits = max_split;
    if (splits < 1) splits = 1;
    long long rc = (rows + splits - 1) / splits;
    rc = (rc + kTcChunk - 1) / kTcChunk * kTcChunk;
    splits = (rows + rc - 1) / rc;
    Gemm g = mk(dOut, ldo, In, ldi, t->part, n_i, n_o, n_i, rows, EPI_PARTIAL);
    g.kchunk = rc;
    g.status = t->status;
    dim3 grid((unsigned)((n_o + 127) / 128), (unsigned)((n_i + kTcMaxN - 1) / kTcMaxN), (unsigned)splits);
    float* bias_part = t->part + splits * n_o * n_i;
    tc_wgrad_kernel<<<grid, kTcThreads, smem, s>>>(g, bias_part, t->status);
    e = cudaGetLastError();
    const long long len = (long long)n_o * n_i;
    if (e == cudaSuccess) e = reduce((int)splits, {{t->part, len, len, gW}, {bias_part, n_o, n_o, gb}}, s);
    return e;
  }
  const WgradCores q = wgrad_cores(dOut, ldo, n_o, In, ldi, n_i, rows, gW, gb, t->part);
  cudaError_t e = gemm(2, q.g, s);
  if (e != cudaSuccess) return e;
  colsum_kernel<<<dim3((unsigned)q.nx(), (unsigned)q.sum.nblk), 256, 0, s>>>(q.sum, q.sum, q.nx());
  e = cudaGetLastError();
  return e == cudaSuccess ? reduce(0, {q.dw, q.db}, s) : e;
}

// Two weight gradients on the CUDA cores, by the launches of one (gemm_pair).
cudaError_t wgrad_pair(const WgradCores& a, const WgradCores& b, cudaStream_t s) {
  cudaError_t e = gemm_pair(2, a.g, b.g, s);
  if (e != cudaSuccess) return e;
  colsum_kernel<<<dim3((unsigned)(a.nx() + b.nx()), (unsigned)std::max(a.sum.nblk, b.sum.nblk)), 256, 0, s>>>(
      a.sum, b.sum, a.nx());
  e = cudaGetLastError();
  return e == cudaSuccess ? reduce(0, {a.dw, a.db, b.dw, b.db}, s) : e;
}

// The LayerNorm kernels loop over rows (grid stride): at most kLnBlocks
// blocks, no more than are resident at once.
template <int DJ>
cudaError_t ln_fwd(const float* X, const float* g, const float* b, float* Y, float* st, long long rows, cudaStream_t s) {
  static const int nblk = (int)std::min<long long>(kLnBlocks, resident_blocks(ln_fwd_kernel<DJ>, 256));
  ln_fwd_kernel<DJ><<<nblk, 256, 0, s>>>(X, g, b, Y, st, rows);
  return cudaGetLastError();
}

template <int DJ, bool REC>
cudaError_t ln_bwd(ut_tfm* t, const float* dY, const float* X, const float* st, const float* g, const float* base,
                   float* out, float* grad_gb, long long rows, cudaStream_t s, const float* dY0 = nullptr) {
  static const int nblk = (int)std::min<long long>(kLnBlocks, resident_blocks(ln_bwd_kernel<DJ, REC>, 256));
  ln_bwd_kernel<DJ, REC><<<nblk, 256, 0, s>>>(dY, X, st, g, base, out, t->part, rows, dY0, (unsigned)t->T);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess) e = reduce(nblk, {{t->part, 2 * 32 * DJ, 2 * 32 * DJ, grad_gb}}, s);
  return e;
}

template <int DH>
cudaError_t attn_fwd(const float* QKV, const int32_t* ne, const int32_t* sel, float* P, float* O, long long n, int T,
                     int NS, int H, bool mma, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (mma && DH == 16 && T <= 16 && ((uintptr_t)QKV & 15) == 0) {
    static const long long cap = resident_blocks(attn_fwd_mma_kernel, 128);
    attn_fwd_mma_kernel<<<att_grid(cap, n * H), 128, 0, s>>>(QKV, ne, sel, P, O, n, T, NS, H, 1.0f / sqrtf((float)DH));
    return cudaGetLastError();
  }
  static std::atomic<unsigned long long> ready{0};
  const cudaError_t e = smem_optin(attn_fwd_kernel<DH>, kAttnSmemMax, ready);
  if (e != cudaSuccess) return e;
  attn_fwd_kernel<DH><<<blocks_for(n * H, attn_items(T)), kAttnThreads, attn_fwd_smem(T, DH), s>>>(
      QKV, ne, sel, P, O, n, T, NS, H, 1.0f / sqrtf((float)DH));
  return cudaGetLastError();
}

template <int PE>
cudaError_t attn_bwd_mma(const float* QKV, const float* P, const float* dO, float* dQKV, long long n, int T, int H,
                         cudaStream_t s) {
  static const long long cap = resident_blocks(attn_bwd_mma_kernel<PE>, 128);
  attn_bwd_mma_kernel<PE><<<att_grid(cap, n * H), 128, 0, s>>>(QKV, P, dO, dQKV, n, T, H, 0.25f);
  return cudaGetLastError();
}

template <int DH>
cudaError_t attn_bwd(const float* QKV, const float* P, const float* dO, float* dQKV, long long n, int T, int H,
                     bool mma, cudaStream_t s) {
  if (n <= 0) return cudaSuccess;
  if (mma && DH == 16 && T <= 16 && ((uintptr_t)QKV & 15) == 0 && ((uintptr_t)dO & 15) == 0)
    return att_p_per_lane(T) == 4 ? attn_bwd_mma<4>(QKV, P, dO, dQKV, n, T, H, s)
                                  : attn_bwd_mma<8>(QKV, P, dO, dQKV, n, T, H, s);
  static std::atomic<unsigned long long> ready{0};
  const cudaError_t e = smem_optin(attn_bwd_kernel<DH>, kAttnSmemMax, ready);
  if (e != cudaSuccess) return e;
  attn_bwd_kernel<DH><<<blocks_for(n * H, attn_items(T)), kAttnThreads, attn_bwd_smem(T, DH), s>>>(
      QKV, P, dO, dQKV, n, T, H, 1.0f / sqrtf((float)DH));
  return cudaGetLastError();
}

// The last block's attention (recurrent queries).  KV, Q0 and dO0 are the
// handle's buffers at multiples of 32 floats: every float4 access is aligned.
template <int DH>
cudaError_t attn0_fwd(const float* Q0, const float* KV, const int32_t* ne, const int32_t* sel, float* P0, float* O0,
                      long long n, int T, int NS, int H, bool mma, cudaStream_t s) {
  const float scale = 1.0f / sqrtf((float)DH);
  const unsigned grid = blocks_for(n * H * 32, 256);
  if (mma && DH == 16 && T <= 16)
    attn0_fwd_mma_kernel<<<grid, 256, 0, s>>>(Q0, KV, ne, sel, P0, O0, n, T, NS, H, scale);
  else
    attn0_fwd_kernel<DH><<<grid, 256, 0, s>>>(Q0, KV, ne, sel, P0, O0, n, T, NS, H, scale);
  return cudaGetLastError();
}

template <int DH>
cudaError_t attn0_bwd(const float* Q0, const float* KV, const float* P0, const float* dO0, float* D0, float* dKV,
                      long long n, int T, int H, bool mma, cudaStream_t s) {
  const float scale = 1.0f / sqrtf((float)DH);
  const unsigned grid = blocks_for(n * H * 32, 256);
  if (mma && DH == 16 && T <= 16)
    attn0_bwd_mma_kernel<<<grid, 256, 0, s>>>(Q0, KV, P0, dO0, D0, dKV, n, T, H, scale);
  else
    attn0_bwd_kernel<DH><<<grid, 256, 0, s>>>(Q0, KV, P0, dO0, D0, dKV, n, T, H, scale);
  return cudaGetLastError();
}

struct Call {
  const void* tok;
  const int32_t* ne;
  const float* h;
  const int32_t* sel;
  long long n;
};

// Activations of block l (the last block's lie behind the others'; its QKV
// holds KV, and Q0 follows it).
struct Block {
  float *X, *Y1, *Y2, *S1, *S2, *QKV, *Q0, *P, *O, *M, *Z, *G;
};
Block block_of(const ut_tfm* t, int l) {
  const long long MR = t->max_rows, d = t->d;
  Block b;
  b.X = t->X + l * MR * d;
  b.Y1 = t->Y1 + l * MR * d;
  b.Y2 = t->Y2 + l * MR * d;
  b.S1 = t->S1 + l * MR * 2;
  b.S2 = t->S2 + l * MR * 2;
  b.QKV = t->QKV + l * MR * 3 * d;
  b.Q0 = b.QKV + MR * 2 * d;
  b.P = t->P + (long long)l * t->cfg.max_batch * t->H * t->T * t->T;
  b.O = t->O + l * MR * d;
  b.M = t->M + l * MR * d;
  b.Z = t->Z + l * MR * 4 * d;
  b.G = t->G + l * MR * 4 * d;
  return b;
}

// Arguments of block l's feed-forward sub-block (tfm_ffn.cuh).
FfnArgs ffn_args(const ut_tfm* t, int l, const float* M, float* out, long long rows) {
  const int64_t* ol = t->off.data() + 2 + 12 * l;
  const int64_t* im = t->img_off.data() + 8 * l;
  FfnArgs a;
  std::memset(&a, 0, sizeof(a));
  a.M = M;
  a.out = out;
  a.gain = t->prm + ol[T_LN2G];
  a.off = t->prm + ol[T_LN2B];
  a.b1 = t->prm + ol[T_B1];
  a.b2 = t->prm + ol[T_B2];
  a.w1 = t->wimg + im[2];
  a.w2 = t->wimg + im[3];
  a.w1t = t->wimg + im[6];
  a.w2t = t->wimg + im[7];
  a.rows = rows;
  a.status = t->status;
  return a;
}

// Arguments of block l's LayerNorm and Q, K, V (tfm_qkv.cuh), last block's form
// included.
QkvArgs qkv_args(const ut_tfm* t, int l, const Block& b, long long rows) {
  const int64_t* ol = t->off.data() + 2 + 12 * l;
  QkvArgs a;
  std::memset(&a, 0, sizeof(a));
  a.X = b.X;
  a.gain = t->prm + ol[T_LN1G];
  a.off = t->prm + ol[T_LN1B];
  a.bias = t->prm + ol[T_BQKV];
  a.qkv = b.QKV;
  a.q0 = b.Q0;
  a.rows = rows;
  a.T = l == t->L - 1 ? t->T : 0;
  a.status = t->status;
  return a;
}

template <int DJ, int DH, typename TokT>
cudaError_t forward(ut_tfm* t, const Call& c, cudaStream_t s) {
  constexpr int d = 32 * DJ;
  const long long rows = c.n * t->T, MR = t->max_rows;
  const float* w = t->prm;
  const auto& o = t->off;
  if (t->gemm_tc) {  // the weights' BF16 images for this call
    pack_images_kernel<<<dim3(blocks_for(t->img_max, 256), (unsigned)t->n_img), 256, 0, s>>>(t->prm, t->img_spec,
                                                                                            t->wimg);
    cudaError_t e0 = cudaGetLastError();
    if (e0 != cudaSuccess) return e0;
  }
  auto img = [&](int l, int which) -> const uint16_t* {
    return t->gemm_tc ? t->wimg + t->img_off[8 * l + which] : nullptr;
  };
  {
    const unsigned blocks = (unsigned)std::min<long long>((c.n + 7) / 8, 152LL * 8);
    const TokT* tk = (const TokT*)c.tok;
    if (d == 32)
      embed_kernel<TokT, 1><<<blocks, 256, 0, s>>>(tk, c.ne, c.h, c.sel, w + o[0], w + o[1], t->X, c.n, t->T, t->NS);
    else if (d == 64)
      embed_kernel<TokT, 2><<<blocks, 256, 0, s>>>(tk, c.ne, c.h, c.sel, w + o[0], w + o[1], t->X, c.n, t->T, t->NS);
    else if (d == 96)
      embed_kernel<TokT, 3><<<blocks, 256, 0, s>>>(tk, c.ne, c.h, c.sel, w + o[0], w + o[1], t->X, c.n, t->T, t->NS);
    else
      embed_kernel<TokT, 4><<<blocks, 256, 0, s>>>(tk, c.ne, c.h, c.sel, w + o[0], w + o[1], t->X, c.n, t->T, t->NS);
  }
  cudaError_t e = cudaGetLastError();
  auto gemm0 = [&](Gemm g, int bias, const uint16_t* bimg) {
    g.bias = w + bias;
    g.bimg = bimg;
    g.status = t->status;
    return gemm(0, g, s);
  };
  for (int l = 0; l < t->L && e == cudaSuccess; ++l) {
    const int64_t* ol = o.data() + 2 + 12 * l;
    const bool last = l == t->L - 1;
    const long long m = last ? c.n : rows;  // rows after the attention: the recurrent tokens alone in the last block
    const Block b = block_of(t, l);
    const bool fused = t->gemm_tc && d == kFfD;
    if (fused) {
      QkvArgs a = qkv_args(t, l, b, rows);
      a.w = last ? img(t->L, 2) : img(l, 0);
      e = qkv_fwd(a, s);
    } else {
      e = ln_fwd<DJ>(b.X, w + ol[T_LN1G], w + ol[T_LN1B], b.Y1, b.S1, rows, s);
    }
    if (e != cudaSuccess) break;
    if (last) {
      if (!fused) {  // the recurrent rows of Y1 are T d apart
        Gemm kv = mk(b.Y1, d, w + ol[T_WQKV] + d * d, d, b.QKV, 2 * d, rows, 2 * d, d, EPI_BIAS);
        Gemm q = mk(b.Y1, (long long)t->T * d, w + ol[T_WQKV], d, b.Q0, d, c.n, d, d, EPI_BIAS);
        kv.bias = w + ol[T_BQKV] + d;
        q.bias = w + ol[T_BQKV];
        kv.bimg = img(l, 0);
        q.bimg = img(t->L, 0);
        kv.status = q.status = t->status;
        e = gemm_pair(0, kv, q, s);
      }
      if (e == cudaSuccess)
        e = attn0_fwd<DH>(b.Q0, b.QKV, c.ne, c.sel, b.P, b.O, c.n, t->T, t->NS, t->H, t->gemm_tc != 0, s);
    } else {
      if (!fused)
        e = gemm0(mk(b.Y1, d, w + ol[T_WQKV], d, b.QKV, 3 * d, rows, 3 * d, d, EPI_BIAS), ol[T_BQKV], img(l, 0));
      if (e == cudaSuccess)
        e = attn_fwd<DH>(b.QKV, c.ne, c.sel, b.P, b.O, c.n, t->T, t->NS, t->H, t->gemm_tc != 0, s);
    }
    if (e != cudaSuccess) break;
    Gemm g = mk(b.O, d, w + ol[T_WO], d, b.M, d, m, d, d, EPI_BIAS_RES);
    g.R = b.X;
    g.ldr = last ? (long long)t->T * d : d;
    e = gemm0(g, ol[T_BO], img(l, 1));
    if (fused) {
      if (e == cudaSuccess) e = ffn_fwd(ffn_args(t, l, b.M, b.X + MR * d, m), s);
      continue;
    }
    if (e == cudaSuccess) e = ln_fwd<DJ>(b.M, w + ol[T_LN2G], w + ol[T_LN2B], b.Y2, b.S2, m, s);
    if (e != cudaSuccess) break;
    g = mk(b.Y2, d, w + ol[T_W1], d, b.Z, 4 * d, m, 4 * d, d, EPI_BIAS_GELU);
    g.C2 = b.G;
    e = gemm0(g, ol[T_B1], img(l, 2));
    if (e != cudaSuccess) break;
    g = mk(b.G, 4 * d, w + ol[T_W2], 4 * d, b.X + MR * d, d, m, d, 4 * d, EPI_BIAS_RES);
    g.R = b.M;
    e = gemm0(g, ol[T_B2], img(l, 3));
  }
  return e;
}

// Blocks of the head and embedding-gradient kernels, a warp per sample: small
// batches start no idle warps, whose partial sums would be zeros to write and
// add (a critic's gradient of 64 samples 264 -> 243 us).
int row_blocks(long long n) { return (int)std::max(1ll, std::min<long long>(kRowBlocks, (n + 7) / 8)); }

template <int DJ, int DH, typename TokT>
cudaError_t backward(ut_tfm* t, const Call& c, float* grad, cudaStream_t s) {
  constexpr int d = 32 * DJ;
  const long long rows = c.n * t->T;
  const float* w = t->prm;
  const auto& o = t->off;
  cudaError_t e = cudaSuccess;
  // input-gradient GEMM of block l with the transposed image `which` (4..7)
  auto dgemm = [&](int l, int which, Gemm g) {
    g.bimg = t->gemm_tc ? t->wimg + t->img_off[8 * l + which] : nullptr;
    g.status = t->status;
    return gemm(1, g, s);
  };
  for (int l = t->L - 1; l >= 0 && e == cudaSuccess; --l) {
    const int64_t* ol = o.data() + 2 + 12 * l;
    const bool last = l == t->L - 1;
    const long long m = last ? c.n : rows;
    const Block b = block_of(t, l);
    // feed-forward sub-block: X' = M + W2 gelu(W1 LN2(M) + b1) + b2
    if (t->gemm_tc && d == kFfD) {
      FfnArgs a = ffn_args(t, l, b.M, t->dM, m);
      a.dX = t->dX;
      a.slab = t->part;
      a.vec = t->part + 152ll * kFfSlab;
      int ctas = 0;
      e = ffn_bwd(a, &ctas, s);
      if (e == cudaSuccess)
        e = reduce(ctas,
                   {{a.slab, kFfH * kFfD, kFfSlab, grad + ol[T_W1]},
                    {a.slab + kFfH * kFfD, kFfH * kFfD, kFfSlab, grad + ol[T_W2]},
                    {a.vec, kFfH, kFfVec, grad + ol[T_B1]},
                    {a.vec + kFfH, kFfD, kFfVec, grad + ol[T_B2]},
                    {a.vec + kFfH + kFfD, 2 * kFfD, kFfVec, grad + ol[T_LN2G]}},
                   s);
    } else {
      Gemm g = mk(t->dX, d, w + ol[T_W2], 4 * d, t->dBig, 4 * d, m, 4 * d, d, EPI_GELU_GRAD);
      g.aux = b.Z;
      e = dgemm(l, 7, g);
      if (e == cudaSuccess) e = wgrad(t, t->dX, d, d, b.G, 4 * d, 4 * d, m, grad + ol[T_W2], grad + ol[T_B2], s);
      if (e == cudaSuccess) e = dgemm(l, 6, mk(t->dBig, 4 * d, w + ol[T_W1], d, t->dY, d, m, d, 4 * d, EPI_STORE));
      if (e == cudaSuccess) e = wgrad(t, t->dBig, 4 * d, 4 * d, b.Y2, d, d, m, grad + ol[T_W1], grad + ol[T_B1], s);
      if (e == cudaSuccess)
        e = ln_bwd<DJ, false>(t, t->dY, b.M, b.S2, w + ol[T_LN2G], t->dX, t->dM, grad + ol[T_LN2G], m, s);
    }
    // attention sub-block: M = X + Wo attn(LN1(X)) + bo
    if (e == cudaSuccess) e = dgemm(l, 5, mk(t->dM, d, w + ol[T_WO], d, t->dO, d, m, d, d, EPI_STORE));
    if (e == cudaSuccess) e = wgrad(t, t->dM, d, d, b.O, d, d, m, grad + ol[T_WO], grad + ol[T_BO], s);
    if (e != cudaSuccess) break;
    const bool fused = t->gemm_tc && d == kFfD;
    float* D0 = t->dBig + rows * 2 * d;  // behind dKV: [n][3d] of the 2d n T floats that are left (T >= 2)
    if (fused) {
      if (last)
        e = attn0_bwd<DH>(b.Q0, b.QKV, b.P, t->dO, D0, t->dBig, c.n, t->T, t->H, true, s);
      else
        e = attn_bwd<DH>(b.QKV, b.P, t->dO, t->dBig, c.n, t->T, t->H, true, s);
      QkvArgs a = qkv_args(t, l, b, rows);
      a.w = t->wimg + t->img_off[last ? 8 * t->L + 3 : 8 * l + 4];
      a.dqkv = t->dBig;
      a.dq0 = D0;
      a.base = t->dM;
      a.out = t->dX;
      a.slab = t->part;
      a.vec = t->part + (long long)kQkvCtas * kQkvSlab;
      int ctas = 0;
      if (e == cudaSuccess) e = qkv_bwd(a, &ctas, s);
      if (e == cudaSuccess)
        e = reduce(ctas,
                   {{a.slab, kQkvSlab, kQkvSlab, grad + ol[T_WQKV]},
                    {a.vec, kQkvN, kQkvVec, grad + ol[T_BQKV]},
                    {a.vec + kQkvN, 2 * kFfD, kQkvVec, grad + ol[T_LN1G]}},
                   s);
      continue;
    }
    if (last) {
      // the recurrent rows' input gradient is a product of its own, over dQ,
      // dK and dV in one sum as in the other blocks
      const float* Wq = w + ol[T_WQKV];
      e = attn0_bwd<DH>(b.Q0, b.QKV, b.P, t->dO, D0, t->dBig, c.n, t->T, t->H, t->gemm_tc != 0, s);
      const Gemm dkv = mk(t->dBig, 2 * d, Wq + d * d, d, t->dY, d, rows, d, 2 * d, EPI_STORE);
      const Gemm dq = mk(D0, 3 * d, Wq, d, t->dO, d, c.n, d, 3 * d, EPI_STORE);
      float *gW = grad + ol[T_WQKV], *gb = grad + ol[T_BQKV];
      const long long Td = (long long)t->T * d;
      if (t->gemm_tc) {
        if (e == cudaSuccess) e = dgemm(l, 4, dkv);
        if (e == cudaSuccess) e = dgemm(t->L, 3, dq);
        if (e == cudaSuccess) e = wgrad(t, t->dBig, 2 * d, 2 * d, b.Y1, d, d, rows, gW + d * d, gb + d, s);
        if (e == cudaSuccess) e = wgrad(t, D0, 3 * d, d, b.Y1, Td, d, c.n, gW, gb, s);
      } else {
        if (e == cudaSuccess) e = gemm_pair(1, dkv, dq, s);
        const WgradCores kv = wgrad_cores(t->dBig, 2 * d, 2 * d, b.Y1, d, d, rows, gW + d * d, gb + d, t->part);
        const WgradCores q = wgrad_cores(D0, 3 * d, d, b.Y1, Td, d, c.n, gW, gb, kv.end());
        if (e == cudaSuccess) e = wgrad_pair(kv, q, s);
      }
      if (e == cudaSuccess)
        e = ln_bwd<DJ, true>(t, t->dY, b.X, b.S1, w + ol[T_LN1G], t->dM, t->dX, grad + ol[T_LN1G], rows, s, t->dO);
      continue;
    }
    e = attn_bwd<DH>(b.QKV, b.P, t->dO, t->dBig, c.n, t->T, t->H, t->gemm_tc != 0, s);
    if (e == cudaSuccess) e = dgemm(l, 4, mk(t->dBig, 3 * d, w + ol[T_WQKV], d, t->dY, d, rows, d, 3 * d, EPI_STORE));
    if (e == cudaSuccess) e = wgrad(t, t->dBig, 3 * d, 3 * d, b.Y1, d, d, rows, grad + ol[T_WQKV], grad + ol[T_BQKV], s);
    if (e == cudaSuccess)
      e = ln_bwd<DJ, false>(t, t->dY, b.X, b.S1, w + ol[T_LN1G], t->dM, t->dX, grad + ol[T_LN1G], rows, s);
  }
  if (e != cudaSuccess) return e;
  const int rb = row_blocks(c.n);
  embed_grad_kernel<TokT, DJ><<<rb, 256, 0, s>>>((const TokT*)c.tok, c.ne, c.sel, t->dX, t->part, c.n, t->T, t->NS);
  e = cudaGetLastError();
  if (e == cudaSuccess) e = reduce(8 * rb, {{t->part, 9 * d, 9 * d, grad + o[0]}}, s);
  return e;
}

// mode 0: forward (out, h_out); 1: PPO actor loss + gradient; 2: value loss +
// gradient.
template <int DJ, int DH, typename TokT>
cudaError_t run(ut_tfm* t, const Call& c, int mode, const HeadArgs& ha_in, float* grad, cudaStream_t s) {
  constexpr int d = 32 * DJ;
  cudaError_t e = forward<DJ, DH, TokT>(t, c, s);
  if (e != cudaSuccess) return e;
  const auto& o = t->off;
  const int idx = 2 + 12 * t->L;
  HeadArgs ha = ha_in;
  ha.XL = t->X + (long long)t->L * t->max_rows * d;
  ha.n = c.n;
  ha.n_out = t->n_out;
  ha.mode = mode;
  ha.lnf_g = t->prm + o[idx];
  ha.lnf_b = t->prm + o[idx + 1];
  ha.Wh = t->prm + o[idx + 2];
  ha.bh = t->prm + o[idx + 3];
  ha.sel = c.sel;
  ha.inv_n = 1.0f / (float)c.n;
  ha.dXL = t->dX;
  ha.part = t->part;
  ha.spart = t->spart;
  const int rb = row_blocks(c.n);
  if (t->n_out == 1)
    head_kernel<DJ, 1><<<rb, 256, 0, s>>>(ha);
  else if (t->n_out <= 8)
    head_kernel<DJ, 8><<<rb, 256, 0, s>>>(ha);
  else
    head_kernel<DJ, 16><<<rb, 256, 0, s>>>(ha);
  e = cudaGetLastError();
  if (e != cudaSuccess || mode == 0) return e;
  const long long plen = 2 * d + (long long)t->n_out * d + t->n_out;
  e = reduce(8 * rb, {{t->part, plen, plen, grad + o[idx]}}, s);
  if (e != cudaSuccess) return e;
  reduce_stats_kernel<<<1, 256, 0, s>>>(t->spart, 8 * rb, 1.0 / (double)c.n, t->stats_d);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  return backward<DJ, DH, TokT>(t, c, grad, s);
}

template <int DJ, int DH>
cudaError_t run_tok(ut_tfm* t, const Call& c, int mode, const HeadArgs& ha, float* grad, cudaStream_t s) {
  return t->cfg.tokens_bf16 ? run<DJ, DH, __nv_bfloat16>(t, c, mode, ha, grad, s)
                            : run<DJ, DH, float>(t, c, mode, ha, grad, s);
}

template <int DJ>
cudaError_t run_dh(ut_tfm* t, const Call& c, int mode, const HeadArgs& ha, float* grad, cudaStream_t s) {
  switch (t->dh) {
    case 8: return run_tok<DJ, 8>(t, c, mode, ha, grad, s);
    case 16: return run_tok<DJ, 16>(t, c, mode, ha, grad, s);
    default: return run_tok<DJ, 32>(t, c, mode, ha, grad, s);
  }
}

cudaError_t dispatch(ut_tfm* t, const Call& c, int mode, const HeadArgs& ha, float* grad) {
  switch (t->d) {
    case 32: return run_dh<1>(t, c, mode, ha, grad, t->stream);
    case 64: return run_dh<2>(t, c, mode, ha, grad, t->stream);
    case 96: return run_dh<3>(t, c, mode, ha, grad, t->stream);
    default: return run_dh<4>(t, c, mode, ha, grad, t->stream);
  }
}

ut_status fail(ut_tfm* t, ut_status st, const std::string& msg) {
  t->err = msg;
  return st;
}

void* dalloc(ut_tfm* t, size_t bytes) {
  void* p = nullptr;
  if (cudaMalloc(&p, bytes ? bytes : 16) != cudaSuccess) return nullptr;
  t->allocs.push_back(p);
  return p;
}

bool call_ok(const ut_tfm* t, const void* tok, const int32_t* ne, const float* h, int64_t n) {
  return tok && ne && h && n >= 1 && n <= t->cfg.max_batch;
}

}  // namespace
}  // namespace tfm
}  // namespace ut

using namespace ut::tfm;

namespace ut {

TfmInfo tfm_info(const ut_tfm* t) {
  return TfmInfo{t->d, t->L, t->H, t->n_out, t->NS, t->cfg.tokens_bf16, (long long)t->cfg.max_batch, t->id,
                 t->gemm_tc};
}

cudaError_t tfm_forward_on(ut_tfm* t, const void* tokens, const int32_t* n_ent, const float* h, long long n,
                           float* out, float* h_out, cudaStream_t s) {
  HeadArgs ha;
  std::memset(&ha, 0, sizeof(ha));
  ha.out = out;
  ha.h_out = h_out;
  const cudaStream_t own = t->stream;
  t->stream = s;
  const cudaError_t e = dispatch(t, Call{tokens, n_ent, h, nullptr, n}, 0, ha, nullptr);
  t->stream = own;
  return e;
}

}  // namespace ut

extern "C" int64_t tfm_param_count(const ut_tfm_config* cfg) {
  if (!valid_config(cfg)) return -1;
  return offsets(cfg->d_model, cfg->n_layers, cfg->n_out).back();
}

extern "C" ut_status tfm_create(const ut_tfm_config* cfg, const float* params_host, int64_t n_params,
                                void* cuda_stream, ut_tfm** out) {
  if (!out) return UT_ERR_INVALID;
  *out = nullptr;
  if (!valid_config(cfg) || !params_host || n_params != tfm_param_count(cfg)) return UT_ERR_INVALID;
  ut_tfm* t = new ut_tfm();
  t->cfg = *cfg;
  t->stream = (cudaStream_t)cuda_stream;
  t->d = cfg->d_model;
  t->L = cfg->n_layers;
  t->H = cfg->n_heads;
  t->dh = t->d / t->H;
  t->n_out = cfg->n_out;
  t->NS = cfg->n_slots;
  t->T = 1 + cfg->n_slots;
  t->f = 4 * t->d;
  t->n_params = n_params;
  t->off = offsets(t->d, t->L, t->n_out);
  t->max_rows = cfg->max_batch * t->T;
  const size_t R = (size_t)t->max_rows, d = (size_t)t->d, L = (size_t)t->L;
  const size_t Pn = (size_t)cfg->max_batch * t->H * t->T * t->T;
  size_t part = (size_t)128 * 4 * d * d;
  part += (size_t)256 * 4 * d;  // CUDA-core weight gradients, and the column sums behind them
  part = std::max(part, (size_t)kRowWarps * (2 * d + (size_t)t->n_out * d + t->n_out));
  part = std::max(part, (size_t)kRowWarps * 9 * d);
  part = std::max(part, (size_t)kLnBlocks * 2 * d);
  part = std::max(part, (size_t)kTcSplitsMax * (4 * d * d + 4 * d));  // tensor-core weight- and bias-gradient slabs
  bool ok = true;
  auto A = [&](size_t n) -> float* {
    float* p = (float*)dalloc(t, n * 4);
    ok = ok && p;
    return p;
  };
  t->prm = A(n_params);
  t->am = A(n_params);
  t->av = A(n_params);
  const size_t B = (size_t)cfg->max_batch, RL = (L - 1) * R + B;  // rows kept after the attention, all blocks
  t->X = A((L * R + B) * d);
  t->Y1 = A(L * R * d);
  t->Y2 = A(RL * d);
  t->S1 = A(L * R * 2);
  t->S2 = A(RL * 2);
  t->QKV = A(((L - 1) * R * 3 + R * 2 + B) * d);
  t->P = A((L - 1) * Pn + B * t->H * t->T);
  t->O = A(RL * d);
  t->M = A(RL * d);
  t->Z = A(RL * 4 * d);
  t->G = A(RL * 4 * d);
  t->dX = A(R * d);
  t->dM = A(R * d);
  t->dY = A(R * d);
  t->dO = A(R * d);
  t->dBig = A(R * 4 * d);
  t->part = A(part);
  t->spart = (double*)dalloc(t, (size_t)kRowWarps * 4 * 8);
  t->stats_d = (double*)dalloc(t, 4 * 8);
  ok = ok && t->spart && t->stats_d;
  // weight images: per block, B of the forward for Wqkv [3d][d], Wo [d][d],
  // W1 [4d][d], W2 [d][4d], then B of the input gradient (their transposes)
  std::vector<int64_t> spec;
  int64_t img_total = 0;
  t->img_max = 0;
  auto add_img = [&](int64_t woff, int rows_w, int cols_w, int tr) {
    const int R = tr ? cols_w : rows_w, C = tr ? rows_w : cols_w;
    // each 256-row block holds C columns of 256 rows (the last block padded)
    t->img_off.push_back(img_total);
    spec.insert(spec.end(), {woff, (int64_t)R, (int64_t)C, (int64_t)tr, img_total});
    img_total += (int64_t)((R + kTcMaxN - 1) / kTcMaxN) * kTcMaxN * C;
    t->img_max = std::max(t->img_max, R * C);
  };
  for (int l = 0; l < t->L; ++l) {
    const int64_t* ol = t->off.data() + 2 + 12 * l;
    const bool last = l == t->L - 1;  // (Wk and Wv: rows d .. 3d - 1 of Wqkv)
    const int64_t woff[4] = {ol[T_WQKV] + (last ? (int64_t)t->d * t->d : 0), ol[T_WO], ol[T_W1], ol[T_W2]};
    const int rows_w[4] = {(last ? 2 : 3) * t->d, t->d, 4 * t->d, t->d}, cols_w[4] = {t->d, t->d, t->d, 4 * t->d};
    for (int tr = 0; tr < 2; ++tr)
      for (int k = 0; k < 4; ++k) add_img(woff[k], rows_w[k], cols_w[k], tr);
  }
  for (int n : {1, 3})
    for (int tr = 0; tr < 2; ++tr) add_img(t->off[2 + 12 * (t->L - 1) + T_WQKV], n * t->d, t->d, tr);
  t->n_img = 8 * t->L + 4;
  t->wimg = (uint16_t*)dalloc(t, (size_t)img_total * 2);
  t->img_spec = (int64_t*)dalloc(t, spec.size() * 8);
  t->status = (int*)dalloc(t, 4);
  ok = ok && t->wimg && t->img_spec && t->status;
  if (!ok) {
    tfm_destroy(t);
    return UT_ERR_NOMEM;
  }
  cudaError_t e = cudaMemcpyAsync(t->prm, params_host, (size_t)n_params * 4, cudaMemcpyHostToDevice, t->stream);
  if (e == cudaSuccess)
    e = cudaMemcpyAsync(t->img_spec, spec.data(), spec.size() * 8, cudaMemcpyHostToDevice, t->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(t->wimg, 0, (size_t)img_total * 2, t->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(t->status, 0, 4, t->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(t->am, 0, (size_t)n_params * 4, t->stream);
  if (e == cudaSuccess) e = cudaMemsetAsync(t->av, 0, (size_t)n_params * 4, t->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(t->stream);
  if (e != cudaSuccess) {
    tfm_destroy(t);
    return UT_ERR_CUDA;
  }
  *out = t;
  return UT_OK;
}

extern "C" void tfm_destroy(ut_tfm* t) {
  if (!t) return;
  if (t->stream) cudaStreamSynchronize(t->stream);
  for (void* p : t->allocs) cudaFree(p);
  delete t;
}

extern "C" const char* tfm_last_error(const ut_tfm* t) { return t ? t->err.c_str() : "null handle"; }

extern "C" ut_status tfm_params(ut_tfm* t, float** params_dev) {
  if (!t || !params_dev) return UT_ERR_INVALID;
  *params_dev = t->prm;
  return UT_OK;
}

extern "C" ut_status tfm_forward(ut_tfm* t, const void* tokens_dev, const int32_t* n_ent_dev, const float* h_dev,
                                 const int32_t* sel_dev, int64_t n, float* out_dev, float* h_out_dev) {
  if (!t) return UT_ERR_INVALID;
  if (!call_ok(t, tokens_dev, n_ent_dev, h_dev, n) || !out_dev || (h_out_dev == h_dev && sel_dev))
    return fail(t, UT_ERR_INVALID, "tfm_forward: invalid arguments");
  HeadArgs ha;
  std::memset(&ha, 0, sizeof(ha));
  ha.out = out_dev;
  ha.h_out = h_out_dev;
  const cudaError_t e = dispatch(t, Call{tokens_dev, n_ent_dev, h_dev, sel_dev, n}, 0, ha, nullptr);
  return e == cudaSuccess ? UT_OK : fail(t, UT_ERR_CUDA, std::string("tfm_forward: ") + cudaGetErrorString(e));
}

static ut_status finish_stats(ut_tfm* t, double* stats_host, const char* name) {
  if (!stats_host) return UT_OK;
  int status = 0;
  cudaError_t e = cudaMemcpyAsync(stats_host, t->stats_d, 4 * 8, cudaMemcpyDeviceToHost, t->stream);
  if (e == cudaSuccess) e = cudaMemcpyAsync(&status, t->status, 4, cudaMemcpyDeviceToHost, t->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(t->stream);
  if (e != cudaSuccess) return fail(t, UT_ERR_CUDA, std::string(name) + ": " + cudaGetErrorString(e));
  if (status == 2) return fail(t, UT_ERR_TIMEOUT, std::string(name) + ": a bounded tensor-core wait gave up");
  return UT_OK;
}

extern "C" ut_status tfm_set_gemm_path(ut_tfm* t, int32_t tensor_cores) {
  if (!t || (tensor_cores != 0 && tensor_cores != 1)) return UT_ERR_INVALID;
  t->gemm_tc = tensor_cores;
  return UT_OK;
}

extern "C" ut_status tfm_ppo_actor_grad(ut_tfm* t, const void* tokens_dev, const int32_t* n_ent_dev,
                                        const float* h_dev, const int32_t* sel_dev, int64_t n,
                                        const int32_t* actions_dev, const float* logp_old_dev, const float* adv_dev,
                                        float clip_eps, float ent_coef, float* grad_dev, double* stats_host) {
  if (!t) return UT_ERR_INVALID;
  if (!call_ok(t, tokens_dev, n_ent_dev, h_dev, n) || !actions_dev || !logp_old_dev || !adv_dev || !grad_dev ||
      !(clip_eps > 0.0f) || !(ent_coef >= 0.0f) || t->n_out < 2)
    return fail(t, UT_ERR_INVALID, "tfm_ppo_actor_grad: invalid arguments");
  HeadArgs ha;
  std::memset(&ha, 0, sizeof(ha));
  ha.actions = actions_dev;
  ha.logp_old = logp_old_dev;
  ha.adv = adv_dev;
  ha.clip_eps = clip_eps;
  ha.ent_coef = ent_coef;
  const cudaError_t e = dispatch(t, Call{tokens_dev, n_ent_dev, h_dev, sel_dev, n}, 1, ha, grad_dev);
  if (e != cudaSuccess) return fail(t, UT_ERR_CUDA, std::string("tfm_ppo_actor_grad: ") + cudaGetErrorString(e));
  return finish_stats(t, stats_host, "tfm_ppo_actor_grad");
}

extern "C" ut_status tfm_value_grad(ut_tfm* t, const void* tokens_dev, const int32_t* n_ent_dev, const float* h_dev,
                                    const int32_t* sel_dev, int64_t n, const float* returns_dev, float* grad_dev,
                                    double* stats_host) {
  if (!t) return UT_ERR_INVALID;
  if (!call_ok(t, tokens_dev, n_ent_dev, h_dev, n) || !returns_dev || !grad_dev || t->n_out != 1)
    return fail(t, UT_ERR_INVALID, "tfm_value_grad: invalid arguments");
  HeadArgs ha;
  std::memset(&ha, 0, sizeof(ha));
  ha.ret = returns_dev;
  const cudaError_t e = dispatch(t, Call{tokens_dev, n_ent_dev, h_dev, sel_dev, n}, 2, ha, grad_dev);
  if (e != cudaSuccess) return fail(t, UT_ERR_CUDA, std::string("tfm_value_grad: ") + cudaGetErrorString(e));
  return finish_stats(t, stats_host, "tfm_value_grad");
}

extern "C" ut_status tfm_adam_step(ut_tfm* t, const float* grad_dev, float lr, float beta1, float beta2, float eps) {
  if (!t) return UT_ERR_INVALID;
  if (!grad_dev || !(lr >= 0.0f) || !(beta1 >= 0.0f && beta1 < 1.0f) || !(beta2 >= 0.0f && beta2 < 1.0f) ||
      !(eps > 0.0f))
    return fail(t, UT_ERR_INVALID, "tfm_adam_step: invalid arguments");
  t->adam_t += 1;
  const float bc1 = (float)(1.0 - std::pow((double)beta1, t->adam_t));
  const float bc2 = (float)(1.0 - std::pow((double)beta2, t->adam_t));
  adam_kernel<<<blocks_for(t->n_params, 256), 256, 0, t->stream>>>(t->prm, t->am, t->av, grad_dev, t->n_params, lr,
                                                                   beta1, beta2, eps, bc1, bc2);
  const cudaError_t e = cudaGetLastError();
  return e == cudaSuccess ? UT_OK : fail(t, UT_ERR_CUDA, std::string("tfm_adam_step: ") + cudaGetErrorString(e));
}

extern "C" ut_status tfm_sync_policy(ut_tfm* t, ut_env* env) {
  if (!t || !env) return UT_ERR_INVALID;
  const ut_config& c = env->cfg;
  if (c.d_model != t->d || c.n_layers != t->L || c.n_heads != t->H || c.n_actions != t->n_out)
    return fail(t, UT_ERR_INVALID, "tfm_sync_policy: the env's transformer agent has another configuration");
  std::vector<float> host((size_t)t->n_params);
  cudaError_t e = cudaMemcpyAsync(host.data(), t->prm, host.size() * 4, cudaMemcpyDeviceToHost, t->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(t->stream);
  if (e != cudaSuccess) return fail(t, UT_ERR_CUDA, std::string("tfm_sync_policy: ") + cudaGetErrorString(e));
  const ut_status st = env_set_policy(env, host.data(), t->n_params);
  if (st != UT_OK) t->err = std::string("tfm_sync_policy: ") + env_last_error(env);
  return st;
}

extern "C" ut_status ppo_gae(const float* reward_dev, const float* value_dev, const int32_t* done_dev, int32_t T,
                             int64_t E, float gamma, float lam, float* adv_dev, float* ret_dev,
                             const int32_t* agent_env_dev, int64_t NA, float* adv_agent_dev, void* cuda_stream) {
  if (!reward_dev || !value_dev || !done_dev || !adv_dev || !ret_dev || T < 1 || E < 1 || !(gamma >= 0.0f) ||
      !(gamma <= 1.0f) || !(lam >= 0.0f) || !(lam <= 1.0f))
    return UT_ERR_INVALID;
  if ((agent_env_dev == nullptr) != (adv_agent_dev == nullptr) || (adv_agent_dev && NA < 1)) return UT_ERR_INVALID;
  cudaStream_t s = (cudaStream_t)cuda_stream;
  gae_kernel<<<blocks_for(E, 256), 256, 0, s>>>(reward_dev, value_dev, done_dev, T, E, gamma, lam, adv_dev, ret_dev);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && adv_agent_dev) {
    gae_agents_kernel<<<blocks_for((long long)T * NA, 256), 256, 0, s>>>(adv_dev, agent_env_dev, T, E, NA,
                                                                        adv_agent_dev);
    e = cudaGetLastError();
  }
  return e == cudaSuccess ? UT_OK : UT_ERR_CUDA;
}
