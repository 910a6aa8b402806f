// First half of the training transformer's attention sub-block at d = 64, one
// kernel per direction (included by tfm.cu, inside namespace ut::tfm after
// tfm_ffn.cuh), tensor-core path:
//
//   forward   Q, K, V = Wqkv LN1(X) + bqkv
//   backward  dX from dQ, dK, dV and the residual path's gradient, and the
//             gradients of Wqkv, bqkv and the LayerNorm
//
// Both are bound by HBM: the forward reads X and writes Q, K, V (1 KB per token
// row; LayerNorm and GEMM as two kernels moved 1.5 KB), the backward reads dQ,
// dK, dV, X and the residual's gradient and writes dX (1.5 KB; input gradient,
// weight gradient and LayerNorm backward as three kernels moved 3.3 KB).  The
// LayerNorm output is made again in the backward; the staged gradient tile is
// the K-major operand of the input gradient and, read MN-major, the operand of
// the weight gradient, which accumulates in tensor memory over a CTA's tiles
// (tfm_ffn.cuh).  Two CTAs per SM hide each other's stages.  The arithmetic of
// every value is that of the separate kernels.  1.80 M rows: forward 309 us (6.0
// TB/s; as LayerNorm and GEMM about 450), backward 0.70 ms (3.9 TB/s; as four
// kernels 1.3); what holds the backward is the latency of its staging, half of
// a tile's cycles.
//
// T > 0 marks the last block: dQ and Q are kept for the recurrent rows alone
// (row s T at s), K and V as [rows][128], and the residual's gradient is zero
// outside the recurrent rows.
#pragma once

constexpr int kQkvN = 3 * kFfD;
constexpr size_t kQkvW = (size_t)kQkvN * kFfD * 2;            // weight image (24 KB)
constexpr size_t kQkvE = (size_t)128 * 64 * 4;                // staging tile (32 KB)
constexpr size_t kQkvFwdSmem = kQkvW + kRowA + 2 * kQkvE;     // 104 KB
constexpr size_t kQkvBwdSmem = kQkvW + 3 * kFfA + kRowA;      // 88 KB
constexpr int kQkvSlab = kQkvN * kFfD;                        // per-CTA partials: dWqkv
constexpr int kQkvVec = kQkvN + 2 * kFfD;                     // and dbqkv, d(ln1 gain), d(ln1 offset)

struct QkvArgs {
  const float* X;            // [rows][64]
  const float *gain, *off, *bias;
  const uint16_t* w;         // image of Wqkv (forward) or its transpose (backward)
  float *qkv, *q0;           // forward: [rows][192], or K, V [rows][128] and Q [n][64]
  const float *dqkv, *dq0;   // backward: dQ, dK, dV [rows][192], or dK, dV [rows][128] and dQ (rows of [n][192])
  const float* base;         // residual's gradient [rows][64] or [n][64]
  float* out;                // dX [rows][64]
  float *slab, *vec;
  long long rows;
  int T;                     // 0, or tokens per sample of the last block
  int* status;
};

__global__ void __launch_bounds__(256, 2) qkv_fwd_kernel(QkvArgs a) {
  extern __shared__ __align__(128) unsigned char sm_tile[];
  unsigned char* sW = sm_tile;
  unsigned char* sY = sW + kQkvW;
  float* sE = reinterpret_cast<float*>(sY + kRowA);  // two staging tiles
  __shared__ __align__(8) uint64_t bars[2];         // products, weights
  __shared__ uint32_t tbase;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, row = tid & 127, half = tid >> 7;
  if (warp == 0) {
    tc::tmem_alloc(&tbase, 256);
    tc::tmem_relinquish();
  }
  if (tid == 32) {
    tc::mbar_init(&bars[0], 1);
    tc::mbar_init(&bars[1], 1);
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tbase, tl = tmem + ((uint32_t)(warp & 3) << 21);
  const uint32_t aY = tc::smem_addr(sY), aW = tc::smem_addr(sW);
  if (tid == 0) {
    tc::mbar_expect_tx(&bars[1], (uint32_t)kQkvW);
    tc::bulk_g2s(sW, a.w, (uint32_t)kQkvW, &bars[1]);
  }
  const float g0 = a.gain[lane], g1 = a.gain[lane + 32], f0 = a.off[lane], f1 = a.off[lane + 32];
  const long long tiles = (a.rows + 127) / 128;
  Bar done{&bars[0], 0};
  bool ok = true, first = true;
  float x[16][2];
  auto fetch = [&](long long mt) {
    // (rows past the end repeat the last one: nothing of theirs is stored)
    const long long r0 = mt * 128 + warp * 16;
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const float* src = a.X + min(r0 + i, a.rows - 1) * 64 + lane;
      x[i][0] = __ldg(src);
      x[i][1] = __ldg(src + 32);
    }
  };
  fetch(blockIdx.x);
  for (long long mt = blockIdx.x; mt < tiles; mt += gridDim.x, first = false) {
    {
      float rs[16];
      rows_normalise(x, rs);
#pragma unroll
      for (int i = 0; i < 16; i += 2) {
        st_bf_rows(sY, kRowGrp, warp * 16 + i, 0, x[i][0] * g0 + f0, x[i + 1][0] * g0 + f0);
        st_bf_rows(sY, kRowGrp, warp * 16 + i, 32, x[i][1] * g1 + f1, x[i + 1][1] * g1 + f1);
      }
    }
    fetch(mt + gridDim.x);  // in flight during this tile's product and stores
    ffn_publish();
    if (tid == 0) {
      if (first) ok &= tc::mbar_wait(&bars[1], 0u, kTcPolls);
      constexpr uint32_t idesc = tc::idesc_bf16(128, kQkvN);
      const uint64_t ad = tc::smem_desc(aY, kRowGrp, 128), bd = tc::smem_desc(aW, kQkvN * 16, 128);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        tc::mma_bf16(tmem, tc::desc_advance(ad, j * 2 * kRowGrp), tc::desc_advance(bd, j * 2 * kQkvN * 16), idesc,
                     j > 0 ? 1u : 0u);
      tc::mma_commit(&bars[0]);
    }
    ok &= done.wait();
    tc::fence_after_sync();
    ok = __syncthreads_and(ok);  // (the tensor-memory loads below are warp-collective)
    if (!ok) break;
#pragma unroll 1
    for (int j = 0; j < 3; ++j) {  // Q, K, V
      float* e = sE + (j & 1) * (128 * 64);
      {
        float v[32];
        tc::tmem_ld32(tl + 64 * j + half * 32, v);
#pragma unroll
        for (int k = 0; k < 8; ++k)
          *reinterpret_cast<float4*>(e + epi_pos(row, half * 8 + k)) =
              make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
      }
      tc::fence_before_sync();
      __syncthreads();
      tc::fence_after_sync();
      const int c4 = tid & 15;
      const float4 b = __ldg(reinterpret_cast<const float4*>(a.bias + 64 * j) + c4);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = (tid >> 4) + 16 * i;
        const long long m = mt * 128 + r;
        if (m >= a.rows) break;
        const float4 v = *reinterpret_cast<const float4*>(e + epi_pos(r, c4));
        float* dst;
        if (a.T == 0) {
          dst = a.qkv + m * 192 + 64 * j;
        } else if (j > 0) {
          dst = a.qkv + m * 128 + 64 * (j - 1);
        } else {
          const unsigned s = (unsigned)m / (unsigned)a.T;  // (rows < 2^32)
          if (m != (long long)s * a.T) continue;
          dst = a.q0 + (long long)s * 64;
        }
        reinterpret_cast<float4*>(dst)[c4] = make_float4(v.x + b.x, v.y + b.y, v.z + b.z, v.w + b.w);
      }
      // (a staging tile is written again two blocks later, behind a barrier)
    }
  }
  if (!ok && tid == 0) {  // no weight copy may still be landing when the CTA exits
    tc::mbar_wait(&bars[1], 0u, kTcPolls);
    raise_status(a.status, 2);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 256);
}

__global__ void __launch_bounds__(256, 2) qkv_bwd_kernel(QkvArgs a) {
  extern __shared__ __align__(128) unsigned char sm_tile[];
  unsigned char* sW = sm_tile;       // Wqkv^T [192 / 8][64][8]
  unsigned char* sD = sW + kQkvW;    // dQ, dK, dV operand [192 / 8][128][8]
  unsigned char* sY = sD + 3 * kFfA; // LayerNorm output (and, read as features 192 .. 255 of sD, ignored rows)
  float* sE = reinterpret_cast<float*>(sD);  // staging [128][64] of dY, once every MMA has read sD
  __shared__ __align__(8) uint64_t bars[2];  // products, weights
  __shared__ uint32_t tbase;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, row = tid & 127, half = tid >> 7;
  if (warp == 0) {
    tc::tmem_alloc(&tbase, 256);
    tc::tmem_relinquish();
  }
  if (tid == 32) {
    tc::mbar_init(&bars[0], 1);
    tc::mbar_init(&bars[1], 1);
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tbase, tl = tmem + ((uint32_t)(warp & 3) << 21);
  const uint32_t aY = tc::smem_addr(sY), aD = tc::smem_addr(sD), aW = tc::smem_addr(sW);
  constexpr uint32_t kDw = 0, kDy = 128;  // dWqkv of features 0 .. 127, 128 .. 191 (64 columns each); dY
  if (tid == 0) {
    tc::mbar_expect_tx(&bars[1], (uint32_t)kQkvW);
    tc::bulk_g2s(sW, a.w, (uint32_t)kQkvW, &bars[1]);
  }
  const float g0 = a.gain[lane], g1 = a.gain[lane + 32], f0 = a.off[lane], f1 = a.off[lane + 32];
  float pg[2] = {0.0f, 0.0f}, pb[2] = {0.0f, 0.0f};
  float pbias[6] = {0.f, 0.f, 0.f, 0.f, 0.f, 0.f};  // dbqkv: see the staging
  const long long tiles = (a.rows + 127) / 128;
  Bar done{&bars[0], 0};
  bool ok = true, first = true;
  const int r8 = lane & 7, q4 = lane >> 3;
  for (long long mt = blockIdx.x; mt < tiles; mt += gridDim.x, first = false) {
    const long long r0 = mt * 128 + warp * 16;
    // the warp's 16 rows of dQ, dK, dV: lane = row r8 (+ 8) x 8 columns of a
    // 32-column block, so a load touches whole sectors of 8 rows and the
    // 16-byte operand stores are free of conflicts; pbias[b] collects column
    // 32 b + 8 q4 + bitrev(r8) (a lane keeps one of 8 columns per halving).
    // Every load is made, from a row that exists, and what does not belong to
    // the tile is zeroed afterwards: the loads of three blocks stay in flight
    // together (behind branches each waited for itself, 12 k cycles a tile).
    const float *pq[2], *pk[2];  // the lane's columns of Q, and of K and V, in its two rows
    bool vk[2], vq[2];
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const long long m = r0 + r8 + 8 * i, mc = m < a.rows ? m : a.rows - 1;
      vk[i] = m < a.rows;
      if (a.T == 0) {
        pq[i] = a.dqkv + mc * 192 + 8 * q4;
        pk[i] = pq[i] + 64;
        vq[i] = vk[i];
      } else {
        const unsigned smp = (unsigned)mc / (unsigned)a.T;  // (rows < 2^32)
        pq[i] = a.dq0 + (long long)smp * 192 + 8 * q4;
        pk[i] = a.dqkv + mc * 128 + 8 * q4;
        vq[i] = vk[i] && mc == (long long)smp * a.T;
      }
    }
    float xh[16][2], rs[16];
#pragma unroll
    for (int b0 = 0; b0 < 6; b0 += 3) {
      float4 u[3][2][2];  // block, row, half of the 8 columns
#pragma unroll
      for (int h = 0; h < 3; ++h) {
        const int b = b0 + h;
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const float4* src = reinterpret_cast<const float4*>(b < 2 ? pq[i] + 32 * b : pk[i] + 32 * (b - 2));
          u[h][i][0] = __ldg(src);
          u[h][i][1] = __ldg(src + 1);
        }
      }
      if (b0 == 3) {  // the rows of X behind the last gradients
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          const long long mc = r0 + i < a.rows ? r0 + i : a.rows - 1;
          xh[i][0] = __ldg(a.X + mc * 64 + lane);
          xh[i][1] = __ldg(a.X + mc * 64 + lane + 32);
        }
      }
#pragma unroll
      for (int h = 0; h < 3; ++h) {
        const int b = b0 + h, col = 32 * b + 8 * q4;
        float s[8];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const bool on = b < 2 ? vq[i] : vk[i];
          float v[8] = {u[h][i][0].x, u[h][i][0].y, u[h][i][0].z, u[h][i][0].w,
                        u[h][i][1].x, u[h][i][1].y, u[h][i][1].z, u[h][i][1].w};
#pragma unroll
          for (int k = 0; k < 8; ++k) {
            v[k] = on ? v[k] : 0.0f;
            s[k] = i ? s[k] + v[k] : v[k];
          }
          st8_bf(sD, warp * 16 + r8 + 8 * i, col, v);
        }
        float t4[4], t2[2];
#pragma unroll
        for (int k = 0; k < 4; ++k)
          t4[k] = ((lane & 1) ? s[k + 4] : s[k]) + __shfl_xor_sync(0xffffffffu, (lane & 1) ? s[k] : s[k + 4], 1);
#pragma unroll
        for (int k = 0; k < 2; ++k)
          t2[k] = ((lane & 2) ? t4[k + 2] : t4[k]) + __shfl_xor_sync(0xffffffffu, (lane & 2) ? t4[k] : t4[k + 2], 2);
        pbias[b] += ((lane & 4) ? t2[1] : t2[0]) + __shfl_xor_sync(0xffffffffu, (lane & 4) ? t2[0] : t2[1], 4);
      }
    }
    rows_normalise(xh, rs);
#pragma unroll
    for (int i = 0; i < 16; i += 2) {
      st_bf_rows(sY, kRowGrp, warp * 16 + i, 0, xh[i][0] * g0 + f0, xh[i + 1][0] * g0 + f0);
      st_bf_rows(sY, kRowGrp, warp * 16 + i, 32, xh[i][1] * g1 + f1, xh[i + 1][1] * g1 + f1);
    }
    ffn_publish();
    if (tid == 0) {
      if (first) ok &= tc::mbar_wait(&bars[1], 0u, kTcPolls);
      constexpr uint32_t idesc = tc::idesc_bf16(128, 64);
      const uint64_t ad = tc::smem_desc(aD, 128 * 16, 128), bd = tc::smem_desc(aW, 64 * 16, 128);
#pragma unroll
      for (int j = 0; j < kQkvN / 16; ++j)
        tc::mma_bf16(tmem + kDy, tc::desc_advance(ad, j * 2 * 128 * 16), tc::desc_advance(bd, j * 2 * 64 * 16), idesc,
                     j > 0 ? 1u : 0u);
      ffn_mma_rows(tmem + kDw, aD, aY, !first);
      ffn_mma_rows(tmem + kDw + 64, aD + 16 * 2048, aY, !first);
      tc::mma_commit(&bars[0]);
    }
    // the rows of the tile after the next into L2 meanwhile, a 128-byte line per
    // thread and turn (two launches of 1.8 M rows: 1399 us, the next tile's 1492)
    {
      const long long nm = (mt + 2 * gridDim.x) * 128, w = a.T ? 128 : 192;
      const long long lines = (a.rows - nm < 128 ? a.rows - nm : 128) * w / 32;  // (none past the last tile)
      for (long long i = tid; i < lines; i += 256)
        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.dqkv + nm * w + i * 32));
      for (long long i = tid; i < lines * 64 / w; i += 256) {
        asm volatile("prefetch.global.L2 [%0];" ::"l"(a.X + nm * 64 + i * 32));
        if (a.T == 0) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.base + nm * 64 + i * 32));
      }
    }
    ok &= done.wait();
    tc::fence_after_sync();
    ok = __syncthreads_and(ok);  // (the tensor-memory loads below are warp-collective)
    if (!ok) break;
    {
      float v[32];
      tc::tmem_ld32(tl + kDy + half * 32, v);
#pragma unroll
      for (int k = 0; k < 8; ++k)
        *reinterpret_cast<float4*>(sE + epi_pos(row, half * 8 + k)) =
            make_float4(v[4 * k], v[4 * k + 1], v[4 * k + 2], v[4 * k + 3]);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    // sample and token of the warp's first row (last block's form)
    unsigned smp = a.T ? (unsigned)r0 / (unsigned)a.T : 0u, tok = a.T ? (unsigned)r0 - smp * (unsigned)a.T : 0u;
#pragma unroll
    for (int h = 0; h < 16; h += 8) {
      float y[8][2], res[8][2];  // (all of the residual's loads before the first store)
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const long long m = r0 + h + i, mc = m < a.rows ? m : a.rows - 1;
        const float* b = a.base + (a.T ? (long long)(m < a.rows ? smp : 0u) : mc) * 64 + lane;
        const bool on = a.T == 0 || tok == 0;
        res[i][0] = __ldg(b);
        res[i][1] = __ldg(b + 32);
        if (!on) res[i][0] = res[i][1] = 0.0f;
        if (a.T && ++tok == (unsigned)a.T) {
          tok = 0;
          ++smp;
        }
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const int r = warp * 16 + h + i;
        y[i][0] = sE[epi_pos(r, lane >> 2) + (lane & 3)];
        y[i][1] = sE[epi_pos(r, 8 + (lane >> 2)) + (lane & 3)];
      }
      rows_ln_bwd(y, xh + h, rs + h, res, g0, g1, pg, pb);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        const long long m = r0 + h + i;
        if (m < a.rows) {
          a.out[m * 64 + lane] = y[i][0];
          a.out[m * 64 + lane + 32] = y[i][1];
        }
      }
    }
    __syncthreads();  // the staging tile is read: the next tile's gradients go over it
  }
  if (ok) {
    float* slab = a.slab + (long long)blockIdx.x * kQkvSlab;
    // lane = feature: 0 .. 127 (half 0) and 128 .. 191 (half 1)
    const int feat = half * 128 + row;
#pragma unroll 1
    for (int c0 = 0; c0 < 64; c0 += 16) {
      float v[16];
      tc::tmem_ld16(tl + kDw + half * 64 + c0, v);
      if (feat < kQkvN) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          *reinterpret_cast<float4*>(slab + feat * 64 + c0 + 4 * j) =
              make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
      }
    }
    // vector gradients over the 8 warps, in order
    float* s_l = sE;  // [8][kQkvVec]
    float* l = s_l + warp * kQkvVec;
    const int rev = ((r8 & 1) << 2) | (r8 & 2) | (r8 >> 2);
#pragma unroll
    for (int b = 0; b < 6; ++b) l[32 * b + 8 * q4 + rev] = pbias[b];
    l[kQkvN + lane] = pg[0];
    l[kQkvN + 32 + lane] = pg[1];
    l[kQkvN + 64 + lane] = pb[0];
    l[kQkvN + 96 + lane] = pb[1];
    __syncthreads();
    float* vec = a.vec + (long long)blockIdx.x * kQkvVec;
    for (int i = tid; i < kQkvVec; i += 256) {
      float t = 0.0f;
#pragma unroll
      for (int w = 0; w < 8; ++w) t += s_l[w * kQkvVec + i];
      vec[i] = t;
    }
  } else if (tid == 0) {  // no weight copy may still be landing when the CTA exits
    tc::mbar_wait(&bars[1], 0u, kTcPolls);
    raise_status(a.status, 2);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 256);
}

constexpr int kQkvCtas = 2 * 152;

cudaError_t qkv_fwd(const QkvArgs& a, cudaStream_t s) {
  static std::atomic<unsigned long long> ready{0};
  const cudaError_t e = smem_optin(qkv_fwd_kernel, kQkvFwdSmem, ready);
  if (e != cudaSuccess) return e;
  qkv_fwd_kernel<<<(unsigned)std::min<long long>((a.rows + 127) / 128, kQkvCtas), 256, kQkvFwdSmem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t qkv_bwd(const QkvArgs& a, int* ctas, cudaStream_t s) {
  static std::atomic<unsigned long long> ready{0};
  const cudaError_t e = smem_optin(qkv_bwd_kernel, kQkvBwdSmem, ready);
  if (e != cudaSuccess) return e;
  *ctas = (int)std::min<long long>((a.rows + 127) / 128, kQkvCtas);
  qkv_bwd_kernel<<<(unsigned)*ctas, 256, kQkvBwdSmem, s>>>(a);
  return cudaGetLastError();
}
