// Feed-forward sub-block of the training transformer at d = 64 in one kernel
// per direction (included by tfm.cu, inside namespace ut::tfm after
// tfm_tc.cuh), tensor-core path:
//
//   forward   X' = M + W2 gelu(W1 LN2(M) + b1) + b2
//   backward  dM from dX' and every parameter gradient of the sub-block
//
// As separate kernels it moved 11.8 KB per token row through HBM (the LayerNorm
// output, the 4d-wide pre-activations, GELU outputs and their gradients, each
// FP32 and read up to three times).  Here a 128-row tile stays on chip: the
// forward reads M and writes X' (512 B per row), the backward reads M and dX',
// makes the LayerNorm output and the pre-activations again (the same MMAs and
// arithmetic, the same bits) and writes dM (768 B per row); its weight
// gradients accumulate in tensor memory over all of a CTA's tiles.  What
// bounds both is the CUDA cores' work per hidden value (erf, and in the
// backward the exponential of its derivative; issue 69 % active forward, 60 %
// backward) and the chain of stages within a tile.  1.97 M rows (163,840 samples' two blocks): forward 0.77 ms, backward
// 1.46 ms; the actor's gradient step 14.3 -> 10.4 ms, the critic's (32,768
// samples) 3.24 -> 2.33.  It also serves small calls: 5 launches and 5
// reductions become 1 and 5.
//
// The arithmetic of every value is that of the separate kernels (ln_fwd,
// tc_rows with its epilogues, ln_bwd); only the sums over token rows of the
// parameter gradients associate differently.
//
// An operand tile of 128 token rows is stored [feature / 8][row][8] BF16
// (K-major, tc.cuh).  Read with the MN-major descriptor (8-row groups 128 B
// apart along K, 8-feature groups 2048 B apart) the same bytes are its
// transpose, so one image serves the product over features and the weight
// gradient over rows.
#pragma once

constexpr int kFfD = 64, kFfH = 256;                 // width, hidden width
constexpr size_t kFfW = (size_t)kFfD * kFfH * 2;     // one weight image (32 KB)
constexpr size_t kFfA = (size_t)128 * 64 * 2;        // operand tile of 64 features (16 KB)
// Tiles written a row per warp have their 8-feature groups 2048 + 32 bytes
// apart: the four groups of a store fall into different banks.  (Not in the
// forward here, where 112 KB is the most that two CTAs per SM can have.)
constexpr uint32_t kRowGrp = 2048 + 32;
constexpr size_t kRowA = 8 * (size_t)kRowGrp;
constexpr size_t kFfFwdSmem = 2 * kFfW + 3 * kFfA;  // W1, W2; Y2, two G chunks
constexpr size_t kFfBwdSmem = 3 * kFfW + 2 * kRowA + 4 * kFfA + 128 * 64 * 4;  // 224 KB, one CTA per SM
constexpr int kFfSlab = 2 * kFfD * kFfH;             // per-CTA partials: dW1 [256][64], dW2 [64][256]
constexpr int kFfVec = kFfH + 3 * kFfD;              // and db1, db2, d(ln2 gain), d(ln2 offset)
constexpr uint32_t kMnMajorA = 1u << 15, kMnMajorB = 1u << 16;  // instruction descriptor: transposed operands

struct FfnArgs {
  const float* M;    // [rows][64]
  const float* dX;   // [rows][64] (backward)
  float* out;        // X' or dM
  const float *gain, *off, *b1, *b2;
  const uint16_t *w1, *w2;    // images of W1, W2 (forward)
  const uint16_t *w2t, *w1t;  // of their transposes (backward)
  float* slab;       // [CTAs][kFfSlab]
  float* vec;        // [CTAs][kFfVec]
  long long rows;
  int* status;
};

// D[128 x 64] (+)= A[128 x 64] B[64 x 64]^T, both K-major; A's 8-feature groups
// `a_grp` bytes apart, B's image `b_rows` rows high.
__device__ __forceinline__ void ffn_mma(uint32_t d_tmem, uint32_t a, uint32_t a_grp, uint32_t b, uint32_t b_rows,
                                        bool accumulate) {
  constexpr uint32_t idesc = tc::idesc_bf16(128, 64);
  const uint64_t ad = tc::smem_desc(a, a_grp, 128), bd = tc::smem_desc(b, b_rows * 16, 128);
#pragma unroll
  for (int j = 0; j < 4; ++j)
    tc::mma_bf16(d_tmem, tc::desc_advance(ad, j * 2 * a_grp), tc::desc_advance(bd, j * 2 * b_rows * 16), idesc,
                 (accumulate || j > 0) ? 1u : 0u);
}
// D[128 x 64] (+)= A^T B over the tile's 128 token rows: A 128 features (groups
// 2048 bytes apart), B 64 (kRowGrp).
__device__ __forceinline__ void ffn_mma_rows(uint32_t d_tmem, uint32_t a, uint32_t b, bool accumulate) {
  constexpr uint32_t idesc = tc::idesc_bf16(128, 64) | kMnMajorA | kMnMajorB;
  const uint64_t ad = tc::smem_desc(a, 128, 128 * 16), bd = tc::smem_desc(b, 128, kRowGrp);
#pragma unroll
  for (int j = 0; j < 8; ++j)
    tc::mma_bf16(d_tmem, tc::desc_advance(ad, j * 256), tc::desc_advance(bd, j * 256), idesc,
                 (accumulate || j > 0) ? 1u : 0u);
}
__device__ __forceinline__ void ffn_publish() {
  tc::fence_async_smem();
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
}
// Rows `row` and `row` + 1 of a tile from lanes that hold one column of each
// (column c0 + lane): neighbouring lanes trade, so that each stores two columns
// of one row.
__device__ __forceinline__ void st_bf_rows(unsigned char* img, uint32_t grp, int row, int c0, float va, float vb) {
  const int odd = threadIdx.x & 1, c = c0 + (threadIdx.x & 30);
  const float got = __shfl_xor_sync(0xffffffffu, odd ? va : vb, 1);
  *reinterpret_cast<uint32_t*>(img + (c >> 3) * grp + (row + odd) * 16 + (c & 7) * 2) =
      odd ? pack_bf2(got, vb) : pack_bf2(va, got);
}
// LayerNorm of N rows on the warp, lane: columns `lane` and `lane` + 32 of each
// (the arithmetic of ln_fwd_kernel): x becomes (x - mean) rstd, rs the rstd.
template <int N>
__device__ __forceinline__ void rows_normalise(float (&x)[N][2], float (&rs)[N]) {
  float v[N];
#pragma unroll
  for (int i = 0; i < N; ++i) v[i] = x[i][0] + x[i][1];
  const float mean = row_sums(v) * (1.0f / 64);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float m = row_get<N>(mean, i);
    x[i][0] -= m;
    x[i][1] -= m;
    v[i] = 0.0f;
    v[i] += x[i][0] * x[i][0];
    v[i] += x[i][1] * x[i][1];
  }
  const float rstd = 1.0f / sqrtf(row_sums(v) * (1.0f / 64) + 1e-5f);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    rs[i] = row_get<N>(rstd, i);
    x[i][0] *= rs[i];
    x[i][1] *= rs[i];
  }
}
// LayerNorm backward of N rows (the arithmetic of ln_bwd_kernel): y the
// gradient at the LayerNorm output, xh and rs from rows_normalise; y becomes
// the residual's gradient res plus the gradient at its input (one rounding), pg
// and pb gather the gain's and offset's.
template <int N>
__device__ __forceinline__ void rows_ln_bwd(float (&y)[N][2], const float (*xh)[2], const float* rs,
                                            const float (*res)[2], float g0, float g1, float (&pg)[2],
                                            float (&pb)[2]) {
  float s1[N], s2[N];
#pragma unroll
  for (int i = 0; i < N; ++i) {
    pg[0] = fmaf(y[i][0], xh[i][0], pg[0]);
    pg[1] = fmaf(y[i][1], xh[i][1], pg[1]);
    pb[0] += y[i][0];
    pb[1] += y[i][1];
    y[i][0] *= g0;
    y[i][1] *= g1;
    s1[i] = y[i][0] + y[i][1];
    s2[i] = fmaf(y[i][1], xh[i][1], y[i][0] * xh[i][0]);
  }
  const float t1 = row_sums(s1) * (1.0f / 64), t2 = row_sums(s2) * (1.0f / 64);
#pragma unroll
  for (int i = 0; i < N; ++i) {
    const float m1 = row_get<N>(t1, i), m2 = row_get<N>(t2, i);
    y[i][0] = fmaf(rs[i], y[i][0] - m1 - xh[i][0] * m2, res[i][0]);
    y[i][1] = fmaf(rs[i], y[i][1] - m1 - xh[i][1] * m2, res[i][1]);
  }
}
__device__ __forceinline__ void st8_bf(unsigned char* img, int row, int c, const float* v) {
  *reinterpret_cast<uint4*>(img + tc::kmajor_offset(row, c, 128)) =
      make_uint4(pack_bf2(v[0], v[1]), pack_bf2(v[2], v[3]), pack_bf2(v[4], v[5]), pack_bf2(v[6], v[7]));
}

// Bounded waits on an mbarrier with its phase.
struct Bar {
  uint64_t* m;
  uint32_t parity;
  __device__ __forceinline__ bool wait() {
    const bool ok = tc::mbar_wait(m, parity, kTcPolls);
    parity ^= 1u;
    return ok;
  }
};

// 256 threads: LayerNorm and residual with a warp per row (16 rows per warp,
// the row's values kept in registers), GELU with a thread per row and half of
// a 64-wide hidden chunk.  The MMAs of chunk c + 1's pre-activations and of
// chunk c - 1's output product run during chunk c's GELU.
__global__ void __launch_bounds__(256, 2) ffn_fwd_kernel(FfnArgs a) {
  extern __shared__ __align__(128) unsigned char sm_tile[];  // (a wider alignment would cost the second CTA)
  unsigned char* sW1 = sm_tile;
  unsigned char* sW2 = sW1 + kFfW;
  unsigned char* sY = sW2 + kFfW;
  unsigned char* sG = sY + kFfA;               // two chunks
  float* sE = reinterpret_cast<float*>(sG);    // output staging [128][64] over them
  __shared__ __align__(8) uint64_t bars[5];    // pre-activations 0, 1; output product 0, 1; weights
  __shared__ uint32_t tbase;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, row = tid & 127, half = tid >> 7;
  if (warp == 0) {
    tc::tmem_alloc(&tbase, 256);
    tc::tmem_relinquish();
  }
  if (tid == 32)
    for (int k = 0; k < 5; ++k) tc::mbar_init(&bars[k], 1);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tbase, tl = tmem + ((uint32_t)(warp & 3) << 21);
  const uint32_t aY = tc::smem_addr(sY), aG = tc::smem_addr(sG), aW1 = tc::smem_addr(sW1), aW2 = tc::smem_addr(sW2);
  constexpr uint32_t kOut = 128;  // column of the output product (pre-activations: 0 and 64)
  if (tid == 0) {
    tc::mbar_expect_tx(&bars[4], 2 * (uint32_t)kFfW);
    tc::bulk_g2s(sW1, a.w1, (uint32_t)kFfW, &bars[4]);
    tc::bulk_g2s(sW2, a.w2, (uint32_t)kFfW, &bars[4]);
  }
  Bar z0{&bars[0], 0}, z1{&bars[1], 0}, o0{&bars[2], 0}, o1{&bars[3], 0};
  const float g0 = a.gain[lane], g1 = a.gain[lane + 32], f0 = a.off[lane], f1 = a.off[lane + 32];
  const float c0 = a.b2[lane], c1 = a.b2[lane + 32];
  const long long tiles = (a.rows + 127) / 128;
  bool ok = true, first = true;
  for (long long mt = blockIdx.x; mt < tiles; mt += gridDim.x, first = false) {
    const long long r0 = mt * 128 + warp * 16;
    float x[16][2];
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const bool in = r0 + i < a.rows;
      x[i][0] = in ? __ldg(a.M + (r0 + i) * 64 + lane) : 0.0f;
      x[i][1] = in ? __ldg(a.M + (r0 + i) * 64 + lane + 32) : 0.0f;
    }
    {
      float y[16][2], rs[16];
#pragma unroll
      for (int i = 0; i < 16; ++i) y[i][0] = x[i][0], y[i][1] = x[i][1];
      rows_normalise(y, rs);
#pragma unroll
      for (int i = 0; i < 16; i += 2) {
        st_bf_rows(sY, 2048, warp * 16 + i, 0, y[i][0] * g0 + f0, y[i + 1][0] * g0 + f0);
        st_bf_rows(sY, 2048, warp * 16 + i, 32, y[i][1] * g1 + f1, y[i + 1][1] * g1 + f1);
      }
    }
    ffn_publish();
    if (tid == 0) {
      if (first) ok &= tc::mbar_wait(&bars[4], 0u, kTcPolls);
      ffn_mma(tmem, aY, 2048, aW1, kFfH, false);
      tc::mma_commit(&bars[0]);
    }
    {  // the next tile's rows into L2 meanwhile, a 128-byte line per thread (783 -> 770 us)
      const long long nm = (mt + gridDim.x) * 128 + (tid >> 1);
      if (nm < a.rows) asm volatile("prefetch.global.L2 [%0];" ::"l"(a.M + nm * 64 + (tid & 1) * 32));
    }
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
      ok &= (c & 1) ? z1.wait() : z0.wait();
      if (c >= 2) ok &= (c & 1) ? o1.wait() : o0.wait();  // chunk c - 2's output product has read G buffer c & 1
      tc::fence_after_sync();
      if (tid == 0 && c < 3) {
        ffn_mma(tmem + 64 * ((c + 1) & 1), aY, 2048, aW1 + (c + 1) * 64 * 16, kFfH, false);
        tc::mma_commit(&bars[(c + 1) & 1]);
      }
      unsigned char* g = sG + (c & 1) * kFfA;
      const float4* b4 = reinterpret_cast<const float4*>(a.b1 + c * 64 + half * 32);
      float v[32];
      tc::tmem_ld32(tl + 64 * (c & 1) + half * 32, v);
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const float4 b = __ldg(b4 + j);
        v[4 * j] = gelu_f(v[4 * j] + b.x);
        v[4 * j + 1] = gelu_f(v[4 * j + 1] + b.y);
        v[4 * j + 2] = gelu_f(v[4 * j + 2] + b.z);
        v[4 * j + 3] = gelu_f(v[4 * j + 3] + b.w);
      }
#pragma unroll
      for (int j = 0; j < 32; j += 8) st8_bf(g, row, half * 32 + j, v + j);
      ffn_publish();
      if (tid == 0) {
        ffn_mma(tmem + kOut, aG + (c & 1) * (uint32_t)kFfA, 2048, aW2 + c * 8 * 64 * 16, kFfD, c > 0);
        tc::mma_commit(&bars[2 + (c & 1)]);
      }
    }
    ok &= o0.wait();
    ok &= o1.wait();
    tc::fence_after_sync();
    ok = __syncthreads_and(ok);  // (the tensor-memory loads below are warp-collective)
    if (!ok) break;
    {
      float v[32];
      tc::tmem_ld32(tl + kOut + half * 32, v);
#pragma unroll
      for (int j = 0; j < 8; ++j)
        *reinterpret_cast<float4*>(sE + epi_pos(row, half * 8 + j)) =
            make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
#pragma unroll
    for (int i = 0; i < 16; ++i) {
      const int r = warp * 16 + i;
      const float v0 = sE[epi_pos(r, lane >> 2) + (lane & 3)], v1 = sE[epi_pos(r, 8 + (lane >> 2)) + (lane & 3)];
      if (r0 + i < a.rows) {
        a.out[(r0 + i) * 64 + lane] = v0 + c0 + x[i][0];
        a.out[(r0 + i) * 64 + lane + 32] = v1 + c1 + x[i][1];
      }
    }
    // (the next tile's LayerNorm writes sY alone; its GELU comes after a barrier)
  }
  if (!ok && tid == 0) {  // no weight copy may still be landing when the CTA exits
    tc::mbar_wait(&bars[4], 0u, kTcPolls);
    raise_status(a.status, 2);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 256);
}

// 512 threads, one CTA per SM (its weight gradients fill half of the tensor
// memory): LayerNorm and its backward with a warp per row (8 rows per warp),
// GELU and its derivative with a thread per row and quarter of a 64-wide
// hidden chunk.
__global__ void __launch_bounds__(512, 1) ffn_bwd_kernel(FfnArgs a) {
  extern __shared__ __align__(128) unsigned char sm_tile[];
  unsigned char* sW1 = sm_tile;            // W1: pre-activations
  unsigned char* sW2t = sW1 + kFfW;        // W2^T: gradient at the GELU output
  unsigned char* sW1t = sW2t + kFfW;       // W1^T: gradient at the LayerNorm output
  unsigned char* sY = sW1t + kFfW;         // LayerNorm output
  unsigned char* sD = sY + kRowA;          // dX'
  unsigned char* sG = sD + kRowA;          // GELU outputs of a 128-wide hidden pair of chunks
  unsigned char* sZ = sG + 2 * kFfA;       // gradients at its pre-activations
  float* sE = reinterpret_cast<float*>(sZ + 2 * kFfA);  // staging [128][64]
  __shared__ __align__(8) uint64_t bars[4];  // chunk products, pair products, output product, weights
  __shared__ uint32_t tbase;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, row = tid & 127, part = tid >> 7;
  if (warp == 0) {
    tc::tmem_alloc(&tbase, 512);
    tc::tmem_relinquish();
  }
  if (tid == 32)
    for (int k = 0; k < 4; ++k) tc::mbar_init(&bars[k], 1);
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tbase, tl = tmem + ((uint32_t)(warp & 3) << 21);
  const uint32_t aY = tc::smem_addr(sY), aD = tc::smem_addr(sD), aG = tc::smem_addr(sG), aZ = tc::smem_addr(sZ);
  const uint32_t aW1 = tc::smem_addr(sW1), aW2t = tc::smem_addr(sW2t), aW1t = tc::smem_addr(sW1t);
  // tensor memory: dW1 of hidden 0-127 and 128-255, dW2^T of the same, then
  // pre-activations, gradient at the GELU output, gradient at the LN output
  constexpr uint32_t kW1 = 0, kW2 = 128, kPre = 256, kGrad = 320, kDy = 384;
  if (tid == 0) {
    tc::mbar_expect_tx(&bars[3], 3 * (uint32_t)kFfW);
    tc::bulk_g2s(sW1, a.w1, (uint32_t)kFfW, &bars[3]);
    tc::bulk_g2s(sW2t, a.w2t, (uint32_t)kFfW, &bars[3]);
    tc::bulk_g2s(sW1t, a.w1t, (uint32_t)kFfW, &bars[3]);
  }
  Bar chunk{&bars[0], 0}, pair{&bars[1], 0}, dy_bar{&bars[2], 0};
  const float g0 = a.gain[lane], g1 = a.gain[lane + 32], f0 = a.off[lane], f1 = a.off[lane + 32];
  float pg[2] = {0.0f, 0.0f}, pb[2] = {0.0f, 0.0f}, pd0 = 0.0f, pd1 = 0.0f;  // LN gain, offset; db2
  float pz[4] = {0.0f, 0.0f, 0.0f, 0.0f};  // db1 of hidden 64 c + 16 part + lane % 16 over this warp's rows
  const long long tiles = (a.rows + 127) / 128;
  bool ok = true, first = true;
  float xn[8][2], dn[8][2];  // the next tile's rows of M and dX', in flight during the current one
  auto fetch = [&](long long mt) {
    const long long r0 = mt * 128 + warp * 8;
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      const bool in = mt < tiles && r0 + i < a.rows;
      xn[i][0] = in ? __ldg(a.M + (r0 + i) * 64 + lane) : 0.0f;
      xn[i][1] = in ? __ldg(a.M + (r0 + i) * 64 + lane + 32) : 0.0f;
      dn[i][0] = in ? __ldg(a.dX + (r0 + i) * 64 + lane) : 0.0f;
      dn[i][1] = in ? __ldg(a.dX + (r0 + i) * 64 + lane + 32) : 0.0f;
    }
  };
  fetch(blockIdx.x);
  for (long long mt = blockIdx.x; mt < tiles; mt += gridDim.x, first = false) {
    const long long r0 = mt * 128 + warp * 8;
    float xh[8][2], dx[8][2], rs[8];  // normalised rows, dX', 1 / std
#pragma unroll
    for (int i = 0; i < 8; ++i) xh[i][0] = xn[i][0], xh[i][1] = xn[i][1];
    rows_normalise(xh, rs);
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      dx[i][0] = dn[i][0];
      dx[i][1] = dn[i][1];
      pd0 += dx[i][0];
      pd1 += dx[i][1];
    }
#pragma unroll
    for (int i = 0; i < 8; i += 2) {
      const int r = warp * 8 + i;
      st_bf_rows(sY, kRowGrp, r, 0, xh[i][0] * g0 + f0, xh[i + 1][0] * g0 + f0);
      st_bf_rows(sY, kRowGrp, r, 32, xh[i][1] * g1 + f1, xh[i + 1][1] * g1 + f1);
      st_bf_rows(sD, kRowGrp, r, 0, dx[i][0], dx[i + 1][0]);
      st_bf_rows(sD, kRowGrp, r, 32, dx[i][1], dx[i + 1][1]);
    }
    ffn_publish();
    if (tid == 0) {
      if (first) ok &= tc::mbar_wait(&bars[3], 0u, kTcPolls);
      ffn_mma(tmem + kPre, aY, kRowGrp, aW1, kFfH, false);
      ffn_mma(tmem + kGrad, aD, kRowGrp, aW2t, kFfH, false);
      tc::mma_commit(&bars[0]);
    }
#pragma unroll 1
    for (int c = 0; c < 4; ++c) {
      ok &= chunk.wait();
      if (c == 2) ok &= pair.wait();  // the first pair's products have read sG and sZ
      tc::fence_after_sync();
      float z[16], v[16];
      tc::tmem_ld16(tl + kPre + part * 16, z);
      tc::tmem_ld16(tl + kGrad + part * 16, v);
      if (c < 3) {  // both are in registers: the next chunk's products may overwrite them
        tc::fence_before_sync();
        __syncthreads();
        tc::fence_after_sync();
        if (tid == 0) {
          ffn_mma(tmem + kPre, aY, kRowGrp, aW1 + (c + 1) * 64 * 16, kFfH, false);
          ffn_mma(tmem + kGrad, aD, kRowGrp, aW2t + (c + 1) * 64 * 16, kFfH, false);
          tc::mma_commit(&bars[0]);
        }
      }
      const float4* b4 = reinterpret_cast<const float4*>(a.b1 + c * 64 + part * 16);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float4 b = __ldg(b4 + j);
        z[4 * j] += b.x;
        z[4 * j + 1] += b.y;
        z[4 * j + 2] += b.z;
        z[4 * j + 3] += b.w;
      }
#pragma unroll
      for (int j = 0; j < 16; ++j) {  // gelu_grad_f and gelu_f of one erf
        const float e1 = 1.0f + erff(z[j] * 0.70710678118654752f);
        v[j] *= 0.5f * e1 + z[j] * expf(-0.5f * z[j] * z[j]) * 0.39894228040143268f;
        z[j] = 0.5f * z[j] * e1;
      }
      const int hc = (c & 1) * 64 + part * 16;
      st8_bf(sG, row, hc, z);
      st8_bf(sG, row, hc + 8, z + 8);
      st8_bf(sZ, row, hc, v);
      st8_bf(sZ, row, hc + 8, v + 8);
      const float s = colsum16(v);
#pragma unroll
      for (int k = 0; k < 4; ++k)
        if (k == c) pz[k] += s;
      ffn_publish();
      if (tid == 0) {
        ffn_mma(tmem + kDy, aZ + (c & 1) * 8 * 2048, 2048, aW1t + c * 8 * 64 * 16, kFfD, c > 0);
        if (c & 1) {
          ffn_mma_rows(tmem + kW1 + (c >> 1) * 64, aZ, aY, !first);
          ffn_mma_rows(tmem + kW2 + (c >> 1) * 64, aG, aD, !first);
          tc::mma_commit(&bars[c == 1 ? 1 : 2]);
        }
      }
    }
    fetch(mt + gridDim.x);
    ok &= dy_bar.wait();  // every MMA of the tile is done
    tc::fence_after_sync();
    ok = __syncthreads_and(ok);  // (the tensor-memory loads below are warp-collective)
    if (!ok) break;
    {
      float v[16];
      tc::tmem_ld16(tl + kDy + part * 16, v);
#pragma unroll
      for (int j = 0; j < 4; ++j)
        *reinterpret_cast<float4*>(sE + epi_pos(row, part * 4 + j)) =
            make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
    }
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    {
      float y[8][2];
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        y[i][0] = sE[epi_pos(warp * 8 + i, lane >> 2) + (lane & 3)];
        y[i][1] = sE[epi_pos(warp * 8 + i, 8 + (lane >> 2)) + (lane & 3)];
      }
      rows_ln_bwd(y, xh, rs, dx, g0, g1, pg, pb);
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        if (r0 + i < a.rows) {
          a.out[(r0 + i) * 64 + lane] = y[i][0];
          a.out[(r0 + i) * 64 + lane + 32] = y[i][1];
        }
      }
    }
    // (the next tile's LayerNorm writes sY and sD, whose MMAs are done; sE is
    // written again after several barriers)
  }
  if (ok) {
    // this CTA's slabs: column part 0, 1: dW1 of the two hidden halves (lane =
    // hidden unit), 2, 3: dW2^T of the same
    const int hid = (part & 1) * 128 + row;
    float* slab = a.slab + (long long)blockIdx.x * kFfSlab;
    const uint32_t col = part < 2 ? kW1 + part * 64 : kW2 + (part - 2) * 64;
#pragma unroll 1
    for (int c0 = 0; c0 < 64; c0 += 16) {
      float v[16];
      tc::tmem_ld16(tl + col + c0, v);
      if (part < 2) {
#pragma unroll
        for (int j = 0; j < 4; ++j)
          *reinterpret_cast<float4*>(slab + hid * 64 + c0 + 4 * j) =
              make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) slab[kFfD * kFfH + (c0 + j) * kFfH + hid] = v[j];
      }
    }
    // vector gradients: db1 over the four row quarters, the rest over the 16
    // warps, in order (sE is free: a barrier follows its last reads)
    __syncthreads();
    float* s_z = sE;             // [4][256]
    float* s_l = sE + 4 * kFfH;  // [16][192]: db2, gain, offset
    if (lane < 16) {
#pragma unroll
      for (int c = 0; c < 4; ++c) s_z[(warp & 3) * kFfH + c * 64 + part * 16 + lane] = pz[c];
    }
    float* l = s_l + warp * 192;
    l[lane] = pd0;
    l[lane + 32] = pd1;
    l[64 + lane] = pg[0];
    l[96 + lane] = pg[1];
    l[128 + lane] = pb[0];
    l[160 + lane] = pb[1];
    __syncthreads();
    float* vec = a.vec + (long long)blockIdx.x * kFfVec;
    if (tid < kFfH) {
      vec[tid] = ((s_z[tid] + s_z[kFfH + tid]) + s_z[2 * kFfH + tid]) + s_z[3 * kFfH + tid];
    } else if (tid < kFfH + 192) {
      float t = 0.0f;
#pragma unroll
      for (int w = 0; w < 16; ++w) t += s_l[w * 192 + tid - kFfH];
      vec[tid] = t;
    }
  } else if (tid == 0) {  // no weight copy may still be landing when the CTA exits
    tc::mbar_wait(&bars[3], 0u, kTcPolls);
    raise_status(a.status, 2);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 512);
}

// X' of the sub-block over `rows` token rows.
cudaError_t ffn_fwd(const FfnArgs& a, cudaStream_t s) {
  static std::atomic<unsigned long long> ready{0};
  const cudaError_t e = smem_optin(ffn_fwd_kernel, kFfFwdSmem, ready);
  if (e != cudaSuccess) return e;
  const long long tiles = (a.rows + 127) / 128;
  ffn_fwd_kernel<<<(unsigned)std::min<long long>(tiles, 2 * 152), 256, kFfFwdSmem, s>>>(a);
  return cudaGetLastError();
}

// dM, and the partial gradients of its CTAs (returned count) into a.slab, a.vec.
cudaError_t ffn_bwd(const FfnArgs& a, int* ctas, cudaStream_t s) {
  static std::atomic<unsigned long long> ready{0};
  const cudaError_t e = smem_optin(ffn_bwd_kernel, kFfBwdSmem, ready);
  if (e != cudaSuccess) return e;
  *ctas = (int)std::min<long long>((a.rows + 127) / 128, 152);
  ffn_bwd_kernel<<<(unsigned)*ctas, 512, kFfBwdSmem, s>>>(a);
  return cudaGetLastError();
}
