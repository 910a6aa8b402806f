// Learned range-only estimator kernels: forward (inference and training),
// input-gradient pass, weight-gradient pass, Adam, feature recording.
//
// All three hidden layers run on the tensor cores (tcgen05.mma, BF16 x BF16 ->
// FP32 in TMEM) with 128 rows per CTA, four threads per row in the epilogues.
// The first layer's inputs are FP32 features split into a BF16
// high part and a BF16 remainder that are multiplied by the same weights and
// accumulated together: ranges of hundreds of metres keep ~1e-5 relative
// precision instead of BF16's 4e-3, which matters for metre-level tracking.
// The 2-wide output layer runs on CUDA cores.
#include "estimator.cuh"
#include "gelu.cuh"
#include "tc.cuh"
#include "warp_sums.cuh"

#include <cmath>
#include <cstring>

namespace ut {
namespace est {
namespace {

constexpr int kT = 128;
constexpr uint32_t TAG_BATCH = 14;
constexpr float kMaxCorr = 3.0f;  // largest correction per step, in units of L
constexpr size_t kImgA = (size_t)kT * HID * 2;  // one tile's operand image [HID / 8][128 rows][8] (64 KB)
constexpr size_t kImgX = (size_t)kT * IN * 2;   // of the features (24 KB)

// Derivative of erf-GELU for the backward pass: Phi(x) + x phi(x).  (The
// forward passes evaluate GELU with gelu.cuh's form, within 5.4e-6 of the
// erf form.)
__device__ __forceinline__ float gelu_grad(float x) {
  return 0.5f * (1.0f + erff(x * 0.70710678118654752f)) + x * 0.39894228040143268f * __expf(-0.5f * x * x);
}

__device__ __forceinline__ void store8(unsigned char* img, int row, int k0, int rows, const float* v) {
  uint4 p;
  p.x = bf16x2_bits(v[0], v[1]);
  p.y = bf16x2_bits(v[2], v[3]);
  p.z = bf16x2_bits(v[4], v[5]);
  p.w = bf16x2_bits(v[6], v[7]);
  *reinterpret_cast<uint4*>(img + tc::kmajor_offset(row, k0, rows)) = p;
}

// x[i] += p[i] over 4 M values of read-only memory, p 16-byte aligned.
template <int M>
__device__ __forceinline__ void add4(float* x, const float* p) {
#pragma unroll
  for (int i = 0; i < M; ++i) {
    const float4 b = __ldg(reinterpret_cast<const float4*>(p) + i);
    x[4 * i] += b.x;
    x[4 * i + 1] += b.y;
    x[4 * i + 2] += b.z;
    x[4 * i + 3] += b.w;
  }
}

// o0, o1 += the output layer's two sums over 4 M hidden units a from unit c0 on,
// in order.
template <int M>
__device__ __forceinline__ void out_sums(const float* mst, int c0, const float* a, float& o0, float& o1) {
  const float4* w4 = reinterpret_cast<const float4*>(mst + W4_OFF + c0);
#pragma unroll
  for (int i = 0; i < M; ++i) {
    const float4 w0 = __ldg(w4 + i), w1 = __ldg(w4 + HID / 4 + i);
    o0 = fmaf(w0.x, a[4 * i], o0);
    o1 = fmaf(w1.x, a[4 * i], o1);
    o0 = fmaf(w0.y, a[4 * i + 1], o0);
    o1 = fmaf(w1.y, a[4 * i + 1], o1);
    o0 = fmaf(w0.z, a[4 * i + 2], o0);
    o1 = fmaf(w1.z, a[4 * i + 2], o1);
    o0 = fmaf(w0.w, a[4 * i + 3], o0);
    o1 = fmaf(w1.w, a[4 * i + 3], o1);
  }
}

// 24 consecutive features of a row from column c0 (a multiple of 8) on, as BF16
// high parts and remainders in two operand images.
__device__ __forceinline__ void store_features(unsigned char* hi_img, unsigned char* lo_img, int row, int c0,
                                               const float (&x)[24]) {
#pragma unroll
  for (int k = 0; k < 24; k += 8) {
    float hi[8], lo[8];
#pragma unroll
    for (int i = 0; i < 8; ++i) {
      hi[i] = bf_bits2f(f2bf_bits(x[k + i]));
      lo[i] = x[k + i] - hi[i];
    }
    store8(hi_img, row, c0 + k, 128, hi);
    store8(lo_img, row, c0 + k, 128, lo);
  }
}

// Estimator features of filter f for its update at step g (reading C18):
// in the local frame of the filter's current estimate e1 (units of L), each
// of the 16 most recent pings, newest first, as [(q - e1) / L, range
// innovation (r - |q - e1|_3D) / L, (g - g_m) / 16, 1], then the last motion
// of the estimate (e1 - e2) / L and its smoothed motion v / L (the velocity
// EMA including this update's e1 - e2); zero padded to 96.  The network's
// output is the correction (x - e1) / L.
// Columns LO .. LO + N - 1 of them.  STEP: the sum of squares with the step's
// own roundings (its low bits decide BF16 roundings, so the order is fixed here
// and not left to the compiler).
template <int LO, bool STEP, int N>
__device__ __forceinline__ void ring_features(const EnvDev& d, int f, uint32_t g, float e1x, float e1y, float e2x,
                                              float e2y, float vx, float vy, float (&x)[N]) {
  const int it = d.filt_target[f];
  const float dz = UT_IN_BOUNDS(it >= 0 && it < d.NT, d.status) ? d.tz[it] : 0.0f;  // target depth; senders at the surface
  const float L = d.est_scale;
  const int head = d.ring_head[f], cnt = d.ring_count[f];
  const float4* ring = reinterpret_cast<const float4*>(d.ring) + (long long)f * kRing;
#pragma unroll
  for (int i = 0; i < N; ++i) x[i] = 0.0f;
#pragma unroll
  for (int s = 0; s < kRing; ++s) {
    if (5 * s + 4 < LO || 5 * s >= LO + N) continue;  // (compile time: none of its columns wanted)
    float4 e = make_float4(0.f, 0.f, 0.f, 0.f);
    const bool on = s < cnt;
    if (on) e = ring[(head - 1 - s) & (kRing - 1)];
    const float dx = e.x - e1x, dy = e.y - e1y;
    const float rho = sqrtf(STEP ? __fadd_rn(fmaf(dx, dx, dy * dy), __fmul_rn(dz, dz)) : dx * dx + dy * dy + dz * dz);
    const float v[5] = {on ? dx / L : 0.0f, on ? dy / L : 0.0f, on ? (e.z - rho) / L : 0.0f,
                        on ? ((float)g - e.w) / 16.0f : 0.0f, on ? 1.0f : 0.0f};
#pragma unroll
    for (int k = 0; k < 5; ++k)
      if (5 * s + k >= LO && 5 * s + k < LO + N) x[5 * s + k - LO] = v[k];
  }
  const float m[4] = {(e1x - e2x) / L, (e1y - e2y) / L, vx / L, vy / L};
#pragma unroll
  for (int k = 0; k < 4; ++k)
    if (5 * kRing + k >= LO && 5 * kRing + k < LO + N) x[5 * kRing + k - LO] = m[k];
}

// acc[128 x 128] (+)= A[128 x 16 ksteps] B[128 x 16 ksteps]^T, issued by the
// calling thread (both images 128 rows high).
__device__ __forceinline__ void issue_mma(uint32_t d_tmem, uint32_t a, uint32_t b, int ksteps, bool accumulate) {
  constexpr uint32_t idesc = tc::idesc_bf16(128, 128);
  uint64_t ad = tc::smem_desc(a, 128 * 16, 128), bd = tc::smem_desc(b, 128 * 16, 128);
#pragma unroll 2
  for (int k = 0; k < ksteps; ++k) {
    tc::mma_bf16(d_tmem, ad, bd, idesc, (accumulate || k > 0) ? 1u : 0u);
    ad = tc::desc_advance(ad, 2 * 128 * 16);
    bd = tc::desc_advance(bd, 2 * 128 * 16);
  }
}

// ---------------------------------------------------------------------------
// Estimator step in the environment (learned form): one CTA of 512 threads
// per 128 filters, thread = filter row x one of 4 column parts.  Each part
// builds its 24 of the row's features (one thread per row built all 96: 13 k of
// a tile's 48 k cycles; 102,400 filters 144 -> 124 us); the hidden-layer epilogues (bias, erf-GELU of
// gelu.cuh in packed pairs, BF16 operand) split
// the 256 hidden units 4 ways; the weight images (N-halves
// of W1, W2, W3) stream through two shared-memory slots by the bulk-copy
// engine, so the next layer's weights arrive during the current epilogue.
// ---------------------------------------------------------------------------
constexpr int kTE = 512;
constexpr int kParts = kTE / 128;
constexpr int kEnvStages = 6;                               // W1, W2, W3, two N-halves each
constexpr size_t kEnvSlot = (size_t)128 * HID * 2;          // largest half image (64 KB)
constexpr size_t kEnvSmem = 65536 + 2 * kEnvSlot;           // A operand + two weight slots
constexpr uint32_t kEnvPolls = 1u << 22;

__device__ __forceinline__ void env_stage(int s, size_t& off, uint32_t& bytes) {
  if (s < 2) {
    off = IMG_W1_OFF + (size_t)s * 128 * IN * 2;
    bytes = (uint32_t)(128 * IN * 2);
  } else {
    const int l = (s - 2) >> 1, h = (s - 2) & 1;
    off = (l == 0 ? IMG_W2_OFF : IMG_W3_OFF) + (size_t)h * 128 * HID * 2;
    bytes = (uint32_t)(128 * HID * 2);
  }
}

// test_wait_polls > 0 (test hook, env_test_wait_timeout): first a bounded
// wait on a barrier that nothing signals, then the timed-out exit (status 2)
// before any copy or MMA is issued.
__global__ void __launch_bounds__(kTE, 1) fwd_env_kernel(Net net, EnvDev d, int stale, uint32_t test_wait_polls) {
  pdl_wait();  // (dependents launch as this grid's CTAs exit)
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* sA = smem;           // features hi | lo [2 x 128 x 96], then hidden activations [128 x 256]
  unsigned char* sW = smem + 65536;   // two weight slots
  __shared__ __align__(8) uint64_t full[2];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ __align__(8) uint64_t never;  // test hook: a barrier nothing signals
  __shared__ uint32_t tbase;
  __shared__ float sOut[kParts][2][128];
  __shared__ int bad;
  const int tid = threadIdx.x, warp = tid >> 5, row = tid & 127, part = tid >> 7;
  const long long f = (long long)blockIdx.x * 128 + row;
  const bool valid = f < d.F;

  if (warp == 0) {
    tc::tmem_alloc(&tbase, 256);
    tc::tmem_relinquish();
  }
  if (tid == 32) {
    tc::mbar_init(&full[0], 1);
    tc::mbar_init(&full[1], 1);
    tc::mbar_init(&mbar, 1);
    tc::mbar_init(&never, 1);
    bad = 0;
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tbase;
  if (test_wait_polls) {
    if (tid == 32 && !tc::mbar_wait(&never, 0u, test_wait_polls)) bad = 1;
    __syncthreads();
    if (bad) {
      if (tid == 0) raise_status(d.status, 2);
      if (warp == 0) tc::tmem_dealloc(tmem, 256);
      return;
    }
  }
  const uint32_t tl = tmem + ((uint32_t)(warp & 3) << 21);  // this warp's lane quarter
  const uint32_t aA = tc::smem_addr(sA), aW = tc::smem_addr(sW);
  auto fetch = [&](int st) {  // thread 0: stage st into slot st % 2
    size_t off;
    uint32_t bytes;
    env_stage(st, off, bytes);
    tc::mbar_expect_tx(&full[st & 1], bytes);
    tc::bulk_g2s(sW + (st & 1) * kEnvSlot, net.img + off, bytes, &full[st & 1]);
  };
  if (tid == 0) {
    fetch(0);
    fetch(1);
  }

  // this part's features of the row -> A operand as BF16 high and low parts
  float e1x = 0.0f, e1y = 0.0f, vnx = 0.0f, vny = 0.0f;
  bool fresh = false;  // (part 0) a ping received this step
  {
    float x[24];
    if (valid) {
      e1x = d.estx[f];
      e1y = d.esty[f];
      const float e2x = d.prev_estx[f], e2y = d.prev_esty[f];
      vnx = fmaf(kVelKeep, d.velx[f], (1.0f - kVelKeep) * (e1x - e2x));
      vny = fmaf(kVelKeep, d.vely[f], (1.0f - kVelKeep) * (e1y - e2y));
      const uint32_t g = d.counters[0] + 1u;
      if (part == 0) {
        ring_features<0, true>(d, (int)f, g, e1x, e1y, e2x, e2y, vnx, vny, x);
        fresh = x[3] == 0.0f && x[4] == 1.0f;
      } else if (part == 1) {
        ring_features<24, true>(d, (int)f, g, e1x, e1y, e2x, e2y, vnx, vny, x);
      } else if (part == 2) {
        ring_features<48, true>(d, (int)f, g, e1x, e1y, e2x, e2y, vnx, vny, x);
      } else {
        ring_features<72, true>(d, (int)f, g, e1x, e1y, e2x, e2y, vnx, vny, x);
      }
    } else {
#pragma unroll
      for (int i = 0; i < 24; ++i) x[i] = 0.0f;
    }
    store_features(sA, sA + 128 * IN * 2, row, part * 24, x);
  }

  bool ok = true;
  uint32_t mphase = 0;
  int stage = 0;
  const float* mst = net.master;
  float o0 = 0.0f, o1 = 0.0f;
  for (int l = 0; l < 3; ++l) {
    // MMA group of layer l: both N-halves (and, for layer 1, both feature parts)
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (tid == 0) {
      for (int h = 0; h < 2; ++h) {
        ok &= tc::mbar_wait(&full[(stage + h) & 1], (uint32_t)(((stage + h) >> 1) & 1), kEnvPolls);
        const uint32_t bB = aW + (uint32_t)(((stage + h) & 1) * kEnvSlot);
        issue_mma(tmem + 128 * h, aA, bB, (l == 0 ? IN : HID) / 16, false);
        if (l == 0) issue_mma(tmem + 128 * h, aA + (uint32_t)(128 * IN * 2), bB, IN / 16, true);
      }
      tc::mma_commit(&mbar);
    }
    ok &= tc::mbar_wait(&mbar, mphase, kEnvPolls);
    mphase ^= 1u;
    tc::fence_after_sync();
    stage += 2;
    if (tid == 0 && stage < kEnvStages) {  // both slots are free again: next layer's weights
      fetch(stage);
      fetch(stage + 1);
    }
    // epilogue of hidden layer l on this thread's 64 hidden units
    const float* bias = mst + (l == 0 ? B1_OFF : (l == 1 ? B2_OFF : B3_OFF));
#pragma unroll 1
    for (int c0 = part * (HID / kParts); c0 < (part + 1) * (HID / kParts); c0 += 32) {
      float av[32];
      tc::tmem_ld32(tl + c0, av);
      add4<8>(av, bias + c0);  // (every layer's biases start at a multiple of 4)
#pragma unroll
      for (int i = 0; i < 32; i += 2) gelu2(av[i], av[i + 1]);  // erf-GELU, packed pairs
      if (l < 2) {
#pragma unroll
        for (int i = 0; i < 32; i += 8) store8(sA, row, c0 + i, 128, av + i);
      } else {
        out_sums<8>(mst, c0, av, o0, o1);
      }
    }
  }
  sOut[part][0][row] = o0;
  sOut[part][1][row] = o1;
  if (!ok) atomicExch(&bad, 1);
  __syncthreads();
  if (part == 0 && valid && bad == 0) {
    o0 = __ldg(mst + B4_OFF);
    o1 = __ldg(mst + B4_OFF + 1);
#pragma unroll
    for (int k = 0; k < kParts; ++k) {
      o0 += sOut[k][0][row];
      o1 += sOut[k][1][row];
    }
    const int it0 = d.filt_target[f];
    const int it = UT_IN_BOUNDS(it0 >= 0 && it0 < d.NT, d.status) ? it0 : 0;
    // Bounded update (dropped if not finite): with a ping received this step
    // the estimate may move up to kMaxCorr L.  Without one, the rule chosen
    // by the mode applies: hold the estimate (stale inputs cannot drive the
    // closed loop away), apply the network all the same, or coast by the
    // estimate's smoothed motion v (constant velocity).
    const float lim = (fresh || stale == 1) ? kMaxCorr : 0.0f;
    float c0 = isfinite(o0) ? fminf(fmaxf(o0, -lim), lim) : 0.0f;
    float c1 = isfinite(o1) ? fminf(fmaxf(o1, -lim), lim) : 0.0f;
    if (!fresh && stale == 2) {
      c0 = fminf(fmaxf(vnx / d.est_scale, -kMaxCorr), kMaxCorr);
      c1 = fminf(fmaxf(vny / d.est_scale, -kMaxCorr), kMaxCorr);
    }
    const float ex = e1x + d.est_scale * c0, ey = e1y + d.est_scale * c1;
    d.prev2_estx[f] = d.prev_estx[f];
    d.prev2_esty[f] = d.prev_esty[f];
    d.prev_estx[f] = e1x;
    d.prev_esty[f] = e1y;
    d.velx[f] = vnx;
    d.vely[f] = vny;
    d.estx[f] = ex;
    d.esty[f] = ey;
    const float dx = ex - d.tx[it], dy = ey - d.ty[it];
    d.err[f] = sqrtf(dx * dx + dy * dy);
  }
  if (bad && tid == 0) {
    // no copy may still be landing in shared memory when the CTA exits
    for (int st = kEnvStages - 2; st < kEnvStages; ++st)
      tc::mbar_wait(&full[st & 1], (uint32_t)((st >> 1) & 1), kEnvPolls);
    raise_status(d.status, 2);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 256);
}

// ---------------------------------------------------------------------------
// The network on feature rows: forward (est_forward), and in training also
// the loss, the input-gradient pass and the sums that need no contraction.
// One CTA of 512 threads per 128 rows, thread = row x one of 4 column parts,
// weights as in fwd_env_kernel (the transposed W3 and W2 follow as stages
// 6 .. 9).  Training keeps what the weight gradients contract as BF16 operand
// images in HBM (features, a1, a2 and dz1 .. dz3 of each tile, written with
// 16-byte stores, 512 contiguous bytes per warp); z2 and z3 stay in tensor
// memory until their derivative is needed, z1 goes through HBM.
//
// 128 CTAs of a 16,384-row batch are one wave, so the pass is the latency of
// one tile, 65 us; on one thread per row and kernel, with a five-step warp sum
// for each of 1,280 columns, the forward took 86 us and the backward 185.
// ---------------------------------------------------------------------------
constexpr int kTrainStages = 10;  // W1, W2, W3, W3^T, W2^T, two N-halves each

__device__ __forceinline__ void train_stage(int s, size_t& off, uint32_t& bytes) {
  if (s < kEnvStages) {
    env_stage(s, off, bytes);
  } else {
    const int h = (s - kEnvStages) & 1;
    off = (s < kEnvStages + 2 ? IMG_W3T_OFF : IMG_W2T_OFF) + (size_t)h * 128 * HID * 2;
    bytes = (uint32_t)(128 * HID * 2);
  }
}

template <bool TRAIN>
__global__ void __launch_bounds__(kTE, 1) mlp_kernel(Net net, const float* __restrict__ X,
                                                     const int32_t* __restrict__ rows, int B, float* __restrict__ out,
                                                     TrainBufs t, int* status, uint32_t test_wait_polls) {
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* sA = smem;          // features hi | lo, then the current A operand [128 x 256]
  unsigned char* sW = smem + 65536;  // two weight slots
  __shared__ __align__(8) uint64_t full[2];
  __shared__ __align__(8) uint64_t mbar;
  __shared__ __align__(8) uint64_t never;  // test hook: a barrier nothing signals
  __shared__ uint32_t tbase;
  __shared__ float sOut[2][128];
  __shared__ float s_red[TRAIN ? 4 : 1][TRAIN ? NB_PART : 1];  // column sums of each 32-row quarter
  __shared__ double s_loss[4];
  __shared__ int bad;
  constexpr uint32_t kCols = TRAIN ? 512 : 256;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, row = tid & 127, part = tid >> 7, quarter = warp & 3;
  const long long b = (long long)blockIdx.x * kT + row;
  const bool valid = b < B;
  const long long src = valid ? (rows ? (long long)rows[b] : b) : 0;

  if (warp == 0) {
    tc::tmem_alloc(&tbase, kCols);
    tc::tmem_relinquish();
  }
  if (tid == 32) {
    tc::mbar_init(&full[0], 1);
    tc::mbar_init(&full[1], 1);
    tc::mbar_init(&mbar, 1);
    tc::mbar_init(&never, 1);
    bad = 0;
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tbase;
  if (test_wait_polls) {  // as in fwd_env_kernel
    if (tid == 32 && !tc::mbar_wait(&never, 0u, test_wait_polls)) bad = 1;
    __syncthreads();
    if (bad) {
      if (tid == 0) raise_status(status, 2);
      if (warp == 0) tc::tmem_dealloc(tmem, kCols);
      return;
    }
  }
  const uint32_t tl = tmem + ((uint32_t)quarter << 21);  // this warp's lane quarter
  const uint32_t aA = tc::smem_addr(sA), aW = tc::smem_addr(sW);
  constexpr int kStages = TRAIN ? kTrainStages : kEnvStages;
  auto fetch = [&](int st) {  // thread 0: stage st into slot st % 2
    size_t off;
    uint32_t bytes;
    train_stage(st, off, bytes);
    tc::mbar_expect_tx(&full[st & 1], bytes);
    tc::bulk_g2s(sW + (st & 1) * kEnvSlot, net.img + off, bytes, &full[st & 1]);
  };
  if (tid == 0) {
    fetch(0);
    fetch(1);
  }
  // features of this row, columns 24 part .. + 23, as BF16 high and low parts
  {
    float x[24];
#pragma unroll
    for (int i = 0; i < 24; i += 4) {
      const float4 v = __ldg(reinterpret_cast<const float4*>(X + src * IN + part * 24 + i));
      x[i] = v.x; x[i + 1] = v.y; x[i + 2] = v.z; x[i + 3] = v.w;
    }
    if (!valid) {  // (row 0 of X was read)
#pragma unroll
      for (int i = 0; i < 24; ++i) x[i] = 0.0f;
    }
    store_features(sA, sA + 128 * IN * 2, row, part * 24, x);
    if (TRAIN) {
#pragma unroll
      for (int k = 0; k < 24; k += 8) store8(t.x_img + (size_t)blockIdx.x * kImgX, row, part * 24 + k, 128, x + k);
    }
  }

  bool ok = true;
  uint32_t mphase = 0;
  int stage = 0;
  const float* mst = net.master;
  // D[128 x 256] at column `col` = A (sA; the hi and lo features of layer 1)
  // times the next two stages' weights; every thread calls it
  auto product = [&](uint32_t col, int K, int n_a) {
    tc::fence_async_smem();
    tc::fence_before_sync();
    __syncthreads();
    tc::fence_after_sync();
    if (tid == 0) {
      for (int h = 0; h < 2; ++h) {
        ok &= tc::mbar_wait(&full[(stage + h) & 1], (uint32_t)(((stage + h) >> 1) & 1), kEnvPolls);
        const uint32_t bB = aW + (uint32_t)(((stage + h) & 1) * kEnvSlot);
        issue_mma(tmem + col + 128 * h, aA, bB, K / 16, false);
        if (n_a == 2) issue_mma(tmem + col + 128 * h, aA + (uint32_t)(128 * IN * 2), bB, K / 16, true);
      }
      tc::mma_commit(&mbar);
    }
    ok &= tc::mbar_wait(&mbar, mphase, kEnvPolls);
    mphase ^= 1u;
    tc::fence_after_sync();
    stage += 2;
    if (tid == 0 && stage < kStages) {  // both slots are free again
      fetch(stage);
      fetch(stage + 1);
    }
  };
  const int c_lo = part * (HID / kParts), c_hi = c_lo + HID / kParts;
  constexpr uint32_t kZ2 = TRAIN ? 256 : 0;  // column of layer 2's accumulator (layers 1 and 3: 0)
  for (int l = 0; l < 2; ++l) {
    const uint32_t col = l == 1 ? kZ2 : 0u;
    product(col, l == 0 ? IN : HID, l == 0 ? 2 : 1);
    const float* bias = mst + (l == 0 ? B1_OFF : B2_OFF);
#pragma unroll 1
    for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
      float v[16];
      tc::tmem_ld16(tl + col + c0, v);
      add4<4>(v, bias + c0);
      if (TRAIN && l == 0) {
        float4* zr = reinterpret_cast<float4*>(t.z + b * HID + c0);
#pragma unroll
        for (int i = 0; i < 4; ++i) zr[i] = make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]);
      }
#pragma unroll
      for (int i = 0; i < 16; i += 2) gelu2(v[i], v[i + 1]);  // erf-GELU, packed pairs
      store8(sA, row, c0, 128, v);
      store8(sA, row, c0 + 8, 128, v + 8);
      if (TRAIN) {
        unsigned char* img = t.a_img + ((size_t)l * gridDim.x + blockIdx.x) * kImgA;
        store8(img, row, c0, 128, v);
        store8(img, row, c0 + 8, 128, v + 8);
      }
    }
  }
  // layer 3, and the output layer's two sums over the hidden units in order:
  // the four parts take their turns (their errors feed the BF16 gradients, and
  // a small batch shows another order)
  product(0, HID, 1);
  float o0 = 0.0f, o1 = 0.0f;
  {
    float a3[HID / kParts];
#pragma unroll
    for (int k = 0; k < HID / kParts; k += 32) {
      float v[32];
      tc::tmem_ld32(tl + c_lo + k, v);
#pragma unroll
      for (int i = 0; i < 32; ++i) a3[k + i] = v[i];
      add4<8>(a3 + k, mst + B3_OFF + c_lo + k);
    }
#pragma unroll
    for (int i = 0; i < HID / kParts; i += 2) gelu2(a3[i], a3[i + 1]);
#pragma unroll 1
    for (int turn = 0; turn < kParts; ++turn) {
      if (part == turn) {  // (warp-uniform)
        if (turn > 0) {
          o0 = sOut[0][row];
          o1 = sOut[1][row];
        }
        out_sums<HID / kParts / 4>(mst, c_lo, a3, o0, o1);
        sOut[0][row] = o0;
        sOut[1][row] = o1;
      }
      __syncthreads();
    }
    o0 = sOut[0][row] + __ldg(mst + B4_OFF);
    o1 = sOut[1][row] + __ldg(mst + B4_OFF + 1);
  }
  if constexpr (TRAIN) {
    // output layer: dL/dout / B; loss per row: sum over the two outputs of
    // e^2 / 2 (Huber with delta > 0: quadratic inside |e| <= delta, linear
    // outside).  The row's four threads hold the same values.
    float d0 = 0.0f, d1 = 0.0f;
    double se = 0.0;
    if (valid) {
      const float e[2] = {o0 - t.Y[src * OUT], o1 - t.Y[src * OUT + 1]};
      float g[2];
#pragma unroll
      for (int c = 0; c < 2; ++c) {
        const float ae = fabsf(e[c]);
        if (t.huber > 0.0f && ae > t.huber) {
          g[c] = copysignf(t.huber, e[c]);
          se += (double)t.huber * ((double)ae - 0.5 * t.huber);
        } else {
          g[c] = e[c];
          se += 0.5 * (double)e[c] * e[c];
        }
      }
      d0 = g[0] / (float)B;
      d1 = g[1] / (float)B;
    }
    float* red = s_red[quarter];  // dW4, db3, db2, db1, db4
    if (part == 0) {
      se = warp_sum_d(se);
      const float r0 = warp_sum(d0), r1 = warp_sum(d1);
      if (lane == 0) {
        s_loss[quarter] = se;
        red[5 * HID] = r0;
        red[5 * HID + 1] = r1;
      }
    }
    // dz3 = (W4^T dout) GELU'(z3), then dz2 and dz1 through the transposed
    // weights; each is the next product's A operand and an operand image of
    // the weight gradients
    for (int l = 2; l >= 0; --l) {
      if (l < 2) product(0, HID, 1);
      const float* bias = mst + (l == 0 ? B1_OFF : (l == 1 ? B2_OFF : B3_OFF));
      unsigned char* img = t.dz_img + ((size_t)l * gridDim.x + blockIdx.x) * kImgA;
#pragma unroll 1
      for (int c0 = c_lo; c0 < c_hi; c0 += 16) {
        float v[16], z[16];
        if (l == 0) {
          const float4* zr = reinterpret_cast<const float4*>(t.z + b * HID + c0);  // (this thread's own stores)
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 q = zr[i];
            z[4 * i] = q.x; z[4 * i + 1] = q.y; z[4 * i + 2] = q.z; z[4 * i + 3] = q.w;
          }
        } else {
          tc::tmem_ld16(tl + (l == 1 ? kZ2 : 0u) + c0, z);
          add4<4>(z, bias + c0);
        }
        if (l == 2) {
          float a[16], a1[16];
#pragma unroll
          for (int i = 0; i < 16; ++i) a[i] = z[i];
#pragma unroll
          for (int i = 0; i < 16; i += 2) gelu2(a[i], a[i + 1]);
#pragma unroll
          for (int i = 0; i < 4; ++i) {
            const float4 w0 = __ldg(reinterpret_cast<const float4*>(mst + W4_OFF + c0) + i);
            const float4 w1 = __ldg(reinterpret_cast<const float4*>(mst + W4_OFF + HID + c0) + i);
            v[4 * i] = d0 * w0.x + d1 * w1.x;
            v[4 * i + 1] = d0 * w0.y + d1 * w1.y;
            v[4 * i + 2] = d0 * w0.z + d1 * w1.z;
            v[4 * i + 3] = d0 * w0.w + d1 * w1.w;
          }
#pragma unroll
          for (int i = 0; i < 16; ++i) {
            a1[i] = d1 * a[i];
            a[i] = d0 * a[i];
          }
          const float w0 = colsum16(a), w1 = colsum16(a1);
          if (lane < 16) {
            red[c0 + lane] = w0;
            red[HID + c0 + lane] = w1;
          }
        } else {
          tc::tmem_ld16(tl + c0, v);
        }
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = valid ? v[i] * gelu_grad(z[i]) : 0.0f;
        const float sb = colsum16(v);
        if (lane < 16) red[(4 - l) * HID + c0 + lane] = sb;
        store8(img, row, c0, 128, v);
        store8(img, row, c0 + 8, 128, v + 8);
        if (l > 0) {
          store8(sA, row, c0, 128, v);
          store8(sA, row, c0 + 8, 128, v + 8);
        }
      }
    }
    __syncthreads();
    // the CTA's partial sums: the four quarters' values added in order
    float* pb = t.part_b + (long long)blockIdx.x * NB_PART;
    for (int i = tid; i < NB_PART; i += kTE) pb[i] = ((s_red[0][i] + s_red[1][i]) + s_red[2][i]) + s_red[3][i];
    if (tid == 0) t.part_loss[blockIdx.x] = ((s_loss[0] + s_loss[1]) + s_loss[2]) + s_loss[3];
  }
  if (!ok) atomicExch(&bad, 1);
  __syncthreads();
  if (!TRAIN && part == 0 && valid && bad == 0) {
    out[b * OUT] = o0;
    out[b * OUT + 1] = o1;
  }
  if (bad && tid == 0) {
    // no copy may still be landing in shared memory when the CTA exits
    for (int st = kStages - 2; st < kStages; ++st)
      tc::mbar_wait(&full[st & 1], (uint32_t)((st >> 1) & 1), kEnvPolls);
    raise_status(status, 2);
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, kCols);
}

// ---------------------------------------------------------------------------
// Weight gradients dW_l = dz_l^T a_{l-1} summed over the batch: M = 128 output
// features (one half), N = input features, K = the rows.  An operand image of
// mlp_kernel [feature / 8][row][8] is also the MN-major form of its transpose
// (descriptor: 8-row groups 128 B apart in K, 8-feature groups 128 * 16 B
// apart in M / N), so a tile's two images go from HBM to the tensor core by
// bulk copies, two tiles in flight, with no thread touching them (16,384 rows:
// 14.5 us, against 77 when each CTA transposed its operands element by
// element).  The
// CTA's range of tiles accumulates in TMEM and is written to the split's slab,
// summed over the splits in order by grad_reduce_kernel.  grid = (batch
// splits, output half, layer).
// ---------------------------------------------------------------------------
constexpr size_t kWgradStage = kImgA / 2 + kImgA;  // half of dz's features, all of a's
constexpr size_t kWgradSmem = 2 * kWgradStage;

__global__ void __launch_bounds__(kT, 1) wgrad_kernel(TrainBufs t, int* status) {
  extern __shared__ __align__(1024) unsigned char smem[];
  __shared__ __align__(8) uint64_t full[2];
  __shared__ __align__(8) uint64_t done[2];
  __shared__ uint32_t tbase;
  __shared__ int bad;
  const int tid = threadIdx.x, warp = tid >> 5;
  const int layer = blockIdx.z, half = blockIdx.y;
  const int n_in = layer == 0 ? IN : HID;
  const int n_tiles = (t.B + kT - 1) / kT;
  const int per = (n_tiles + gridDim.x - 1) / gridDim.x;
  const int begin = blockIdx.x * per, n = min(n_tiles, begin + per) - begin;  // n <= 0: no rows left for this split

  if (warp == 0) {
    tc::tmem_alloc(&tbase, 256);
    tc::tmem_relinquish();
  }
  if (tid == 0) {
    for (int k = 0; k < 2; ++k) {
      tc::mbar_init(&full[k], 1);
      tc::mbar_init(&done[k], 1);
    }
    bad = 0;
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  const uint32_t tmem = tbase;
  if (tid == 0 && n > 0) {
    const uint32_t bytes_b = (uint32_t)(kT * n_in * 2);
    auto fetch = [&](int c) {
      const size_t tile = (size_t)begin + c;
      unsigned char* dst = smem + (c & 1) * kWgradStage;
      const unsigned char* dz = t.dz_img + ((size_t)layer * n_tiles + tile) * kImgA + half * (kImgA / 2);
      const unsigned char* a =
          layer == 0 ? t.x_img + tile * kImgX : t.a_img + ((size_t)(layer - 1) * n_tiles + tile) * kImgA;
      tc::mbar_expect_tx(&full[c & 1], (uint32_t)(kImgA / 2) + bytes_b);
      tc::bulk_g2s(dst, dz, (uint32_t)(kImgA / 2), &full[c & 1]);
      tc::bulk_g2s(dst + kImgA / 2, a, bytes_b, &full[c & 1]);
    };
    const uint32_t idesc = tc::idesc_bf16(128, (uint32_t)n_in) | (1u << 15) | (1u << 16);  // both MN-major
    bool ok = true;
    int fetched = min(n, 2);
    for (int c = 0; c < fetched; ++c) fetch(c);
    for (int c = 0; c < n && ok; ++c) {
      ok = tc::mbar_wait(&full[c & 1], (uint32_t)((c >> 1) & 1), kEnvPolls);
      if (!ok) break;
      const uint32_t aa = tc::smem_addr(smem + (c & 1) * kWgradStage), bb = aa + (uint32_t)(kImgA / 2);
      const uint64_t ad = tc::smem_desc(aa, 128, kT * 16), bd = tc::smem_desc(bb, 128, kT * 16);
#pragma unroll
      for (int j = 0; j < kT / 16; ++j)
        tc::mma_bf16(tmem, tc::desc_advance(ad, j * 256), tc::desc_advance(bd, j * 256), idesc,
                     (c > 0 || j > 0) ? 1u : 0u);
      tc::mma_commit(&done[c & 1]);
      if (c + 1 < n) {  // refill the other stage once its MMAs (tile c - 1) are through
        if (c >= 1 && fetched < n) {
          ok = tc::mbar_wait(&done[(c - 1) & 1], (uint32_t)(((c - 1) >> 1) & 1), kEnvPolls);
          if (ok) fetch(fetched++);
        }
      }
    }
    if (ok) ok = tc::mbar_wait(&done[(n - 1) & 1], (uint32_t)(((n - 1) >> 1) & 1), kEnvPolls);
    if (!ok) {  // no copy may still be landing when the CTA exits
      bad = 1;
      for (int c = max(0, fetched - 2); c < fetched; ++c)
        tc::mbar_wait(&full[c & 1], (uint32_t)((c >> 1) & 1), kEnvPolls);
      raise_status(status, 2);
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  tc::fence_after_sync();
  if (!bad) {
    // this split's slab: dW1 [256][96], then dW2 and dW3 [256][256]
    const long long w_off = layer == 0 ? 0 : (long long)HID * IN + (long long)(layer - 1) * HID * HID;
    float* pw = t.part_w + (long long)blockIdx.x * NW_PART + w_off + (long long)(half * 128 + tid) * n_in;
    const uint32_t lane = tmem + ((uint32_t)(warp * 32) << 16);
    for (int c0 = 0; c0 < n_in; c0 += 16) {
      float v[16];
      if (n > 0) {
        tc::tmem_ld16(lane + c0, v);
      } else {
#pragma unroll
        for (int i = 0; i < 16; ++i) v[i] = 0.0f;
      }
#pragma unroll
      for (int i = 0; i < 16; i += 4)
        *reinterpret_cast<float4*>(pw + c0 + i) = make_float4(v[i], v[i + 1], v[i + 2], v[i + 3]);
    }
  }
  tc::fence_before_sync();
  __syncthreads();
  if (warp == 0) tc::tmem_dealloc(tmem, 256);
}

// Canonical parameter offset of a slab position: `which` 0 for the bias /
// output-layer slab, 1 for the hidden weight slab.
__device__ __forceinline__ long long part_dst(int which, long long i) {
  if (which == 0) {
    if (i < 2 * HID) return W4_OFF + i;
    if (i < 3 * HID) return B3_OFF + (i - 2 * HID);
    if (i < 4 * HID) return B2_OFF + (i - 3 * HID);
    if (i < 5 * HID) return B1_OFF + (i - 4 * HID);
    return B4_OFF + (i - 5 * HID);
  }
  if (i < (long long)HID * IN) return W1_OFF + i;
  if (i < (long long)HID * IN + (long long)HID * HID) return W2_OFF + (i - (long long)HID * IN);
  return W3_OFF + (i - (long long)HID * IN - (long long)HID * HID);
}

// Gradient and loss from the partial slabs, every sum in a fixed order.
// Blocks 0 .. kRedW - 1: four hidden weights per thread, over the splits in
// order (the slabs' tensors start at multiples of 4, so a thread's four stay
// in one tensor; 4 us for all three kinds, 34 as three kernels).  The next
// kRedB: 32 entries of the bias slab each, thread
// row g the parts p = g (mod 8), then the 8 row sums in order.  The last: the
// loss, parts p = i (mod 256), then warp and block sums.
constexpr int kRedW = (int)((NW_PART / 4 + 255) / 256), kRedB = (NB_PART + 31) / 32;

__global__ void __launch_bounds__(256) grad_reduce_kernel(TrainBufs t, int splits, int n_cta) {
  const int tid = threadIdx.x;
  // partial sums of a pass that gave up, or of an earlier one, go no further
  // (looked at behind the sums: its load is in flight during theirs)
  const int gave_up = t.result->status;
  if (blockIdx.x < kRedW) {
    const long long i = ((long long)blockIdx.x * 256 + tid) * 4;
    if (i >= NW_PART) return;
    float4 s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll 8
    for (int p = 0; p < splits; ++p) {
      const float4 v = *reinterpret_cast<const float4*>(t.part_w + (long long)p * NW_PART + i);
      s.x += v.x; s.y += v.y; s.z += v.z; s.w += v.w;
    }
    if (gave_up) return;
    float* g = t.grad + part_dst(1, i);
    g[0] = s.x; g[1] = s.y; g[2] = s.z; g[3] = s.w;
    return;
  }
  if (blockIdx.x < kRedW + kRedB) {
    __shared__ float red[8][33];
    const int c = tid & 31, g = tid >> 5, i = ((int)blockIdx.x - kRedW) * 32 + c;
    float s = 0.0f;
    if (i < NB_PART) {
#pragma unroll 8
      for (int p = g; p < n_cta; p += 8) s += t.part_b[(long long)p * NB_PART + i];
    }
    red[g][c] = s;
    __syncthreads();
    if (g == 0 && i < NB_PART && !gave_up) {
      float acc = 0.0f;
#pragma unroll
      for (int k = 0; k < 8; ++k) acc += red[k][c];
      t.grad[part_dst(0, i)] = acc;
    }
    return;
  }
  __shared__ double sl[8];
  double s = 0.0;
  for (int p = tid; p < n_cta; p += 256) s += t.part_loss[p];
  s = warp_sum_d(s);
  if ((tid & 31) == 0) sl[tid >> 5] = s;
  __syncthreads();
  if (tid == 0 && !gave_up) {
    double acc = 0.0;
#pragma unroll
    for (int k = 0; k < 8; ++k) acc += sl[k];
    t.result->loss = acc / t.B;
  }
}

// Image position of weight element (layer, out, in) in the forward operand
// (chunks of 128 output rows) and, for layers 2 and 3, in the transposed one.
__device__ __forceinline__ void write_images(unsigned char* img, long long i, float w) {
  const uint16_t bits = f2bf_bits(w);
  if (i >= W1_OFF && i < B1_OFF) {
    const int o = (int)((i - W1_OFF) / IN), in = (int)((i - W1_OFF) % IN);
    *reinterpret_cast<uint16_t*>(img + IMG_W1_OFF + (size_t)(o / 128) * 128 * IN * 2 +
                                 tc::kmajor_offset(o % 128, in, 128)) = bits;
  } else if ((i >= W2_OFF && i < B2_OFF) || (i >= W3_OFF && i < B3_OFF)) {
    const bool l2 = i < B2_OFF;
    const long long r = i - (l2 ? W2_OFF : W3_OFF);
    const int o = (int)(r / HID), in = (int)(r % HID);
    const size_t fw = l2 ? IMG_W2_OFF : IMG_W3_OFF, bw = l2 ? IMG_W2T_OFF : IMG_W3T_OFF;
    *reinterpret_cast<uint16_t*>(img + fw + (size_t)(o / 128) * 128 * HID * 2 + tc::kmajor_offset(o % 128, in, 128)) =
        bits;
    *reinterpret_cast<uint16_t*>(img + bw + (size_t)(in / 128) * 128 * HID * 2 + tc::kmajor_offset(in % 128, o, 128)) =
        bits;
  }
}

__global__ void adam_kernel(float* master, float* m, float* v, const float* grad, float lr, float beta1, float beta2,
                            float eps, float c1, float c2, unsigned char* img, EstResult* result) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= NPARAM) return;
  const int gave_up = result ? result->status : 0;
  const float g = grad[i];
  const float mi = beta1 * m[i] + (1.0f - beta1) * g;
  const float vi = beta2 * v[i] + (1.0f - beta2) * g * g;
  const float th = master[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
  if (gave_up) return;
  if (result && i == 0) ++result->updates;
  m[i] = mi;
  v[i] = vi;
  master[i] = th;
  write_images(img, i, th);
}

__global__ void pack_kernel(const float* master, unsigned char* img) {
  const long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (i < NPARAM) write_images(img, i, master[i]);
}

__global__ void batch_rows_kernel(int32_t* rows, int B, uint32_t n_rows, uint64_t seed, uint32_t step) {
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  if (b >= B) return;
  Rand4 r = philox((uint32_t)b, step, 0u, TAG_BATCH, seed);
  rows[b] = (int32_t)__umulhi(r.x[0], n_rows);
}

__global__ void record_kernel(EnvDev d, float* feat, float* label) {
  const int f = blockIdx.x * blockDim.x + threadIdx.x;
  if (f >= d.F) return;
  // after the step: the update's inputs are the estimate history
  const float e1x = d.prev_estx[f], e1y = d.prev_esty[f];
  float x[IN];
  ring_features<0, false>(d, f, d.counters[0], e1x, e1y, d.prev2_estx[f], d.prev2_esty[f], d.velx[f], d.vely[f], x);
#pragma unroll
  for (int i = 0; i < IN; i += 4)
    *reinterpret_cast<float4*>(feat + (long long)f * IN + i) = make_float4(x[i], x[i + 1], x[i + 2], x[i + 3]);
  const int it = d.filt_target[f];
  label[(long long)f * 2] = (d.tx[it] - e1x) / d.est_scale;
  label[(long long)f * 2 + 1] = (d.ty[it] - e1y) / d.est_scale;
}

}  // namespace

cudaError_t launch_forward(const Net& net, const float* X, int B, float* out, int* status, uint32_t test_wait_polls,
                           cudaStream_t s) {
  static std::atomic<unsigned long long> ready{0};
  cudaError_t e = smem_optin(mlp_kernel<false>, kEnvSmem, ready);
  if (e != cudaSuccess) return e;
  if (B <= 0) return cudaSuccess;
  mlp_kernel<false><<<(B + kT - 1) / kT, kTE, kEnvSmem, s>>>(net, X, nullptr, B, out, TrainBufs{}, status,
                                                              test_wait_polls);
  return cudaGetLastError();
}

cudaError_t launch_forward_env(const Net& net, const EnvDev& d, int stale, uint32_t test_wait_polls,
                               cudaStream_t s) {
  static std::atomic<unsigned long long> ready{0};
  cudaError_t e = smem_optin(fwd_env_kernel, kEnvSmem, ready);
  if (e != cudaSuccess) return e;
  if (d.F <= 0) return cudaSuccess;
  launch_pdl(fwd_env_kernel, dim3((d.F + 127) / 128), dim3(kTE), kEnvSmem, s, net, d, stale, test_wait_polls);
  return cudaGetLastError();
}

cudaError_t launch_record(const EnvDev& d, float* feat, float* label, cudaStream_t s) {
  if (d.F <= 0) return cudaSuccess;
  record_kernel<<<(d.F + 127) / 128, 128, 0, s>>>(d, feat, label);
  return cudaGetLastError();
}

cudaError_t launch_loss_grad(const Net& net, const TrainBufs& t, cudaStream_t s) {
  static std::atomic<unsigned long long> ready_m{0}, ready_w{0};
  cudaError_t e = smem_optin(mlp_kernel<true>, kEnvSmem, ready_m);
  if (e == cudaSuccess) e = smem_optin(wgrad_kernel, kWgradSmem, ready_w);
  if (e != cudaSuccess) return e;
  if (t.B <= 0) return cudaSuccess;
  const int n_cta = (t.B + kT - 1) / kT;
  mlp_kernel<true><<<n_cta, kTE, kEnvSmem, s>>>(net, t.X, t.rows, t.B, nullptr, t, &t.result->status,
                                                t.test_wait_polls);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int splits = n_cta < kWgradSplits ? n_cta : kWgradSplits;
  wgrad_kernel<<<dim3(splits, 2, 3), kT, kWgradSmem, s>>>(t, &t.result->status);
  e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  grad_reduce_kernel<<<kRedW + kRedB + 1, 256, 0, s>>>(t, splits, n_cta);
  return cudaGetLastError();
}

cudaError_t launch_adam(float* master, float* m, float* v, const float* grad, int step, float lr, float beta1,
                        float beta2, float eps, unsigned char* img, EstResult* result, cudaStream_t s) {
  const double c1 = 1.0 - std::pow((double)beta1, step), c2 = 1.0 - std::pow((double)beta2, step);
  adam_kernel<<<(unsigned)((NPARAM + 255) / 256), 256, 0, s>>>(master, m, v, grad, lr, beta1, beta2, eps, (float)c1,
                                                              (float)c2, img, result);
  return cudaGetLastError();
}

cudaError_t launch_pack(const float* master, unsigned char* img, cudaStream_t s) {
  pack_kernel<<<(unsigned)((NPARAM + 255) / 256), 256, 0, s>>>(master, img);
  return cudaGetLastError();
}

cudaError_t launch_batch_rows(int32_t* rows, int B, int64_t n_rows, uint64_t seed, uint32_t step, cudaStream_t s) {
  batch_rows_kernel<<<(B + 255) / 256, 256, 0, s>>>(rows, B, (uint32_t)n_rows, seed, step);
  return cudaGetLastError();
}

}  // namespace est
}  // namespace ut
