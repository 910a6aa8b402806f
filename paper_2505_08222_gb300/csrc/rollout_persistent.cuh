// Persistent rollout: T environment steps in one launch, one CTA per
// environment.
//
// Environments are independent (the step vectorises over them, Sec.
// III-A.3), so a CTA can advance its own environment through all T steps
// with block barriers only, no grid-wide synchronisation.  The filter step of
// each of the environment's filters runs on NT threads (the same device code
// as pf_step_kernel); one more warp owns the environment.  With random actions
// a step's move, pings and messages do not depend on the filters, so while they
// run step t that warp already prepares step t + 1 (its measurement lists go to
// one of two shared-memory copies) and then takes step t - 1's errors into the
// metrics: a step lasts as long as its filters.  Observation tokens are written
// for the last step alone: no other step's can be read.  (64 environments of
// one filter of 1000 particles: the environment's stages in line with the
// filter took 7.3 us per step, this 4.0.)  An environment with a single
// filter keeps that filter's particles in registers for the whole rollout: they
// are read from HBM once before the first step and written once after the last.
// The counters and the episode-end flag follow the step-by-step rollout exactly
// (global step g = counters[0] + 1 + t), so the results equal the graph
// rollout's bit for bit when both use the same filter launch shape (NT, PPT);
// the device metrics are the same sums added in another order.
//
// Actions are the environment's uniform random actions: the transformer
// agent and the learned estimator run as their own kernels and keep the
// graph rollout.
#pragma once

#include "env_step.cuh"
#include "pf_kernel.cuh"

namespace ut {
namespace persist {

// Threads of the kernel: the environment's warp beside the filter's, or (NT =
// 1024, a CTA's limit) the filter's warp 0 in turn.
template <int NT>
constexpr int rollout_threads() {
  return NT < 1024 ? NT + 32 : NT;
}
// Shared-memory copies of what the environment's stage and the filters hand
// each other within a step: measurement lists, headers, errors; two of each.
inline size_t rollout_stage_bytes(int filters, int AM) { return 2 * (size_t)filters * (AM * 16 + 16 + 4) + 16; }

// CTAs per SM that the registers must allow when there are more environments than
// SMs: small filters leave room for several on an SM, and left to itself the
// compiler gives the environment's stage that room (202 to 216 registers at 4
// particles per thread and up to 128 threads; 80 to 128 capped).  (50 steps of
// 2000 environments of 1000 particles: 2984 us with one CTA per SM, 1729 with two;
// 600 of 400: 950 and 517.  Up to one environment per SM the registers are worth
// more: 64 of 2 x 2, 100 particles: 580 us, 614 with the cap.)
template <int NT, int PPT>
constexpr int rollout_min_blocks() {
  if (PPT > 4) return NT <= 64 ? 4 : (NT <= 128 ? 2 : 1);
  return NT <= 32 ? 12 : (NT <= 64 ? 6 : (NT <= 128 ? 3 : (NT <= 256 ? 2 : 1)));
}

template <int NT, int PPT, int MODE, int MINB>
__global__ void __launch_bounds__(rollout_threads<NT>(), MINB) rollout_kernel(EnvDev d, int T, int max_filters) {
  constexpr bool kOwnWarp = rollout_threads<NT>() > NT;
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ EnvWarpSmem ew;
  const int e = blockIdx.x;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t g0 = d.counters[0], t0 = d.counters[1];
  const int f0 = d.filter_off[e], nf = d.filter_off[e + 1] - f0;
  const int a0 = d.agent_off[e], A = d.agent_off[e + 1] - a0, k0 = d.target_off[e], K = d.target_off[e + 1] - k0;
  const bool resident = nf == 1;  // (CTA-uniform)
  const bool env_warp = kOwnWarp ? warp == NT / 32 : warp == 0;
  const bool filter_warp = warp < NT / 32;
  // step t's lists, headers and errors of this environment's filters: one of two
  // copies in shared memory; the last step's go to the handle's own buffers
  float4* s_meas = reinterpret_cast<float4*>(smem_raw + pf::step_smem_bytes(NT, PPT));
  float4* s_hdr = s_meas + 2 * max_filters * d.AM;
  float* s_err = reinterpret_cast<float*>(s_hdr + 2 * max_filters);
  auto lists = [&](int t) {
    if (t + 1 >= T || !UT_IN_BOUNDS(nf <= max_filters, d.status)) return StepLists{d.meas, d.meas_hdr, d.err};
    const int c = t & 1;
    return StepLists{s_meas + c * max_filters * d.AM - (long long)f0 * d.AM, s_hdr + c * max_filters - f0,
                     s_err + c * max_filters - f0};
  };
  float x[PPT], y[PPT], vx[PPT], vy[PPT];
  if (resident && filter_warp) pf::load_particles<NT, PPT, MODE>(d, f0, x, y, vx, vy);
  StepMetrics acc;
  PosReward pos, pos_prev;
  auto account = [&](int t, const PosReward& q) {  // step t's reward and errors (all but the last step)
    double se;
    const float r = reward_errors(d, q, A, K, nf, lists(t).err() + f0, se);
    acc.sq += se;
    acc.rw += (double)r;
    acc.n_err += (unsigned long long)nf;
    acc.n_crash += (unsigned long long)q.cr;
    acc.n_agents += (unsigned long long)A;
  };
  if (env_warp) step_env_warp(d, lists(0), e, nullptr, g0 + 1u, ew);
  __syncthreads();  // measurement lists and headers of step 0
  for (int t = 0; t < T; ++t) {
    if (filter_warp) {
      const StepLists in = lists(t);
      const uint32_t g = g0 + 1u + (uint32_t)t;
      if (resident) {
        pf::pf_step_body<NT, PPT, MODE, false, true, kOwnWarp>(d, in, f0, g, x, y, vx, vy);
      } else {
        for (int k = 0; k < nf; ++k) {
          pf::pf_step_body<NT, PPT, MODE, false, false, kOwnWarp>(d, in, f0 + k, g, x, y, vx, vy);
          if (k + 1 < nf) pf::filter_bar<NT, kOwnWarp>();
        }
      }
    }
    if (env_warp && t + 1 < T) {
      pos_prev = pos;
      pos = reward_positions(d, a0, A, k0, K);  // of step t, before the move of step t + 1
      if (kOwnWarp) step_env_warp(d, lists(t + 1), e, nullptr, g0 + 2u + (uint32_t)t, ew);
      if (kOwnWarp && t > 0) account(t - 1, pos_prev);
    }
    __syncthreads();  // step t's errors, step t + 1's lists; the filter's shared memory free again
    if (!kOwnWarp && t + 1 < T) {
      if (env_warp) {
        step_env_warp(d, lists(t + 1), e, nullptr, g0 + 2u + (uint32_t)t, ew);
        account(t, pos);
      }
      __syncthreads();
    }
  }
  if (env_warp) {
    if (kOwnWarp && T > 1) account(T - 2, pos);
    StepMetrics m;
    obs_reward_warp(d, e, 0, t0 + (uint32_t)T, m);
    acc.sq += m.sq;
    acc.rw += m.rw;
    acc.n_err += m.n_err;
    acc.n_crash += m.n_crash;
    acc.n_agents += m.n_agents;
  }
  if (resident && filter_warp) pf::store_particles<NT, PPT, MODE>(d, f0, x, y, vx, vy);
  if (env_warp && lane == 0) {
    atomicAdd(&d.metrics_d[0], acc.sq);
    atomicAdd(&d.metrics_d[1], acc.rw);
    atomicAdd(&d.metrics_u[0], acc.n_err);
    atomicAdd(&d.metrics_u[1], acc.n_crash);
    atomicAdd(&d.metrics_u[2], acc.n_agents);
  }
}

template <int NT, int PPT, int MODE, int MINB>
cudaError_t launch_blocks(const EnvDev& d, int T, cudaStream_t s) {
  static std::atomic<unsigned long long> ready{0};
  auto k = rollout_kernel<NT, PPT, MODE, MINB>;
  const int filters = d.shared_filter ? d.TM : d.AM * d.TM;
  const cudaError_t e =
      smem_optin(k, pf::step_smem_bytes(NT, PPT) + rollout_stage_bytes(kMaxAgents * kMaxTargets, kMaxAgents), ready);
  if (e != cudaSuccess) return e;
  const size_t smem = pf::step_smem_bytes(NT, PPT) + rollout_stage_bytes(filters, d.AM);
  k<<<d.E, rollout_threads<NT>(), smem, s>>>(d, T, filters);
  return cudaGetLastError();
}

template <int NT, int PPT, int MODE>
cudaError_t launch_mode(const EnvDev& d, int T, cudaStream_t s) {
  return d.E > 152 ? launch_blocks<NT, PPT, MODE, rollout_min_blocks<NT, PPT>()>(d, T, s)
                   : launch_blocks<NT, PPT, MODE, 1>(d, T, s);
}

template <int NT, int PPT>
cudaError_t launch_shape(const EnvDev& d, int T, cudaStream_t s) {
  if (d.P > NT * PPT) return cudaErrorInvalidValue;
  if (d.P == NT * PPT) return launch_mode<NT, PPT, 2>(d, T, s);
  if (d.P % 4 == 0) return launch_mode<NT, PPT, 1>(d, T, s);
  return launch_mode<NT, PPT, 0>(d, T, s);
}

}  // namespace persist
}  // namespace ut
