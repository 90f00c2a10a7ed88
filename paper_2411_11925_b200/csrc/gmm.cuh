// Gaussian-mixture output heads (the paper's appendix on model variants): per token an explicit mixture
// p(x) = sum_k pi_k N(x; mu_k, diag(sigma_k^2)) instead of a diffusion head.  Both densities are closed forms, so a
// round is: draft samples x_i ~ q_i, ratio p_i(x_i) / q_i(x_i), accepted prefix (Sec. 3.1 rule, Alg. 1), and
// acceptance-rejection resampling of the first rejected position from max(0, p - q)/Z (Eq. 5, Eq. 9-11) with
// proposals from p.
//
// These kernels are a few microseconds of dependent memory trips and shuffles, so each lane does whole pieces of work
// instead of one coordinate of a shared one: a lane evaluates a component over all coordinates (densities of one row) or
// a proposal over all components (resampling).  The sums over coordinates keep the order of a butterfly over 32 lanes
// and the sums over components run in component order, so a row's bits do not depend on which kernel evaluates it, and
// identical mixtures give identical bits.  C <= 32.
#pragma once
#include <cuda_runtime.h>
#include <stdint.h>

#include "rowops.cuh"

namespace csd {

constexpr int kGmmC = 32;   // widest token

struct GmmView {
  int K;
  const float* logw;       // [rows, K] unnormalised log-weights
  const float* mu;         // [rows, K, C]
  const float* log_sigma;  // [rows, K, C]
};

constexpr float kHalfLog2Pi = 0.9189385332046727f;

// Butterfly-ordered sum of 32 values of which those beyond C are zero (C <= 16: the first level adds zeros only).
template <int CP> __device__ __forceinline__ float gmm_tree_sum(float* v) {
#pragma unroll
  for (int o = CP / 2; o > 0; o >>= 1)
#pragma unroll
    for (int c = 0; c < o; ++c) v[c] = __fadd_rn(v[c], v[c + o]);
  return v[0];
}

// log of the weights' normaliser, log sum_k exp(logw_k), by WIDTH lanes together: the exponentials in parallel, their
// sum in component order.
template <int WIDTH>
__device__ __forceinline__ float gmm_log_norm(const float* lw, int K, int sub) {
  float mx = -INFINITY;
  for (int k = sub; k < K; k += WIDTH) mx = fmaxf(mx, lw[k]);
#pragma unroll
  for (int o = WIDTH / 2; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, o, WIDTH));
  float se = 0.0f;
  // (both halves of the warp take as many turns as the longer mixture needs: the shuffles are warp-wide)
  const int turns = __reduce_max_sync(0xffffffffu, K);
  for (int g = 0; g < turns; g += WIDTH) {
    const float e = g + sub < K ? expf(lw[g + sub] - mx) : 0.0f;
    for (int j = 0; j < WIDTH && g + j < turns; ++j) se += __shfl_sync(0xffffffffu, e, j, WIDTH);   // zeros beyond K
  }
  return mx + logf(se);
}

// One more component of a running log-sum-exp.
__device__ __forceinline__ void gmm_lse_add(float comp, float& run_m, float& run_s) {
  if (comp > run_m) { run_s = run_s * expf(run_m - comp) + 1.0f; run_m = comp; }
  else run_s += expf(comp - run_m);
}

// log-densities of one row under two mixtures by one warp: lanes 0..15 evaluate components of p, lanes 16..31 of q, each
// lane a component over all coordinates (xs: the row's token in shared memory, zero padded).  Returns the lane half's
// own density.
template <int CP>
__device__ __forceinline__ float gmm_row_logpdf_pair(const GmmView& m, size_t row, int C, int lane, const float* xs) {
  const int sub = lane & 15;
  const float* lw = m.logw + row * m.K;
  const float lse = gmm_log_norm<16>(lw, m.K, sub);
  const int turns = __reduce_max_sync(0xffffffffu, m.K);
  float run_m = -INFINITY, run_s = 0.0f;
  for (int g = 0; g < turns; g += 16) {
    const int k = g + sub;
    float comp = 0.0f;
    if (k < m.K) {
      const float* mu = m.mu + (row * m.K + k) * C;
      const float* ls = m.log_sigma + (row * m.K + k) * C;
      float t[CP], sl[CP];
#pragma unroll
      for (int c = 0; c < CP; ++c) { sl[c] = c < C ? ls[c] : 0.0f; t[c] = c < C ? mu[c] : 0.0f; }
#pragma unroll
      for (int c = 0; c < CP; ++c) {
        const float d = (xs[c] - t[c]) * expf(-sl[c]);
        t[c] = c < C ? __fmul_rn(d, d) : 0.0f;
      }
      const float st = gmm_tree_sum<CP>(t), ss = gmm_tree_sum<CP>(sl);
      comp = (lw[k] - lse) - ss - 0.5f * st - kHalfLog2Pi * C;
    }
    for (int j = 0; j < 16 && g + j < turns; ++j) {
      const float cj = __shfl_sync(0xffffffffu, comp, j, 16);
      if (g + j < m.K) gmm_lse_add(cj, run_m, run_s);
    }
  }
  return run_m + logf(run_s);
}

// Draft samples: x[row] = mu_k + sigma_k * noise[row], k = CDF inverse of the weights at u_comp[row]: the component
// whose cumulative weight first reaches u (the last one if rounding leaves the total short).  One warp per row.
__global__ void __launch_bounds__(128)
gmm_sample_kernel(int R, int C, GmmView q, const float* __restrict__ u_comp, const float* __restrict__ noise,
                  float* __restrict__ x, int32_t* __restrict__ comp) {
  griddep_enter();
  const int row = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (row >= R) return;
  const float u = u_comp[row];
  const float nz = lane < C ? noise[static_cast<size_t>(row) * C + lane] : 0.0f;
  const float* lw = q.logw + static_cast<size_t>(row) * q.K;
  const float lse = gmm_log_norm<32>(lw, q.K, lane);
  float cum = 0.0f;
  int k = q.K - 1;
  for (int g = 0; g < q.K - 1 && k == q.K - 1; g += 32) {
    const float e = g + lane < q.K ? expf(lw[g + lane] - lse) : 0.0f;
    for (int j = 0; j < 32 && g + j < q.K - 1; ++j) {
      cum += __shfl_sync(0xffffffffu, e, j);
      if (!(cum < u)) { k = g + j; break; }
    }
  }
  if (lane < C) {
    const size_t o = (static_cast<size_t>(row) * q.K + k) * C + lane;
    x[static_cast<size_t>(row) * C + lane] = fmaf(expf(q.log_sigma[o]), nz, q.mu[o]);
  }
  if (comp && lane == 0) comp[row] = k;
}

// One block per sequence, warp i = draft position i (gamma <= 32): logratio = log p(x) - log q(x), accept iff
// log u <= logratio, n_accept = number of leading accepts.
template <int CP>
__global__ void __launch_bounds__(1024)
gmm_verify_kernel(int B, int gamma, int C, GmmView q, GmmView p, const float* __restrict__ x, const float* __restrict__ u,
                  float* __restrict__ logratio, int32_t* __restrict__ n_accept, uint32_t* __restrict__ accept_mask) {
  __shared__ int acc_s[32];
  __shared__ float xs[32][kGmmC];
  griddep_enter();
  const int b = blockIdx.x, i = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const size_t row = static_cast<size_t>(b) * gamma + i;
  const float uv = u[row];
  xs[i][lane] = lane < C ? x[row * C + lane] : 0.0f;
  __syncwarp();
  const float lpq = gmm_row_logpdf_pair<CP>(lane < 16 ? p : q, row, C, lane, xs[i]);
  const float lq = __shfl_sync(0xffffffffu, lpq, 16);
  const float lr = __fsub_rn(lpq, lq);
  if (lane == 0) { logratio[row] = lr; acc_s[i] = logf(uv) <= lr ? 1 : 0; }
  __syncthreads();
  if (threadIdx.x < 32) {
    const uint32_t mask = __ballot_sync(0xffffffffu, lane < gamma && acc_s[lane] != 0);
    if (lane == 0) {
      const uint32_t rej = ~mask & (gamma >= 32 ? 0xffffffffu : ((1u << gamma) - 1u));
      n_accept[b] = rej ? (__ffs(rej) - 1) : gamma;
      if (accept_mask) accept_mask[b] = mask;
    }
  }
}

// Resampling: one block per sequence, 64 proposals x' of the first rejected row at a time, alpha_s = max(0, 1 - q(x') / p(x'));
// the first accepted one in order is taken.  Warps 0 and 2 evaluate log p of proposals 0..31 and 32..63, warps 1 and 3 log
// q, a lane per proposal.  What the proposals share (means, standard deviations and their reciprocals, per-component
// constants, component weights) is put in shared memory once when it fits (SMEM), else read and formed on the fly.
// Evaluating proposals one after the other instead (a warp per sequence, a lane per coordinate) took 30 us at 37
// sequences, K = 6, C = 16, where some sequences need tens of proposals; this form is a few dependent trips to memory.
struct GmmResampleParams {
  int B, gamma, C, cap;
  GmmView q, p;
  const int32_t* n_accept;
  const float *w, *xi, *v;
  float* x_new;
  int32_t* n_prop;
  uint32_t* flags;
  int32_t* cap_hits;
  unsigned long long* tally;
};
constexpr int kGmmProposals = 64;   // proposals per pass
__host__ __device__ inline size_t gmm_resample_smem_floats(int Kq, int Kp, int C) {
  return static_cast<size_t>(3 * Kp + 2 * Kq) * C + 2 * Kp + Kq;
}

template <int CP, bool SMEM>
__global__ void __launch_bounds__(128) gmm_resample_kernel(const GmmResampleParams p) {
  extern __shared__ float sm[];
  __shared__ float dens[2][kGmmProposals];
  __shared__ int first_s;
  const int b = blockIdx.x, tid = threadIdx.x, lane = tid & 31, C = p.C, Kp = p.p.K, Kq = p.q.K;
  const int side = (tid >> 5) & 1, slot = (tid >> 6) * 32 + lane;   // side 0: p, 1: q
  griddep_enter();
  const int n = p.n_accept[b];
  int hit = 0;
  if (n >= p.gamma) {
    if (tid == 0) { p.n_prop[b] = 0; p.flags[b] = 0u; }
  } else {
    const size_t row = static_cast<size_t>(b) * p.gamma + n;
    const float *gmu_p = p.p.mu + row * Kp * C, *gls_p = p.p.log_sigma + row * Kp * C;
    const float *gmu_q = p.q.mu + row * Kq * C, *gls_q = p.q.log_sigma + row * Kq * C;
    const float *lw_p = p.p.logw + row * Kp;
    float *mu_p = sm, *inv_p = mu_p + Kp * C, *sig_p = inv_p + Kp * C, *mu_q = sig_p + Kp * C, *inv_q = mu_q + Kq * C;
    float *base_p = inv_q + Kq * C, *wt_p = base_p + Kp, *base_q = wt_p + Kp;
    // this warp's mixture
    const int K = side ? Kq : Kp;
    const float *gmu = side ? gmu_q : gmu_p, *gls = side ? gls_q : gls_p, *lw = side ? p.q.logw + row * Kq : lw_p;
    const float *mu = side ? mu_q : mu_p, *inv = side ? inv_q : inv_p;
    float* base = side ? base_q : base_p;
    if (SMEM) {
      for (int i = tid; i < Kp * C; i += 128) { const float s = gls_p[i]; mu_p[i] = gmu_p[i]; inv_p[i] = expf(-s); sig_p[i] = expf(s); }
      for (int i = tid; i < Kq * C; i += 128) { mu_q[i] = gmu_q[i]; inv_q[i] = expf(-gls_q[i]); }
    }
    const float lse = gmm_log_norm<32>(lw, K, lane);
    const float lse_p = SMEM ? lse : gmm_log_norm<32>(lw_p, Kp, lane);   // (used by the p warps only when SMEM)
    // (log weight - normaliser) - sum of log sigma of one component
    auto comp_base = [&](int k) {
      float sl[CP];
#pragma unroll
      for (int c = 0; c < CP; ++c) sl[c] = c < C ? gls[k * C + c] : 0.0f;
      return (lw[k] - lse) - gmm_tree_sum<CP>(sl);
    };
    if (SMEM) {
      if (tid < 64) for (int k = lane; k < K; k += 32) { base[k] = comp_base(k); if (side == 0) wt_p[k] = expf(lw_p[k] - lse_p); }
      __syncthreads();
    }
    int k = p.cap;
    bool done = false;
    for (int k0 = 0; k0 < p.cap && !done; k0 += kGmmProposals) {
      const int kk = k0 + slot < p.cap ? k0 + slot : p.cap - 1;
      const size_t pr = static_cast<size_t>(b) * p.cap + kk;
      const float u = p.w[pr], vk = p.v[pr];
      float x[CP];
#pragma unroll
      for (int c = 0; c < CP; ++c) x[c] = c < C ? p.xi[pr * C + c] : 0.0f;
      float cum = 0.0f;
      int kc = 0;
      for (; kc < Kp - 1; ++kc) {
        cum += SMEM ? wt_p[kc] : expf(lw_p[kc] - lse_p);
        if (!(cum < u)) break;
      }
#pragma unroll
      for (int c = 0; c < CP; ++c) {
        const int i = kc * C + c;
        if (c < C) x[c] = fmaf(SMEM ? sig_p[i] : expf(gls_p[i]), x[c], SMEM ? mu_p[i] : gmu_p[i]);
      }
      float run_m = -INFINITY, run_s = 0.0f;
      for (int j = 0; j < K; ++j) {
        float t[CP];
#pragma unroll
        for (int c = 0; c < CP; ++c) {
          const int i = j * C + c;
          t[c] = 0.0f;
          if (c < C) { const float d = (x[c] - (SMEM ? mu[i] : gmu[i])) * (SMEM ? inv[i] : expf(-gls[i])); t[c] = __fmul_rn(d, d); }
        }
        gmm_lse_add((SMEM ? base[j] : comp_base(j)) - 0.5f * gmm_tree_sum<CP>(t) - kHalfLog2Pi * C, run_m, run_s);
      }
      dens[side][slot] = run_m + logf(run_s);
      if (tid == 0) first_s = kGmmProposals;
      __syncthreads();
      if (side == 0) {
        const float alpha = fmaxf(0.0f, -expm1f(fminf(0.0f, dens[1][slot] - dens[0][slot])));
        if (k0 + slot < p.cap && vk <= alpha) atomicMin(&first_s, slot);
      }
      __syncthreads();
      const int first = first_s;
      done = first < kGmmProposals;
      const int last = min(p.cap - k0, kGmmProposals) - 1;
      const int take = done ? first : last;
      if (done) k = k0 + first + 1;
      // the thread that evaluated the proposal taken (the last one when the cap is reached) writes it
      if (side == 0 && slot == take && (done || k0 + kGmmProposals >= p.cap)) {
#pragma unroll
        for (int c = 0; c < CP; ++c)
          if (c < C) p.x_new[static_cast<size_t>(b) * C + c] = x[c];
      }
      __syncthreads();                      // before the next pass reuses dens and first_s
    }
    if (tid == 0) { p.n_prop[b] = k; p.flags[b] = 1u | (done ? 0u : 2u); }
    hit = done ? 0 : 1;
  }
  tally_cap_hits(hit, p.tally, p.cap_hits);
}

}  // namespace csd
