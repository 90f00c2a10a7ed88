// Row-parallel kernels around the GEMM chain: timestep embedding, the per-step boundary kernel
// (eps_hat reduction, classifier-free guidance, DDPM update, input projection, LayerNorm partials,
// condition vector s), and the verification / resampling kernels.
#pragma once
#include <type_traits>
#include "epilogue.cuh"
#include "ptx.cuh"

namespace csd {

// C[m, n] = act(sum_k A[m, k] B[n, k] + bias[n]), fp32, k in ascending order: the timestep embeddings of all steps wherever the
// layer kernels or a chain of tensor-core products read them.  The order is part of the result: one fp32 ulp of te flips
// 16-bit roundings of s that T steps carry on (summed lane-wise and through a butterfly, as rows_gemm_kernel sums, the rounds
// of 4096 rows moved by 1e-4 to 4e-4 of their norm), so a sum is one chain of K FMAs and a thread runs 4 MR of them side by
// side.  Bound by shared-memory loads and that chain.  Tile 8 MR x 32, 64 threads; operands arrive by cp.async, four pieces of
// 32 k ahead.  MR = 4 for the schedules of ~100 steps (one CTA per SM at W = 1024), MR = 1 where few rows leave more SMs idle
// than the wider tile saves loads.
constexpr int kEmbK = 32, kEmbStages = 4, kEmbLd = kEmbK + 4;   // (row stride of nine 16-byte units: conflict-free)

// Element-sized or 16-byte asynchronous copy to shared memory; nothing is read where n is 0 (the destination is zeroed).
template <int BYTES> __device__ __forceinline__ void cp_async(float* dst, const float* src, int n) {
  if constexpr (BYTES == 16) asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(n) : "memory");
  else asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(smem_u32(dst)), "l"(src), "r"(n) : "memory");
}

template <int MR, bool SILU>
__global__ void __launch_bounds__(64) embed_kernel(const float* __restrict__ A, const float* __restrict__ B, const float* __restrict__ bias,
                                                   float* __restrict__ C, int M, int N, int K) {
  __shared__ __align__(16) float sm[kEmbStages][(8 * MR + 32) * kEmbLd];
  const int tid = threadIdx.x, mi = tid >> 3, ni = tid & 7, m0 = blockIdx.y * 8 * MR, n0 = blockIdx.x * 32;
  const bool vec = K % 4 == 0 && ((reinterpret_cast<uintptr_t>(A) | reinterpret_cast<uintptr_t>(B)) & 15) == 0;
  const int pieces = (K + kEmbK - 1) / kEmbK;
  griddep_enter();
  auto fetch = [&](int p) {       // rows 0 .. 8 MR - 1: A, the other 32: B; zero beyond M, N, K
    if (p < pieces) {
      float* s = sm[p % kEmbStages];
      const int w = vec ? 4 : 1;
      for (int i = tid; i < (8 * MR + 32) * (kEmbK / w); i += 64) {
        const int r = i / (kEmbK / w), k = i % (kEmbK / w) * w, row = r < 8 * MR ? m0 + r : n0 + r - 8 * MR;
        const bool in = p * kEmbK + k < K && row < (r < 8 * MR ? M : N);
        const float* src = r < 8 * MR ? A : B;
        if (in) src += static_cast<size_t>(row) * K + p * kEmbK + k;
        if (vec) cp_async<16>(s + r * kEmbLd + k, src, in ? 16 : 0);
        else cp_async<4>(s + r * kEmbLd + k, src, in ? 4 : 0);
      }
    }
    asm volatile("cp.async.commit_group;" ::: "memory");
  };
  float acc[MR][4];
#pragma unroll
  for (int i = 0; i < MR; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.0f;
  for (int p = 0; p < kEmbStages - 1; ++p) fetch(p);
  for (int p = 0; p < pieces; ++p) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kEmbStages - 2) : "memory");
    __syncthreads();              // piece p is there, and everybody is done with the one whose place is taken next
    fetch(p + kEmbStages - 1);
    const float* a = sm[p % kEmbStages] + mi * kEmbLd;
    const float* b = sm[p % kEmbStages] + (8 * MR + ni) * kEmbLd;
#pragma unroll
    for (int k = 0; k < kEmbK; k += 4) {
      float4 av[MR], bv[4];
#pragma unroll
      for (int i = 0; i < MR; ++i) av[i] = *reinterpret_cast<const float4*>(a + 8 * i * kEmbLd + k);
#pragma unroll
      for (int j = 0; j < 4; ++j) bv[j] = *reinterpret_cast<const float4*>(b + 8 * j * kEmbLd + k);
#pragma unroll
      for (int i = 0; i < MR; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          float s = acc[i][j];
          s = fmaf(av[i].x, bv[j].x, s); s = fmaf(av[i].y, bv[j].y, s); s = fmaf(av[i].z, bv[j].z, s); s = fmaf(av[i].w, bv[j].w, s);
          acc[i][j] = s;
        }
    }
  }
#pragma unroll
  for (int i = 0; i < MR; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int m = m0 + mi + 8 * i, n = n0 + ni + 8 * j;
      if (m < M && n < N) {
        const float v = acc[i][j] + bias[n];
        C[static_cast<size_t>(m) * N + n] = SILU ? silu_f(v) : v;
      }
    }
}

template <typename ACT>
__global__ void convert_act_kernel(const float* __restrict__ src, ACT* __restrict__ dst, size_t n) {
  const size_t i = static_cast<size_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  if (i < n) dst[i] = to_act<ACT>(src[i]);
}

// Token and guidance row of row rho of a chain whose rows come in groups of G: with guidance G / 2 tokens' conditional rows,
// then their unconditional twins.
template <int G>
__device__ __forceinline__ int group_row_token(int rho, int cfg, int* rep) {
  const int blk = rho / G, r = rho % G;
  if (!cfg) { *rep = 0; return rho; }
  *rep = r / (G / 2);
  return blk * (G / 2) + r % (G / 2);
}

// s_t = SiLU(cz + te_t) of every step, in that row order and operand format: s_all[(t - 1) rows + rho][col]; rows of tokens
// beyond R are zero.  rows rows from rho0 on, T steps from te on.  A block keeps its row of cz in registers over kCondSteps steps: one step per block was bound by the
// trip to memory (115 us for 1024 rows of 1024 and 100 steps, 210 MB written).
constexpr int kCondSteps = 10;
template <typename ACT, int G>
__global__ void __launch_bounds__(128) cond_all_kernel(const float* __restrict__ cz, const float* __restrict__ te, ACT* __restrict__ s_all,
                                                       int R, int cfg, int W, int rows, int rho0, int T) {
  const int rho = blockIdx.x, t0 = blockIdx.y * kCondSteps, t1 = min(T, t0 + kCondSteps);
  int rep;
  const int i = group_row_token<G>(rho0 + rho, cfg, &rep);
  for (int j = threadIdx.x; j < W / 8; j += blockDim.x) {
    uint4* dst = reinterpret_cast<uint4*>(s_all + static_cast<size_t>(rho) * W) + j;     // 8 values per store
    const size_t step = static_cast<size_t>(rows) * W / 8;
    if (i >= R) {
      for (int t = t0; t < t1; ++t) dst[t * step] = make_uint4(0u, 0u, 0u, 0u);
      continue;
    }
    const float4* c4 = reinterpret_cast<const float4*>(cz + (static_cast<size_t>(rep) * R + i) * W) + 2 * j;
    const float4 a = c4[0], b = c4[1];
#pragma unroll 2
    for (int t = t0; t < t1; ++t) {
      const float4* t4 = reinterpret_cast<const float4*>(te + static_cast<size_t>(t) * W) + 2 * j;
      const float4 ta = __ldg(t4), tb = __ldg(t4 + 1);
      __align__(16) ACT o[8];
      o[0] = to_act<ACT>(silu_f(a.x + ta.x)); o[1] = to_act<ACT>(silu_f(a.y + ta.y));
      o[2] = to_act<ACT>(silu_f(a.z + ta.z)); o[3] = to_act<ACT>(silu_f(a.w + ta.w));
      o[4] = to_act<ACT>(silu_f(b.x + tb.x)); o[5] = to_act<ACT>(silu_f(b.y + tb.y));
      o[6] = to_act<ACT>(silu_f(b.z + tb.z)); o[7] = to_act<ACT>(silu_f(b.w + tb.w));
      dst[t * step] = *reinterpret_cast<const uint4*>(o);
    }
  }
}

enum StepMode : int { STEP_INIT = 0, STEP_MID = 1, STEP_LAST = 2 };

// Arithmetic of the step boundary, spelled with explicit roundings so that every kernel that
// finishes a step produces the same bits.
// guidance: eps_u + s (eps_c - eps_u)
__device__ __forceinline__ float cfg_combine(float ec, float eu, float scale) { return fmaf(scale, __fsub_rn(ec, eu), eu); }
// Eq. 3 mean: a x - b eps_hat
__device__ __forceinline__ float ddpm_mean(float a, float x, float b, float e) { return fmaf(-b, e, __fmul_rn(a, x)); }
// x_{t-1} = mu + sigma eps
__device__ __forceinline__ float ddpm_sample(float mu, float sigma, float eps) { return fmaf(sigma, eps, mu); }

// h = Win x + bin for the two columns (64 g + lane, 64 g + 32 + lane) of one row, and the (mean, M2)
// LayerNorm partial of the row's 64-column group g (warp-wide; every lane returns the same partial).
// wa / wb: the two columns' rows of Win (16 floats each), ba / bb their biases, xs: the row's x (16).
__device__ __forceinline__ void input_proj_group(const float* wa, const float* wb, float ba, float bb, const float* xs,
                                                 float acc[2], float& mean, float& m2) {
  float a0 = ba, a1 = bb;
#pragma unroll
  for (int c = 0; c < kCPad; ++c) { a0 = fmaf(wa[c], xs[c], a0); a1 = fmaf(wb[c], xs[c], a1); }
  acc[0] = a0; acc[1] = a1;
  float sum = __fadd_rn(a0, a1);
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
  mean = sum * (1.0f / kStatCols);
  const float d0 = a0 - mean, d1 = a1 - mean;
  m2 = fmaf(d1, d1, __fmul_rn(d0, d0));
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) m2 += __shfl_xor_sync(0xffffffffu, m2, o);
}

// h and the LayerNorm partials of up to RB consecutive token rows (their guidance twins hold the same values) over the
// 64-column group g, by one warp: lane holds columns 64 g + lane and + 32 in acc.  Tiled layout (tensor-core path): the values
// pass through tile_s [RB][64] so that the rows' 16-byte quads, which are neighbours in memory, are written together.
template <bool TILED, int RB>
__device__ __forceinline__ void write_h_group(float* h, float* stats, const float (&acc)[RB][2], const float (&mean)[RB], const float (&m2)[RB],
                                              float* tile_s, int g, int r0, int nrow, int nrep, int R, int W, int lane) {
  const int M = R * nrep, G = W / kStatCols;
  if (!TILED) {
#pragma unroll
    for (int rr = 0; rr < RB; ++rr)
      for (int rep = 0; rr < nrow && rep < nrep; ++rep) {
        const size_t row = static_cast<size_t>(r0 + rr) + static_cast<size_t>(rep) * R;
        if (lane == 0) reinterpret_cast<float2*>(stats)[row * G + g] = make_float2(mean[rr], m2[rr]);
        h[row * W + g * kStatCols + lane] = acc[rr][0];
        h[row * W + g * kStatCols + 32 + lane] = acc[rr][1];
      }
    return;
  }
  __syncwarp();
#pragma unroll
  for (int rr = 0; rr < RB; ++rr) { tile_s[rr * kStatCols + lane] = acc[rr][0]; tile_s[rr * kStatCols + 32 + lane] = acc[rr][1]; }
  __syncwarp();
  for (int rep = 0; rep < nrep; ++rep) {
#pragma unroll
    for (int rr = 0; rr < RB; ++rr)
      if (rr < nrow && lane == rr) reinterpret_cast<float2*>(stats)[tiled_stat_off(r0 + rr + rep * R, g, M, G)] = make_float2(mean[rr], m2[rr]);
#pragma unroll
    for (int k = 0; k < (RB * 16 + 31) / 32; ++k) {
      const int idx = k * 32 + lane, rr = idx % RB, c4 = idx / RB;
      if (c4 < 16 && rr < nrow)
        *reinterpret_cast<float4*>(h + tiled_off(r0 + rr + rep * R, g * 16 + c4, M, W)) = *reinterpret_cast<const float4*>(tile_s + rr * kStatCols + c4 * 4);
    }
  }
}

struct StepParams {
  int R, cfg, C, W, NT;          // token rows, guidance flag, token dim, width, number of column tiles
  float cfg_scale, a, b, sigma;  // coefficients of the step being finished (t)
  int sample_last;               // STEP_LAST: also draw x0 = mu1 + sigma eps
  const float* epart;            // [Rh, NT, 16] eps_hat partial sums of step t
  const float* bout;             // [16] (zero padded)
  const float* eps_t;            // [R, C] noise of step t
  const float* x_src;            // STEP_INIT: x_T
  float* x;                      // [R, C] current state (in/out)
  float *x0, *mu1, *x1;          // STEP_LAST outputs (x0, x1 may be null)
  const float* win;              // [W, 16] (zero padded), bin [W]
  const float* bin;
  const float* cz;               // [Rh, W]
  const float* te_next;          // [W] embedding of the step being prepared
  float* h;                      // [Rh, W] (16-bit operands: tiled layout, as stats)
  float* stats;                  // [Rh, W/64, 2]
  void* s;                       // [Rh, W] activations: s of the step te_next belongs to (null: none)
  void* s_b;                     // a second s to prepare (first boundary only), with its embedding te_b
  const float* te_b;
  float* traj_x;                 // TRAJ kernels: where the state this boundary produces is recorded ([R, C])
  float* traj_mu;                // TRAJ kernels: where the mean of the step being finished is recorded ([R, C])
  int* status;                   // set to 1 when a mean or state of this step is not finite (csd_sync reports it)
  // learned-variance heads (LV kernels): epart rows are 32 wide, [eps partials | variance-parameter partials]
  float lv_min, lv_max;          // bounds of the log-variance at the step being finished
  float* lv1;                    // STEP_LAST: [R, C] log-variance of the last step
  float* half_logdet;            // [R]: (1/2) sum over steps t >= 2 and coordinates of the log-variance (zeroed by STEP_INIT)
};

// log-variance of one coordinate from the head's variance output w: lv_min + (w + 1)/2 (lv_max - lv_min)
__device__ __forceinline__ float lv_interp(float w, float lv_min, float lv_max) {
  return fmaf(__fmul_rn(0.5f, __fadd_rn(w, 1.0f)), __fsub_rn(lv_max, lv_min), lv_min);
}

// RB token rows per block.  Finishes step t (unless STEP_INIT) and prepares the next one:
//   eps_hat = sum of tile partials + bout; guidance; mu = a x - b eps_hat; x <- mu + sigma eps_t
//   h = Win x + bin (same for both guidance rows), LayerNorm partials per 64 columns,
//   s = SiLU(cz + te_next) of the step after that (s is double-buffered, see the host code).
// With one row per block the kernel is bound by re-reading Win (64 B per column and row) through L1; RB = 4 reads a
// group's columns once for four rows.  The arithmetic of a row does not depend on RB.
// TRAJ: also record the whole trajectory (every state and every mean), for the single-path ratio of Eq. 2.
// LV: the head also predicts its transition's diagonal variance (Eq. 3 in its general form): the noise is scaled per
// coordinate by exp(lv / 2), the row's half log-determinant is accumulated for Sigma of Eq. 7.
template <typename ACT, int RB, bool TRAJ = false, bool LV = false>
__global__ void __launch_bounds__(256, RB == 4 ? 3 : 0) step_kernel(StepParams p, int mode) {
  constexpr int EPW = LV ? kCPad2 : kCPad;
  __shared__ float xs[RB][kCPad];
  __shared__ float eh[RB][2][kCPad];
  __shared__ float wv[LV ? RB : 1][kCPad];
  constexpr bool kTiled = !std::is_same<ACT, float>::value;
  __shared__ __align__(16) float tile_s[kTiled ? 8 : 1][RB * kStatCols];
  const int r0 = blockIdx.x * RB, tid = threadIdx.x;
  const int nrep = p.cfg ? 2 : 1;
  const int nrow = min(RB, p.R - r0);
  griddep_wait();
  if (tid == 0) griddep_launch_dependents();
  if (mode == STEP_INIT) {
    if (tid < RB * kCPad) {
      const int rr = tid / kCPad, c = tid % kCPad;
      float v = 0.0f;
      if (rr < nrow && c < p.C) {
        v = p.x_src[static_cast<size_t>(r0 + rr) * p.C + c];
        p.x[static_cast<size_t>(r0 + rr) * p.C + c] = v;
        if (TRAJ) p.traj_x[static_cast<size_t>(r0 + rr) * p.C + c] = v;
        if (LV && c == 0) p.half_logdet[r0 + rr] = 0.0f;
      }
      xs[rr][c] = v;
    }
    __syncthreads();
  } else {
    if (tid < RB * 2 * kCPad) {
      const int c = tid % kCPad, rep = (tid / kCPad) & 1, rr = tid / (2 * kCPad);
      if (rr < nrow && rep < nrep) {
        const float* e = p.epart + (static_cast<size_t>(r0 + rr + rep * p.R) * p.NT) * EPW + c;
        float acc = 0.0f;
        for (int nt = 0; nt < p.NT; ++nt) acc += e[nt * EPW];
        eh[rr][rep][c] = acc + p.bout[c];
        if (LV && rep == 0) {       // the variance parameter is the conditional row's own
          float accv = 0.0f;
          for (int nt = 0; nt < p.NT; ++nt) accv += e[nt * EPW + kCPad];
          wv[rr][c] = accv + p.bout[kCPad + c];
        }
      }
    }
    __syncthreads();
    if (tid < RB * kCPad) {
      const int rr = tid / kCPad, c = tid % kCPad;
      float xn = 0.0f;
      if (rr < nrow && c < p.C) {
        const size_t o = static_cast<size_t>(r0 + rr) * p.C + c;
        float e = eh[rr][0][c];
        if (p.cfg) e = cfg_combine(eh[rr][0][c], eh[rr][1][c], p.cfg_scale);
        const float xo = p.x[o];
        const float mu = ddpm_mean(p.a, xo, p.b, e);
        float sigma = p.sigma, lv = 0.0f;
        if (LV) { lv = lv_interp(wv[rr][c], p.lv_min, p.lv_max); sigma = expf(0.5f * lv); }
        xn = ddpm_sample(mu, sigma, p.eps_t[o]);
        // an activation beyond the 16-bit operand range became inf further up and arrives here as inf or NaN
        if (!(fabsf(xn) <= 3.0e38f)) *p.status = 1;
        if (LV && mode == STEP_LAST) p.lv1[o] = lv;
        if (mode == STEP_LAST) {
          p.mu1[o] = mu;
          if (p.x1) p.x1[o] = xo;
          if (p.sample_last && p.x0) p.x0[o] = xn;
        } else {
          p.x[o] = xn;
          if (TRAJ) { p.traj_x[o] = xn; p.traj_mu[o] = mu; }
        }
      }
      xs[rr][c] = xn;
      if (LV && mode != STEP_LAST) {
        // (1/2) sum_d lv of this step, coordinates in order (lanes 0..15 of a half-warp hold one row)
        float hsum = (rr < nrow && c < p.C) ? 0.5f * lv_interp(wv[rr][c], p.lv_min, p.lv_max) : 0.0f;
        constexpr unsigned kRowLanes = RB * kCPad >= 32 ? 0xffffffffu : 0x0000ffffu;   // threads inside this branch
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) hsum += __shfl_xor_sync(kRowLanes, hsum, o);
        if (rr < nrow && c == 0) p.half_logdet[r0 + rr] += hsum;
      }
    }
    if (mode == STEP_LAST) return;
    __syncthreads();
  }
  // prepare: each warp handles 64 consecutive columns at a time (lane, lane + 32): one LayerNorm partial
  const int lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
  ACT* s = reinterpret_cast<ACT*>(p.s);
  ACT* s_b = reinterpret_cast<ACT*>(p.s_b);
  for (int g = warp; g < p.W / kStatCols; g += nwarp) {
    float wa[kCPad], wb[kCPad];
    const int na = g * kStatCols + lane, nb = na + 32;
#pragma unroll
    for (int c4 = 0; c4 < kCPad / 4; ++c4) {
      const float4 qa = reinterpret_cast<const float4*>(p.win + static_cast<size_t>(na) * kCPad)[c4];
      const float4 qb = reinterpret_cast<const float4*>(p.win + static_cast<size_t>(nb) * kCPad)[c4];
      wa[4 * c4] = qa.x; wa[4 * c4 + 1] = qa.y; wa[4 * c4 + 2] = qa.z; wa[4 * c4 + 3] = qa.w;
      wb[4 * c4] = qb.x; wb[4 * c4 + 1] = qb.y; wb[4 * c4 + 2] = qb.z; wb[4 * c4 + 3] = qb.w;
    }
    const float ba = p.bin[na], bb = p.bin[nb];
    float te[2] = {0.0f, 0.0f}, teb[2] = {0.0f, 0.0f};
    if (s) { te[0] = p.te_next[na]; te[1] = p.te_next[nb]; }
    if (s_b) { teb[0] = p.te_b[na]; teb[1] = p.te_b[nb]; }
    // every cz value of the group first: the loads are independent, but behind the stores below the compiler must
    // assume they are not, and each row would wait for its own trip to memory
    float czv[RB][2][2];
#pragma unroll
    for (int rr = 0; rr < RB; ++rr)
#pragma unroll
      for (int rep = 0; rep < 2; ++rep)
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const size_t row = static_cast<size_t>(r0 + rr) + static_cast<size_t>(rep) * p.R;
          czv[rr][rep][j] = (rr < nrow && rep < nrep && (s || s_b)) ? __ldg(p.cz + row * p.W + g * kStatCols + j * 32 + lane) : 0.0f;
        }
    float acc[RB][2], mean[RB], m2[RB];
#pragma unroll
    for (int rr = 0; rr < RB; ++rr) input_proj_group(wa, wb, ba, bb, xs[rr], acc[rr], mean[rr], m2[rr]);   // (rows beyond nrow: x = 0)
    write_h_group<kTiled, RB>(p.h, p.stats, acc, mean, m2, tile_s[kTiled ? warp : 0], g, r0, nrow, nrep, p.R, p.W, lane);
#pragma unroll
    for (int rr = 0; rr < RB; ++rr) {
      if (rr >= nrow) break;
#pragma unroll
      for (int rep = 0; rep < 2; ++rep) {
        if (rep >= nrep) break;
        const size_t row = static_cast<size_t>(r0 + rr) + static_cast<size_t>(rep) * p.R;
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const int n = g * kStatCols + j * 32 + lane;
          if (s) s[row * p.W + n] = to_act<ACT>(silu_f(czv[rr][rep][j] + te[j]));
          if (s_b) s_b[row * p.W + n] = to_act<ACT>(silu_f(czv[rr][rep][j] + teb[j]));
        }
      }
    }
  }
}

// ---------------------------------------------------------------------------------------------
// Single-path ratio (Eq. 2): the target head scores the DRAFT's trajectory, so its T evaluations do not depend
// on one another and several steps are evaluated as one batch of rows.  Token row r' = j * Rin + r of a pass is
// row r of trajectory slot j0 + j (timestep t = T - j0 - j); with guidance its head rows are r' and Rtok + r'.
struct BatchParams {
  int Rin, Rtok, cfg, C, W, NT, T, j0;   // rows per step, token rows of the pass, ..., first trajectory slot
  float cfg_scale;
  const float* sched;    // device [5, T] of the target / draft pair: a, b, log-constant, 1/(2 sigma_p^2), 1/(2 sigma_q^2)
  const float* traj_x;   // [T + 1, Rin, C]: slot j holds x_{T-j}
  const float* win;      // [W, 16] (zero padded), bin [W]
  const float* bin;
  const float* cz;       // [Rin (1 + cfg), W]: one condition projection per row, shared by all steps
  const float* te;       // [T, W]
  float* h;              // [Rh, W]
  float* stats;          // [Rh, W/64, 2]
  void* s;               // [Rh, W] activations
  const float* epart;    // [Rh, NT, 16] eps_hat partial sums
  const float* bout;     // [16]
  float* mu_p;           // [Rtok, C] out: mean of the target's transition at the draft's state
  int* status;           // set to 1 when a mean is not finite
};

// Prepares a pass: h = Win x + bin, its LayerNorm partials and s = SiLU(cz + te_t), four token rows per block,
// with the arithmetic of step_kernel (the same device functions), so a row gets the bits it gets there.
template <typename ACT>
__global__ void __launch_bounds__(256) batch_prepare_kernel(BatchParams p) {
  constexpr int RB = 4;
  __shared__ float xs[RB][kCPad];
  constexpr bool kTiled = !std::is_same<ACT, float>::value;
  __shared__ __align__(16) float tile_s[kTiled ? 8 : 1][RB * kStatCols];
  const int r0 = blockIdx.x * RB, tid = threadIdx.x;
  const int nrep = p.cfg ? 2 : 1;
  const int nrow = min(RB, p.Rtok - r0);
  griddep_wait();
  if (tid == 0) griddep_launch_dependents();
  if (tid < RB * kCPad) {
    const int rr = tid / kCPad, c = tid % kCPad;
    float v = 0.0f;
    if (rr < nrow && c < p.C) v = p.traj_x[(static_cast<size_t>(p.j0) * p.Rin + r0 + rr) * p.C + c];
    xs[rr][c] = v;
  }
  __syncthreads();
  const int lane = tid & 31, warp = tid >> 5, nwarp = blockDim.x >> 5;
  ACT* s = reinterpret_cast<ACT*>(p.s);
  for (int g = warp; g < p.W / kStatCols; g += nwarp) {
    float wa[kCPad], wb[kCPad];
    const int na = g * kStatCols + lane, nb = na + 32;
#pragma unroll
    for (int c4 = 0; c4 < kCPad / 4; ++c4) {
      const float4 qa = reinterpret_cast<const float4*>(p.win + static_cast<size_t>(na) * kCPad)[c4];
      const float4 qb = reinterpret_cast<const float4*>(p.win + static_cast<size_t>(nb) * kCPad)[c4];
      wa[4 * c4] = qa.x; wa[4 * c4 + 1] = qa.y; wa[4 * c4 + 2] = qa.z; wa[4 * c4 + 3] = qa.w;
      wb[4 * c4] = qb.x; wb[4 * c4 + 1] = qb.y; wb[4 * c4 + 2] = qb.z; wb[4 * c4 + 3] = qb.w;
    }
    const float ba = p.bin[na], bb = p.bin[nb];
    // every cz and te value of the group first: independent loads in flight together (one trip to memory per
    // group instead of one per row)
    float czv[RB][2][2], tev[RB][2];
#pragma unroll
    for (int rr = 0; rr < RB; ++rr) {
      const int rt = min(r0 + rr, p.Rtok - 1), j = rt / p.Rin, ri = rt - j * p.Rin;
      const float* te = p.te + static_cast<size_t>(p.T - 1 - p.j0 - j) * p.W;
      tev[rr][0] = te[na]; tev[rr][1] = te[nb];
#pragma unroll
      for (int rep = 0; rep < 2; ++rep) {
        const size_t zrow = static_cast<size_t>(ri) + static_cast<size_t>(rep < nrep ? rep : 0) * p.Rin;
        czv[rr][rep][0] = __ldg(p.cz + zrow * p.W + na);
        czv[rr][rep][1] = __ldg(p.cz + zrow * p.W + nb);
      }
    }
    float acc[RB][2], mean[RB], m2[RB];
#pragma unroll
    for (int rr = 0; rr < RB; ++rr) input_proj_group(wa, wb, ba, bb, xs[rr], acc[rr], mean[rr], m2[rr]);   // (rows beyond nrow: x = 0)
    write_h_group<kTiled, RB>(p.h, p.stats, acc, mean, m2, tile_s[kTiled ? warp : 0], g, r0, nrow, nrep, p.Rtok, p.W, lane);
#pragma unroll
    for (int rr = 0; rr < RB; ++rr) {
      if (rr >= nrow) break;
#pragma unroll
      for (int rep = 0; rep < 2; ++rep) {
        if (rep >= nrep) break;
        const size_t row = static_cast<size_t>(r0 + rr) + static_cast<size_t>(rep) * p.Rtok;
        s[row * p.W + na] = to_act<ACT>(silu_f(czv[rr][rep][0] + tev[rr][0]));
        s[row * p.W + nb] = to_act<ACT>(silu_f(czv[rr][rep][1] + tev[rr][1]));
      }
    }
  }
}

// Finishes a pass: eps_hat = sum of tile partials + bout, guidance, mu^p_t = a_t x_t - b_t eps_hat (Eq. 3 mean),
// 16 token rows per block of 256 threads (thread = row, coordinate).
__global__ void __launch_bounds__(256) batch_finish_kernel(BatchParams p) {
  const int rt = blockIdx.x * 16 + (threadIdx.x >> 4), c = threadIdx.x & 15;
  griddep_wait();
  if (rt >= p.Rtok || c >= p.C) return;
  float e[2] = {0.0f, 0.0f};
  for (int rep = 0; rep < (p.cfg ? 2 : 1); ++rep) {
    const float* ep = p.epart + (static_cast<size_t>(rt) + static_cast<size_t>(rep) * p.Rtok) * p.NT * kCPad + c;
    float acc = 0.0f;
    for (int nt = 0; nt < p.NT; ++nt) acc += ep[nt * kCPad];
    e[rep] = acc + p.bout[c];
  }
  const float eh = p.cfg ? cfg_combine(e[0], e[1], p.cfg_scale) : e[0];
  const int ti = p.T - 1 - p.j0 - rt / p.Rin;   // t - 1
  const float x = p.traj_x[(static_cast<size_t>(p.j0) * p.Rin + rt) * p.C + c];
  const float mu = ddpm_mean(p.sched[ti], x, p.sched[p.T + ti], eh);
  if (!(fabsf(mu) <= 3.0e38f)) *p.status = 1;
  p.mu_p[static_cast<size_t>(rt) * p.C + c] = mu;
}

// Per-step terms of the log-ratio of Eq. 2 for the steps of one pass, one thread per (step, token row):
//   term_t = C (log sigma_q,t - log sigma_p,t) - |x_{t-1} - mu^p_t|^2 / (2 sigma_p,t^2) + |x_{t-1} - mu^q_t|^2 / (2 sigma_q,t^2).
// The two quadratic forms are rounded separately, so identical means give a term of exactly zero.
__global__ void __launch_bounds__(128)
single_path_terms_kernel(int Rin, int C, int T, int j0, int nsteps, const float* __restrict__ sched,
                         const float* __restrict__ traj_x, const float* __restrict__ traj_mu,
                         const float* __restrict__ mu_p, float* __restrict__ terms) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= nsteps * Rin) return;
  const int j = i / Rin, r = i - j * Rin;
  const int ti = T - 1 - j0 - j;
  const float* xn = traj_x + (static_cast<size_t>(j0 + j + 1) * Rin + r) * C;
  const float* mq = traj_mu + (static_cast<size_t>(j0 + j) * Rin + r) * C;
  const float* mp = mu_p + static_cast<size_t>(i) * C;
  float dp = 0.0f, dq = 0.0f;
  for (int c = 0; c < C; ++c) {
    const float x = xn[c];
    const float ep = x - mp[c], eq = x - mq[c];
    dp = fmaf(ep, ep, dp);
    dq = fmaf(eq, eq, dq);
  }
  terms[static_cast<size_t>(j0 + j) * Rin + r] =
      sched[2 * T + ti] + __fsub_rn(__fmul_rn(dq, sched[4 * T + ti]), __fmul_rn(dp, sched[3 * T + ti]));
}

// Sum of the T terms in trajectory order (in double, so the order of magnitude of the early terms does not cost the
// late ones their digits), then the accept test and prefix scan of Alg. 1: one warp per sequence.
__global__ void __launch_bounds__(128)
single_path_accept_kernel(int B, int gamma, int T, const float* __restrict__ terms, const float* __restrict__ u,
                          float* __restrict__ logratio, int32_t* __restrict__ n_accept,
                          uint32_t* __restrict__ accept_mask) {
  const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (b >= B) return;
  bool ok = true;
  if (lane < gamma) {
    const size_t row = static_cast<size_t>(b) * gamma + lane;
    const size_t R = static_cast<size_t>(B) * gamma;
    double total = 0.0;
    for (int j = 0; j < T; ++j) total += static_cast<double>(terms[j * R + row]);
    const float lr = static_cast<float>(total);
    logratio[row] = lr;
    ok = logf(u[row]) <= lr;
  }
  const uint32_t ballot = __ballot_sync(0xffffffffu, ok);
  if (lane == 0) {
    const uint32_t rej = ~ballot;
    int n = rej ? (__ffs(rej) - 1) : gamma;
    if (n > gamma) n = gamma;
    n_accept[b] = n;
    if (accept_mask) accept_mask[b] = (gamma >= 32) ? ballot : (ballot & ((1u << gamma) - 1u));
  }
}

// The C coordinates of one row or proposal, zero beyond C; 16-byte loads where the row allows them.
__device__ __forceinline__ void load_coords(const float* __restrict__ src, int C, float* z) {
  if (C == kCPad && (reinterpret_cast<uintptr_t>(src) & 15) == 0) {
#pragma unroll
    for (int c4 = 0; c4 < kCPad / 4; ++c4) {
      const float4 q = __ldg(reinterpret_cast<const float4*>(src) + c4);
      z[4 * c4] = q.x; z[4 * c4 + 1] = q.y; z[4 * c4 + 2] = q.z; z[4 * c4 + 3] = q.w;
    }
  } else {
#pragma unroll
    for (int c = 0; c < kCPad; ++c) z[c] = c < C ? __ldg(src + c) : 0.0f;
  }
}

// ---------------------------------------------------------------------------------------------
// Verification: one warp per sequence, lane i = draft position i (gamma <= 32).
//   logratio = log_sigma + C (log sq1 - log sp1) - |x0 - mu_p|^2 / (2 sp1^2) + |x0 - mu_q|^2 / (2 sq1^2)
//   accept iff log u <= logratio;  n_accept = number of leading accepts (ballot + find-first-set).
__global__ void __launch_bounds__(128)
accept_scan_kernel(int B, int gamma, int C, float log_const, float inv2vp, float inv2vq,
                   const float* __restrict__ x0, const float* __restrict__ mu_q,
                   const float* __restrict__ mu_p, const float* __restrict__ u,
                   float* __restrict__ logratio, int32_t* __restrict__ n_accept,
                   uint32_t* __restrict__ accept_mask, const float* __restrict__ offset = nullptr) {
  griddep_enter();
  const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (b >= B) return;
  bool acc = true;  // lanes beyond gamma do not reject
  if (lane < gamma) {
    const size_t row = static_cast<size_t>(b) * gamma + lane;
    float dp = 0.0f, dq = 0.0f;
    float xv[kCPad], pv[kCPad], qv[kCPad];       // every load of the row in flight at once
    load_coords(x0 + row * C, C, xv); load_coords(mu_p + row * C, C, pv); load_coords(mu_q + row * C, C, qv);
#pragma unroll
    for (int c = 0; c < kCPad; ++c) {            // (coordinates beyond C add exact zeros)
      const float ep = xv[c] - pv[c], eq = xv[c] - qv[c];
      dp = fmaf(ep, ep, dp);
      dq = fmaf(eq, eq, dq);
    }
    // Both products are rounded separately (no FMA contraction), so that identical draft and target
    // means give a difference of exactly zero.
    float lr = log_const + __fsub_rn(__fmul_rn(dq, inv2vq), __fmul_rn(dp, inv2vp));
    if (offset) lr = __fadd_rn(lr, offset[row]);   // terms of the steps t >= 2 when the noise is not shared
    logratio[row] = lr;
    acc = logf(u[row]) <= lr;
  }
  const uint32_t ballot = __ballot_sync(0xffffffffu, acc);
  if (lane == 0) {
    const uint32_t rej = ~ballot;
    int n = rej ? (__ffs(rej) - 1) : gamma;
    if (n > gamma) n = gamma;
    n_accept[b] = n;
    if (accept_mask) accept_mask[b] = (gamma >= 32) ? ballot : (ballot & ((1u << gamma) - 1u));
  }
}

// Without trajectory alignment the exponentials of the steps t >= 2 of Eq. 4 do not cancel: x^m_{t-1} - mu^m_t =
// sigma_m,t eps^m_t, so step t contributes (|eps^q_t|^2 - |eps^p_t|^2) / 2 beyond the Sigma term.  One thread per
// token row, steps in order, double accumulation; identical noise gives exactly 0.
__global__ void __launch_bounds__(128)
noise_norm_term_kernel(int R, int C, int T, const float* __restrict__ eps_q, const float* __restrict__ eps_p,
                       float* __restrict__ offset) {
  const int r = blockIdx.x * blockDim.x + threadIdx.x;
  if (r >= R) return;
  double total = 0.0;
  for (int t = 1; t < T; ++t) {   // slices 1..T-1 = steps 2..T
    const float* a = eps_q + (static_cast<size_t>(t) * R + r) * C;
    const float* b = eps_p + (static_cast<size_t>(t) * R + r) * C;
    float nq = 0.0f, np = 0.0f;
    for (int c = 0; c < C; ++c) { nq = fmaf(a[c], a[c], nq); np = fmaf(b[c], b[c], np); }
    total += 0.5 * (static_cast<double>(nq) - static_cast<double>(np));
  }
  offset[r] = static_cast<float>(total);
}

// All-accepted branch of Alg. 1: sequence b keeps its sample of position gamma + 1 only if n_accept[b] == gamma.
__global__ void __launch_bounds__(256)
bonus_select_kernel(int B, int C, int gamma, const int32_t* __restrict__ n_accept, const float* __restrict__ x0,
                    float* __restrict__ x_bonus, uint32_t* __restrict__ taken) {
  const int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i >= B * C) return;
  const int b = i / C;
  const bool all = n_accept[b] >= gamma;
  if (all) x_bonus[i] = x0[i];
  if (taken && i == b * C) taken[b] = all ? 1u : 0u;
}

// Verification with predicted diagonal variances.  Per token  log Sigma = half_logdet_q - half_logdet_p  (Eq. 7: the
// product over t >= 2 of sqrt|Sigma_q,t| / sqrt|Sigma_p,t|, accumulated by the two chains), and
//   logratio = log Sigma + log N(x0; mu_p, diag(exp(lv_p))) - log N(x0; mu_q, diag(exp(lv_q)))      (Eq. 8).
// Each model's exponent-plus-normaliser sum is formed by the same instruction sequence, so identical draft and target
// values give a difference of exactly zero.
__device__ __forceinline__ float diag_neg_logpdf(const float* x, const float* mu, const float* lv, int C) {
  float acc = 0.0f;     // sum_d [ lv_d / 2 + (x - mu)_d^2 / (2 exp(lv_d)) ]
  for (int c = 0; c < C; ++c) {
    const float e = x[c] - mu[c];
    acc = __fadd_rn(acc, __fadd_rn(__fmul_rn(0.5f, lv[c]), __fmul_rn(__fmul_rn(0.5f, __fmul_rn(e, e)), expf(-lv[c]))));
  }
  return acc;
}

__global__ void __launch_bounds__(128)
accept_scan_lv_kernel(int B, int gamma, int C, const float* __restrict__ x0, const float* __restrict__ mu_q,
                      const float* __restrict__ lv_q, const float* __restrict__ hld_q, const float* __restrict__ mu_p,
                      const float* __restrict__ lv_p, const float* __restrict__ hld_p, const float* __restrict__ u,
                      float* __restrict__ logratio, float* __restrict__ log_sigma_rows, int32_t* __restrict__ n_accept,
                      uint32_t* __restrict__ accept_mask) {
  griddep_enter();
  const int b = blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  if (b >= B) return;
  bool acc = true;
  if (lane < gamma) {
    const size_t row = static_cast<size_t>(b) * gamma + lane;
    const float ls = __fsub_rn(hld_q[row], hld_p[row]);
    const float nq = diag_neg_logpdf(x0 + row * C, mu_q + row * C, lv_q + row * C, C);
    const float np = diag_neg_logpdf(x0 + row * C, mu_p + row * C, lv_p + row * C, C);
    const float lr = __fadd_rn(ls, __fsub_rn(nq, np));
    log_sigma_rows[row] = ls;
    logratio[row] = lr;
    acc = logf(u[row]) <= lr;
  }
  const uint32_t ballot = __ballot_sync(0xffffffffu, acc);
  if (lane == 0) {
    const uint32_t rej = ~ballot;
    int n = rej ? (__ffs(rej) - 1) : gamma;
    if (n > gamma) n = gamma;
    n_accept[b] = n;
    if (accept_mask) accept_mask[b] = (gamma >= 32) ? ballot : (ballot & ((1u << gamma) - 1u));
  }
}

// Sum over the 16 (padded) coordinates in the order of a butterfly reduction over 32 lanes whose upper half holds zeros.
__device__ __forceinline__ float coord_tree_sum(float* v) {
#pragma unroll
  for (int o = kCPad / 2; o > 0; o >>= 1)
#pragma unroll
    for (int c = 0; c < o; ++c) v[c] = __fadd_rn(v[c], v[c + o]);
  return v[0];
}

// The number of sequences whose cap was reached, summed over the blocks without a memset before the launch: every block
// adds (its hits, 1) to one 64-bit word, the last one to arrive has the sum and leaves the word at zero for the context's
// next call.  The word serves one launch at a time: launches that others of the context may overlap (captured ones, whose
// graphs run on any stream) get none and add to a cap_hits zeroed before them.  hits: this block's count, valid in thread 0.
__device__ __forceinline__ void tally_cap_hits(int hits, unsigned long long* tally, int32_t* cap_hits) {
  if (threadIdx.x != 0) return;
  if (!tally) {
    if (hits) atomicAdd(cap_hits, hits);
    return;
  }
  unsigned long long before = 0;
  if (gridDim.x > 1) {
    before = atomicAdd(tally, (static_cast<unsigned long long>(hits) << 32) | 1ull);
    if (static_cast<unsigned>(before) != gridDim.x - 1) return;
    *tally = 0ull;
  }
  *cap_hits = static_cast<int32_t>(before >> 32) + hits;
}

// Resampling (Cor. 1), one warp per sequence, 32 proposals at a time: lane j evaluates proposal k0 + j over all
// coordinates, the first accepted one in order is taken.  (A warp per proposal, lane = coordinate, walks the proposals
// one by one, each a trip to memory for xi and v and ten dependent shuffles; the sums keep that form's order.)
// LV: diagonal final-step covariances, x' = mu_p + exp(lv_p / 2) xi with the rejected token's own Sigma.
struct ResampleParams {
  int B, gamma, C, cap;
  float log_sigma, sp1, sq1, log_sp1, log_sq1;   // fixed variances
  const float *log_sigma_rows, *lv_p, *lv_q;     // LV
  const int32_t* n_accept;
  const float *mu_p, *mu_q, *xi, *v;
  float* x_new;
  int32_t* n_prop;
  uint32_t* flags;
  int32_t* cap_hits;
  unsigned long long* tally;
};

template <bool LV>
__global__ void __launch_bounds__(128) resample_kernel(const ResampleParams p) {
  __shared__ int hit_s[4];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int b = blockIdx.x * (blockDim.x >> 5) + warp;
  int hit = 0;
  griddep_enter();
  const int n = b < p.B ? p.n_accept[b] : p.gamma;
  // the first 32 proposals do not depend on the row: their loads travel with n_accept's
  float z[kCPad], vk = 0.0f;
  auto fetch = [&](int k0) {
    const size_t pr = static_cast<size_t>(b) * p.cap + (k0 + lane < p.cap ? k0 + lane : p.cap - 1);
    load_coords(p.xi + pr * p.C, p.C, z);
    vk = __ldg(p.v + pr);
  };
  if (b < p.B) fetch(0);
  if (n >= p.gamma) {
    if (b < p.B && lane == 0) { p.n_prop[b] = 0; p.flags[b] = 0u; }
  } else {
    const size_t row = static_cast<size_t>(b) * p.gamma + n;
    const bool on = lane < p.C;
    const size_t o = row * p.C + lane;
    const float mp = on ? p.mu_p[o] : 0.0f, mq = on ? p.mu_q[o] : 0.0f;
    float sp = p.sp1, ivp = 0.5f / (p.sp1 * p.sp1), ivq = 0.5f / (p.sq1 * p.sq1), ls = p.log_sigma, hl = 0.0f;
    if (LV) {
      const float lp_d = on ? p.lv_p[o] : 0.0f, lq_d = on ? p.lv_q[o] : 0.0f;
      sp = expf(0.5f * lp_d); ivp = 0.5f * expf(-lp_d); ivq = 0.5f * expf(-lq_d);
      ls = p.log_sigma_rows[row];
      hl = on ? 0.5f * (lq_d - lp_d) : 0.0f;       // (1/2) sum_d (lv_q - lv_p): the normalisers' part of lp - lq
#pragma unroll
      for (int s = 16; s > 0; s >>= 1) hl += __shfl_xor_sync(0xffffffffu, hl, s);
    }
    int k = p.cap;
    bool done = false;
    for (int k0 = 0; k0 < p.cap && !done; k0 += 32) {
      if (k0 > 0) fetch(k0);
      float ep[kCPad], eq[kCPad];
#pragma unroll
      for (int c = 0; c < kCPad; ++c) {
        const float mpc = __shfl_sync(0xffffffffu, mp, c), mqc = __shfl_sync(0xffffffffu, mq, c);
        const float spc = LV ? __shfl_sync(0xffffffffu, sp, c) : sp;
        const float x = fmaf(spc, z[c], mpc);
        const float dp = x - mpc, dq = x - mqc;
        ep[c] = __fmul_rn(dp, dp); eq[c] = __fmul_rn(dq, dq);
        if (LV) { ep[c] = __fmul_rn(ep[c], __shfl_sync(0xffffffffu, ivp, c)); eq[c] = __fmul_rn(eq[c], __shfl_sync(0xffffffffu, ivq, c)); }
        if (c >= p.C) { ep[c] = 0.0f; eq[c] = 0.0f; }
      }
      const float se = coord_tree_sum(ep), sq = coord_tree_sum(eq);
      float d;                                       // log q(x') - log Sigma - log p(x')
      if (LV) d = (se - sq) - hl - ls;               // lq - lp = -(1/2) sum lv_q - sq + (1/2) sum lv_p + se
      else {
        const float lp = -p.C * p.log_sp1 - se * ivp;
        const float lq = -p.C * p.log_sq1 - sq * ivq;
        d = lq - ls - lp;
      }
      const float alpha = fmaxf(0.0f, -expm1f(fminf(0.0f, d)));
      const uint32_t ok = __ballot_sync(0xffffffffu, k0 + lane < p.cap && vk <= alpha);
      if (ok) { k = k0 + __ffs(ok); done = true; }
    }
    // the proposal taken (the last one when the cap was reached)
    if (on) p.x_new[static_cast<size_t>(b) * p.C + lane] = fmaf(sp, p.xi[(static_cast<size_t>(b) * p.cap + k - 1) * p.C + lane], mp);
    if (lane == 0) { p.n_prop[b] = k; p.flags[b] = 1u | (done ? 0u : 2u); }
    hit = done ? 0 : 1;
  }
  if (lane == 0) hit_s[warp] = hit;
  __syncthreads();
  tally_cap_hits(hit_s[0] + hit_s[1] + hit_s[2] + hit_s[3], p.tally, p.cap_hits);
}

}  // namespace csd
