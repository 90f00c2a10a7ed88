// fp32 heads (CSD_F32): one persistent kernel per chain instead of one kernel per layer, and the small fp32 products
// before it.
//
// A head is a per-token MLP: rows never exchange data.  The head rows are cut into groups of G (with guidance G / 2 tokens'
// conditional rows and their unconditional twins) and a cluster of 8 CTAs owns a group for all layers and steps; CTA r
// owns output columns [r W/8, (r + 1) W/8) of every layer.  The group's activations (condition vector s, u, v) live in
// every CTA's shared memory, each CTA broadcasting the columns it produced to its peers (distributed shared memory); the
// only synchronisation is the cluster's hardware barrier, three per block and two per step, and the products of s (AdaLN
// shift | scale | gate, which wait for nothing) are computed between arriving at a barrier and waiting for it.  Groups never
// wait for each other, so any number of clusters may be resident.
//
// A product is a warp's: 2 or 4 weight rows against the group's G rows, lanes split K (weights read coalesced, 16 bytes per
// lane; activations from shared memory, G CW FMAs per lane for G + CW loads), then a transposing butterfly that leaves each
// lane with G CW / 32 finished sums.  What bounds it: few rows: barriers and the trip to L2 for the weights (the layer
// kernels before: one launch per layer and a 128-thread block per 32 x 128 tile, 3.8 ms for the smallest workload, 1 x 4
// tokens, 10 steps); many rows: shared-memory loads and FMAs in balance.
#pragma once
#include "gemm.cuh"
#include "rowops.cuh"

namespace csd {

constexpr int kFcCluster = 8;
// Threads per CTA: as many as the rows' accumulators leave registers for.
template <int G> struct FcThreads { static constexpr int value = G <= 8 ? 512 : 384; };
constexpr int kFcMaxSteps = 128;    // steps per launch: their coefficients travel as kernel parameters

// ------------------------------------------------------------------------------------------------ warp-level products
// First two 16-byte pieces of each weight row for this lane: requested before a barrier, used after it.
template <int CW> struct FcPre { float4 w[2][CW]; };

template <int CW>
__device__ __forceinline__ void fc_preload(FcPre<CW>& pre, const float* w0, int ldw, int K, int lane) {
#pragma unroll
  for (int i = 0; i < 2; ++i)
#pragma unroll
    for (int c = 0; c < CW; ++c) {
      const int k = lane * 4 + 128 * i;
      pre.w[i][c] = k < K ? __ldg(reinterpret_cast<const float4*>(w0 + static_cast<size_t>(c) * ldw + k)) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
    }
}

// acc[g CW + c] = this lane's part of sum_k xs[g][k] w[c][k] (rows w0 + c ldw); K a multiple of 4, pre = fc_preload of the same rows.
template <int G, int CW>
__device__ __forceinline__ void fc_dots(float (&acc)[G * CW], FcPre<CW>& pre, const float* w0, int ldw, const float* xs,
                                        int ldx, int K, int lane) {
#pragma unroll
  for (int i = 0; i < G * CW; ++i) acc[i] = 0.0f;
#pragma unroll 1
  for (int k = lane * 4; k < K; k += 128) {
    float4 w[CW];
#pragma unroll
    for (int c = 0; c < CW; ++c) {
      w[c] = pre.w[0][c];
      pre.w[0][c] = pre.w[1][c];
      if (k + 256 < K) pre.w[1][c] = __ldg(reinterpret_cast<const float4*>(w0 + static_cast<size_t>(c) * ldw + k + 256));
    }
#pragma unroll
    for (int g = 0; g < G; ++g) {
      const float4 x = *reinterpret_cast<const float4*>(xs + g * ldx + k);
#pragma unroll
      for (int c = 0; c < CW; ++c) {
        float a = acc[g * CW + c];
        a = fmaf(w[c].x, x.x, a); a = fmaf(w[c].y, x.y, a); a = fmaf(w[c].z, x.z, a); a = fmaf(w[c].w, x.w, a);
        acc[g * CW + c] = a;
      }
    }
  }
}

// Sums N values over the warp, transposing: lane l ends with values [l N/32, (l + 1) N/32) in v[0..] (N >= 32), or value
// l N/32 (N < 32: 32/N lanes share a value).
template <int N>
__device__ __forceinline__ void fc_reduce(float (&v)[N], int lane) {
  int n = N;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    if (n > 1) {
      n >>= 1;
      const bool up = (lane & o) != 0;
#pragma unroll
      for (int i = 0; i < N / 2; ++i)
        if (i < n) {
          const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
          v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
        }
    } else v[0] += __shfl_xor_sync(0xffffffffu, v[0], o);
  }
}

// ------------------------------------------------------------------------------------------------ products before the chain
// C[m, n] = act(sum_k A[m, k] B[n, k] + bias[n]), fp32: timestep embedding and (fp32 heads) condition projection.  Eight rows
// of A in shared memory, a warp takes four rows of B at a time.  Two independent products may share a launch.
struct RowsGemm {
  const float *A, *B, *bias;
  float* C;
  int M, N, K, silu;
  int blocks_n;      // N / 32 (N is a head's width, a multiple of 128)
};
struct RowsGemmPair {
  RowsGemm g[2];
  int split;         // first block of the second product
};
constexpr int kRgRows = 8, kRgCols = 32, kRgKc = 1024;   // K is walked in pieces of 1024 (32 KB of A)

__global__ void __launch_bounds__(256) rows_gemm_kernel(const RowsGemmPair pr) {
  __shared__ __align__(16) float as[kRgRows * kRgKc];
  const bool second = static_cast<int>(blockIdx.x) >= pr.split;
  const RowsGemm p = second ? pr.g[1] : pr.g[0];
  const int blk = static_cast<int>(blockIdx.x) - (second ? pr.split : 0);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int m0 = (blk / p.blocks_n) * kRgRows, n0 = (blk % p.blocks_n) * kRgCols + warp * 4;
  const bool vec = p.K % 4 == 0 && ((reinterpret_cast<uintptr_t>(p.A) | reinterpret_cast<uintptr_t>(p.B)) & 15) == 0;
  griddep_enter();
  float sum[kRgRows * 4];
#pragma unroll
  for (int i = 0; i < kRgRows * 4; ++i) sum[i] = 0.0f;
  for (int k0 = 0; k0 < p.K; k0 += kRgKc) {
    const int kc = min(kRgKc, p.K - k0);
    if (k0) __syncthreads();
    if (vec) {
      for (int i = tid; i < kRgRows * (kc / 4); i += 256) {
        const int r = i / (kc / 4), k = (i - r * (kc / 4)) * 4;
        const float4 a = m0 + r < p.M ? *reinterpret_cast<const float4*>(p.A + static_cast<size_t>(m0 + r) * p.K + k0 + k) : make_float4(0.0f, 0.0f, 0.0f, 0.0f);
        *reinterpret_cast<float4*>(as + r * kRgKc + k) = a;
      }
    } else {
      for (int i = tid; i < kRgRows * kc; i += 256) {
        const int r = i / kc, k = i - r * kc;
        as[r * kRgKc + k] = m0 + r < p.M ? p.A[static_cast<size_t>(m0 + r) * p.K + k0 + k] : 0.0f;
      }
    }
    const float* w0 = p.B + static_cast<size_t>(n0) * p.K + k0;
    if (vec) {
      FcPre<4> pre;
      fc_preload<4>(pre, w0, p.K, kc, lane);
      __syncthreads();
      float acc[kRgRows * 4];
      fc_dots<kRgRows, 4>(acc, pre, w0, p.K, as, kRgKc, kc, lane);
#pragma unroll
      for (int i = 0; i < kRgRows * 4; ++i) sum[i] += acc[i];
    } else {
      __syncthreads();
      for (int k = lane; k < kc; k += 32)
#pragma unroll
        for (int c = 0; c < 4; ++c) {
          const float w = __ldg(w0 + static_cast<size_t>(c) * p.K + k);
#pragma unroll
          for (int r = 0; r < kRgRows; ++r) sum[r * 4 + c] = fmaf(w, as[r * kRgKc + k], sum[r * 4 + c]);
        }
    }
  }
  fc_reduce<kRgRows * 4>(sum, lane);       // lane = 4 row + column
  const int m = m0 + (lane >> 2), n = n0 + (lane & 3);
  if (m < p.M) {
    const float v = sum[0] + p.bias[n];
    p.C[static_cast<size_t>(m) * p.N + n] = p.silu ? silu_f(v) : v;
  }
}

// ------------------------------------------------------------------------------------------------ the chain
struct FcParams {
  int R, cfg, C, W, L, T;        // T: steps of the whole schedule
  int t_hi, t_lo;                // steps of this launch: t_hi down to t_lo
  int per;                       // tokens per group
  int sample_last, lv;
  float cfg_scale;
  const float* w;                // per block [shift | scale: 2 W rows][gate: W][first layer: W][second layer: W], then final [2 W]
  const float* bias;             // per block shift, scale, gate, first, second layer [W] each, then final shift, scale
  const float *win, *bin, *wout_t, *bout;
  const float *cz, *te;          // [Rh, W], [T, W]
  const float *x_T, *eps;
  float *x, *x0, *mu1, *x1;      // x: [R, C] state between launches
  float *traj_x, *traj_mu;       // optional records
  float *lv1, *half_logdet;
  int* status;
  float a[kFcMaxSteps], b[kFcMaxSteps], s0[kFcMaxSteps], s1[kFcMaxSteps];   // index t - t_lo; s0 = sigma or lv_min, s1 = lv_max
};

// Shared memory of a CTA in floats; wc = W / 8 columns per CTA.
constexpr int kFcWinLd = kCPad + 1;   // a row of Win and its bias in shared memory (odd: lanes walk rows)
struct FcLayout { int s, u, v, mods, h, stats, part, win, wout, bout, x, total; };
__host__ __device__ inline FcLayout fc_layout(int G, int W, int epw) {
  const int wc = W / kFcCluster;
  FcLayout l{};
  int o = 0;
  auto take = [&](int n) { const int r = o; o += (n + 3) & ~3; return r; };
  l.s = take(G * W); l.u = take(G * W); l.v = take(G * W);
  l.mods = take(3 * G * wc); l.h = take(G * wc);
  l.stats = take(kFcCluster * G * 2); l.part = take(kFcCluster * G * epw);
  l.win = take(wc * kFcWinLd); l.wout = take(wc * epw); l.bout = take(epw); l.x = take(G * kCPad);
  l.total = o;
  return l;
}

__device__ __forceinline__ void fc_st_cluster(uint32_t addr, float v) { asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(addr), "f"(v) : "memory"); }

// The cluster barrier's instructions want converged warps.
__device__ __forceinline__ void fc_arrive() { __syncwarp(); cluster_arrive(); }
__device__ __forceinline__ void fc_wait() { __syncwarp(); cluster_wait(); }

// CWD: columns per task of the dependent layers (two when the CTA's columns are few, to keep more warps busy)
template <int G, int CWD>
__global__ void __launch_bounds__(FcThreads<G>::value, 1) f32_chain_kernel(const __grid_constant__ FcParams p) {
  constexpr int kFcThreads = FcThreads<G>::value, kFcWarps = kFcThreads / 32;
  extern __shared__ __align__(16) float sm[];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int W = p.W, L = p.L, wc = W / kFcCluster, EPW = p.lv ? kCPad2 : kCPad, nrep = p.cfg ? 2 : 1;
  const int rank = static_cast<int>(cluster_ctarank()), grp = static_cast<int>(blockIdx.x) / kFcCluster;
  const int c0 = rank * wc;                                  // first column of this CTA
  const FcLayout lo = fc_layout(G, W, EPW);
  float *s = sm + lo.s, *u = sm + lo.u, *v = sm + lo.v, *mods = sm + lo.mods, *h = sm + lo.h, *stats = sm + lo.stats,
        *part = sm + lo.part, *win = sm + lo.win, *wout = sm + lo.wout, *bout = sm + lo.bout, *xs = sm + lo.x;
  const int per = p.per;                                     // tokens per group; row g: token g % per, guidance half g / per
  const int tok0 = grp * per;
  const size_t W2 = static_cast<size_t>(W) * W;

#pragma unroll 1
  for (int i = tid; i < wc * kCPad; i += kFcThreads) win[(i / kCPad) * kFcWinLd + i % kCPad] = p.win[static_cast<size_t>(c0) * kCPad + i];
#pragma unroll 1
  for (int i = tid; i < wc; i += kFcThreads) win[i * kFcWinLd + kCPad] = p.bin[c0 + i];
#pragma unroll 1
  for (int i = tid; i < EPW; i += kFcThreads) bout[i] = p.bout[i];
#pragma unroll 1
  for (int i = tid; i < wc * EPW; i += kFcThreads) wout[i] = p.wout_t[static_cast<size_t>(c0) * EPW + i];
  griddep_wait();
  if (tid == 0) griddep_launch_dependents();
  fc_arrive(); fc_wait();                          // every CTA of the cluster runs: its shared memory may be written

  auto bcast = [&](const float* dst, float val) {            // the same location in every CTA of the cluster
    const uint32_t a = smem_u32(dst);
#pragma unroll
    for (int r = 0; r < kFcCluster; ++r) fc_st_cluster(mapa_shared(a, static_cast<uint32_t>(r)), val);
  };
  // First weight row of a task and its bias: kind 0 / 1 / 2 = shift / scale / gate of block k, 3 / 4 = first / second layer.
  // The final pair is kinds 0 and 1 of block L.  Shift and scale rows are interleaved in groups of 64; a task's two or
  // four columns are consecutive rows in every matrix.
  auto row_ptr = [&](int kind, int k, int col) -> const float* {
    const int j = c0 + col;
    const int row = kind < 2 ? (j >> 6) * 128 + (j & 63) + kind * 64 : kind * W + j;
    return p.w + static_cast<size_t>(k) * 5 * W2 + static_cast<size_t>(row) * W;
  };
  auto bias_of = [&](int kind, int k, int col) -> float { return __ldg(p.bias + (static_cast<size_t>(k) * 5 + kind) * W + c0 + col); };
  // (mean, M2) of each row over this CTA's columns of h, to every CTA: one warp per row.
  auto send_stats = [&]() {
#pragma unroll 1
    for (int g = warp; g < G; g += kFcWarps) {
      float sum = 0.0f;
      for (int j = lane; j < wc; j += 32) sum += h[g * wc + j];
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) sum += __shfl_xor_sync(0xffffffffu, sum, o);
      const float mean = sum / static_cast<float>(wc);
      float m2 = 0.0f;
      for (int j = lane; j < wc; j += 32) { const float d = h[g * wc + j] - mean; m2 = fmaf(d, d, m2); }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) m2 += __shfl_xor_sync(0xffffffffu, m2, o);
      if (lane < kFcCluster) {
        const uint32_t off = static_cast<uint32_t>((lo.stats + (rank * G + g) * 2) * 4), base = mapa_shared(smem_u32(sm), static_cast<uint32_t>(lane)) + off;
        fc_st_cluster(base, mean);
        fc_st_cluster(base + 4, m2);
      }
    }
    __syncwarp();
  };
  auto row_norm = [&](int g, float& mean, float& rstd) {     // merge of the eight equal-count partials
    float sm8 = 0.0f, m2 = 0.0f, q = 0.0f;
#pragma unroll
    for (int r = 0; r < kFcCluster; ++r) { sm8 += stats[(r * G + g) * 2]; m2 += stats[(r * G + g) * 2 + 1]; }
    mean = sm8 * (1.0f / kFcCluster);
#pragma unroll
    for (int r = 0; r < kFcCluster; ++r) { const float d = stats[(r * G + g) * 2] - mean; q = fmaf(d, d, q); }
    rstd = 1.0f / sqrtf(fmaf(static_cast<float>(wc), q, m2) / static_cast<float>(W) + 1e-6f);
  };
  // Products of s into mods[kind][g][col]: shift | scale | gate of block k, or the final pair (nk = 2).
  auto make_mods = [&](int k, int nk) {
    constexpr int CW = 4, N = G * CW;
    const int per_kind = wc / CW, ntask = nk * per_kind;
#pragma unroll 1
    for (int t = warp; t < ntask; t += kFcWarps) {
      const int kind = t / per_kind, col = (t - kind * per_kind) * CW;
      const float* w0 = row_ptr(kind, k, col);
      FcPre<CW> pre;
      fc_preload<CW>(pre, w0, W, W, lane);
      constexpr int PER = N >= 32 ? N / 32 : 1, SHARE = N >= 32 ? 1 : 32 / N;
      float bv[PER];                                         // the biases of this lane's sums, requested ahead
#pragma unroll
      for (int e = 0; e < PER; ++e) bv[e] = bias_of(kind, k, col + (lane / SHARE * PER + e) % CW);
      float acc[N];
      fc_dots<G, CW>(acc, pre, w0, W, s, W, W, lane);
      fc_reduce<N>(acc, lane);
      if (lane % SHARE == 0) {
#pragma unroll
        for (int e = 0; e < PER; ++e) {
          const int i = lane / SHARE * PER + e, g = i / CW, c = i % CW;
          mods[(kind * G + g) * wc + col + c] = acc[e] + bv[e];
        }
      }
      __syncwarp();
    }
  };
  // One MLP layer over this CTA's columns.  second = false: v = SiLU(W1 u + b1), broadcast; true: h += gate (W2 v + b2).
  // The first task's weights are requested before the barrier that makes the operand complete.
  auto layer = [&](int k, bool second) {
    constexpr int CW = CWD, N = G * CW;
    const int ntask = wc / CW;
    const int kind = second ? 4 : 3;
    const float* w0 = row_ptr(kind, k, warp * CW);
    FcPre<CW> pre;
    if (warp < ntask) fc_preload<CW>(pre, w0, W, W, lane);
    fc_wait();
#pragma unroll 1
    for (int t = warp; t < ntask; t += kFcWarps) {
      if (t != warp) { w0 = row_ptr(kind, k, t * CW); fc_preload<CW>(pre, w0, W, W, lane); }
      constexpr int PER = N >= 32 ? N / 32 : 1, SHARE = N >= 32 ? 1 : 32 / N;
      float bv[PER];
#pragma unroll
      for (int e = 0; e < PER; ++e) bv[e] = bias_of(kind, k, t * CW + (lane / SHARE * PER + e) % CW);
      float acc[N];
      fc_dots<G, CW>(acc, pre, w0, W, second ? v : u, W, W, lane);
      fc_reduce<N>(acc, lane);
      if (lane % SHARE == 0) {
#pragma unroll
        for (int e = 0; e < PER; ++e) {
          const int i = lane / SHARE * PER + e, g = i / CW, col = t * CW + i % CW;
          const float y = acc[e] + bv[e];
          if (!second) bcast(v + g * W + c0 + col, silu_f(y));
          else h[g * wc + col] = fmaf(mods[(2 * G + g) * wc + col], y, h[g * wc + col]);
        }
      }
      __syncwarp();
    }
  };
  auto make_s = [&](int t) {                                 // s = SiLU(cz + te_t), the whole rows, by every CTA
    const float4* te = reinterpret_cast<const float4*>(p.te + static_cast<size_t>(t - 1) * W);
#pragma unroll 1
    for (int i = tid; i < G * (W / 4); i += kFcThreads) {
      const int g = i / (W / 4), j = i - g * (W / 4), tok = tok0 + g % per, rep = g / per;
      float4 o = make_float4(0.0f, 0.0f, 0.0f, 0.0f);
      if (rep < nrep && tok < p.R) {
        const float4 c = *(reinterpret_cast<const float4*>(p.cz + (static_cast<size_t>(rep) * p.R + tok) * W) + j), e = te[j];
        o = make_float4(silu_f(c.x + e.x), silu_f(c.y + e.y), silu_f(c.z + e.z), silu_f(c.w + e.w));
      }
      *reinterpret_cast<float4*>(s + g * W + 4 * j) = o;
    }
  };

  // state of the group's tokens, in every CTA
  const bool first_launch = p.t_hi == p.T;
#pragma unroll 1
  for (int i = tid; i < G * kCPad; i += kFcThreads) {
    const int q = i / kCPad, c = i % kCPad, tok = tok0 + q;
    float xv = 0.0f;
    if (q < per && tok < p.R && c < p.C) {
      const size_t o = static_cast<size_t>(tok) * p.C + c;
      xv = first_launch ? p.x_T[o] : p.x[o];
      if (first_launch && rank == 0) {
        if (p.traj_x) p.traj_x[o] = xv;
        if (p.lv && c == 0) p.half_logdet[tok] = 0.0f;
      }
    }
    xs[i] = xv;
  }
  make_s(p.t_hi);
  __syncthreads();

#pragma unroll 1
  for (int t = p.t_hi; t >= p.t_lo; --t) {
    // h = Win x + bin over this CTA's columns
#pragma unroll 1
    for (int i = tid; i < G * wc; i += kFcThreads) {
      const int g = i / wc, col = i - g * wc;
      const float* xr = xs + (g % per) * kCPad;
      const float* wr = win + col * kFcWinLd;
      float a = wr[kCPad];
#pragma unroll
      for (int c = 0; c < kCPad; ++c) a = fmaf(wr[c], xr[c], a);
      h[i] = a;
    }
    // (k = -1: only what precedes block 0)
#pragma unroll 1
    for (int k = -1; k < L; ++k) {
      if (k >= 0) {
#pragma unroll 1
        for (int i = tid; i < G * wc; i += kFcThreads) {     // u = LN(h)(1 + scale) + shift
          const int g = i / wc, col = i - g * wc;
          float mean, rstd;
          row_norm(g, mean, rstd);
          const float nv = __fmul_rn(__fsub_rn(h[i], mean), rstd);
          bcast(u + g * W + c0 + col, fmaf(nv, __fadd_rn(1.0f, mods[(G + g) * wc + col]), mods[g * wc + col]));
        }
#pragma unroll 1
        for (int second = 0; second < 2; ++second) { fc_arrive(); layer(k, second != 0); }
      }
      __syncthreads();
      send_stats();
      fc_arrive();
      make_mods(k + 1, k + 1 < L ? 3 : 2);
      fc_wait();
      __syncthreads();
    }
    // output projection: this CTA's columns' part of eps_hat (and of the variance parameter), to every CTA
    float* uf = u + c0;                                      // own columns: nobody else reads them before the next barrier
#pragma unroll 1
    for (int i = tid; i < G * wc; i += kFcThreads) {
      const int g = i / wc, col = i - g * wc;
      float mean, rstd;
      row_norm(g, mean, rstd);
      const float nv = __fmul_rn(__fsub_rn(h[i], mean), rstd);
      uf[g * W + col] = fmaf(nv, __fadd_rn(1.0f, mods[(G + g) * wc + col]), mods[g * wc + col]);
    }
    __syncthreads();
#pragma unroll 1
    for (int i = tid; i < G * EPW; i += kFcThreads) {
      const int g = i / EPW, c = i - g * EPW;
      float a0 = 0.0f, a1 = 0.0f;                            // two chains (wc is even)
      for (int col = 0; col < wc; col += 2) {
        a0 = fmaf(uf[g * W + col], wout[col * EPW + c], a0);
        a1 = fmaf(uf[g * W + col + 1], wout[(col + 1) * EPW + c], a1);
      }
      bcast(part + (rank * G + g) * EPW + c, a0 + a1);
    }
    fc_arrive();
    float noise = 0.0f;                                      // per 16 <= the block's threads: one value each
    if (tid < per * kCPad && tok0 + tid / kCPad < p.R && tid % kCPad < p.C)
      noise = p.eps[(static_cast<size_t>(t - 1) * p.R + tok0 + tid / kCPad) * p.C + tid % kCPad];
    if (t > p.t_lo) make_s(t - 1);
    fc_wait();
    // guidance and the transition of Eq. 3, by every CTA alike (CTA 0 writes what leaves the chip)
    if (const int i = tid; i < per * kCPad) {
      const int q = i / kCPad, c = i % kCPad, tok = tok0 + q;
      auto out = [&](int g, int cc) {
        float e = 0.0f;
#pragma unroll
        for (int r = 0; r < kFcCluster; ++r) e += part[(r * G + g) * EPW + cc];
        return e + bout[cc];
      };
      const bool on = tok < p.R && c < p.C;
      float xn = 0.0f, lv = 0.0f;
      if (on) {
        const size_t o = static_cast<size_t>(tok) * p.C + c;
        float e = out(q, c);
        if (p.cfg) e = cfg_combine(e, out(per + q, c), p.cfg_scale);
        const float xo = xs[i], mu = ddpm_mean(p.a[t - p.t_lo], xo, p.b[t - p.t_lo], e);
        float sigma = p.s0[t - p.t_lo];
        if (p.lv) { lv = lv_interp(out(q, kCPad + c), p.s0[t - p.t_lo], p.s1[t - p.t_lo]); sigma = expf(0.5f * lv); }
        xn = ddpm_sample(mu, sigma, noise);
        if (rank == 0) {
          if (!(fabsf(xn) <= 3.0e38f)) *p.status = 1;
          if (t == 1) {
            if (p.lv) p.lv1[o] = lv;
            p.mu1[o] = mu;
            if (p.x1) p.x1[o] = xo;
            if (p.sample_last && p.x0) p.x0[o] = xn;
          } else {
            if (t == p.t_lo) p.x[o] = xn;                    // the next launch starts from it
            if (p.traj_x) {
              const size_t slot = static_cast<size_t>(p.R) * p.C;
              p.traj_x[static_cast<size_t>(p.T - t + 1) * slot + o] = xn;
              p.traj_mu[static_cast<size_t>(p.T - t) * slot + o] = mu;
            }
          }
        }
      }
      xs[i] = xn;
      if (p.lv && t > 1) {                                   // (1/2) sum_d lv: a half-warp holds one token (per 16 divides the block)
        float hs = on ? 0.5f * lv : 0.0f;
        const unsigned mask = per * kCPad >= 32 ? 0xffffffffu : 0x0000ffffu;
#pragma unroll
        for (int o = 8; o > 0; o >>= 1) hs += __shfl_xor_sync(mask, hs, o);
        if (rank == 0 && on && c == 0) p.half_logdet[tok] += hs;
      }
    }
    __syncthreads();
  }
  fc_arrive(); fc_wait();                          // no CTA leaves while a peer may still write to it
}

}  // namespace csd
