// A denoising chain of few rows (W in {512, 1024, 1536}, 16-bit operands) in two parts:
//
// 1. mods_gemm_kernel: everything a head takes from the condition vector - shifts, scales, gates: three fifths of its
//    multiply-adds - does not depend on x_t.  It is formed for many steps at once, as one dense product over the rows of a chunk
//    of steps, in fp32.
// 2. group_chain_kernel: what depends on x_t.  Token rows never exchange data, so the rows are cut into groups of 16 (with
//    guidance 8 tokens' conditional rows and their unconditional twins) and a cluster of W / 128 CTAs owns a group for all
//    steps of the chunk; CTA r owns output columns [128 r, 128 r + 128) of every layer.  Groups never wait for each other and
//    nothing waits for a kernel that runs beside it, so any number of chains may run at a time.
//
// Few rows are bound by latency: per layer a CTA multiplies its 128 weight rows (the MMA's M operand, streamed ahead through
// a ring) with the group's 16 rows (its N), 64 instructions or 2.6 k cycles at W = 1024, and the results have to reach the
// other CTAs of the cluster.  They do so by bulk copies from shared memory to shared memory (4 KB to each, 0.7 to 2 k cycles;
// a CTA's turn order starts with its own tile), counted in by mbarriers: no
// trip through L2, no cluster barrier.  The two activation buffers (a', v) need no hand-back: a CTA sends its
// part of one only after its product on the other, which took every peer's part of that.  LayerNorm partials travel as
// 8-byte remote stores, the residual stream h stays in registers (a thread owns 8 rows of a column), and every CTA of the
// cluster updates the group's token states x_t for itself from the exchanged output-projection partials.
//
// Two forms.  Plain (the default mode): the operand of a block's first layer is u = LN(h)(1 + scale) + shift, rounded once, as in
// the layer kernels, and the LayerNorm partials are awaited before it can leave.  FOLD (CSD_CHAIN_SMALL_BATCH up to 128 head rows):
// the folded blocks of fold.cuh, first-layer terms P1 | P2 among the products of s; what leaves is a' = h (1 + scale), which waits
// for nothing.  Folding rounds the fused weights as well, and the mean goes only after the product: against float64 its error
// is 1.02 to 1.20 times that of the layer kernels (geometric means over 12 draws of 9 to 91 tokens each; 2 x 512 to 12 x 1536, both
// formats), the plain form's 0.90 to 1.03 times.  The wait costs 1 to 9 %: 3 x 1024, T = 40, 12 tokens with guidance 1.03 -> 1.07 ms,
// 12 x 1536 5.8 -> 6.3 ms (layer kernels 2.2 and 9.6).
#pragma once
#include "fold.cuh"

namespace csd {

// ------------------------------------------------------------------------------------------ products of s_t
constexpr int kMgStages = 6, kMgStageBytes = 32768;   // per stage: 128 weight rows | 128 rows of s, one k-block of 64
constexpr int kMgEpiWarps = 8;
constexpr int kMgThreads = (kMgEpiWarps + 3) * 32;
constexpr int kMgSmemBytes = 1024 + kMgStages * kMgStageBytes + 256;

__device__ __forceinline__ void gc_settle(const int* err) { if (*reinterpret_cast<const volatile int*>(err) != 0) settle(); }

struct MgParams {
  int nkb, tiles_n, units;     // k-blocks; tiles of 256 rows of s; tiles in all (s fastest: the weights stream past once)
  const int* wrow;             // first row of each tile of 256 weight rows in the first matrix, or ~row in the second
  int s_row0;                  // first row of s
  float4* out;                 // [weight row / 128][row of s / 4][128 weight rows][4 rows of s]
  int* err;
};

// out = weights s^T in 256 x 256 tiles per CTA pair, written from registers: a lane holds one weight row, so a warp's 16-byte
// stores cover 512 contiguous bytes, and a group's 16 rows of one column tile are one contiguous 8 KB block.  128 rows, 100
// steps, 14 sections of 1024: 0.53 ms in all on the 84 SMs that the chain leaves, 715 TFLOP/s, hidden behind it.
template <int AB_FMT>
__global__ void __launch_bounds__(kMgThreads, 1)
mods_gemm_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmX, const __grid_constant__ CUtensorMap tmS,
                 const MgParams p) {
  constexpr int S = kMgStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + S * kMgStageBytes);
  uint64_t* empty_bar = full_bar + S;
  uint64_t* acc_full = empty_bar + S;     // [2]
  uint64_t* acc_empty = acc_full + 2;     // [2], every epilogue warp of both CTAs
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(acc_empty + 2);     // and whether the context is free of errors

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int unit0 = static_cast<int>(blockIdx.x >> 1), nunits = static_cast<int>(gridDim.x >> 1);
  const int my_tiles = (p.units - unit0 + nunits - 1) / nunits;
  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmW); tma_prefetch_desc(&tmX); tma_prefetch_desc(&tmS);
    for (int s = 0; s < S; ++s) { mbar_init(&full_bar[s], 2); mbar_init(&empty_bar[s], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 2 * kMgEpiWarps); }
    tmem_base_s[1] = *reinterpret_cast<const volatile int*>(p.err) == 0;    // one reading for all warps
    fence_mbar_init();
  }
  if (warp == 1) { tmem_alloc_pair(tmem_base_s, 512); tmem_relinquish_pair(); }
  tc_fence_before_sync();
  __syncthreads();
  cluster_arrive(); cluster_wait();       // the peer's barriers exist before anything signals them
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_base_s;
  const bool run = tmem_base_s[1] != 0;

  if (run && (warp == 0 || warp == kMgEpiWarps + 2)) {
    const bool is_w = warp == 0;
    if (lane == 0) {
      bool ok = true;
      int it = 0, next = is_w ? __ldg(p.wrow + unit0 / p.tiles_n) : 0;
      for (int i = 0; i < my_tiles && ok; ++i) {
        const int u = unit0 + i * nunits;
        const CUtensorMap* const tm = !is_w ? &tmS : next < 0 ? &tmX : &tmW;
        const int row = (!is_w ? p.s_row0 + u % p.tiles_n * 256 : next < 0 ? ~next : next) + rank * 128;
        if (is_w && i + 1 < my_tiles) next = __ldg(p.wrow + (u + nunits) / p.tiles_n);
        for (int kb = 0; kb < p.nkb; ++kb, ++it) {
          const int s = it % S;
          if (it >= S && !ch_wait<false>(&empty_bar[s], ((it / S) & 1) ^ 1, p.err)) { ch_fail(p.err, DEV_ERR_TMA_WAIT, 1, it); ok = false; break; }
          if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], 32768);     // both CTAs' bytes of this operand
          tma_load_2d_pair(smem + s * kMgStageBytes + (is_w ? 0 : 16384), tm, mapa_shared(smem_u32(&full_bar[s]), 0), kb * kBlockK, row);
        }
      }
    }
    __syncwarp();
  } else if (run && warp == 1 && rank == 0) {
    const bool leader = elect_one();
    constexpr uint32_t idesc = umma_idesc_f16(256, AB_FMT, 256);
    bool ok = true;
    int it = 0;
    for (int i = 0; i < my_tiles && ok; ++i) {
      const int ab = i & 1;
      if (i >= 2 && !ch_wait<true>(&acc_empty[ab], ((i >> 1) - 1) & 1, p.err)) { if (leader) ch_fail(p.err, DEV_ERR_MMA_WAIT, 1, i); ok = false; break; }
      tc_fence_after_sync();
      for (int kb = 0; kb < p.nkb; ++kb, ++it) {
        const int s = it % S;
        if (!ch_wait<false>(&full_bar[s], (it / S) & 1, p.err)) { if (leader) ch_fail(p.err, DEV_ERR_MMA_WAIT, 2, it); ok = false; break; }
        tc_fence_after_sync();
        if (leader) {
          const uint32_t sa = smem_u32(smem + s * kMgStageBytes);
          const uint64_t da = umma_smem_desc_sw128(sa), db = umma_smem_desc_sw128(sa + 16384);
#pragma unroll
          for (int k = 0; k < kBlockK / 16; ++k) umma_f16_pair(tmem_base + ab * 256, da + 2 * k, db + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
          umma_commit_pair(&empty_bar[s]);
        }
        __syncwarp();
      }
      if (ok && leader) umma_commit_pair(&acc_full[ab]);
      __syncwarp();
    }
  } else if (run && warp >= 2 && warp < kMgEpiWarps + 2) {
    const int q = warp & 3, half = (warp - 2) >> 2;
    bool ok = true;
    for (int i = 0; i < my_tiles && ok; ++i) {
      const int u = unit0 + i * nunits, ab = i & 1;
      ok = ch_wait<false>(&acc_full[ab], (i >> 1) & 1, p.err);
      if (!ok) ch_fail(p.err, DEV_ERR_EPI_WAIT, 1, i);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after_sync();
      const uint32_t trow = tmem_base + ab * 256 + half * 128 + (static_cast<uint32_t>(q * 32) << 16);
      float4* o = p.out + ((static_cast<size_t>(u / p.tiles_n) * 2 + rank) * (p.tiles_n * 64) + (u % p.tiles_n) * 64 + half * 32) * 128 + q * 32 + lane;
#pragma unroll
      for (int c = 0; c < 4; ++c) {
        float a[kChunk];
        tmem_ld32(trow + c * kChunk, a);
        tmem_ld_wait();
        if (c == 3) {            // this warp's last read of the buffer
          tc_fence_before_sync();
          __syncwarp();
          if (lane == 0) mbar_arrive_cluster_tmem(mapa_shared(smem_u32(&acc_empty[ab]), 0));
        }
#pragma unroll
        for (int j = 0; j < kChunk / 4; ++j) o[(c * 8 + j) * 128] = make_float4(a[4 * j], a[4 * j + 1], a[4 * j + 2], a[4 * j + 3]);
      }
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  gc_settle(p.err);
  cluster_arrive(); cluster_wait();   // neither CTA leaves while the pair's MMAs or signals may touch it
  if (warp == 1) tmem_dealloc_pair(tmem_base, 512);
}

// ------------------------------------------------------------------------------------------ the chain
constexpr int kGcRows = 16;               // rows of a group = MMA N
constexpr int kGcHalf = kGcRows / 2;      // rows of an epilogue thread
constexpr int kGcEpi = 256;               // warps 0..7: epilogue
// Three pairs of a loading warp (11..13) and an MMA-issuing warp (8..10), each with its own part of the weight ring and its own
// accumulator, take k-blocks in turn (the same ones in every phase: the sums, hence the bits, do not depend on where a launch starts).  One pair spends 370 cycles on loading and 530 on issuing a k-block (waits, the
// instructions' own latency, the commit), which the tensor pipe finishes in 160.  The ring is divided because waits on a
// barrier's parity are only sound for one warp that follows its phases in order.
constexpr int kGcMma = 3;
constexpr int kGcThreads = kGcEpi + 2 * kGcMma * 32;
constexpr int kGcMaxW = 1536;
constexpr int kGcMaxCl = kGcMaxW / 128;
constexpr int kGcTile = kGcRows * 256;    // bytes of one CTA's part of an activation buffer: two k-blocks of [16 rows][128 B]
constexpr int kGcMaxStages = 12;          // of one k-block of [128 weight rows][128 B]; a multiple of the pairs

struct GcLayout { int act, ring, stages, part, wout, stats, misc, total; };
__host__ __device__ inline GcLayout gc_layout(int W) {
  GcLayout l{};
  int o = 0;
  auto take = [&](int n) { const int r = o; o += n; return r; };
  l.act = take(2 * kGcRows * W * 2);      // a' | v
  l.wout = take(128 * kCPad * 4);
  l.stats = take(W / 32 * kGcRows * 8);   // [32-column group][row] (mean, M2)
  l.part = take(kGcRows * kCPad * 4);     // the outgoing output-projection partial
  l.misc = take(1024 + 512 + 512);        // x [16 tokens][16], (mean, rstd) per epilogue warp [8][8], barriers
  l.stages = (226 * 1024 - o) / 16384;    // all that is left streams weights: 9, 9, 6 stages at W = 512, 1024, 1536
  l.stages = (l.stages > kGcMaxStages ? kGcMaxStages : l.stages) / kGcMma * kGcMma;
  l.ring = take(0);
  o = (o + 1023) / 1024 * 1024;
  l.ring = o;
  o += l.stages * 16384;
  l.total = o;
  return l;
}

constexpr int kGcMaxSteps = 128;          // steps per launch: their coefficients travel as kernel parameters

struct GcParams {
  int R, cfg, W, L, C, T, t_hi, t_lo, rows, sample_last;   // rows: kernel rows (groups x 16)
  float cfg_scale;
  const CUtensorMap* maps;     // [2 L]: W1_k, W2_k in boxes of 128 rows
  const float4* mods; int nq;  // products of the chunk, nq row quads per weight row
  const float *c1, *bsh, *bsc, *bg, *b1, *b2, *bfsh, *bfsc;   // block 0; c1_k | c2_k (FOLD) are 2 W floats a block, the others 5 W apart
  const float *win, *bin, *wout_t, *bout;
  const float *x_T, *eps;
  float *x, *x0, *mu1, *x1, *traj_x, *traj_mu;
  int* err;
  int* status;
  float ca[kGcMaxSteps], cb[kGcMaxSteps], sigma[kGcMaxSteps];   // index t - t_lo
};

// Shared memory of this CTA -> the same or another CTA of the cluster, completion counted in bytes on a barrier there.
__device__ __forceinline__ void gc_copy(uint32_t dst_cluster, const void* src, uint32_t bytes, uint32_t bar_cluster) {
  asm volatile("cp.async.bulk.shared::cluster.shared::cta.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];"
               ::"r"(dst_cluster), "r"(smem_u32(src)), "r"(bytes), "r"(bar_cluster) : "memory");
}
__device__ __forceinline__ void gc_st_async(uint32_t dst_cluster, float a, float b, uint32_t bar_cluster) {
  const unsigned long long v = (static_cast<unsigned long long>(__float_as_uint(b)) << 32) | __float_as_uint(a);
  asm volatile("st.async.shared::cluster.mbarrier::complete_tx::bytes.b64 [%0], %1, [%2];" ::"r"(dst_cluster), "l"(v), "r"(bar_cluster) : "memory");
}
// Sums 8 values over the warp, transposing: lane l ends with value l / 4.
__device__ __forceinline__ float gc_reduce8(const float (&in)[kGcHalf], int lane) {
  float v[kGcHalf];
#pragma unroll
  for (int i = 0; i < kGcHalf; ++i) v[i] = in[i];
#pragma unroll
  for (int n = 4; n >= 1; n >>= 1) {
    const int o = 4 * n;
    const bool up = (lane & o) != 0;
#pragma unroll
    for (int i = 0; i < 4; ++i)
      if (i < n) {
        const float send = up ? v[i] : v[i + n], keep = up ? v[i + n] : v[i];
        v[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
      }
  }
  v[0] += __shfl_xor_sync(0xffffffffu, v[0], 2);
  return v[0] + __shfl_xor_sync(0xffffffffu, v[0], 1);
}
// Issued where it stands: the products of a phase are on their way while its MMAs run.
__device__ __forceinline__ float4 gc_ld(const float4* p) {
  float4 v;
  asm volatile("ld.global.nc.L1::no_allocate.v4.f32 {%0, %1, %2, %3}, [%4];" : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w) : "l"(p));
  return v;
}

template <typename ACT, int AB_FMT, bool FOLD>
__global__ void __launch_bounds__(kGcThreads, 1) group_chain_kernel(const __grid_constant__ GcParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int W = p.W, L = p.L, T = p.T, CL = W / 128;
  const GcLayout lo = gc_layout(W);
  const int act_bytes = kGcRows * W * 2;
  const int SR = lo.stages / kGcMma;       // stages of a pair
  uint8_t* act = smem + lo.act;
  float4* part_out = reinterpret_cast<float4*>(smem + lo.part);
  float* wout_s = reinterpret_cast<float*>(smem + lo.wout);
  float2* stats_s = reinterpret_cast<float2*>(smem + lo.stats);
  float* xs = reinterpret_cast<float*>(smem + lo.misc);
  float2* norm_all = reinterpret_cast<float2*>(smem + lo.misc + 1024);
  uint64_t* bars = reinterpret_cast<uint64_t*>(smem + lo.misc + 1536);
  uint64_t *w_full = bars, *w_empty = w_full + kGcMaxStages, *act_full = w_empty + kGcMaxStages, *acc_full = act_full + 2 * kGcMaxCl,
           *stats_full = acc_full + 1, *part_full = stats_full + 1;
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(part_full + 1);     // and whether the context is free of errors
  // free at the end of a step, when every product that reads them is complete here and every peer has its copy: the columns'
  // modulated h (read by this CTA only), the peers' output-projection partials
  float* uf_s = reinterpret_cast<float*>(act);                       // [16][kUfLd]
  float* part_s = reinterpret_cast<float*>(act + act_bytes);         // [CL][16][16]
  constexpr int kUfLd = 132;

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = static_cast<int>(cluster_ctarank()), grp = static_cast<int>(blockIdx.x) / CL;
  const int n_base = rank * 128;
  if (tid == 0) {
    for (int s = 0; s < kGcMaxStages; ++s) { mbar_init(&w_full[s], 1); mbar_init(&w_empty[s], 1); }
    for (int i = 0; i < 2 * kGcMaxCl; ++i) mbar_init(&act_full[i], 1);
    mbar_init(acc_full, kGcMma); mbar_init(stats_full, 1); mbar_init(part_full, 1);
    tmem_base_s[1] = *reinterpret_cast<const volatile int*>(p.err) == 0;    // one reading for all warps
    fence_mbar_init();
  }
  if (warp == 8) { tmem_alloc(tmem_base_s, 64); tmem_relinquish(); }
  for (int i = tid; i < 128 * kCPad; i += kGcThreads) wout_s[i] = p.wout_t[static_cast<size_t>(n_base) * kCPad + i];
  tc_fence_before_sync();
  __syncthreads();
  cluster_arrive(); cluster_wait();       // the peers' barriers exist before anything signals them
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_base_s;
  const bool run = tmem_base_s[1] != 0;

  // (a CTA that gives up on a wait goes on through its barriers without waiting: its peers' waits end by the context's
  // error word)
  if (run && warp >= 8 + kGcMma) {
    // ---------------------------------------------------------------- weights, k-blocks in this CTA's turn order
    if (lane == 0) {
      const int m = warp - 8 - kGcMma;
      int s = 0;
      uint32_t par = 1;
      bool ok = true;
      for (int t = p.t_hi; t >= p.t_lo && ok; --t)
        for (int ph = 0; ph < 2 * L && ok; ++ph)
          for (int j = m; j < 2 * CL; j += kGcMma) {
            const int kb = 2 * rank + j < 2 * CL ? 2 * rank + j : 2 * rank + j - 2 * CL, st = m * SR + s;
            if (!ch_wait<false>(&w_empty[st], par, p.err)) { ch_fail(p.err, DEV_ERR_TMA_WAIT, 1, ph); ok = false; break; }   // (fresh: passes)
            mbar_arrive_expect_tx(&w_full[st], 16384);
            tma_load_2d(smem + lo.ring + st * 16384, p.maps + ph, &w_full[st], kb * kBlockK, n_base);
            if (++s == SR) { s = 0; par ^= 1; }
          }
    }
    __syncwarp();
  } else if (run && warp >= 8) {
    // ---------------------------------------------------------------- MMA issue, into 16 columns per pair (the epilogue adds
    // the pairs' up)
    const bool leader = elect_one();
    constexpr uint32_t idesc = umma_idesc_f16(kGcRows, AB_FMT);
    const int m = warp - 8;
    const uint32_t acc = tmem_base + m * kGcRows;
    bool ok = true;
    int s = 0;
    uint32_t par = 0, use = 0;
    for (int t = p.t_hi; t >= p.t_lo && ok; --t)
      for (int ph = 0; ph < 2 * L && ok; ++ph) {
        const int buf = ph & 1;
        uint64_t* const tile = act_full + buf * kGcMaxCl;
        if (m == 0 && lane < CL && lane != rank) mbar_arrive_expect_tx(&tile[lane], kGcTile);   // (its own: the epilogue arrives)
        __syncwarp();
        ok = ch_wait<false>(&tile[rank], use & 1, p.err);      // this CTA's tile is also the word that the accumulators are free
        uint32_t more = 0;
        for (int j = m; j < 2 * CL; j += kGcMma) {
          const int src = rank + (j >> 1) < CL ? rank + (j >> 1) : rank + (j >> 1) - CL, st = m * SR + s;
          // half of the lanes wait for the weights, half for the tile (one after the other: 2.79 instead of 2.73 ms a call of
          // 128 rows, 3 x 1024, 100 steps)
          ok = ok && ch_wait<false>(lane & 1 ? &w_full[st] : &tile[src], lane & 1 ? par : use & 1, p.err);
          ok = __all_sync(0xffffffffu, ok);
          __syncwarp();        // (a vote orders no memory: the leader issues on what the other lanes have waited for)
          if (!ok) { if (leader) ch_fail(p.err, DEV_ERR_MMA_WAIT, 2, ph); break; }
          tc_fence_after_sync();
          if (leader) {
            const uint64_t da = umma_smem_desc_sw128(smem_u32(smem + lo.ring + st * 16384)),
                           db = umma_smem_desc_sw128(smem_u32(act + buf * act_bytes + src * kGcTile + (j & 1) * (kGcRows * 128)));
#pragma unroll
            for (int k = 0; k < kBlockK / 16; ++k) umma_f16(acc, da + 2 * k, db + 2 * k, idesc, k > 0 ? 1u : more);
            umma_commit(&w_empty[st]);
          }
          more = 1;
          __syncwarp();
          if (++s == SR) { s = 0; par ^= 1; }
        }
        if (ok && leader) umma_commit(acc_full);
        __syncwarp();
        if (buf == 1) ++use;
      }
  } else if (run && warp < 8) {
    // ---------------------------------------------------------------- epilogue: thread = 8 rows of the group in one column
    const int ew = warp, et = tid, q4 = ew & 3, half = ew >> 2, c = q4 * 32 + lane, col = n_base + c, r0 = half * kGcHalf;
    const int per = p.cfg ? 8 : 16, tok0 = grp * per;        // tokens of the group; row i is token i % per
    float2* norm_s = norm_all + ew * kGcHalf;                // this warp's copy of its rows' (mean, rstd)
    bool ok = true;
    uint32_t n_acc = 0, n_stat = 0, n_part = 0;
    auto epi_sync = [&]() { asm volatile("bar.sync 1, 256;" ::: "memory"); };
    auto wait = [&](uint64_t* bar, uint32_t parity, int site) {
      if (ok && !ch_wait<true>(bar, parity, p.err)) { ch_fail(p.err, DEV_ERR_EPI_WAIT, site, static_cast<int>(n_acc)); ok = false; }
    };
    const float4* const mods0 = p.mods + (grp * (kGcRows / 4) + r0 / 4) * 128;
    // product of step t with row `row` of tile `tile` of 128 weight rows, for this thread's rows of the group
    auto take_row = [&](float (&m)[kGcHalf], int t, int tile, int row) {
      const float4* src = mods0 + ((tile * p.nq + (t - p.t_lo) * (p.rows / 4)) * 128 + row);
      const float4 a = gc_ld(src), b = gc_ld(src + 128);
      m[0] = a.x; m[1] = a.y; m[2] = a.z; m[3] = a.w; m[4] = b.x; m[5] = b.y; m[6] = b.z; m[7] = b.w;
    };
    // two matrices whose rows are interleaved in groups of 64, from tile `base`, in this thread's column
    auto take_pair = [&](float (&u)[kGcHalf], float (&v)[kGcHalf], int t, int base) {
      const int tile = base + 2 * rank + (c >> 6);
      take_row(u, t, tile, c & 63); take_row(v, t, tile, 64 + (c & 63));
    };
    // Plain: per block shift | scale, gate; the final pair.  FOLD: gate_k | scale_{k+1} (k < L - 1), P1_k | P2_k (k = 1.., then 0),
    // shift_0 | scale_0, the last gate, the final pair.
    const int tail = (2 * L - 1) * 2 * CL;
    auto take_ss = [&](float (&sh)[kGcHalf], float (&sc)[kGcHalf], int t, int k) { take_pair(sh, sc, t, 3 * CL * k); };
    auto take_p12 = [&](float (&p1)[kGcHalf], float (&p2)[kGcHalf], int t, int k) { take_pair(p1, p2, t, 2 * CL * (k == 0 ? 2 * (L - 1) : L - 2 + k)); };
    auto take_gate = [&](float (&m)[kGcHalf], int t, int k) { take_row(m, t, 3 * CL * k + 2 * CL + rank, c); };
    // 16-bit tile of this CTA's columns: into its own activation buffer `buf`, and from there into every peer's
    auto send_tile = [&](const float (&v)[kGcHalf], int buf) {
      uint8_t* const out = act + buf * act_bytes + rank * kGcTile;
      uint8_t* kb = out + (c >> 6) * (kGcRows * 128) + r0 * 128;
      const int u = (c & 63) >> 3, b = (c & 7) * 2;
#pragma unroll
      for (int i = 0; i < kGcHalf; ++i) *reinterpret_cast<ACT*>(kb + i * 128 + ((u ^ i) << 4) + b) = to_act<ACT>(v[i]);
      fence_proxy_async_smem();
      epi_sync();
      if (ok && ew == 0 && lane < CL) {
        const uint32_t bar = smem_u32(&act_full[buf * kGcMaxCl + rank]);
        const int peer = rank + lane < CL ? rank + lane : rank + lane - CL;
        if (lane == 0) mbar_arrive(&act_full[buf * kGcMaxCl + rank]);
        else gc_copy(mapa_shared(smem_u32(out), peer), out, kGcTile, mapa_shared(bar, peer));
      }
      __syncwarp();
    };
    // (mean, M2) of each row over this warp's 32 columns, to every CTA
    auto send_stats = [&](const float (&v)[kGcHalf]) {
      const float mean = gc_reduce8(v, lane) * (1.0f / 32.0f);      // of row lane / 4
      float d[kGcHalf];
#pragma unroll
      for (int i = 0; i < kGcHalf; ++i) { const float e = v[i] - __shfl_sync(0xffffffffu, mean, 4 * i); d[i] = e * e; }
      const float m2 = gc_reduce8(d, lane);
      const uint32_t at = smem_u32(stats_s + (rank * 4 + q4) * kGcRows + r0 + (lane >> 2)), bar = smem_u32(stats_full);
      for (int r = lane & 3; ok && r < CL; r += 4) gc_st_async(mapa_shared(at, r), mean, m2, mapa_shared(bar, r));
    };
    const uint32_t stats_bytes = static_cast<uint32_t>(CL) * 4 * kGcRows * 8, part_bytes = static_cast<uint32_t>(CL) * kGcRows * kCPad * 4;
    // the rows' (mean, rstd) from all partials, into norm_s (32-column groups merged as equal-count partials)
    auto norms = [&]() {
      wait(stats_full, n_stat & 1, 5);
      if (et == 0) mbar_arrive_expect_tx(stats_full, stats_bytes);   // the next phase's
      ++n_stat;
      const int row = lane & 7, h = lane >> 3;                       // four lanes per row, a quarter of the W / 32 partials each
      const float2* src = stats_s + h * CL * kGcRows + r0 + row;
      float sm = 0.0f, m2 = 0.0f, q = 0.0f;
#pragma unroll 4
      for (int g = 0; g < CL; ++g) { const float2 v = src[g * kGcRows]; sm += v.x; m2 += v.y; }
      sm += __shfl_xor_sync(0xffffffffu, sm, 8);
      sm += __shfl_xor_sync(0xffffffffu, sm, 16);
      const float mean = sm / static_cast<float>(4 * CL);
#pragma unroll 4
      for (int g = 0; g < CL; ++g) { const float d = src[g * kGcRows].x - mean; q = fmaf(d, d, q); }
      m2 = fmaf(32.0f, q, m2);
      m2 += __shfl_xor_sync(0xffffffffu, m2, 8);
      m2 += __shfl_xor_sync(0xffffffffu, m2, 16);
      if (lane < kGcHalf) norm_s[row] = make_float2(mean, 1.0f / sqrtf(m2 / static_cast<float>(W) + 1e-6f));
      __syncwarp();
    };
    auto acc_load = [&](float (&a)[kGcHalf]) {
      wait(acc_full, n_acc & 1, 6);
      ++n_acc;
      tc_fence_after_sync();
      float b[kGcMma][kGcHalf];
#pragma unroll
      for (int m = 0; m < kGcMma; ++m) tmem_ld8(tmem_base + (static_cast<uint32_t>(q4 * 32) << 16) + m * kGcRows + r0, b[m]);
      tmem_ld_wait();
#pragma unroll
      for (int i = 0; i < kGcHalf; ++i) a[i] = (b[0][i] + b[1][i]) + b[2][i];
      tc_fence_before_sync();
    };

    if (et == 0) { mbar_arrive_expect_tx(stats_full, stats_bytes); mbar_arrive_expect_tx(part_full, part_bytes); }
    // state of the group's tokens
    const bool first = p.t_hi == T;
    if (et < per * kCPad) {
      const int tok = tok0 + (et >> 4), e = et & 15;
      float v = 0.0f;
      if (tok < p.R && e < p.C) {
        const size_t o = static_cast<size_t>(tok) * p.C + e;
        v = first ? p.x_T[o] : p.x[o];
        if (first && rank == 0 && p.traj_x) p.traj_x[o] = v;
      }
      xs[et] = v;
    }
    float h[kGcHalf], m0[kGcHalf], m1[kGcHalf], m2[FOLD ? 1 : kGcHalf], a[kGcHalf];
    // Plain: u = LN(h)(1 + scale) + shift of block k to every CTA
    auto send_u = [&](const float (&sh)[kGcHalf], const float (&sc)[kGcHalf], float bsh, float bsc) {
      norms();
#pragma unroll
      for (int i = 0; i < kGcHalf; ++i) {
        const float2 nr = norm_s[i];
        a[i] = fmaf(__fmul_rn(__fsub_rn(h[i], nr.x), nr.y), __fadd_rn(1.0f, sc[i] + bsc), sh[i] + bsh);
      }
      send_tile(a, 0);
    };
    float4 w0, w1, w2, w3;                                   // the column's input weights, on their way while the partials meet
    const float4* const win4 = reinterpret_cast<const float4*>(p.win + static_cast<size_t>(col) * kCPad);
    const float bi = __ldg(p.bin + col), bs = __ldg(p.bsc + col), bh = FOLD ? 0.0f : __ldg(p.bsh + col);
    auto take_win = [&]() { w0 = gc_ld(win4); w1 = gc_ld(win4 + 1); w2 = gc_ld(win4 + 2); w3 = gc_ld(win4 + 3); };
    auto take_first = [&](int t) { if constexpr (FOLD) take_row(m0, t, tail + 2 * rank + (c >> 6), 64 + (c & 63)); else take_ss(m0, m1, t, 0); };
    take_first(p.t_hi);
    take_win();
    epi_sync();
    for (int t = p.t_hi; t >= p.t_lo; --t) {
      // ---- h = Win x + bin for the column; a' = h (1 + scale_0), or u
      {
#pragma unroll
        for (int i = 0; i < kGcHalf; ++i) {
          const float4* xq = reinterpret_cast<const float4*>(xs + ((p.cfg ? 0 : r0) + i) * kCPad);
          const float4 x0 = xq[0], x1 = xq[1], x2 = xq[2], x3 = xq[3];
          float v = bi;
          v = fmaf(w0.x, x0.x, v); v = fmaf(w0.y, x0.y, v); v = fmaf(w0.z, x0.z, v); v = fmaf(w0.w, x0.w, v);
          v = fmaf(w1.x, x1.x, v); v = fmaf(w1.y, x1.y, v); v = fmaf(w1.z, x1.z, v); v = fmaf(w1.w, x1.w, v);
          v = fmaf(w2.x, x2.x, v); v = fmaf(w2.y, x2.y, v); v = fmaf(w2.z, x2.z, v); v = fmaf(w2.w, x2.w, v);
          v = fmaf(w3.x, x3.x, v); v = fmaf(w3.y, x3.y, v); v = fmaf(w3.z, x3.z, v); v = fmaf(w3.w, x3.w, v);
          h[i] = v;
        }
        if constexpr (FOLD) {
#pragma unroll
          for (int i = 0; i < kGcHalf; ++i) a[i] = __fmul_rn(h[i], __fadd_rn(1.0f, __fadd_rn(m0[i], bs)));
          send_tile(a, 0);
          take_p12(m0, m1, t, 0);
          send_stats(h);
        } else {
          send_stats(h);
          send_u(m0, m1, bh, bs);
        }
      }
#pragma unroll 1
      for (int k = 0; k < L; ++k) {
        // ---- v = SiLU(rstd (a' W1^T - mean (P1 + c1)) + P2 + c2), or SiLU(u W1^T + b1)
        if constexpr (FOLD) {
          const float k0 = __ldg(p.c1 + static_cast<size_t>(2 * k) * W + col), k1 = __ldg(p.c1 + static_cast<size_t>(2 * k + 1) * W + col);
          norms();
          acc_load(a);
#pragma unroll
          for (int i = 0; i < kGcHalf; ++i) {
            const float2 nr = norm_s[i];
            const float t1 = __fsub_rn(a[i], __fmul_rn(nr.x, __fadd_rn(m0[i], k0)));
            a[i] = silu_t<true>(fmaf(nr.y, t1, __fadd_rn(m1[i], k1)));
          }
          send_tile(a, 1);
        } else {
          const float k0 = __ldg(p.b1 + static_cast<size_t>(5 * k) * W + col);
          acc_load(a);
#pragma unroll
          for (int i = 0; i < kGcHalf; ++i) a[i] = silu_t<true>(a[i] + k0);
          send_tile(a, 1);
        }
        // ---- h += gate (v W2^T + b2); the next block's a' = h (1 + scale_{k+1}), or u
        const bool last = k + 1 == L;
        if constexpr (FOLD) {
          if (last) take_row(m0, t, tail + 2 * CL + rank, c);
          else take_pair(m0, m1, t, 2 * CL * k);
          const float kg = __ldg(p.bg + static_cast<size_t>(5 * k) * W + col), kb = __ldg(p.b2 + static_cast<size_t>(5 * k) * W + col),
                      ks = last ? 0.0f : __ldg(p.bsc + static_cast<size_t>(5 * (k + 1)) * W + col);
          acc_load(a);
#pragma unroll
          for (int i = 0; i < kGcHalf; ++i) h[i] = fmaf(__fadd_rn(m0[i], kg), __fadd_rn(a[i], kb), h[i]);
          if (!last) {
#pragma unroll
            for (int i = 0; i < kGcHalf; ++i) a[i] = __fmul_rn(h[i], __fadd_rn(1.0f, __fadd_rn(m1[i], ks)));
            send_tile(a, 0);
          }
          if (last) take_pair(m0, m1, t, tail + 3 * CL);
          else take_p12(m0, m1, t, k + 1);
          send_stats(h);
        } else {
          take_gate(m0, t, k);
          take_ss(m2, m1, t, k + 1);
          const size_t at = static_cast<size_t>(5 * k) * W + col, nx = last ? 0 : at + static_cast<size_t>(5) * W;
          const float kg = __ldg(p.bg + at), kb = __ldg(p.b2 + at), kh = __ldg(p.bsh + nx), ks = __ldg(p.bsc + nx);
          acc_load(a);
#pragma unroll
          for (int i = 0; i < kGcHalf; ++i) { h[i] = fmaf(m0[i] + kg, a[i] + kb, h[i]); m0[i] = m2[i]; }
          send_stats(h);
          if (!last) send_u(m0, m1, kh, ks);
        }
      }
      // ---- output projection of (LN(h)(1 + scale_f) + shift_f): this CTA's columns' part, to every CTA
      const float sa = p.ca[t - p.t_lo], sb = p.cb[t - p.t_lo], sg = p.sigma[t - p.t_lo];
      float noise = 0.0f;
      const int q = et >> 4, e = et & 15, tok = tok0 + q;                 // this thread's entry of the state
      const bool mine = et < per * kCPad && tok < p.R && e < p.C;
      if (mine) noise = p.eps[(static_cast<size_t>(t - 1) * p.R + tok) * p.C + e];
      {
        const float k0 = __ldg(p.bfsh + col), k1 = __ldg(p.bfsc + col);
        norms();
#pragma unroll
        for (int i = 0; i < kGcHalf; ++i) {
          const float2 nr = norm_s[i];
          uf_s[(r0 + i) * kUfLd + c] = fmaf(__fmul_rn(__fsub_rn(h[i], nr.x), nr.y), __fadd_rn(1.0f, m1[i] + k1), m0[i] + k0);
        }
        if (t > p.t_lo) take_first(t - 1);
        epi_sync();
        // four outputs of two rows over 16 columns per thread, the rows 2 ew, 2 ew + 1 in a warp; columns cg, cg + 8, ..
        const int quad = lane & 3, cg = lane >> 2;
        const float* u0 = uf_s + 2 * ew * kUfLd + cg;
        const float4* wq = reinterpret_cast<const float4*>(wout_s) + cg * 4 + quad;
        float o[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) o[i] = 0.0f;
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          const float4 w = wq[j * 32];
          const float a0 = u0[j * 8], a1 = u0[kUfLd + j * 8];
          o[0] = fmaf(a0, w.x, o[0]); o[1] = fmaf(a0, w.y, o[1]); o[2] = fmaf(a0, w.z, o[2]); o[3] = fmaf(a0, w.w, o[3]);
          o[4] = fmaf(a1, w.x, o[4]); o[5] = fmaf(a1, w.y, o[5]); o[6] = fmaf(a1, w.z, o[6]); o[7] = fmaf(a1, w.w, o[7]);
        }
        // sum over cg, transposing: lane (cg, quad) ends with value cg = 4 row + output
#pragma unroll
        for (int n = 4; n >= 1; n >>= 1) {
          const bool up = (cg & n) != 0;
#pragma unroll
          for (int i = 0; i < 4; ++i)
            if (i < n) {
              const float send = up ? o[i] : o[i + n], keep = up ? o[i + n] : o[i];
              o[i] = keep + __shfl_xor_sync(0xffffffffu, send, 4 * n);
            }
        }
        reinterpret_cast<float*>(part_out)[(2 * ew + (cg >> 2)) * kCPad + quad * 4 + (cg & 3)] = o[0];
        fence_proxy_async_smem();
        epi_sync();
        if (ok && ew == 0 && lane < CL)
          gc_copy(mapa_shared(smem_u32(part_s + rank * kGcRows * kCPad), lane), part_out, kGcRows * kCPad * 4, mapa_shared(smem_u32(part_full), lane));
        __syncwarp();
        take_win();
      }
      // ---- guidance and Eq. 3, by every CTA alike (CTA 0 writes what leaves the chip)
      const float bo = mine ? p.bout[e] : 0.0f;
      wait(part_full, n_part & 1, 7);
      if (et == 0) mbar_arrive_expect_tx(part_full, part_bytes);
      ++n_part;
      if (et < per * kCPad) {
        auto out = [&](int row) {
          float s = 0.0f;
          for (int r = 0; r < CL; ++r) s += part_s[(r * kGcRows + row) * kCPad + e];
          return s + bo;
        };
        float xn = 0.0f;
        if (mine) {
          const size_t o = static_cast<size_t>(tok) * p.C + e;
          float ee = out(q);
          if (p.cfg) ee = cfg_combine(ee, out(8 + q), p.cfg_scale);
          const float xo = xs[et], mu = ddpm_mean(sa, xo, sb, ee);
          xn = ddpm_sample(mu, sg, noise);
          if (rank == 0) {
            if (!(fabsf(xn) <= 3.0e38f)) *p.status = 1;
            if (t == 1) {
              p.mu1[o] = mu;
              if (p.x1) p.x1[o] = xo;
              if (p.sample_last && p.x0) p.x0[o] = xn;
            } else {
              if (t == p.t_lo) p.x[o] = xn;                    // the next launch starts from it
              if (p.traj_x) {
                const size_t slot = static_cast<size_t>(p.R) * p.C;
                p.traj_x[static_cast<size_t>(T - t + 1) * slot + o] = xn;
                p.traj_mu[static_cast<size_t>(T - t) * slot + o] = mu;
              }
            }
          }
        }
        xs[et] = xn;
      }
      epi_sync();
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  gc_settle(p.err);
  cluster_arrive(); cluster_wait();       // no CTA leaves while a peer may still write to it
  if (warp == 8) tmem_dealloc(tmem_base, 64);
}

}  // namespace csd
