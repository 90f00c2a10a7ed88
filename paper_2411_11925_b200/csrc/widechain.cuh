// A denoising chain of many rows (more than 256 head rows, W a multiple of 256 from 768 to 2048, 16-bit operands) in two parts:
//
// 1. wide_mods_kernel: everything a head takes from the condition vector - shifts, scales, gates: three fifths of its
//    multiply-adds - does not depend on x_t.  It is formed for several steps at once, as one dense product in fp32, at 8.8 TFLOP/s an SM.
// 2. wide_chain_kernel: what depends on x_t.  Token rows never exchange data, so the rows are cut into slots of 256 (two row
//    blocks of 128: with guidance 64 tokens' conditional rows and their unconditional twins each).  A group of W / 128 CTA pairs
//    owns one or two slots for all steps of a launch; pair n owns output columns [128 n, 128 n + 128) of every layer, one CTA one row
//    block of each slot.  Only the CTAs of a row block wait for each other; nothing waits for a kernel that runs beside it.
//
// A layer is latency: at W = 1024 its product takes 4.5 to 5.5 k cycles (4.1 k of MMAs; shared memory feeds them), and 7 to 10 k go by until
// the next may start - epilogue, stores, release, notice, first operand bytes, and where a LayerNorm lies between, the exchange of its
// partials.  Two forms (HV):
//   2  one slot a group, eight epilogue warps on it: a thread has 64 columns of a row.  A block of 3 and 6 x 1024 heads 22 k cycles.
//   1  two slots a group, four warps each: a layer's product on one slot runs during the other's hand-over.  37 k cycles for both slots: 18 k
//      a slot, on half of the SMs.
// What made the epilogues: words that are polled in one block of assembly (as a C++ loop ptxas held them twice and spilled: 27 k cycles more a
// step), few and wide tensor-memory reads (a read and its wait take some 300 cycles beside running MMAs), rolled loops, projections with
// four rows a thread so that a weight read from shared memory serves four (18 k -> 9 k cycles).  Taken back: sixteen epilogue warps
// (96 registers: spills), a register hand-over between warpgroups by setmaxnreg (illegal instruction: the last warpgroup has three warps), half
// tiles published by a warp of their own (its fence and release wait for all of the SM's stores: 15.7 -> 16.4 ms a round).
//
// 1024 rows each of 3 and 6 x 1024 heads, T = 100: chains alone 8.4 -> 6.8 and 15.1 -> 11.2 ms, a single round 16.6 -> 14.0 ms (repeated for
// seconds 16.7 -> 16.1: the GPU is at its power cap then, at 1.67 GHz instead of 1.76).  Before: one persistent kernel per chain that formed the condition
// products itself, folded blocks.
//
// Accumulators and the residual stream h stay in tensor memory (128 columns each per slot).  The 16-bit operands u and v cross
// global memory in the order in which the MMA wants them in shared memory (no swizzle: [8-column chunk][128 rows][16 bytes]), so
// that an epilogue warp's direct stores cover 512 contiguous bytes; a counter per row block says when all column tiles are there.
// What is small - LayerNorm partials, output-projection partials, the token states - travels as 16-byte words that carry their
// own step number (value | tag, value | tag): the reader polls the data itself and no fence stands in between.
#pragma once
#include "groupchain.cuh"
#include "wideplan.h"

namespace csd {

// ------------------------------------------------------------------------------------------ products of s_t
struct WmParams {
  int nkb, nst, nwt, sb;       // k-blocks; tiles of 256 rows of s, of 256 weight rows; tiles of s that share a pass over the weights
  const int* wrow;             // first row of each weight tile: of shift | scale rows (interleaved by 64), or ~row of gate rows
  const float* bias;           // [nwt][256]
  int* ticket;                 // zeroed before the launch
  float* out;                  // [nwt][row block of s][32768], see the kernel
  int* err;
};

// out = s weights^T + bias in 256 x 256 tiles per CTA pair, as wide_chain_kernel reads it: per weight tile and row block of 128
// rows of s 128 KB, shift | scale tiles as [32-row quarter][8-column group][shift, 1 + scale][2 quads][32 rows][4], gate
// tiles as [128-column half][32-row quarter][16-column group][4 quads][32 rows][4]: a lane holds a row, so a warp's 16-byte accesses
// cover 512 contiguous bytes on both sides.  Tiles are handed out by ticket: pairs that find their SMs late, because a chain still
// has them, take what is left.
template <int AB_FMT>
__global__ void __launch_bounds__(kMgThreads, 1)
wide_mods_kernel(const __grid_constant__ CUtensorMap tmW, const __grid_constant__ CUtensorMap tmS, const WmParams p) {
  constexpr int S = kMgStages;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + S * kMgStageBytes);
  uint64_t* empty_bar = full_bar + S;
  uint64_t* acc_full = empty_bar + S;     // [2]
  uint64_t* acc_empty = acc_full + 2;     // [2], every epilogue warp of both CTAs
  uint64_t* tick_bar = acc_empty + 2;     // [4]
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(tick_bar + 4);     // and whether the context is free of errors
  volatile int* tick_s = reinterpret_cast<volatile int*>(tmem_base_s + 2);   // [4] tickets, written by the leader's first producer

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int units = p.nst * p.nwt;
  if (threadIdx.x == 0) {
    tma_prefetch_desc(&tmW); tma_prefetch_desc(&tmS);
    for (int s = 0; s < S; ++s) { mbar_init(&full_bar[s], 2); mbar_init(&empty_bar[s], 1); }
    for (int i = 0; i < 2; ++i) { mbar_init(&acc_full[i], 1); mbar_init(&acc_empty[i], 2 * kMgEpiWarps); }
    for (int i = 0; i < 4; ++i) mbar_init(&tick_bar[i], 1);
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

  // Ticket of this pair's i-th tile (units or more: none left; -1: gave up).  A slot is written again four tickets on, when the leader's
  // producers have issued three tiles more: their last stages were free, so the MMAs of the third have begun, so every epilogue
  // warp has read the accumulators, and before them the ticket, of the first.
  auto ticket = [&](int i) {
    if (!ch_wait<true>(&tick_bar[i & 3], (i >> 2) & 1, p.err)) { ch_fail(p.err, DEV_ERR_TMA_WAIT, 4, i); return -1; }
    return tick_s[i & 3];
  };
  // tile of weights and of s; all weights pass by sb tiles of s at a time, so that those stay in L2
  auto place = [&](int u, int& wt, int& st) {
    const int b = u / (p.sb * p.nwt), left = p.nst - b * p.sb, n = left < p.sb ? left : p.sb, r = u - b * p.sb * p.nwt;
    wt = r / n; st = b * p.sb + r % n;
  };

  if (run && (warp == 0 || warp == kMgEpiWarps + 2)) {
    const bool is_s = warp == 0;
    if (lane == 0) {
      const bool deals = is_s && rank == 0;
      int it = 0, next = deals ? atomicAdd(p.ticket, 1) : 0;
      bool ok = true;
      for (int i = 0; ok; ++i) {
        int u;
        if (deals) {
          u = next;
          for (int r = 0; r < 2; ++r) {
            const uint32_t a = mapa_shared(smem_u32(const_cast<int*>(tick_s + (i & 3))), static_cast<uint32_t>(r)), b = mapa_shared(smem_u32(&tick_bar[i & 3]), static_cast<uint32_t>(r));
            asm volatile("st.shared::cluster.u32 [%0], %1;" ::"r"(a), "r"(u) : "memory");
            asm volatile("mbarrier.arrive.release.cluster.shared::cluster.b64 _, [%0];" ::"r"(b) : "memory");
          }
          if (u < units) next = atomicAdd(p.ticket, 1);
        } else u = ticket(i);
        if (u < 0 || u >= units) break;
        int wt, st;
        place(u, wt, st);
        const int wr = is_s ? 0 : __ldg(p.wrow + wt);
        const int row = (is_s ? st * 256 : wr < 0 ? ~wr : wr) + rank * 128;
        const CUtensorMap* const tm = is_s ? &tmS : &tmW;
        for (int kb = 0; kb < p.nkb; ++kb, ++it) {
          const int s = it % S;
          if (it >= S && !ch_wait<false>(&empty_bar[s], ((it / S) & 1) ^ 1, p.err)) { ch_fail(p.err, DEV_ERR_TMA_WAIT, 1, it); ok = false; break; }
          if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], 32768);     // both CTAs' bytes of this operand
          tma_load_2d_pair(smem + s * kMgStageBytes + (is_s ? 0 : 16384), tm, mapa_shared(smem_u32(&full_bar[s]), 0), kb * kBlockK, row);
        }
      }
    }
    __syncwarp();
  } else if (run && warp == 1 && rank == 0) {
    const bool leader = elect_one();
    constexpr uint32_t idesc = umma_idesc_f16(256, AB_FMT, 256);
    bool ok = true;
    int it = 0;
    for (int i = 0; ok; ++i) {
      const int u = __shfl_sync(0xffffffffu, ticket(i), 0);
      if (u < 0 || u >= units) break;
      const int ab = i & 1;
      if (i >= 2 && !ch_wait<true>(&acc_empty[ab], ((i >> 1) - 1) & 1, p.err)) { if (leader) ch_fail(p.err, DEV_ERR_MMA_WAIT, 1, i); break; }
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
    for (int i = 0;; ++i) {
      const int u = __shfl_sync(0xffffffffu, ticket(i), 0);
      if (u < 0 || u >= units) break;
      int wt, st;
      place(u, wt, st);
      const int ab = i & 1;
      const bool gate = __ldg(p.wrow + wt) < 0;
      bool ok = ch_wait<false>(&acc_full[ab], (i >> 1) & 1, p.err);
      if (!ok) ch_fail(p.err, DEV_ERR_EPI_WAIT, 1, i);
      ok = __all_sync(0xffffffffu, ok);
      if (!ok) break;
      tc_fence_after_sync();
      const uint32_t trow = tmem_base + ab * 256 + half * 128 + (static_cast<uint32_t>(q * 32) << 16);
      const float4* const b4 = reinterpret_cast<const float4*>(p.bias + static_cast<size_t>(wt) * 256 + half * 128);
      float4* const o = reinterpret_cast<float4*>(p.out) + ((static_cast<size_t>(wt) * p.nst + st) * 2 + rank) * 8192 + lane;
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
        for (int j = 0; j < kChunk / 4; ++j) {
          const float4 b = __ldg(b4 + c * 8 + j);
          float4 v = make_float4(a[4 * j] + b.x, a[4 * j + 1] + b.y, a[4 * j + 2] + b.z, a[4 * j + 3] + b.w);
          if (gate) o[half * 4096 + q * 1024 + (c * 2 + (j >> 2)) * 128 + (j & 3) * 32] = v;
          else {                 // columns of this half: 64 of shift, 64 of scale
            if (c >= 2) v = make_float4(__fadd_rn(1.0f, v.x), __fadd_rn(1.0f, v.y), __fadd_rn(1.0f, v.z), __fadd_rn(1.0f, v.w));
            o[q * 2048 + (half * 8 + (c & 1) * 4 + (j >> 1)) * 128 + ((c >> 1) * 2 + (j & 1)) * 32] = v;
          }
        }
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
constexpr int kWcMmaWarp = 8, kWcActWarp = 9, kWcWeightWarp = 10;
constexpr int kWcThreads = 11 * 32;
constexpr int kWcAhead = 4;               // pieces of the products that an epilogue thread has in flight
constexpr int kWcStageBytes = 24576;      // one k-block: 128 rows of u or v | 64 weight rows
constexpr int kWcMaxStages = 8, kWcMinStages = 4;
constexpr int kWcMaxSteps = 64;           // steps per launch: their coefficients travel as kernel parameters
constexpr int kWcMaxCt = 16;              // column tiles: W up to 2048

struct WcLayout { int ring, stages, win, wout, bias, bin, xch, eh, bars, total; };
__host__ __device__ inline WcLayout wc_layout(int L, int epw, int halves) {
  WcLayout l{};
  int o = 0;
  auto take = [&](int n) { const int r = o; o += n; return r; };
  l.win = take(128 * kCPad * 4);
  l.wout = take(128 * epw * 4);
  l.bias = take(2 * L * 128 * 4);
  l.bin = take(128 * 4);
  l.xch = take(halves == 2 ? 128 * 8 : 0);          // a row's partial, of the second half of the columns
  l.eh = take(halves == 2 ? 128 * epw * 4 : 0);     // its output-projection sums
  l.bars = take(512);
  o = (o + 1023) / 1024 * 1024;
  l.ring = o;
  l.stages = (226 * 1024 - o) / kWcStageBytes;
  if (l.stages > kWcMaxStages) l.stages = kWcMaxStages;
  l.total = o + l.stages * kWcStageBytes;
  return l;
}

struct WcParams {
  int R, cfg, W, L, C, T, t_hi, t_lo, slot0, slots, sample_last;   // slots [slot0, slot0 + slots) in this launch
  float cfg_scale;
  const CUtensorMap* maps;     // [2 L]: W1_k, W2_k in boxes of 64 rows
  const float* mods;           // products of the launch's steps and slots
  const float *b1, *b2;        // block 0; 5 W apart
  const float *win, *bin, *wout_t, *bout;
  const float *x_T, *eps;
  float *x, *x0, *mu1, *x1, *traj_x, *traj_mu;
  void *u, *v;                 // [row block][W / 8][128][8] operands
  ulonglong2* stats;           // [row block][W / 128][128]   (mean | tag, M2 | tag)
  ulonglong2* epart;           // [row block][W / 128][8 or 16 column pairs][128]
  ulonglong2* xll;             // [row block][8 column pairs][128 tokens]
  unsigned* cnt;               // [row block][u, v] column tiles published, 128 bytes apart
  float* hsum;                 // LV: [row block][128 tokens][16] running half log-determinants
  float *lv1, *half_logdet;
  int* err;
  int* status;
  float ca[kWcMaxSteps], cb[kWcMaxSteps], s0[kWcMaxSteps], s1[kWcMaxSteps];   // index t - t_lo; s0: sigma, or LV the bounds s0, s1
};

__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }
__device__ __forceinline__ void tmem_ld16(uint32_t taddr, float* v) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x16.b32 {%0, %1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15}, [%16];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7]), "=r"(r[8]),
                 "=r"(r[9]), "=r"(r[10]), "=r"(r[11]), "=r"(r[12]), "=r"(r[13]), "=r"(r[14]), "=r"(r[15])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_st16(uint32_t taddr, const float* v) {
  const uint32_t* r = reinterpret_cast<const uint32_t*>(v);
  asm volatile("tcgen05.st.sync.aligned.32x32b.x16.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
                 "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15])
               : "memory");
}

__device__ __forceinline__ void tmem_st8(uint32_t taddr, const float* v) {
  const uint32_t* r = reinterpret_cast<const uint32_t*>(v);
  asm volatile("tcgen05.st.sync.aligned.32x32b.x8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}
// 16 lanes x 16 columns as the accumulator of an m16n8 product, twice: values 4 g + 2 h + b of thread i are of lane i / 4 + 8 h, column
// 8 g + 2 (i % 4) + b.
__device__ __forceinline__ void tmem_ld_frag(uint32_t taddr, float* v) {
  uint32_t* r = reinterpret_cast<uint32_t*>(v);
  asm volatile("tcgen05.ld.sync.aligned.16x256b.x2.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(r[0]), "=r"(r[1]), "=r"(r[2]), "=r"(r[3]), "=r"(r[4]), "=r"(r[5]), "=r"(r[6]), "=r"(r[7])
               : "r"(taddr)
               : "memory");
}
__device__ __forceinline__ void tmem_st_frag(uint32_t taddr, const float* v) {
  const uint32_t* r = reinterpret_cast<const uint32_t*>(v);
  asm volatile("tcgen05.st.sync.aligned.16x256b.x2.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};"
               ::"r"(taddr), "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7])
               : "memory");
}

// Words that carry their own tag: each 64-bit half is written and read in one piece.
__device__ __forceinline__ void wc_put(ulonglong2* p, float a, float b, uint32_t tag) {
  const unsigned long long t = static_cast<unsigned long long>(tag) << 32;
  asm volatile("st.relaxed.gpu.global.v2.b64 [%0], {%1, %2};" ::"l"(p), "l"(t | __float_as_uint(a)), "l"(t | __float_as_uint(b)) : "memory");
}
// Eight words, two (2 KB apart) from each of four places, polled until all carry the tag.  False: the context's error word is up, or
// the wait took longer than the bound of every other one, in cycles of the SM clock.  (One block of assembly: as a C++ loop the words are held twice.)
__device__ __forceinline__ bool wc_poll(ulonglong2 (&w)[8], const ulonglong2* a, const ulonglong2* b, const ulonglong2* c, const ulonglong2* d,
                                        uint32_t tag, const int* err) {
  uint32_t bad;
  asm volatile(
      "{\n\t.reg .pred p;\n\t.reg .b32 x, lo, hi, t0;\n\t.reg .b64 now, most;\n\t"
      "mov.u64 now, %%clock64;\n\tshr.u64 now, now, 10;\n\tcvt.u32.u64 t0, now;\n"      // units of 1024 cycles
      "AGAIN:\n\t"
      "ld.relaxed.gpu.global.v2.b64 {%0, %1}, [%17];\n\t"
      "ld.relaxed.gpu.global.v2.b64 {%2, %3}, [%17 + 2048];\n\t"
      "ld.relaxed.gpu.global.v2.b64 {%4, %5}, [%18];\n\t"
      "ld.relaxed.gpu.global.v2.b64 {%6, %7}, [%18 + 2048];\n\t"
      "ld.relaxed.gpu.global.v2.b64 {%8, %9}, [%19];\n\t"
      "ld.relaxed.gpu.global.v2.b64 {%10, %11}, [%19 + 2048];\n\t"
      "ld.relaxed.gpu.global.v2.b64 {%12, %13}, [%20];\n\t"
      "ld.relaxed.gpu.global.v2.b64 {%14, %15}, [%20 + 2048];\n\t"
      "ld.relaxed.gpu.global.u32 %16, [%22];\n\t"
      "mov.b64 {lo, hi}, %0;\n\txor.b32 x, hi, %21;\n\t"
#define WC_CHECK(r) "mov.b64 {lo, hi}, %" #r ";\n\txor.b32 hi, hi, %21;\n\tor.b32 x, x, hi;\n\t"
      WC_CHECK(1) WC_CHECK(2) WC_CHECK(3) WC_CHECK(4) WC_CHECK(5) WC_CHECK(6) WC_CHECK(7) WC_CHECK(8)
      WC_CHECK(9) WC_CHECK(10) WC_CHECK(11) WC_CHECK(12) WC_CHECK(13) WC_CHECK(14) WC_CHECK(15)
#undef WC_CHECK
      "setp.ne.u32 p, %16, 0;\n\t@p bra DONE;\n\t"
      "setp.eq.u32 p, x, 0;\n\t@p bra DONE;\n\t"
      "mov.u64 now, %%clock64;\n\tshr.u64 now, now, 10;\n\tcvt.u32.u64 x, now;\n\tsub.u32 x, x, t0;\n\t"
      "setp.lt.u32 p, x, 64;\n\t@p bra AGAIN;\n\t"                                           // (the limit is read only then)
      "cvt.u64.u32 now, x;\n\t"
      "ld.volatile.global.u64 most, [%23];\n\tshr.u64 most, most, 10;\n\t"
      "setp.le.u64 p, now, most;\n\t@p bra AGAIN;\n\t"
      "mov.u32 %16, 1;\n"
      "DONE:\n\t}"
      : "=&l"(w[0].x), "=&l"(w[0].y), "=&l"(w[1].x), "=&l"(w[1].y), "=&l"(w[2].x), "=&l"(w[2].y), "=&l"(w[3].x), "=&l"(w[3].y),
        "=&l"(w[4].x), "=&l"(w[4].y), "=&l"(w[5].x), "=&l"(w[5].y), "=&l"(w[6].x), "=&l"(w[6].y), "=&l"(w[7].x), "=&l"(w[7].y), "=&r"(bad)
      : "l"(a), "l"(b), "l"(c), "l"(d), "r"(tag), "l"(err), "l"(&g_wait_limit_cycles)
      : "memory");
  return bad == 0;
}
__device__ __forceinline__ float wc_lo(unsigned long long v) { return __uint_as_float(static_cast<uint32_t>(v)); }

// K-major operand without swizzle: 8-row groups 128 bytes apart, 8-column chunks 2048.
__device__ __forceinline__ uint64_t umma_smem_desc_plain(uint32_t smem_addr) {
  uint64_t d = 0;
  d |= static_cast<uint64_t>((smem_addr & 0x3FFFF) >> 4);
  d |= static_cast<uint64_t>(2048 >> 4) << 16;
  d |= static_cast<uint64_t>(128 >> 4) << 32;
  d |= static_cast<uint64_t>(1) << 46;
  return d;
}

__device__ __forceinline__ void wc_prefetch_l2(const void* p, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;" ::"l"(p), "r"(bytes) : "memory");
}

__device__ __forceinline__ unsigned wc_ld_acquire(const unsigned* p) {
  unsigned v;
  asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(p) : "memory");
  return v;
}
// (after a barrier: cumulative over the writes that the barrier ordered before it)
__device__ __forceinline__ void wc_arrive(unsigned* p) {
  asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(p) : "memory");
}
// One thread waits until the counter has reached target (bounded; gives up once the context's status word is up).
__device__ __forceinline__ bool wc_wait_count(const unsigned* p, unsigned target, const int* err) {
  long long t0 = 0;
  uint32_t spins = 0;
  for (;;) {
    if (wc_ld_acquire(p) >= target) return true;
    if ((++spins & 255u) == 0u) {
      if (*reinterpret_cast<const volatile int*>(err) != 0) return false;
      const long long now = clock64();
      if (t0 == 0) t0 = now;
      else if (now - t0 > *reinterpret_cast<volatile long long*>(&g_wait_limit_cycles)) return false;
    }
  }
}

template <typename ACT, int AB_FMT, bool LV, int HV>
__global__ void __launch_bounds__(kWcThreads, 1)
wide_chain_kernel(const __grid_constant__ CUtensorMap tmU, const __grid_constant__ CUtensorMap tmV, const __grid_constant__ WcParams p) {
  constexpr int EPW = LV ? kCPad2 : kCPad, NC = EPW / 2;
  constexpr int GS = 2 / HV, CW = 128 / HV;      // slots of a group; columns of an epilogue thread
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  const int W = p.W, L = p.L, T = p.T, CT = W / 128, nkb = W / kBlockK;
  const WcLayout lo = wc_layout(L, EPW, HV);
  const int S = lo.stages;
  uint8_t* ring = smem + lo.ring;
  float* win_s = reinterpret_cast<float*>(smem + lo.win);
  float* wout_s = reinterpret_cast<float*>(smem + lo.wout);
  float* bias_s = reinterpret_cast<float*>(smem + lo.bias);      // [2 L][128]: b1_k, b2_k
  float* bin_s = reinterpret_cast<float*>(smem + lo.bin);
  [[maybe_unused]] float2* xch_s = reinterpret_cast<float2*>(smem + lo.xch);
  [[maybe_unused]] float* eh_s = reinterpret_cast<float*>(smem + lo.eh);
  uint64_t* full_bar = reinterpret_cast<uint64_t*>(smem + lo.bars);
  uint64_t* empty_bar = full_bar + kWcMaxStages;
  uint64_t* acc_full = empty_bar + kWcMaxStages;    // [slot]
  uint64_t* acc_empty = acc_full + 2;               // [slot], 4 warps of each CTA
  uint32_t* tmem_base_s = reinterpret_cast<uint32_t*>(acc_empty + 2);       // and whether the context is free of errors

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int cl = static_cast<int>(blockIdx.x >> 1), grp = cl / CT, tile_n = cl % CT, n_base = tile_n * 128;
  const int nslot = p.slots - GS * grp < GS ? 1 : GS;
  const int rb0 = 2 * (p.slot0 + GS * grp) + rank;                // row block of slot 0; of slot 1: + 2
  if (tid == 0) {
    tma_prefetch_desc(&tmU); tma_prefetch_desc(&tmV);
    for (int s = 0; s < kWcMaxStages; ++s) { mbar_init(&full_bar[s], 2); mbar_init(&empty_bar[s], 1); }
    for (int s = 0; s < 2; ++s) { mbar_init(&acc_full[s], 1); mbar_init(&acc_empty[s], 8 * HV); }
    tmem_base_s[1] = *reinterpret_cast<const volatile int*>(p.err) == 0;    // one reading for all warps
    fence_mbar_init();
  }
  if (warp == kWcMmaWarp) { tmem_alloc_pair(tmem_base_s, 512); tmem_relinquish_pair(); }
  // 16-byte chunks of a column's weights in an order by column pair, so that the four column pairs a warp reads at a time lie in different banks
  auto w_at = [](int col, int c, int epw) { return col * epw + (c ^ ((col & 6) << 1)); };
  for (int i = tid; i < 128 * kCPad; i += kWcThreads) win_s[w_at(i / kCPad, i % kCPad, kCPad)] = p.win[static_cast<size_t>(n_base) * kCPad + i];
  if (tid < 128) bin_s[tid] = p.bin[n_base + tid];
  for (int i = tid; i < 128 * EPW; i += kWcThreads) wout_s[w_at(i / EPW, i % EPW, EPW)] = p.wout_t[static_cast<size_t>(n_base) * EPW + i];
  for (int i = tid; i < L * 128; i += kWcThreads) {
    const int k = i >> 7, c = i & 127;
    bias_s[(2 * k) * 128 + c] = p.b1[static_cast<size_t>(5 * k) * W + n_base + c];
    bias_s[(2 * k + 1) * 128 + c] = p.b2[static_cast<size_t>(5 * k) * W + n_base + c];
  }
  tc_fence_before_sync();
  __syncthreads();
  cluster_arrive(); cluster_wait();       // the peer's barriers exist before anything signals them
  tc_fence_after_sync();
  const uint32_t tmem_base = *tmem_base_s;
  const bool run = tmem_base_s[1] != 0;

  // (a warp that gives up on a wait goes on through its barriers without waiting: other waits end by the context's error word)
  if (run && warp == kWcActWarp) {
    // ---------------------------------------------------------------- operands u and v of this CTA's row blocks
    if (lane == 0) {
      int s = 0;
      uint32_t par = 1;
      bool ok = true;
      for (int t = p.t_hi; t >= p.t_lo && ok; --t)
        for (int ph = 0; ph < 2 * L && ok; ++ph)
          for (int sl = 0; sl < nslot && ok; ++sl) {
            const int rb = rb0 + 2 * sl;
            const CUtensorMap* const tm = (ph & 1) ? &tmV : &tmU;
            const unsigned target = static_cast<unsigned>(((T - t) * L + (ph >> 1) + 1) * CT);
            if (!wc_wait_count(p.cnt + (rb * 2 + (ph & 1)) * 32, target, p.err)) { ch_fail(p.err, DEV_ERR_TMA_WAIT, 3, ph); ok = false; break; }
            for (int kb = 0; kb < nkb; ++kb) {
              if (!ch_wait<false>(&empty_bar[s], par, p.err)) { ch_fail(p.err, DEV_ERR_TMA_WAIT, 1, ph); ok = false; break; }   // (fresh: passes)
              if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], 32768);     // both CTAs' bytes
              tma_load_2d_pair(ring + s * kWcStageBytes, tm, mapa_shared(smem_u32(&full_bar[s]), 0), 0, rb * (W / 2) + kb * 32);
              if (++s == S) { s = 0; par ^= 1; }
            }
          }
    }
    __syncwarp();
  } else if (run && warp == kWcWeightWarp) {
    // ---------------------------------------------------------------- weights: half of the pair's 128 rows
    if (lane == 0) {
      int s = 0;
      uint32_t par = 1;
      bool ok = true;
      for (int t = p.t_hi; t >= p.t_lo && ok; --t)
        for (int ph = 0; ph < 2 * L && ok; ++ph)
          for (int sl = 0; sl < nslot && ok; ++sl)
            for (int kb = 0; kb < nkb; ++kb) {
              if (!ch_wait<false>(&empty_bar[s], par, p.err)) { ch_fail(p.err, DEV_ERR_TMA_WAIT, 2, ph); ok = false; break; }
              if (rank == 0) mbar_arrive_expect_tx(&full_bar[s], 16384);
              tma_load_2d_pair(ring + s * kWcStageBytes + 16384, p.maps + ph, mapa_shared(smem_u32(&full_bar[s]), 0), kb * kBlockK, n_base + rank * 64);
              if (++s == S) { s = 0; par ^= 1; }
            }
    }
    __syncwarp();
  } else if (run && warp == kWcMmaWarp && rank == 0) {
    // ---------------------------------------------------------------- MMA issue (the pair's leader)
    const bool leader = elect_one();
    constexpr uint32_t idesc = umma_idesc_f16(128, AB_FMT, 256);
    bool ok = true;
    int s = 0, it = 0;
    uint32_t par = 0;
    for (int t = p.t_hi; t >= p.t_lo && ok; --t)
      for (int ph = 0; ph < 2 * L && ok; ++ph, ++it)
        for (int sl = 0; sl < nslot && ok; ++sl) {
          if (it > 0 && !ch_wait<true>(&acc_empty[sl], (it - 1) & 1, p.err)) { if (leader) ch_fail(p.err, DEV_ERR_MMA_WAIT, 1, ph); ok = false; break; }
          tc_fence_after_sync();
          for (int kb = 0; kb < nkb; ++kb) {
            if (!ch_wait<false>(&full_bar[s], par, p.err)) { if (leader) ch_fail(p.err, DEV_ERR_MMA_WAIT, 2, ph); ok = false; break; }
            tc_fence_after_sync();
            if (leader) {
              const uint32_t sa = smem_u32(ring + s * kWcStageBytes);
              const uint64_t da = umma_smem_desc_plain(sa), db = umma_smem_desc_sw128(sa + 16384);
#pragma unroll
              for (int k = 0; k < kBlockK / 16; ++k)
                umma_f16_pair(tmem_base + sl * 128, da + 256 * k, db + 2 * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
              umma_commit_pair(&empty_bar[s]);
            }
            __syncwarp();
            if (++s == S) { s = 0; par ^= 1; }
          }
          if (ok && leader) umma_commit_pair(&acc_full[sl]);
          __syncwarp();
        }
  } else if (run && warp < 8 && (HV == 2 || (warp >> 2) < nslot)) {
    // ---------------------------------------------------------------- epilogues of one slot: thread = one row, 128 or 64 columns
    const int sl = HV == 1 ? warp >> 2 : 0, hf = HV == 2 ? warp >> 2 : 0, q = warp & 3, et = tid & 127;
    const int rb = rb0 + 2 * sl, rloc = et;
    const uint32_t trow = tmem_base + (static_cast<uint32_t>(q * 32) << 16);
    const uint32_t t_acc = trow + sl * 128 + hf * CW, t_h = trow + 256 + sl * 128 + hf * CW;
    const int per = p.cfg ? 64 : 128, tk_row = p.cfg ? (rloc & 63) : rloc;       // tokens of a row block; this row's
    bool ok = true;
    auto slot_sync = [&]() { if constexpr (HV == 1) asm volatile("bar.sync %0, 128;" ::"r"(1 + sl) : "memory"); else asm volatile("bar.sync 1, 256;" ::: "memory"); };
    // HV == 2: the second half's warp has left something for the first half's in shared memory
    auto hand_over = [&]() { asm volatile("bar.sync %0, 64;" ::"r"(3 + q) : "memory"); };
    // eight words of this lane, or the word that it gives up
    auto poll = [&](ulonglong2 (&w)[8], const ulonglong2* a, const ulonglong2* b, const ulonglong2* c, const ulonglong2* d, uint32_t tag, int site) {
      const bool got = wc_poll(w, a, b, c, d, tag, p.err);      // (once given up, the error word ends it at once; a branch around it would have the words held twice)
      if (ok && !got) ch_fail(p.err, DEV_ERR_EPI_WAIT, site, static_cast<int>(tag));
      ok = __all_sync(0xffffffffu, ok && got);
    };
    // products of one step: pieces of 2 KB, 16 floats of each lane's row
    const int mrows = 2 * p.slots, nsb = (p.t_hi - p.t_lo + 1) * mrows;
    const int mrb = rb - 2 * p.slot0;
    float4 m[kWcAhead][4];
    auto mod_tile = [&](int t, int tile) { return p.mods + (static_cast<size_t>(tile) * nsb + (t - p.t_lo) * mrows + mrb) * 32768; };
    auto ss_at = [&](int t, int k) { return mod_tile(t, k * (CT + CT / 2) + tile_n) + q * 8192 + hf * 4096; };     // CW / 8 pieces of 8 columns (k = L: the final pair)
    auto gate_at = [&](int t, int k) { return mod_tile(t, k * (CT + CT / 2) + CT + tile_n / 2) + (tile_n & 1) * 16384 + q * 4096 + hf * 2048; };   // CW / 16 of 16
    auto take = [&](float4 (&d)[4], const float* piece) {
#pragma unroll
      for (int j = 0; j < 4; ++j) d[j] = gc_ld(reinterpret_cast<const float4*>(piece) + j * 32 + lane);
    };
    auto take_first = [&](const float* piece) {
#pragma unroll
      for (int i = 0; i < kWcAhead; ++i) take(m[i], piece + i * 512);
    };
    auto ahead = [&](const float* piece, uint32_t bytes) { if (lane == 0) wc_prefetch_l2(piece, bytes); };
    // (mean, M2) of 16 values
    auto stats16 = [&](float& mu, float& m2, const float (&hv)[16]) {
      float a[4], b[4];
#pragma unroll
      for (int j = 0; j < 4; ++j) a[j] = (hv[j] + hv[4 + j]) + (hv[8 + j] + hv[12 + j]);
      mu = ((a[0] + a[1]) + (a[2] + a[3])) * (1.0f / 16.0f);
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float d0 = hv[j] - mu, d1 = hv[4 + j] - mu, d2 = hv[8 + j] - mu, d3 = hv[12 + j] - mu;
        b[j] = fmaf(d0, d0, __fmul_rn(d1, d1)) + fmaf(d2, d2, __fmul_rn(d3, d3));
      }
      m2 = (b[0] + b[1]) + (b[2] + b[3]);
    };
    // i-th group of 16 of this row's columns (i & 3 known at compile time): pairs, fours, eights
    struct Partial { float pm[3], p2[3]; };
    auto partial_add = [&](Partial& s, int i, int four, const float (&hv)[16]) {
      float mu, m2;
      stats16(mu, m2, hv);
      if (i & 1) {
        chan_merge_equal(s.pm[0], s.p2[0], mu, m2, 16.0f);
        if (i == 1) { s.pm[1] = s.pm[0]; s.p2[1] = s.p2[0]; }
        else {
          chan_merge_equal(s.pm[1], s.p2[1], s.pm[0], s.p2[0], 32.0f);
          if (four == 0) { s.pm[2] = s.pm[1]; s.p2[2] = s.p2[1]; } else chan_merge_equal(s.pm[2], s.p2[2], s.pm[1], s.p2[1], 64.0f);
        }
      } else { s.pm[0] = mu; s.p2[0] = m2; }
    };
    // LayerNorm partial of this row's 128 columns, to every column tile
    auto put_stats = [&](float mean, float m2, uint32_t tag) {
      if constexpr (HV == 2) {           // (the giver is here again only after the taker's word has gone round)
        if (hf == 1) xch_s[rloc] = make_float2(mean, m2);
        hand_over();
        if (hf == 1) return;
        const float2 o = xch_s[rloc];
        chan_merge_equal(mean, m2, o.x, o.y, 64.0f);
      }
      wc_put(p.stats + (rb * CT + tile_n) * 128 + rloc, mean, m2, tag);
    };
    // the row's mean and 1 / std
    float mean = 0.0f, rstd = 0.0f;
    auto norms = [&](uint32_t tag) {
      const ulonglong2* src = p.stats + rb * CT * 128 + rloc;
      float mh = 0.0f, m2 = 0.0f;             // of the column tiles so far, eight at a time
#pragma unroll 1
      for (int b = 0; b < CT; b += 8) {
        ulonglong2 w[8];
        const int n = CT - b < 8 ? CT - b : 8;        // even
        const ulonglong2* s0 = src + b * 128;
        poll(w, s0, n > 2 ? s0 + 256 : s0, n > 4 ? s0 + 512 : s0, n > 6 ? s0 + 768 : s0, tag, 5);
        float mb = 0.0f, m2b = 0.0f, qq = 0.0f;
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (j < n) { mb += wc_lo(w[j].x); m2b += wc_lo(w[j].y); }
        mb /= static_cast<float>(n);
#pragma unroll
        for (int j = 0; j < 8; ++j)
          if (j < n) { const float d = wc_lo(w[j].x) - mb; qq = fmaf(d, d, qq); }
        m2b = fmaf(128.0f, qq, m2b);
        const float d = mb - mh, wgt = static_cast<float>(n) / static_cast<float>(b + n);
        mh = fmaf(d, wgt, mh);
        m2 = __fadd_rn(m2, fmaf(__fmul_rn(d, d), wgt * static_cast<float>(b * 128), m2b));
      }
      mean = mh;
      rstd = 1.0f / sqrtf(m2 / static_cast<float>(W) + 1e-6f);
    };
    // LN(h)(1 + scale) + shift of this thread's columns, 8 at a time; the first pieces are on their way
    auto modulate = [&](const float* piece, auto&& sink) {
#pragma unroll 1
      for (int i0 = 0; i0 < CW / 8; i0 += 4) {
        float hv[32];
        tmem_ld32(t_h + i0 * 8, hv);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const float4(&d)[4] = m[i];
          const float sh[8] = {d[0].x, d[0].y, d[0].z, d[0].w, d[1].x, d[1].y, d[1].z, d[1].w};
          const float sc[8] = {d[2].x, d[2].y, d[2].z, d[2].w, d[3].x, d[3].y, d[3].z, d[3].w};
          float o[8];
#pragma unroll
          for (int j = 0; j < 8; ++j) o[j] = fmaf(__fmul_rn(__fsub_rn(hv[i * 8 + j], mean), rstd), sc[j], sh[j]);
          if (i0 + 4 < CW / 8) take(m[i], piece + (i0 + i + 4) * 512);
          sink(i0 + i, o);
        }
      }
    };
    const int act_at = (rb * (W / 8) + tile_n * 16 + hf * (CW / 8)) * 128 + rloc;      // this row's first 8 columns in u and v
    auto put_act = [&](void* buf, int i, const float (&o)[8]) {
      __align__(16) ACT a[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) a[j] = to_act<ACT>(o[j]);
      reinterpret_cast<uint4*>(buf)[act_at + i * 128] = *reinterpret_cast<const uint4*>(a);
    };
    // This column tile's part of the row block's operand is written.  Its readers load it through the async proxy: every writer
    // fences its own stores, all at a time.
    auto publish = [&](int which) {
      asm volatile("fence.proxy.async.global;" ::: "memory");
      slot_sync();
      if (et == 0 && hf == 0) wc_arrive(p.cnt + (rb * 2 + which) * 32);
    };
    auto send_u = [&](const float* piece) { modulate(piece, [&](int i, const float (&o)[8]) { put_act(p.u, i, o); }); publish(0); };
    auto release_acc = [&]() {           // this warp's last read of the accumulators
      tc_fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive_cluster_tmem(mapa_shared(smem_u32(&acc_empty[sl]), 0));
    };
    uint32_t n_acc = 0;
    auto wait_acc = [&]() {
      if (ok && !ch_wait<false>(&acc_full[sl], n_acc & 1, p.err)) { if (lane == 0) ch_fail(p.err, DEV_ERR_EPI_WAIT, 6, static_cast<int>(n_acc)); ok = false; }
      ok = __all_sync(0xffffffffu, ok);
      ++n_acc;
      tc_fence_after_sync();
    };

    // tokens whose state this CTA updates: four coordinates a thread, with guidance the even thread for the conditional row
    const int own = (per + CT - 1) / CT;
    const int rep = p.cfg ? (et & 1) : 0, item = p.cfg ? (et >> 1) : et, cq = item / own, tl = tile_n * own + item % own;
    const bool owns = hf == 0 && cq < kCPad / 4 && tl < per;                       // of a token slot (perhaps beyond the last token)
    const int tok = rb * per + tl;
    const bool live = owns && tok < p.R;
    const bool first = p.t_hi == T;
    const int c0 = 4 * cq;
    float xo[4] = {0.0f, 0.0f, 0.0f, 0.0f}, hl[4] = {0.0f, 0.0f, 0.0f, 0.0f};
    auto state_in = [&](int token, int c) {
      if (token >= p.R || c >= p.C) return 0.0f;
      const size_t o = static_cast<size_t>(token) * p.C + c;
      return first ? p.x_T[o] : p.x[o];
    };
    if (live) {
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        xo[j] = state_in(tok, c0 + j);
        if (first && rep == 0 && c0 + j < p.C && p.traj_x) p.traj_x[static_cast<size_t>(tok) * p.C + c0 + j] = xo[j];
        if (LV && !first) hl[j] = p.hsum[(rb * 128 + tl) * kCPad + c0 + j];
      }
    }
    const bool upd = __any_sync(0xffffffffu, owns);                     // warps with tokens to update

    for (int t = p.t_hi; t >= p.t_lo; --t) {
      const uint32_t step = static_cast<uint32_t>(T - t), tag0 = step * static_cast<uint32_t>(L + 1) + 1;
      // ---- h = Win x + bin
      float xr[kCPad];
      if (t == p.t_hi) {
        const int token = rb * per + tk_row;
#pragma unroll
        for (int c = 0; c < kCPad; ++c) xr[c] = state_in(token, c);
      } else {
        const ulonglong2* src = p.xll + rb * 8 * 128 + tk_row;
        ulonglong2 w[8];
        poll(w, src, src + 256, src + 512, src + 768, step, 7);
#pragma unroll
        for (int j = 0; j < 8; ++j) { xr[2 * j] = wc_lo(w[j].x); xr[2 * j + 1] = wc_lo(w[j].y); }
      }
      {
        // four rows a thread (fragment order), so that a weight read from shared memory serves four: one row a thread would take
        // 512 16-byte reads of 4 cycles each, by each of the SM's warps
        float x4[4][kCPad];
#pragma unroll
        for (int r = 0; r < 4; ++r)
#pragma unroll
          for (int c = 0; c < kCPad; ++c) x4[r][c] = __shfl_sync(0xffffffffu, xr[c], (lane >> 2) + 8 * r);
#pragma unroll 1
        for (int i = 0; i < CW / 16; ++i) {
          float f[2][8];
#pragma unroll
          for (int gb = 0; gb < 4; ++gb) {
            const int col = hf * CW + i * 16 + (gb >> 1) * 8 + 2 * (lane & 3) + (gb & 1);
            const float4* w4 = reinterpret_cast<const float4*>(win_s + col * kCPad);
            const float b = bin_s[col];
            float a[4] = {b, b, b, b};
#pragma unroll
            for (int c4 = 0; c4 < kCPad / 4; ++c4) {
              const float4 w = w4[c4 ^ (lane & 3)];
#pragma unroll
              for (int r = 0; r < 4; ++r) {
                a[r] = fmaf(w.x, x4[r][4 * c4], a[r]); a[r] = fmaf(w.y, x4[r][4 * c4 + 1], a[r]);
                a[r] = fmaf(w.z, x4[r][4 * c4 + 2], a[r]); a[r] = fmaf(w.w, x4[r][4 * c4 + 3], a[r]);
              }
            }
#pragma unroll
            for (int r = 0; r < 4; ++r) f[r >> 1][(gb >> 1) * 4 + (r & 1) * 2 + (gb & 1)] = a[r];
          }
          tmem_st_frag(t_h + i * 16, f[0]);
          tmem_st_frag(t_h + i * 16 + (16u << 16), f[1]);
        }
        tmem_st_wait();
        Partial s;
#pragma unroll 1
        for (int i0 = 0; i0 < CW / 64; ++i0) {
          float hv[4][16];
#pragma unroll
          for (int i = 0; i < 4; ++i) tmem_ld16(t_h + i0 * 64 + i * 16, hv[i]);
          tmem_ld_wait();
#pragma unroll
          for (int i = 0; i < 4; ++i) partial_add(s, i, i0, hv[i]);
        }
        put_stats(s.pm[2], s.p2[2], tag0);
      }
      take_first(ss_at(t, 0));
      norms(tag0);
      send_u(ss_at(t, 0));
#pragma unroll 1
      for (int k = 0; k < L; ++k) {
        // ---- v = SiLU(u W1^T + b1)
        ahead(gate_at(t, k), 16384 / HV);
        ahead(ss_at(t, k + 1), 32768 / HV);
        wait_acc();
#pragma unroll 1
        for (int i = 0; i < CW / 64; ++i) {
          float a[64];
          tmem_ld32(t_acc + i * 64, a);
          tmem_ld32(t_acc + i * 64 + 32, a + 32);
          tmem_ld_wait();
          if (i == CW / 64 - 1) release_acc();
          const float4* b4 = reinterpret_cast<const float4*>(bias_s + (2 * k) * 128 + hf * CW + i * 64);
#pragma unroll
          for (int ii = 0; ii < 8; ++ii) {
            float o[8];
#pragma unroll
            for (int j = 0; j < 2; ++j) {
              const float4 b = b4[2 * ii + j];
              const float* x = a + 8 * ii + 4 * j;
              o[4 * j] = silu_t<true>(x[0] + b.x); o[4 * j + 1] = silu_t<true>(x[1] + b.y);
              o[4 * j + 2] = silu_t<true>(x[2] + b.z); o[4 * j + 3] = silu_t<true>(x[3] + b.w);
            }
            put_act(p.v, i * 8 + ii, o);
          }
        }
        publish(1);
        // ---- h += gate (v W2^T + b2)
        const float* gp = gate_at(t, k);
        take_first(gp);
        wait_acc();
        Partial s;
#pragma unroll
        for (int i = 0; i < CW / 16; ++i) {
          float a[16], hv[16];
          tmem_ld16(t_acc + i * 16, a);
          tmem_ld16(t_h + i * 16, hv);
          tmem_ld_wait();
          if (i == CW / 16 - 1 && k + 1 < L) release_acc();      // (the last block's columns serve the output projection first)
          const float4* b4 = reinterpret_cast<const float4*>(bias_s + (2 * k + 1) * 128 + hf * CW + i * 16);
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            const float4 b = b4[j], g = m[i % kWcAhead][j];
            hv[4 * j] = fmaf(g.x, a[4 * j] + b.x, hv[4 * j]); hv[4 * j + 1] = fmaf(g.y, a[4 * j + 1] + b.y, hv[4 * j + 1]);
            hv[4 * j + 2] = fmaf(g.z, a[4 * j + 2] + b.z, hv[4 * j + 2]); hv[4 * j + 3] = fmaf(g.w, a[4 * j + 3] + b.w, hv[4 * j + 3]);
          }
          if (i + kWcAhead < CW / 16) take(m[i % kWcAhead], gp + (i + kWcAhead) * 512);
          tmem_st16(t_h + i * 16, hv);
          partial_add(s, i & 3, i >> 2, hv);
        }
        put_stats(s.pm[2], s.p2[2], tag0 + k + 1);
        tmem_st_wait();
        take_first(ss_at(t, k + 1));
        norms(tag0 + k + 1);
        if (k + 1 < L) send_u(ss_at(t, k + 1));
      }
      // ---- output projection of (LN(h)(1 + scale_f) + shift_f): this tile's columns' part
      float nz[4] = {0.0f, 0.0f, 0.0f, 0.0f};              // the step's noise, on its way
      if (live && rep == 0)
#pragma unroll
        for (int j = 0; j < 4; ++j)
          if (c0 + j < p.C) nz[j] = __ldg(p.eps + (static_cast<size_t>(t - 1) * p.R + tok) * p.C + c0 + j);
      {
        if (t > p.t_lo) ahead(ss_at(t - 1, 0), 32768 / HV);
        // into the accumulator columns, which the MMAs get back only after it, and back in fragment order: four rows a thread, as above
        modulate(ss_at(t, L), [&](int i, const float (&o)[8]) { tmem_st8(t_acc + i * 8, o); });
        tmem_st_wait();
#pragma unroll 1
        for (int oh = 0; oh < EPW; oh += kCPad) {
          const int row = q * 32 + (lane >> 2) + 8 * (lane & 3);
          float o[kCPad];
          // 64 columns at a time in either form of the kernel, so that both add up in the same order
#pragma unroll 1
          for (int part = 0; part < CW / 64; ++part) {
            float e[4][kCPad];
#pragma unroll
            for (int r = 0; r < 4; ++r)
#pragma unroll
              for (int c = 0; c < kCPad; ++c) e[r][c] = 0.0f;
#pragma unroll 1
            for (int i = 0; i < 4; ++i) {
              float f[2][8];
              tmem_ld_frag(t_acc + part * 64 + i * 16, f[0]);
              tmem_ld_frag(t_acc + part * 64 + i * 16 + (16u << 16), f[1]);
              tmem_ld_wait();
#pragma unroll
              for (int gb = 0; gb < 4; ++gb) {
                const int col = hf * CW + part * 64 + i * 16 + (gb >> 1) * 8 + 2 * (lane & 3) + (gb & 1);
                const float4* w4 = reinterpret_cast<const float4*>(wout_s + col * EPW + oh);
#pragma unroll
                for (int c4 = 0; c4 < kCPad / 4; ++c4) {
                  const float4 w = w4[c4 ^ (lane & 3)];
#pragma unroll
                  for (int r = 0; r < 4; ++r) {
                    const float v = f[r >> 1][(gb >> 1) * 4 + (r & 1) * 2 + (gb & 1)];
                    e[r][4 * c4] = fmaf(v, w.x, e[r][4 * c4]); e[r][4 * c4 + 1] = fmaf(v, w.y, e[r][4 * c4 + 1]);
                    e[r][4 * c4 + 2] = fmaf(v, w.z, e[r][4 * c4 + 2]); e[r][4 * c4 + 3] = fmaf(v, w.w, e[r][4 * c4 + 3]);
                  }
                }
              }
            }
            // sum over the four lanes that share the rows; lane i ends with row i / 4 + 8 (i % 4)
            const bool up2 = (lane & 2) != 0, up1 = (lane & 1) != 0;
#pragma unroll
            for (int c = 0; c < kCPad; ++c) {
              const float s0 = up2 ? e[0][c] : e[2][c], s1 = up2 ? e[1][c] : e[3][c];
              const float k0 = (up2 ? e[2][c] : e[0][c]) + __shfl_xor_sync(0xffffffffu, s0, 2);
              const float k1 = (up2 ? e[3][c] : e[1][c]) + __shfl_xor_sync(0xffffffffu, s1, 2);
              const float v = (up1 ? k1 : k0) + __shfl_xor_sync(0xffffffffu, up1 ? k0 : k1, 1);
              o[c] = part == 0 ? v : o[c] + v;
            }
          }
          if constexpr (HV == 2) {         // the halves' sums: 16 floats a row, 2 KB apart so that the lanes' words lie side by side
            float4* x = reinterpret_cast<float4*>(eh_s) + (oh / kCPad) * 512 + row;
            if (hf == 1) {
#pragma unroll
              for (int c4 = 0; c4 < 4; ++c4) x[c4 * 128] = make_float4(o[4 * c4], o[4 * c4 + 1], o[4 * c4 + 2], o[4 * c4 + 3]);
            }
            hand_over();
            if (hf == 0) {
#pragma unroll
              for (int c4 = 0; c4 < 4; ++c4) { const float4 v = x[c4 * 128]; o[4 * c4] += v.x; o[4 * c4 + 1] += v.y; o[4 * c4 + 2] += v.z; o[4 * c4 + 3] += v.w; }
            }
          }
          if (hf == 0) {
            ulonglong2* dst = p.epart + ((rb * CT + tile_n) * NC + oh / 2) * 128 + row;
#pragma unroll
            for (int c = 0; c < kCPad; c += 2) wc_put(dst + (c / 2) * 128, o[c], o[c + 1], step + 1);
          }
        }
        release_acc();
      }
      // ---- guidance and Eq. 3 for this CTA's tokens; the new state to every column tile
      if (upd) {
        const int ti = t - p.t_lo;
        float ee[4] = {0.0f, 0.0f, 0.0f, 0.0f}, wv[4] = {0.0f, 0.0f, 0.0f, 0.0f};
        if (live)
#pragma unroll
          for (int j = 0; j < 4; ++j)
            if (c0 + j < p.C) {
              ee[j] = p.bout[c0 + j];
              if (LV) wv[j] = p.bout[kCPad + c0 + j];
            }
        auto gather = [&](int col, float (&acc)[4]) {      // sum over the column tiles, in order, then the bias
          const ulonglong2* src = p.epart + (rb * CT * NC + col) * 128 + rep * 64 + (owns ? tl : 0);
          float s[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll 1
          for (int g = 0; g < CT; g += 4) {
            ulonglong2 w[8];
            const int n = CT - g < 4 ? CT - g : 4;
            const ulonglong2* s0 = src + g * NC * 128;
            poll(w, s0, s0 + NC * 128, n > 2 ? s0 + 2 * NC * 128 : s0, n > 2 ? s0 + 3 * NC * 128 : s0, step + 1, 8);
#pragma unroll
            for (int j = 0; j < 4; ++j)
              if (j < n) { s[0] += wc_lo(w[2 * j].x); s[1] += wc_lo(w[2 * j].y); s[2] += wc_lo(w[2 * j + 1].x); s[3] += wc_lo(w[2 * j + 1].y); }
          }
#pragma unroll
          for (int j = 0; j < 4; ++j) acc[j] = s[j] + acc[j];
        };
        gather(owns ? 2 * cq : 0, ee);
        if constexpr (LV) gather(kCPad / 2 + (owns ? 2 * cq : 0), wv);
        float xn[4] = {0.0f, 0.0f, 0.0f, 0.0f};
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float other = __shfl_xor_sync(0xffffffffu, ee[j], 1);
          if (!live || rep != 0 || c0 + j >= p.C) continue;
          const float eh = p.cfg ? cfg_combine(ee[j], other, p.cfg_scale) : ee[j];
          const size_t o = static_cast<size_t>(tok) * p.C + c0 + j;
          const float mu = ddpm_mean(p.ca[ti], xo[j], p.cb[ti], eh);
          float sigma = p.s0[ti], lv = 0.0f;
          if (LV) { lv = lv_interp(wv[j], p.s0[ti], p.s1[ti]); sigma = expf(0.5f * lv); }
          xn[j] = ddpm_sample(mu, sigma, nz[j]);
          if (!(fabsf(xn[j]) <= 3.0e38f)) *p.status = 1;
          if (t == 1) {
            p.mu1[o] = mu;
            if (p.x1) p.x1[o] = xo[j];
            if (p.sample_last && p.x0) p.x0[o] = xn[j];
            if (LV) p.lv1[o] = lv;
          } else {
            if (LV) hl[j] += 0.5f * lv;
            if (t == p.t_lo) p.x[o] = xn[j];                      // the next launch starts from it
            if (p.traj_x) {
              const size_t slot = static_cast<size_t>(p.R) * p.C;
              p.traj_x[static_cast<size_t>(T - t + 1) * slot + o] = xn[j];
              p.traj_mu[static_cast<size_t>(T - t) * slot + o] = mu;
            }
          }
          xo[j] = xn[j];
        }
        if (owns && rep == 0 && t > p.t_lo) {
          ulonglong2* dst = p.xll + (rb * 8 + 2 * cq) * 128 + tl;
          wc_put(dst, xn[0], xn[1], step + 1);
          wc_put(dst + 128, xn[2], xn[3], step + 1);
        }
      }
    }
    if constexpr (LV) {
      // half log-determinants: kept per coordinate between launches, summed over them at the end
      if (live && rep == 0)
#pragma unroll
        for (int j = 0; j < 4; ++j) p.hsum[(rb * 128 + tl) * kCPad + c0 + j] = c0 + j < p.C ? hl[j] : 0.0f;
      slot_sync();
      if (p.t_lo == 1 && live && rep == 0 && cq == 0) {
        float s = 0.0f;
        for (int c = 0; c < p.C; ++c) s += __ldcg(p.hsum + (rb * 128 + tl) * kCPad + c);
        p.half_logdet[tok] = s;
      }
    }
  }
  tc_fence_before_sync();
  __syncthreads();
  gc_settle(p.err);
  cluster_arrive(); cluster_wait();   // neither CTA leaves while the pair's MMAs or signals may touch it
  if (warp == kWcMmaWarp) tmem_dealloc_pair(tmem_base, 512);
}

// Self-test of the bounded waits: one thread polls words that nobody writes, then waits on a barrier on which nobody arrives, so both waits
// run into the limit (csd_set_wait_limit) and give up.  Recorded in the context's error word: role 4, site 1 (2: the poll
// succeeded), and as the iteration the cycles that the poll took, in per cent of the limit.  Nothing else happens: no
// fault, no trap, no wait beyond the limit.
__device__ ulonglong2 g_selftest_words[256];
__global__ void wait_timeout_selftest_kernel(int* err) {
  __shared__ uint64_t bar;
  if (threadIdx.x == 0) { mbar_init(&bar, 1); fence_mbar_init(); }
  __syncthreads();
  if (threadIdx.x != 0) return;
  ulonglong2 w[8];
  const ulonglong2* const a = g_selftest_words;
  const long long t0 = clock64();
  const bool got = wc_poll(w, a, a, a, a, 1, err);
  const long long percent = (clock64() - t0) * 100 / *reinterpret_cast<volatile long long*>(&g_wait_limit_cycles);
  if (!ch_wait<false>(&bar, 0, err)) ch_fail(err, 4, got ? 2 : 1, static_cast<int>(percent < 0xffff ? percent : 0xffff));
}

}  // namespace csd
