// C ABI of the continuous speculative decoding hot path (see include/csd.h for the contract).
// Host side: argument checks, weight packing, workspace, launch sequencing.  Every arithmetic step
// runs in the kernels of gemm.cuh / rowops.cuh.
#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <cstdarg>
#include <cstdio>
#include <cstdlib>
#include <cstring>
#include <new>
#include <type_traits>
#include <vector>

#include "../../include/csd.h"
#include "fold.cuh"
#include "gemm.cuh"
#include "gmm.cuh"
#include "rowops.cuh"
#include "groupchain.cuh"
#include "widechain.cuh"
#include "f32chain.cuh"

using namespace csd;

namespace {

typedef CUresult (*EncodeTiledFn)(CUtensorMap*, CUtensorMapDataType, cuuint32_t, void*, const cuuint64_t*,
                                  const cuuint64_t*, const cuuint32_t*, const cuuint32_t*,
                                  CUtensorMapInterleave, CUtensorMapSwizzle, CUtensorMapL2promotion,
                                  CUtensorMapFloatOOBfill);

struct ChainWs {
  void* base = nullptr;
  size_t cap = 0;
  // carved per call
  void *zc, *s, *u, *v;
  float *cz, *te, *h, *stats, *epart, *x;
  void* s2 = nullptr;   // s of even steps (s of odd steps: s)
  void* ap = nullptr;   // a' = h (1 + scale) of the folded blocks
  float* hid = nullptr; // hidden layer of the timestep embedding [T, W]
  bool owned = true;    // false: base is memory the library did not allocate and must never free or grow
  bool in_graph = false;
};

constexpr int kMaxDevices = 64;   // device ordinals the per-device tables below cover

struct ProfRec { cudaEvent_t a, b; int cls; double flops; };

struct HostIo {  // a device buffer that grows on demand
  void* base = nullptr;
  size_t cap = 0;
  bool in_graph = false;   // a captured call used it: its graph holds the address
};

}  // namespace

struct csd_ctx {
  int device = 0;
  int num_sms = 148;
  cudaStream_t stream = nullptr;
  cudaStream_t side[2] = {nullptr, nullptr};
  cudaEvent_t ev_fork = nullptr, ev_done[2] = {nullptr, nullptr};
  int* d_err = nullptr;
  unsigned long long* tally() const { return reinterpret_cast<unsigned long long*>(d_err + 2); }   // tally_cap_hits
  int64_t launches = 0;
  int chain_mode = CSD_CHAIN_LAYERS;   // csd_set_chain_mode
  EncodeTiledFn encode = nullptr;
  ChainWs ws[3];   // draft chain, target chain, static-scratch calls
  std::vector<void*> in_graphs;   // replaced buffers whose addresses graphs hold: freed with the context
  HostIo io;       // device mirrors for csd_round_host
  HostIo un;       // csd_verify_unaligned: per-row noise terms
  HostIo bn;       // csd_bonus_token: samples of every sequence before the selection
  HostIo sp;       // csd_verify_single_path: schedule constants, mu^p of one pass, running log-ratio
  HostIo gc[2];    // group chain kernel (per chain slot): s of all steps
  HostIo gm[2];    // group and wide chain kernels: condition products of two chunks of steps (wide: s of a chunk before them)
  HostIo wx[2];    // wide chain kernel: what its column tiles exchange
  size_t gc_refused[2] = {SIZE_MAX, SIZE_MAX}, gm_refused[2] = {SIZE_MAX, SIZE_MAX}, wc_refused[2] = {SIZE_MAX, SIZE_MAX};   // sizes that could not be had (wc: gm and wx of a wide chain): asked for again where the device has as much free
  cudaStream_t aux[2] = {nullptr, nullptr};        // (per chain slot) where they are formed
  cudaEvent_t ev_prep[2] = {}, ev_mods[2][2] = {}, ev_read[2][2] = {};   // preparation done; a chunk is written / has been read
  cudaEvent_t ev_on[2] = {};                       // every block of a chunk's chain kernel has its SM
  char err[512] = {0};
  // optional per-launch timing (csd_profile)
  bool prof_on = false;
  std::vector<ProfRec> prof;
  std::vector<cudaEvent_t> ev_pool;
  size_t ev_used = 0;
};

struct csd_head {
  csd_ctx* ctx = nullptr;
  csd_head_desc d{};
  void* wblob = nullptr;   // GEMM weights (bf16 or fp32)
  float* fblob = nullptr;  // fp32 side parameters
  size_t esz = 4;
  // GEMM weights
  void* Wz = nullptr;
  std::vector<void*> Wss, Wg, W1, W2;
  void* Wfss = nullptr;
  // fp32 parameters
  float *bz, *Wt1, *bt1, *Wt2, *bt2, *win, *bin, *bfsh, *bfsc, *wout_t, *bout;
  std::vector<float*> bsh, bsc, bg, b1, b2;
  // tensor maps of the weights (16-bit heads), one set per output-tile width: [0] 64, [1] 128 columns
  struct TmSet {
    CUtensorMap Wz{}, Wfss{};
    std::vector<CUtensorMap> Wss, Wg, W1, W2;
  } tm[2];
  std::vector<CUtensorMap> W1_wide;
  // folded blocks (fold.cuh): packed [Wg_k | Wscale_{k+1}] (k < L-1) and [W1_k Wscale_k | W1_k Wshift_k] (k >= 1),
  // 256-row boxes; c1_k = W1_k (1 + bscale_k), c2_k = W1_k bshift_k + b1_k
  void* xblob = nullptr;
  std::vector<CUtensorMap> Wgs, Wf;
  std::vector<CUtensorMap> Wgs_half, Wf_half;   // the same matrices in 128-row boxes: what one CTA of a pair loads
  std::vector<float*> c1, c2;   // first MLP layer with 256-row boxes (W a multiple of 256)
  // group chain kernel (groupchain.cuh): the dependent layers' maps W1_k, W2_k (device table, boxes of 128 rows); the matrices
  // multiplied by s where they lie (all blocks' rows Wss_0 .. Wfss; xblob), and which tiles of 256 of their rows each form takes
  bool gc_ready = false;
  CUtensorMap* d_gc_maps = nullptr;
  CUtensorMap Wrows{}, Wx{};
  int* d_gc_rows = nullptr;     // plain form, then folded form: first rows (~row: of xblob)
  // wide chain kernel (widechain.cuh): W1_k, W2_k in boxes of 64 rows; per tile of 256 weight rows its first row and its biases
  CUtensorMap* d_wc_maps = nullptr;
  int* d_wc_rows = nullptr;
  float* d_wc_bias = nullptr;
};

namespace {

int fail(csd_ctx* ctx, int code, const char* fmt, ...) {
  if (ctx) {
    va_list ap;
    va_start(ap, fmt);
    vsnprintf(ctx->err, sizeof(ctx->err), fmt, ap);
    va_end(ap);
  }
  return code;
}

#define CSD_CUDA(ctx, call)                                                                          \
  do {                                                                                               \
    cudaError_t e_ = (call);                                                                         \
    if (e_ != cudaSuccess)                                                                           \
      return fail(ctx, CSD_ERR_CUDA, "%s failed: %s (%s:%d)", #call, cudaGetErrorString(e_), __FILE__, \
                  __LINE__);                                                                         \
  } while (0)

// Makes the context's device current for the duration of a call and puts the caller's device back afterwards.
struct DeviceGuard {
  int prev = -1;
  bool ok = true;
  explicit DeviceGuard(int dev) {
    if (cudaGetDevice(&prev) != cudaSuccess) { prev = -1; cudaGetLastError(); }
    if (prev != dev) ok = cudaSetDevice(dev) == cudaSuccess;
  }
  ~DeviceGuard() {
    int cur = -1;
    if (prev >= 0 && cudaGetDevice(&cur) == cudaSuccess && cur != prev) cudaSetDevice(prev);
  }
  DeviceGuard(const DeviceGuard&) = delete;
  DeviceGuard& operator=(const DeviceGuard&) = delete;
};
#define CSD_DEVICE(ctx)                                                                              \
  DeviceGuard device_guard_((ctx)->device);                                                          \
  if (!device_guard_.ok) return fail(ctx, CSD_ERR_CUDA, "cannot make device %d current", (ctx)->device)

cudaEvent_t prof_event(csd_ctx* ctx) {
  if (ctx->ev_used == ctx->ev_pool.size()) {
    cudaEvent_t e = nullptr;
    if (cudaEventCreate(&e) != cudaSuccess) return nullptr;
    ctx->ev_pool.push_back(e);
  }
  return ctx->ev_pool[ctx->ev_used++];
}
// Brackets one launch with events on its own stream when profiling is on.
struct ProfScope {
  csd_ctx* ctx; cudaStream_t st; cudaEvent_t a = nullptr, b = nullptr; int cls; double flops;
  ProfScope(csd_ctx* c, cudaStream_t s, int cls_, double fl) : ctx(c), st(s), cls(cls_), flops(fl) {
    if (ctx->prof_on && (a = prof_event(ctx)) && (b = prof_event(ctx))) cudaEventRecord(a, st);
  }
  ~ProfScope() {
    if (a && b) { cudaEventRecord(b, st); ctx->prof.push_back({a, b, cls, flops}); }
  }
};

inline size_t align_up(size_t v, size_t a) { return (v + a - 1) / a * a; }

uint16_t f32_to_bf16_bits(float f) {
  uint32_t u;
  memcpy(&u, &f, 4);
  if ((u & 0x7fffffffu) > 0x7f800000u) return static_cast<uint16_t>((u >> 16) | 0x40);  // NaN
  const uint32_t bias = ((u >> 16) & 1u) + 0x7fffu;
  return static_cast<uint16_t>((u + bias) >> 16);
}

int make_tmap(csd_ctx* ctx, CUtensorMap* m, int dtype, const void* ptr, uint64_t rows, uint64_t cols, uint64_t ld,
              uint32_t box_rows) {
  const cuuint64_t gdim[2] = {cols, rows};
  const cuuint64_t gstride[1] = {ld * 2};
  const cuuint32_t box[2] = {static_cast<cuuint32_t>(kBlockK), box_rows};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = ctx->encode(m, dtype == CSD_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), gdim, gstride, box,
                                 estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B,
                                 CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(ctx, CSD_ERR_CUDA, "cuTensorMapEncodeTiled failed with code %d", (int)r);
  return CSD_OK;
}

// [lines, 256] elements as they lie, in boxes of 32 lines (16 KB).
int make_plain_tmap(csd_ctx* ctx, CUtensorMap* m, int dtype, const void* ptr, uint64_t lines) {
  const cuuint64_t gdim[2] = {256, lines};
  const cuuint64_t gstride[1] = {512};
  const cuuint32_t box[2] = {256, 32};
  const cuuint32_t estr[2] = {1, 1};
  const CUresult r = ctx->encode(m, dtype == CSD_F16 ? CU_TENSOR_MAP_DATA_TYPE_FLOAT16 : CU_TENSOR_MAP_DATA_TYPE_BFLOAT16, 2, const_cast<void*>(ptr), gdim, gstride, box,
                                 estr, CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_NONE, CU_TENSOR_MAP_L2_PROMOTION_L2_256B, CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE);
  if (r != CUDA_SUCCESS) return fail(ctx, CSD_ERR_CUDA, "cuTensorMapEncodeTiled failed with code %d", (int)r);
  return CSD_OK;
}

// Byte offsets of a chain's intermediates inside its workspace (each piece rounded up to 1 KiB) and their total.
// The one place that knows the layout: the growable workspaces and the fixed static scratch both use it.
struct WsLayout {
  size_t zc, s, u, v, cz, te, h, stats, epart, x, ap, hid, s2, total;
};

WsLayout ws_layout(const csd_head_desc& d, int Rh, int R, int T) {
  const size_t asz = d.dtype == CSD_F32 ? 4 : 2;
  const size_t W = d.W, rh = static_cast<size_t>(Rh);
  size_t off = 0;
  auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 1024); return o; };
  WsLayout l{};
  l.zc = take(rh * d.Dz * asz);
  l.s = take(rh * W * asz); l.u = take(rh * W * asz); l.v = take(rh * W * asz);
  l.cz = take(rh * W * 4); l.te = take(static_cast<size_t>(T) * W * 4); l.h = take(rh * W * 4);
  l.stats = take(rh * (W / kStatCols) * 8);
  l.epart = take(rh * (W / kStatCols) * (d.var_out ? kCPad2 : kCPad) * 4);   // room for 64-wide tiles
  l.x = take(static_cast<size_t>(R) * kCPad * 4);
  l.ap = take(d.dtype == CSD_F32 ? 0 : rh * W * asz);
  l.hid = take(static_cast<size_t>(T) * W * 4);
  l.s2 = take(rh * W * asz);
  l.total = off;
  return l;
}

bool capturing(const csd_ctx* ctx) {
  cudaStreamCaptureStatus s = cudaStreamCaptureStatusNone;
  if (cudaStreamIsCapturing(ctx->stream, &s) != cudaSuccess) { cudaGetLastError(); return false; }
  return s != cudaStreamCaptureStatusNone;
}

// Gives a buffer up, once nothing in flight uses it; what a graph may still use on its next launch stays until csd_destroy.
template <typename Buf>
int give_up(csd_ctx* ctx, Buf& b) {
  void* const base = b.base;
  const bool keep = b.in_graph;
  b.base = nullptr; b.cap = 0; b.in_graph = false;
  if (base && keep) ctx->in_graphs.push_back(base);
  else if (base) CSD_CUDA(ctx, cudaFree(base));
  return CSD_OK;
}

int sync_streams(csd_ctx* ctx) {
  CSD_CUDA(ctx, cudaStreamSynchronize(ctx->stream));
  for (int i = 0; i < 2; ++i) { CSD_CUDA(ctx, cudaStreamSynchronize(ctx->side[i])); CSD_CUDA(ctx, cudaStreamSynchronize(ctx->aux[i])); }
  return CSD_OK;
}

// At least need bytes in b for the call that is being made.
template <typename Buf>
int ensure_buffer(csd_ctx* ctx, Buf& b, size_t need, const char* what) {
  if (need > b.cap) {
    if (int rc = sync_streams(ctx)) return rc;
    if (int rc = give_up(ctx, b)) return rc;
    if (cudaMalloc(&b.base, need) != cudaSuccess) {
      cudaGetLastError();
      b.base = nullptr;
      return fail(ctx, CSD_ERR_WORKSPACE, "cannot allocate %zu bytes for %s", need, what);
    }
    b.cap = need;
  }
  b.in_graph = b.in_graph || capturing(ctx);
  return CSD_OK;
}

// Whether the device has need bytes free, counting `back` that would be given up first, and a little more.
bool room_for(size_t need, size_t back) {
  size_t free = 0, total = 0;
  if (cudaMemGetInfo(&free, &total) != cudaSuccess) { cudaGetLastError(); return false; }
  return free + back >= need + (size_t(32) << 20);
}

int ensure_ws(csd_ctx* ctx, ChainWs& ws, const csd_head_desc& d, int Rh, int R, int T) {
  const WsLayout l = ws_layout(d, Rh, R, T);
  if (l.total > ws.cap && !ws.owned) return fail(ctx, CSD_ERR_WORKSPACE, "the fixed scratch holds %zu bytes, this call needs %zu", ws.cap, l.total);
  if (int rc = ensure_buffer(ctx, ws, l.total, "the workspace")) return rc;
  char* b = static_cast<char*>(ws.base);
  ws.zc = b + l.zc; ws.s = b + l.s; ws.u = b + l.u; ws.v = b + l.v;
  ws.cz = reinterpret_cast<float*>(b + l.cz); ws.te = reinterpret_cast<float*>(b + l.te);
  ws.h = reinterpret_cast<float*>(b + l.h); ws.stats = reinterpret_cast<float*>(b + l.stats);
  ws.epart = reinterpret_cast<float*>(b + l.epart); ws.x = reinterpret_cast<float*>(b + l.x);
  ws.ap = b + l.ap; ws.hid = reinterpret_cast<float*>(b + l.hid);
  ws.s2 = b + l.s2;
  return CSD_OK;
}

template <int EPI, int NSEG, int NMUL, int TN, typename ACT, bool PAIR>
int launch_tc_t(csd_ctx* ctx, cudaStream_t st, const CUtensorMap& a0, const CUtensorMap& b0, const CUtensorMap& a1,
                const CUtensorMap& b1, int K0, int K1, int dep_k, int N, const EpiParams& ep,
                const CUtensorMap* tout = nullptr) {
  constexpr int MMA_N = NMUL * TN;
  auto kern = gemm_tc_kernel<EPI, ACT, NSEG, MMA_N, TN, std::is_same<ACT, __half>::value ? 0 : 1, PAIR>;
  static bool attr_done[kMaxDevices] = {};   // function attributes are per device
  constexpr int smem = TcCfg<EPI, MMA_N, TN, PAIR>::kSmemBytes;
  if (!attr_done[ctx->device]) {
    CSD_CUDA(ctx, cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, smem));
    attr_done[ctx->device] = true;
  }
  // Work units: output tiles, or pair tiles (two row tiles) for CTA pairs.  Persistent: at most one CTA per SM.
  const int tiles_n = N / TN, row_tiles = (ep.M + kTileM - 1) / kTileM;
  const int units = tiles_n * (PAIR ? (row_tiles + 1) / 2 : row_tiles);
  const int max_units = PAIR ? ctx->num_sms / 2 : ctx->num_sms;
  dim3 grid((units < max_units ? units : max_units) * (PAIR ? 2 : 1));
  ProfScope ps(ctx, st, EPI == EPI_MODF2 ? EPI_MODF : EPI, 2.0 * ep.M * static_cast<double>(N) * (K0 + K1) * NMUL);
  cudaLaunchConfig_t cfg{};
  cfg.gridDim = grid; cfg.blockDim = dim3(TcWarps<EPI, TN>::kThreads); cfg.dynamicSmemBytes = smem; cfg.stream = st;
  cudaLaunchAttribute at[2];
  int na = 0;
  if (PAIR) {
    at[na].id = cudaLaunchAttributeClusterDimension;
    at[na].val.clusterDim.x = 2; at[na].val.clusterDim.y = 1; at[na].val.clusterDim.z = 1;
    ++na;
  }
  if (!ctx->prof_on) {   // event pairs between launches defeat the overlap anyway
    at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[na].val.programmaticStreamSerializationAllowed = 1;
    ++na;
  }
  cfg.attrs = at; cfg.numAttrs = na;
  EpiParams e = ep;
  e.nt = N / kStatCols;   // eps partials are per 64-column group for both tile widths
  CSD_CUDA(ctx, cudaLaunchKernelEx(&cfg, kern, a0, b0, a1, b1, tout ? *tout : a0, K0 / kBlockK, K1 / kBlockK, dep_k / kBlockK, tiles_n, units, e,
                                   ctx->d_err));
  ctx->launches++;
  return CSD_OK;
}

// NMUL = 2: B holds the interleaved AdaLN shift | scale rows (two accumulator columns per output column).
// tn: output columns per CTA, 64 or 128; pair: two CTAs share each MMA (needs tn = 128; the B tensor maps
// b0 / b1 then have half-height boxes).  dep_k: first K index (over both segments) whose A operand is
// written by the preceding kernel.
template <int EPI, int NSEG, int NMUL>
int launch_tc(csd_ctx* ctx, int dtype, int tn, bool pair, cudaStream_t st, const CUtensorMap& a0, const CUtensorMap& b0,
              const CUtensorMap& a1, const CUtensorMap& b1, int K0, int K1, int dep_k,
              int N, const EpiParams& ep, const CUtensorMap* tout = nullptr) {
  if (dtype == CSD_F16) {
    if (tn == 64) return launch_tc_t<EPI, NSEG, NMUL, 64, __half, false>(ctx, st, a0, b0, a1, b1, K0, K1, dep_k, N, ep, tout);
    if (pair) return launch_tc_t<EPI, NSEG, NMUL, 128, __half, true>(ctx, st, a0, b0, a1, b1, K0, K1, dep_k, N, ep, tout);
    return launch_tc_t<EPI, NSEG, NMUL, 128, __half, false>(ctx, st, a0, b0, a1, b1, K0, K1, dep_k, N, ep, tout);
  }
  if (tn == 64) return launch_tc_t<EPI, NSEG, NMUL, 64, __nv_bfloat16, false>(ctx, st, a0, b0, a1, b1, K0, K1, dep_k, N, ep, tout);
  if (pair) return launch_tc_t<EPI, NSEG, NMUL, 128, __nv_bfloat16, true>(ctx, st, a0, b0, a1, b1, K0, K1, dep_k, N, ep, tout);
  return launch_tc_t<EPI, NSEG, NMUL, 128, __nv_bfloat16, false>(ctx, st, a0, b0, a1, b1, K0, K1, dep_k, N, ep, tout);
}

template <int EPI, int NSEG, int MMA_N>
int launch_simt(csd_ctx* ctx, cudaStream_t st, const float* A0, int lda0, const float* B0, int K0, const float* A1,
                int lda1, const float* B1, int K1, int N, const EpiParams& ep) {
  dim3 grid(N / kTileN, (ep.M + kSimtRows - 1) / kSimtRows);
  ProfScope ps(ctx, st, EPI == EPI_MODF2 ? EPI_MODF : EPI, 2.0 * ep.M * static_cast<double>(N) * (K0 + K1) * ((NSEG == 1 && MMA_N == 256) ? 2.0 : 1.0));
  EpiParams e = ep;
  e.nt = N / kTileN;
  gemm_simt_kernel<EPI, NSEG, MMA_N><<<grid, 128, 0, st>>>(A0, lda0, B0, K0, K0, A1, lda1, B1, K1, K1, e);
  ctx->launches++;
  CSD_CUDA(ctx, cudaGetLastError());
  return CSD_OK;
}

// Launches of the short kernels: the next one's blocks are set up while the preceding kernel still runs (each waits for it
// before it touches memory), which takes about a microsecond off every kernel boundary.
template <typename... KArgs, typename... Args>
int launch_short(csd_ctx* ctx, cudaStream_t st, void (*kern)(KArgs...), dim3 grid, unsigned block, size_t smem, const Args&... args) {
  cudaLaunchConfig_t lc{};
  lc.gridDim = grid; lc.blockDim = dim3(block); lc.dynamicSmemBytes = smem; lc.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  lc.attrs = at; lc.numAttrs = 1;
  CSD_CUDA(ctx, cudaLaunchKernelEx(&lc, kern, static_cast<KArgs>(args)...));
  ctx->launches++;
  return CSD_OK;
}

int check_sched(csd_ctx* ctx, const csd_schedule* s, bool full) {
  if (!s) return fail(ctx, CSD_ERR_INVALID_ARG, "schedule is null");
  if (s->T < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "schedule T = %d must be >= 1", s->T);
  if (!s->sigma) return fail(ctx, CSD_ERR_INVALID_ARG, "schedule sigma is null");
  if (full && (!s->a || !s->b || !s->tfeat)) return fail(ctx, CSD_ERR_INVALID_ARG, "schedule a/b/tfeat is null");
  for (int t = 0; t < s->T; ++t)
    if (!(s->sigma[t] > 0.0f)) return fail(ctx, CSD_ERR_INVALID_ARG, "schedule sigma[%d] must be > 0", t);
  return CSD_OK;
}

// Folded blocks run as CTA pairs when a layer's row tiles pair up.
#ifndef CSD_FOLD_PAIRS
#define CSD_FOLD_PAIRS 1
#endif
constexpr bool kFoldPairs = CSD_FOLD_PAIRS != 0;

// fp32 heads: the persistent chain kernel for groups of G rows (f32chain.cuh).  False where its shared memory does not fit.
template <int G>
bool fc_ready(const csd_ctx* ctx, const csd_head_desc& d) {
  static int known[kMaxDevices] = {};
  int& k = known[ctx->device];
  if (k == 0) {
    k = cudaFuncSetAttribute(f32_chain_kernel<G, 2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) == cudaSuccess &&
        cudaFuncSetAttribute(f32_chain_kernel<G, 4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) == cudaSuccess ? 1 : -1;
    cudaGetLastError();
  }
  return k == 1 && fc_layout(G, d.W, d.var_out ? kCPad2 : kCPad).total * 4 <= 227 * 1024;
}

// Whether the chain kernel is the faster one for Rh head rows.  Its clusters take turns, about 15 at a time, and every group reads
// all the weights for its 16, 8 or 4 rows (W up to 896, 1664, 3072); the layer kernels' 32 x 128 tiles share them among 32 and cost
// the less per tile the more tiles there are.  ms a step of one block, chain / layer kernels, by head rows (tiles):
//   W =  512: 2048 (256) 0.61 / 0.63, 4096 (512) 1.20 / 1.26, 8192 (1024) 2.34 / 2.12
//   W =  768: 1024 (192) 0.62 / 0.91, 2048 (384) 1.11 / 1.07, 4096 (768) 2.20 / 2.17, 8192 (1536) 4.27 / 3.95
//   W = 1024: 1024 (256) 0.99 / 1.20, 2048 (512) 1.96 / 2.41, 4096 (1024) 3.80 / 3.91, 8192 (2048) 7.51 / 6.57
//   W = 1280: 1024 (320) 1.50 / 1.86, 2048 (640) 2.99 / 3.33, 4096 (1280) 5.82 / 5.09
//   W = 1536:  512 (192) 1.31 / 2.06, 1024 (384) 2.33 / 2.30, 2048 (768) 4.64 / 4.19
//   W = 2048:  256 (128) 1.41 / 2.81,  512 (256) 2.53 / 2.87, 1024 (512) 5.06 / 4.59
//   W = 3072:  256 (192) 2.99 / 4.20,  512 (384) 5.33 / 4.49
// The line: 640 tiles, 256 where a group has four rows only.
bool fc_pays(const csd_ctx* ctx, const csd_head_desc& d, int Rh) {
  return (Rh + 31) / 32 * (d.W / 128) <= (fc_ready<8>(ctx, d) ? 640 : 256);
}

// Rows per group: the fewest that keep all groups of the chains side by side resident at once (a cluster of 8 SMs each,
// about one cluster per GPC stays unused), where a step costs the least time; with more groups than that, the most rows
// that fit, because every group reads all the weights.  0: none fits (W beyond about 4000).  The choice changes no bit.
int fc_rows(const csd_ctx* ctx, const csd_head_desc& d, int R, int cfg, int chains) {
  const int clusters = ctx->num_sms / kFcCluster - 2;
  auto few = [&](int g) { const int per = g / (cfg ? 2 : 1); return (R + per - 1) / per * chains <= clusters; };
  const bool ok4 = fc_ready<4>(ctx, d), ok8 = fc_ready<8>(ctx, d), ok16 = fc_ready<16>(ctx, d);
  if (ok4 && few(4)) return 4;
  if (ok8 && few(8)) return 8;
  return ok16 ? 16 : ok8 ? 8 : ok4 ? 4 : 0;
}

// Shared-memory opt-in of the folded block kernels, once per device and operand type.
bool fold_kernels_ready(const csd_ctx* ctx, const csd_head_desc& d) {
  static int known[kMaxDevices][2] = {};
  int& k = known[ctx->device][d.dtype == CSD_F16 ? 0 : 1];
  if (k == 0) {
    bool ok = true;
    if (d.dtype == CSD_F16) {
      ok = ok && cudaFuncSetAttribute(fold_kernel<__half, 0, FOLD_W1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, FoldCfg<FOLD_W1>::kSmemBytes) == cudaSuccess;
      ok = ok && cudaFuncSetAttribute(fold_kernel<__half, 0, FOLD_GATE, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, FoldCfg<FOLD_GATE>::kSmemBytes) == cudaSuccess;
      ok = ok && cudaFuncSetAttribute(fold_kernel<__half, 0, FOLD_W1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, FoldCfg<FOLD_W1>::kSmemBytes) == cudaSuccess;
      ok = ok && cudaFuncSetAttribute(fold_kernel<__half, 0, FOLD_GATE, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, FoldCfg<FOLD_GATE>::kSmemBytes) == cudaSuccess;
    } else {
      ok = ok && cudaFuncSetAttribute(fold_kernel<__nv_bfloat16, 1, FOLD_W1, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, FoldCfg<FOLD_W1>::kSmemBytes) == cudaSuccess;
      ok = ok && cudaFuncSetAttribute(fold_kernel<__nv_bfloat16, 1, FOLD_GATE, false>, cudaFuncAttributeMaxDynamicSharedMemorySize, FoldCfg<FOLD_GATE>::kSmemBytes) == cudaSuccess;
      ok = ok && cudaFuncSetAttribute(fold_kernel<__nv_bfloat16, 1, FOLD_W1, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, FoldCfg<FOLD_W1>::kSmemBytes) == cudaSuccess;
      ok = ok && cudaFuncSetAttribute(fold_kernel<__nv_bfloat16, 1, FOLD_GATE, true>, cudaFuncAttributeMaxDynamicSharedMemorySize, FoldCfg<FOLD_GATE>::kSmemBytes) == cudaSuccess;
    }
    cudaGetLastError();
    k = ok ? 1 : -1;
  }
  return k == 1;
}

// Clusters of the group chain kernel for width W that the device holds at a time (0: it cannot run), and its opt-ins, once
// per device and operand type.
template <typename ACT, int FMT>
int gchain_clusters_of(const csd_ctx* ctx, int W) {
  static int known[kMaxDevices][kGcMaxCl + 1] = {};
  int& k = known[ctx->device][W / 128];
  if (k == 0) {
    auto kern = group_chain_kernel<ACT, FMT, false>, folded = group_chain_kernel<ACT, FMT, true>;
    auto opt_in = [](auto k) {
      return cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) == cudaSuccess &&
             cudaFuncSetAttribute(k, cudaFuncAttributeNonPortableClusterSizeAllowed, 1) == cudaSuccess;
    };
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = static_cast<unsigned>(W / 128); at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3(static_cast<unsigned>(W / 128)); lc.blockDim = dim3(kGcThreads); lc.dynamicSmemBytes = gc_layout(W).total + 1024;
    lc.attrs = at; lc.numAttrs = 1;
    int n = 0;
    const bool ok = opt_in(kern) && opt_in(folded) &&
                    cudaFuncSetAttribute(mods_gemm_kernel<FMT>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMgSmemBytes) == cudaSuccess &&
                    cudaOccupancyMaxActiveClusters(&n, kern, &lc) == cudaSuccess;
    cudaGetLastError();
    k = ok && n > 0 ? n : -1;
  }
  return k < 0 ? 0 : k;
}
int gchain_clusters(const csd_ctx* ctx, int dtype, int W) {
  return dtype == CSD_F16 ? gchain_clusters_of<__half, 0>(ctx, W) : gchain_clusters_of<__nv_bfloat16, 1>(ctx, W);
}
constexpr size_t kGcChunkBytes = size_t(512) << 20;   // most bytes of condition products of one chunk of steps

// Wide chain kernel (widechain.cuh): the heads it takes.
bool wide_width(const csd_head_desc& d) {
  return d.dtype != CSD_F32 && d.W % 256 == 0 && d.W >= 768 && d.W <= 128 * kWcMaxCt &&
         wc_layout(d.L, d.var_out ? kCPad2 : kCPad, 1).stages >= kWcMinStages;
}
typedef void (*WideKernel)(CUtensorMap, CUtensorMap, WcParams);
template <typename ACT, int FMT>
WideKernel wide_kernel_of(bool lv, int halves) {
  if (halves == 2) return lv ? wide_chain_kernel<ACT, FMT, true, 2> : wide_chain_kernel<ACT, FMT, false, 2>;
  return lv ? wide_chain_kernel<ACT, FMT, true, 1> : wide_chain_kernel<ACT, FMT, false, 1>;
}
WideKernel wide_kernel(int dtype, bool lv, int halves) { return dtype == CSD_F16 ? wide_kernel_of<__half, 0>(lv, halves) : wide_kernel_of<__nv_bfloat16, 1>(lv, halves); }
// CTA pairs of the wide chain kernel that the device holds at a time (0: it cannot run), and the opt-ins, once per device and operand type.
int wide_pairs(const csd_ctx* ctx, int dtype) {
  static int known[kMaxDevices][2] = {};
  int& k = known[ctx->device][dtype == CSD_F16 ? 0 : 1];
  if (k == 0) {
    bool ok = (dtype == CSD_F16 ? cudaFuncSetAttribute(wide_mods_kernel<0>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMgSmemBytes)
                                : cudaFuncSetAttribute(wide_mods_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, kMgSmemBytes)) == cudaSuccess;
    for (int i = 0; i < 4; ++i) ok = ok && cudaFuncSetAttribute(wide_kernel(dtype, (i & 1) != 0, 1 + (i >> 1)), cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024) == cudaSuccess;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3(2); lc.blockDim = dim3(kWcThreads); lc.dynamicSmemBytes = 227 * 1024;
    lc.attrs = at; lc.numAttrs = 1;
    int n = 0;
    ok = ok && cudaOccupancyMaxActiveClusters(&n, wide_kernel(dtype, false, 2), &lc) == cudaSuccess;
    cudaGetLastError();
    k = ok && n > 0 ? n : -1;
  }
  return k < 0 ? 0 : k;
}
WideCut wide_cut(const csd_ctx* ctx, const csd_head_desc& d, int R, int cfg, int halves) {
  return csd::wide_cut(wide_groups(wide_pairs(ctx, d.dtype), d.W), d.W, R, cfg, halves);
}
bool wide_halves(const csd_head_desc& d) { return wc_layout(d.L, d.var_out ? kCPad2 : kCPad, 2).stages >= kWcMinStages; }
// Which form, and whether two chains go side by side, by a model of one step in us, fitted to measured steps (W = 1024, 1024 rows: 3
// blocks 68 in one-slot groups, 82 in two-slot groups; 6 blocks 106 and 158; 12 x 1536 259 and 420).  The choice changes no bit.
double wide_step_us(const csd_head_desc& d, int halves) { return halves == 2 ? 30.0 + 12.7 * d.L * d.W / 1024 : 20.0 + 22.0 * d.L * d.W / 1024; }
double wide_mods_sm_us(const csd_head_desc& d, int slots) { return 2.0 * (3 * d.L + 2) * d.W * d.W * kWcRows * slots / 8.8e6; }   // 8.8 TFLOP/s an SM
// Beside chains that hold at most half of the SMs the products have the rest to themselves; else everything shares the GPU, at about
// 120 of 148 SMs' worth (two chains, which fill each other's gaps: 133).
double wide_us(const csd_ctx* ctx, double chain_us, double chain_sm_us, double mods_sm_us, int held, double share = 0.81) {
  const double other = held <= ctx->num_sms / 2 ? mods_sm_us / (ctx->num_sms - held) : (mods_sm_us + chain_sm_us) / (share * ctx->num_sms);
  return chain_us > other ? chain_us : other;
}
WideCut wide_cut_alone(const csd_ctx* ctx, const csd_head_desc& d, int R, int cfg) {
  const WideCut one = wide_cut(ctx, d, R, cfg, 2), two = wide_cut(ctx, d, R, cfg, 1);
  if (!wide_halves(d) || one.part < one.slots) return two;
  auto us = [&](const WideCut& c) { const double t = wide_step_us(d, c.halves); return wide_us(ctx, t, t * c.ctas, wide_mods_sm_us(d, c.slots), c.ctas); };
  return us(one) <= us(two) ? one : two;
}
constexpr size_t kWcBufferBytes = size_t(2) << 30;    // most bytes of a chunk of steps: s and two buffers of condition products
bool wide_takes(const csd_ctx* ctx, const csd_head* hd, int R, int cfg, int slot, bool batch) {
  const int rows = R * (cfg ? 2 : 1);
  return wide_width(hd->d) && ctx->chain_mode == CSD_CHAIN_LAYERS && slot != 2 && !batch && !ctx->prof_on && wide_pays(hd->d.L, hd->d.W, rows) &&
         wide_groups(wide_pairs(ctx, hd->d.dtype), hd->d.W) >= 1;      // (a device, or a part of one, with fewer SMs than a group has CTAs)
}
// One head's denoising chain for R token rows on stream `st` with workspace slot `slot`:
// begin() enqueues the per-call work (timestep embedding, condition projection, first boundary
// kernel), step(t) enqueues the kernels of step t.  Two chains can be interleaved launch by launch.
struct Chain {
  csd_ctx* ctx; int slot; cudaStream_t st; const csd_head* hd; const csd_schedule* sc;
  int R, cfg; float cfg_scale; const float *z, *x_T, *eps; int sample_last; float *x0, *mu1, *x1;
  int chains = 1;   // chains that run concurrently with this one (itself included)
  int Rh = 0, W = 0, L = 0, T = 0, tn = kTileN;
  bool gck = false, gfold = false;   // the whole chain runs in the group chain kernel (groupchain.cuh), in its folded form
  bool wck = false;       // the whole chain runs in the wide chain kernel (widechain.cuh)
  bool wc_asked = false;  // its buffers have been asked for; wc_most 0: refused
  int beside = 0;         // CTAs that the other chain's wide chain kernel holds meanwhile
  WideCut wc{};
  int wc_most = 0;        // the most steps of a chunk
  struct { WcParams p; CUtensorMap tm_s, tm_u, tm_v; int t_hi, n, launched; } wq{};   // first step and number of steps of the next and the last chunk, launches so far
  int gc_rows = 0, gc_most = 0;      // its rows (groups x 16) and the most steps of a chunk
  int fcg = 0;            // fp32 head: the whole chain runs in the fp32 chain kernel with groups of this many rows (f32chain.cuh)
  bool fold = false;      // blocks 1.. run as two kernels (fold.cuh) instead of three
  CUtensorMap tm_ap{};
  bool mod64 = false;     // modulate kernels in 64-wide tiles although the others use 128
  bool w1_wide = false;   // first MLP layer in 128 x 256 tiles (MMA N = 256)
  bool tc = false, pair = false;
  // s is double-buffered by step parity (index t & 1): the boundary kernel that ends step t writes s of step t - 2,
  // so no product of s ever waits for the kernel right before it
  CUtensorMap tm_z{}, tm_sb[2]{}, tm_u{}, tm_v{}, tm_u_out{}, tm_v_out{};   // _out: boxes of 32 rows, what an epilogue warp stores
  void* sbuf[2] = {nullptr, nullptr};
  int cur_t = 0;
  EpiParams ep{};
  StepParams sp{};
  // trajectory recording (csd_draft_denoise_traj): [T + 1, R, C] states and [T, R, C] means, or null
  float *traj_x = nullptr, *traj_mu = nullptr;
  // learned-variance heads: host arrays [T] of the log-variance bounds, outputs lv1 [R, C] and half_logdet [R]
  const float *lv_min = nullptr, *lv_max = nullptr;
  float *lv1 = nullptr, *half_logdet = nullptr;
  // batched evaluation on a given trajectory (csd_verify_single_path): R = batch_steps * batch_Rin token rows,
  // one pass of the layers; slot batch_j0 of batch_traj is the first step of the pass
  int batch_Rin = 0, batch_j0 = 0, Ts = 0;
  int ws_steps = 0;          // steps the workspace is carved for (the same for every pass of a call, so that the
  bool batch_reuse = false;  // timestep embedding and the condition projection of the first pass stay where they are)
  const float *batch_traj = nullptr, *batch_sched = nullptr;
  float* batch_mu = nullptr;

  template <typename ACT>
  int launch_step_t(cudaLaunchConfig_t& cfg, bool rb4, int mode) {
    if (lv_min) CSD_CUDA(ctx, cudaLaunchKernelEx(&cfg, rb4 ? step_kernel<ACT, 4, false, true> : step_kernel<ACT, 1, false, true>, sp, mode));
    else if (traj_x) CSD_CUDA(ctx, cudaLaunchKernelEx(&cfg, rb4 ? step_kernel<ACT, 4, true> : step_kernel<ACT, 1, true>, sp, mode));
    else CSD_CUDA(ctx, cudaLaunchKernelEx(&cfg, rb4 ? step_kernel<ACT, 4> : step_kernel<ACT, 1>, sp, mode));
    return CSD_OK;
  }

  // kind 0: prepare the pass (h, LayerNorm partials, s); kind 1: finish it (eps_hat, guidance, mu^p)
  int launch_batch(int kind) {
    const csd_head_desc& d = hd->d;
    ChainWs& ws = ctx->ws[slot];
    BatchParams b{};
    b.Rin = batch_Rin; b.Rtok = R; b.cfg = cfg; b.C = d.C; b.W = W; b.NT = tc ? W / kStatCols : W / kTileN;
    b.T = Ts; b.j0 = batch_j0; b.cfg_scale = cfg_scale; b.sched = batch_sched; b.traj_x = batch_traj;
    b.win = hd->win; b.bin = hd->bin; b.cz = ws.cz; b.te = ws.te; b.h = ws.h; b.stats = ws.stats; b.s = ws.s;
    b.epart = ws.epart; b.bout = hd->bout; b.mu_p = batch_mu; b.status = ctx->d_err + 1;
    ProfScope ps(ctx, st, 5, 2.0 * Rh * static_cast<double>(W) * d.C);
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3(kind == 0 ? (R + 3) / 4 : (R + 15) / 16); lc.blockDim = dim3(256); lc.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at; lc.numAttrs = (ctx->prof_on || !tc) ? 0 : 1;
    if (kind == 1) CSD_CUDA(ctx, cudaLaunchKernelEx(&lc, batch_finish_kernel, b));
    else if (d.dtype == CSD_F16) CSD_CUDA(ctx, cudaLaunchKernelEx(&lc, batch_prepare_kernel<__half>, b));
    else if (d.dtype == CSD_BF16) CSD_CUDA(ctx, cudaLaunchKernelEx(&lc, batch_prepare_kernel<__nv_bfloat16>, b));
    else CSD_CUDA(ctx, cudaLaunchKernelEx(&lc, batch_prepare_kernel<float>, b));
    ctx->launches++;
    CSD_CUDA(ctx, cudaGetLastError());
    return CSD_OK;
  }

  int launch_step(int mode) {
    const csd_head_desc& d = hd->d;
    ProfScope ps(ctx, st, 5, 2.0 * Rh * static_cast<double>(W) * d.C);
    cudaLaunchConfig_t cfg{};
    // four token rows per block once that still leaves every SM several blocks (the choice does not change a bit)
    const bool rb4 = R >= 8 * ctx->num_sms;
    cfg.gridDim = dim3(rb4 ? (R + 3) / 4 : R); cfg.blockDim = dim3(256); cfg.dynamicSmemBytes = 0; cfg.stream = st;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    cfg.attrs = at; cfg.numAttrs = (ctx->prof_on || !tc) ? 0 : 1;
    int rc;
    if (d.dtype == CSD_F16) rc = launch_step_t<__half>(cfg, rb4, mode);
    else if (d.dtype == CSD_BF16) rc = launch_step_t<__nv_bfloat16>(cfg, rb4, mode);
    else rc = launch_step_t<float>(cfg, rb4, mode);
    if (rc) return rc;
    ctx->launches++;
    CSD_CUDA(ctx, cudaGetLastError());
    return CSD_OK;
  }

  void sizes() { Rh = R * (cfg ? 2 : 1); W = hd->d.W; L = hd->d.L; Ts = sc->T; }

  int begin() {
    const csd_head_desc& d = hd->d;
    sizes();
    T = batch_Rin ? 1 : Ts;   // a batched pass runs the layers once
    tc = d.dtype != CSD_F32;
    // 64-wide output tiles when 128-wide ones (of all chains running side by side) would occupy at most a
    // quarter of the SMs: a kernel and the early part of its successor should both find free SMs
    tn = (tc && chains * (W / kTileN) * ((Rh + kTileM - 1) / kTileM) <= ctx->num_sms / 4) ? 64 : kTileN;
    // CTA pairs (two row tiles per MMA, half of each weight tile per CTA) need 128-wide tiles; they are
    // used once a kernel has at least two waves of tiles, where L2-to-SM bandwidth is the limit (measured:
    // a few per cent faster at 384 tiles, slower at 64 and 256)
    pair = tc && tn == kTileN && (W / kTileN) * ((Rh + kTileM - 1) / kTileM) >= 2 * ctx->num_sms;
    // First MLP layer: 256-wide MMAs keep the tensor pipe busier per issued instruction (measured about 660 clk
    // per 64-deep k-block and tile against 415 for two 128-wide tiles' worth), but halve the tile count; taken when
    // that does not cost a wave.
    {
      const int row_tiles = (Rh + kTileM - 1) / kTileM, t128 = (W / kTileN) * row_tiles, t256 = (W / 256) * row_tiles;
      const int waves128 = (t128 + ctx->num_sms - 1) / ctx->num_sms, waves256 = (t256 + ctx->num_sms - 1) / ctx->num_sms;
      w1_wide = tc && !pair && tn == kTileN && W % 256 == 0 && waves256 * 664 < waves128 * 415;
    }
    // The modulate kernels' products never wait for the preceding kernel, only their epilogues do: with 64-wide
    // tiles the epilogue a thread runs is half as long.  Taken for a chain that has the GPU to itself and whose
    // 64-wide tiles fit one wave (measured: draft chain of mar256 10.4 -> 9.8 ms, target chain 18.2 -> 17.7 ms;
    // with two chains side by side the extra CTAs cost more than they save).
    mod64 = tc && chains == 1 && tn == kTileN && !pair && 2 * (W / kTileN) * ((Rh + kTileM - 1) / kTileM) <= ctx->num_sms;
    // Folded blocks: one 128-wide tile per CTA, and their early products want idle SMs to overlap the preceding
    // kernel: taken when the layer's tiles fill between an eighth and half of the SMs (measured slower on tiny grids,
    // which run 64-wide tiles, and on a full wave)
    // (the rule looks at this chain alone, so that csd_round and the three separate calls take the same path).
    {
      const int t128 = (W / kTileN) * ((Rh + kTileM - 1) / kTileM);
      fold = tc && (ctx->chain_mode == CSD_CHAIN_LAYERS || ctx->chain_mode == CSD_CHAIN_LAYER_KERNELS) && !pair && L >= 2 && !hd->Wf.empty() &&
             8 * t128 > ctx->num_sms && 2 * t128 <= ctx->num_sms && fold_kernels_ready(ctx, d);
    }
    // Few rows: condition products ahead, one kernel for the rest (groupchain.cuh).  A step takes it as long for one group as
    // for all that are resident (clusters: 33, 15, 7 at W = 512, 1024, 1536), so it wins up to there, even where a round's two
    // chains have to take turns: 240 rows each of the 3 and 6 x 1024 heads, 9.2 ms a round against the layer kernels' 13.2;
    // 7 groups of a 12 x 1536 target, 17.4 against 28.2.  One group more takes two turns by itself (42 ms).  The rule may not
    // look at the other chain: a call of one chain gives the bits that the round gives.
    gck = tc && (ctx->chain_mode == CSD_CHAIN_LAYERS || ctx->chain_mode == CSD_CHAIN_SMALL_BATCH) && hd->gc_ready &&
          slot != 2 && !batch_Rin && !lv_min && !ctx->prof_on &&
          (R + (cfg ? 7 : 15)) / (cfg ? 8 : 16) <= gchain_clusters(ctx, d.dtype, W);
    // Its folded form is a quarter faster a layer and less precise: only in the mode that says so, up to the rows that it names
    gfold = gck && ctx->chain_mode == CSD_CHAIN_SMALL_BATCH && Rh <= 128;
    int rc = CSD_OK;
    if (gck && (rc = reserve_group_chain())) return rc;
    if (gck) { fold = false; pair = false; }
    wck = !gck && wide_takes(ctx, hd, R, cfg, slot, batch_Rin != 0);
    Chain* const self = this;
    if (wck && !wc_asked && (rc = reserve_wide_chains(ctx, &self, 1))) return rc;
    wck = wck && wc_most > 0;
    if (wck) { fold = false; pair = false; }
    // fp32 heads: one persistent kernel per chain, except where a row's bits have to be those of a batched pass
    fcg = !tc && ctx->chain_mode != CSD_CHAIN_LAYERS_PLAIN && !batch_Rin && !ctx->prof_on && fc_pays(ctx, d, Rh) ? fc_rows(ctx, d, R, cfg, chains) : 0;
    ChainWs& ws = ctx->ws[slot];
    rc = batch_Rin ? ensure_ws(ctx, ws, d, ws_steps * batch_Rin * (cfg ? 2 : 1), ws_steps * batch_Rin, Ts)
                       : ensure_ws(ctx, ws, d, Rh, R, Ts);
    if (rc) return rc;
    if (fcg) return launch_f32_chain();
    if (!batch_reuse) {
      if ((rc = launch_embed<true>(sc->tfeat, hd->Wt1, hd->bt1, ws.hid, d.F)) || (rc = launch_embed<false>(ws.hid, hd->Wt2, hd->bt2, ws.te, W))) return rc;
    }
    CSD_CUDA(ctx, cudaGetLastError());
    ep.M = Rh; ep.ldo = W;
    // rows of z: one per head row, or one per row of a step when the steps of a trajectory are batched
    const int Rz = batch_Rin ? batch_Rin * (cfg ? 2 : 1) : Rh;
    if (tc) {
      if (!batch_reuse) {
        const size_t nz = static_cast<size_t>(Rz) * d.Dz;
        const unsigned nblk = static_cast<unsigned>((nz + 255) / 256);
        if (d.dtype == CSD_F16) convert_act_kernel<__half><<<nblk, 256, 0, st>>>(z, static_cast<__half*>(ws.zc), nz);
        else convert_act_kernel<__nv_bfloat16><<<nblk, 256, 0, st>>>(z, static_cast<__nv_bfloat16*>(ws.zc), nz);
        ctx->launches++;
      }
      if ((rc = make_tmap(ctx, &tm_z, d.dtype, ws.zc, Rz, d.Dz, d.Dz, kTileM))) return rc;
      if ((rc = make_tmap(ctx, &tm_sb[1], d.dtype, ws.s, Rh, W, W, kTileM))) return rc;
      if ((rc = make_tmap(ctx, &tm_sb[0], d.dtype, ws.s2, Rh, W, W, kTileM))) return rc;
      if ((rc = make_tmap(ctx, &tm_u, d.dtype, ws.u, Rh, W, W, kTileM))) return rc;
      if ((rc = make_tmap(ctx, &tm_v, d.dtype, ws.v, Rh, W, W, kTileM))) return rc;
      if ((rc = make_tmap(ctx, &tm_u_out, d.dtype, ws.u, Rh, W, W, 32))) return rc;
      if ((rc = make_tmap(ctx, &tm_v_out, d.dtype, ws.v, Rh, W, W, 32))) return rc;
      if ((rc = make_tmap(ctx, &tm_ap, d.dtype, ws.ap, Rh, W, W, kTileM))) return rc;
    }
    // cz = z Wz^T + bz
    const csd_head::TmSet& tmw = hd->tm[(tn == 64 || pair) ? 0 : 1];   // pairs load half of each B tile per CTA
    EpiParams e = ep;
    e.M = Rz;
    e.bias0 = hd->bz; e.out_f32 = ws.cz;
    if (batch_reuse) rc = CSD_OK;
    else if (tc) rc = launch_tc<EPI_BIAS_F32, 1, 1>(ctx, d.dtype, tn, pair, st, tm_z, tmw.Wz, tm_z, tmw.Wz, d.Dz, 0, 0, W, e);
    else rc = launch_simt<EPI_BIAS_F32, 1, 128>(ctx, st, z, d.Dz, static_cast<const float*>(hd->Wz), d.Dz, nullptr, 0,
                                                nullptr, 0, W, e);
    if (rc) return rc;
    sbuf[0] = ws.s2; sbuf[1] = ws.s;
    if (gck) return launch_group_chain();
    if (wck) return begin_wide_chain();
    if (batch_Rin) return launch_batch(0);   // a pass has one step (t = 1): its s is sbuf[1]
    sp.traj_x = traj_x; sp.traj_mu = nullptr; sp.status = ctx->d_err + 1;
    sp.lv1 = lv1; sp.half_logdet = half_logdet; sp.lv_min = 0.0f; sp.lv_max = 0.0f;
    sp.R = R; sp.cfg = cfg; sp.C = d.C; sp.W = W; sp.NT = tc ? W / kStatCols : W / kTileN; sp.cfg_scale = cfg_scale;
    sp.sample_last = sample_last; sp.epart = ws.epart; sp.bout = hd->bout; sp.x_src = x_T; sp.x = ws.x;
    sp.x0 = x0; sp.mu1 = mu1; sp.x1 = x1; sp.win = hd->win; sp.bin = hd->bin; sp.cz = ws.cz; sp.h = ws.h;
    sp.stats = ws.stats; sp.s = sbuf[T & 1];
    sp.te_next = ws.te + static_cast<size_t>(T - 1) * W;
    sp.s_b = T >= 2 ? sbuf[(T - 1) & 1] : nullptr;   // the first boundary also prepares s of step T - 1
    sp.te_b = T >= 2 ? ws.te + static_cast<size_t>(T - 2) * W : nullptr;
    sp.eps_t = eps;
    return launch_step(STEP_INIT);
  }

  int launch_fold(int kind, int k) {
    const csd_head_desc& d = hd->d;
    ChainWs& ws = ctx->ws[slot];
    FoldParams p{};
    p.M = Rh; p.W = W; p.err = ctx->d_err;
    const int tiles_n = W / kTileN, row_tiles = (Rh + kTileM - 1) / kTileM;
    // CTA pairs (two row tiles per MMA) whenever the row tiles pair up
    const bool fp = kFoldPairs && row_tiles % 2 == 0;
    const CUtensorMap *tp, *ta, *tw, *tout;
    if (kind == FOLD_W1) {
      p.c0 = hd->c1[k]; p.c1 = hd->c2[k]; p.c2 = nullptr; p.stats_in = ws.stats; p.out = ws.v;
      tp = fp ? &hd->Wf_half[k] : &hd->Wf[k]; ta = &tm_ap; tw = &hd->tm[fp ? 0 : 1].W1[k]; tout = &tm_v;
    } else {
      p.c0 = hd->bg[k]; p.c1 = hd->b2[k]; p.c2 = hd->bsc[k + 1]; p.stats_out = ws.stats; p.h = ws.h; p.out = ws.ap;
      tp = fp ? &hd->Wgs_half[k] : &hd->Wgs[k]; ta = &tm_v; tw = &hd->tm[fp ? 0 : 1].W2[k]; tout = &tm_ap;
    }
    // algorithmic FLOPs: the block's five W x W products are split 2 (first layer and the modulation folded into
    // it; the kernel executes three products) + 3 (gate, next scale, second layer)
    ProfScope ps(ctx, st, kind == FOLD_W1 ? 1 : 3, 2.0 * Rh * static_cast<double>(W) * W * (kind == FOLD_W1 ? 2.0 : 3.0));
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3(tiles_n * row_tiles); lc.blockDim = dim3(kFoldThreads); lc.stream = st;
    lc.dynamicSmemBytes = kind == FOLD_W1 ? FoldCfg<FOLD_W1>::kSmemBytes : FoldCfg<FOLD_GATE>::kSmemBytes;
    cudaLaunchAttribute at[2];
    int na = 0;
    if (fp) { at[na].id = cudaLaunchAttributeClusterDimension; at[na].val.clusterDim.x = 2; at[na].val.clusterDim.y = 1; at[na].val.clusterDim.z = 1; ++na; }
    if (!ctx->prof_on) { at[na].id = cudaLaunchAttributeProgrammaticStreamSerialization; at[na].val.programmaticStreamSerializationAllowed = 1; ++na; }
    lc.attrs = at; lc.numAttrs = na;
    const CUtensorMap& ts = tm_sb[cur_t & 1];
#define CSD_FOLD_LAUNCH(ACT, FMT, KIND, PAIR) CSD_CUDA(ctx, cudaLaunchKernelEx(&lc, fold_kernel<ACT, FMT, KIND, PAIR>, ts, *tp, *ta, *tw, *tout, tiles_n, p))
    if (d.dtype == CSD_F16) {
      if (kind == FOLD_W1) { if (fp) CSD_FOLD_LAUNCH(__half, 0, FOLD_W1, true); else CSD_FOLD_LAUNCH(__half, 0, FOLD_W1, false); }
      else { if (fp) CSD_FOLD_LAUNCH(__half, 0, FOLD_GATE, true); else CSD_FOLD_LAUNCH(__half, 0, FOLD_GATE, false); }
    } else {
      if (kind == FOLD_W1) { if (fp) CSD_FOLD_LAUNCH(__nv_bfloat16, 1, FOLD_W1, true); else CSD_FOLD_LAUNCH(__nv_bfloat16, 1, FOLD_W1, false); }
      else { if (fp) CSD_FOLD_LAUNCH(__nv_bfloat16, 1, FOLD_GATE, true); else CSD_FOLD_LAUNCH(__nv_bfloat16, 1, FOLD_GATE, false); }
    }
#undef CSD_FOLD_LAUNCH
    ctx->launches++;
    return CSD_OK;
  }

  // One layer of the timestep embedding of all steps: [Ts, W] from [Ts, K].
  template <bool SILU>
  int launch_embed(const float* A, const float* B, const float* bias, float* C, int K) {
    const bool wide = Ts >= 64;
    const int rows = wide ? 32 : 8;
    return launch_short(ctx, st, wide ? embed_kernel<4, SILU> : embed_kernel<1, SILU>, dim3((W + 31) / 32, (Ts + rows - 1) / rows), 64, 0, A, B, bias, C, Ts, W, K);
  }
  static RowsGemm rows_gemm(const float* A, const float* B, const float* bias, float* C, int M, int N, int K, bool silu) {
    return RowsGemm{A, B, bias, C, M, N, K, silu ? 1 : 0, (N + kRgCols - 1) / kRgCols};
  }
  int launch_rows_gemm(const RowsGemm& a, const RowsGemm* b) {
    auto blocks = [](const RowsGemm& g) { return g.blocks_n * ((g.M + kRgRows - 1) / kRgRows); };
    RowsGemmPair pr{{a, b ? *b : a}, blocks(a)};
    return launch_short(ctx, st, rows_gemm_kernel, blocks(a) + (b ? blocks(*b) : 0), 256, 0, pr);
  }

  // fp32 heads: hidden layer of the timestep embedding and condition projection, the embedding, then the chain.
  int launch_f32_chain() {
    const csd_head_desc& d = hd->d;
    ChainWs& ws = ctx->ws[slot];
    const RowsGemm hid = rows_gemm(sc->tfeat, hd->Wt1, hd->bt1, ws.hid, Ts, W, d.F, true), te = rows_gemm(ws.hid, hd->Wt2, hd->bt2, ws.te, Ts, W, W, false),
                   cz = rows_gemm(z, static_cast<const float*>(hd->Wz), hd->bz, ws.cz, Rh, W, d.Dz, false);
    int rc;
    if ((rc = launch_rows_gemm(hid, &cz)) || (rc = launch_rows_gemm(te, nullptr))) return rc;
    FcParams p{};
    p.R = R; p.cfg = cfg; p.C = d.C; p.W = W; p.L = L; p.T = Ts; p.per = fcg / (cfg ? 2 : 1); p.sample_last = sample_last; p.lv = lv_min ? 1 : 0;
    p.cfg_scale = cfg_scale;
    p.w = static_cast<const float*>(hd->Wss[0]); p.bias = hd->bsh[0];   // csd_head_create lays both out block after block
    p.win = hd->win; p.bin = hd->bin; p.wout_t = hd->wout_t; p.bout = hd->bout;
    p.cz = ws.cz; p.te = ws.te; p.x_T = x_T; p.eps = eps; p.x = ws.x; p.x0 = x0; p.mu1 = mu1; p.x1 = x1;
    p.traj_x = traj_x; p.traj_mu = traj_mu; p.lv1 = lv1; p.half_logdet = half_logdet; p.status = ctx->d_err + 1;
    const int groups = (R + p.per - 1) / p.per;
    cudaLaunchConfig_t lc{};
    lc.gridDim = dim3(static_cast<unsigned>(groups) * kFcCluster); lc.blockDim = dim3(fcg == 16 ? FcThreads<16>::value : FcThreads<8>::value); lc.stream = st;
    lc.dynamicSmemBytes = static_cast<size_t>(fc_layout(fcg, W, lv_min ? kCPad2 : kCPad).total) * 4;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = kFcCluster; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[1].val.programmaticStreamSerializationAllowed = 1;
    lc.attrs = at; lc.numAttrs = 2;
    const bool narrow = W / kFcCluster <= 32;
    auto kern = narrow ? (fcg == 16 ? f32_chain_kernel<16, 2> : fcg == 8 ? f32_chain_kernel<8, 2> : f32_chain_kernel<4, 2>)
                       : (fcg == 16 ? f32_chain_kernel<16, 4> : fcg == 8 ? f32_chain_kernel<8, 4> : f32_chain_kernel<4, 4>);
    for (p.t_hi = Ts; p.t_hi >= 1; p.t_hi = p.t_lo - 1) {
      p.t_lo = p.t_hi > kFcMaxSteps ? p.t_hi - kFcMaxSteps + 1 : 1;
      for (int t = p.t_lo; t <= p.t_hi; ++t) {
        const int i = t - p.t_lo;
        p.a[i] = sc->a[t - 1]; p.b[i] = sc->b[t - 1];
        p.s0[i] = lv_min ? lv_min[t - 1] : sc->sigma[t - 1];
        p.s1[i] = lv_min ? lv_max[t - 1] : 0.0f;
      }
      CSD_CUDA(ctx, cudaLaunchKernelEx(&lc, kern, p));
      ctx->launches++;
    }
    return CSD_OK;
  }

  // Weight rows of the condition products, and the bytes of a chunk of steps of them.
  size_t gc_wrows() const { return static_cast<size_t>(gfold ? 4 * L + 3 : 3 * L + 2) * W; }
  size_t gc_chunk_bytes(int steps) const { return gc_wrows() * ((static_cast<size_t>(steps) * gc_rows + 255) / 256) * 256 * 4; }

  // ensure_buffer for buffers that a call can do without: a size that could not be had is asked for again only where there is room.
  int have(HostIo& io, size_t& refused, size_t need, const char* what) {
    if (need > io.cap && need >= refused && (capturing(ctx) || !room_for(need, io.in_graph ? 0 : io.cap))) return CSD_ERR_WORKSPACE;
    const int rc = ensure_buffer(ctx, io, need, what);
    if (rc == CSD_ERR_WORKSPACE && need < refused) refused = need;
    return rc;
  }

  // Buffers of the group chain kernel: bytes by the steps that a call has and the limit, so that no call of fewer steps or rows has to replace
  // them.  Shorter chunks cost a launch each and change no bit, so the buffers are halved until they can be had; where one step does
  // not fit the chain falls back to the layer kernels (gck), which need none of it.
  static int reserve_wide_chains(csd_ctx* ctx, Chain* const* c, int n);
  int reserve_group_chain() {
    gc_rows = (R + (cfg ? 7 : 15)) / (cfg ? 8 : 16) * kGcRows;
    int rc = have(ctx->gc[slot], ctx->gc_refused[slot], static_cast<size_t>(Ts) * gc_rows * W * 2, "the condition vectors of all steps");
    gc_most = Ts < kGcMaxSteps ? Ts : kGcMaxSteps;
    const size_t step = gc_chunk_bytes(1), all = gc_chunk_bytes(gc_most);
    size_t chunk = all < kGcChunkBytes ? all : kGcChunkBytes;
    if (chunk < step) chunk = step;
    while (!rc && (rc = have(ctx->gm[slot], ctx->gm_refused[slot], 2 * chunk, "the condition products")) == CSD_ERR_WORKSPACE && chunk > step) {
      rc = CSD_OK;
      chunk = chunk / 2 < step ? step : chunk / 2;
    }
    while (gc_most > 1 && gc_chunk_bytes(gc_most) > chunk) gc_most = (gc_most + 1) / 2;
    if (rc == CSD_ERR_WORKSPACE) { gck = gfold = false; ctx->err[0] = 0; rc = CSD_OK; }
    return rc;
  }

  // The group chain kernel: s of every step in its row order, then chunk by chunk the condition products (on the slot's
  // own stream, ahead of the chain) and the chain.
  int launch_group_chain() {
    const csd_head_desc& d = hd->d;
    ChainWs& ws = ctx->ws[slot];
    const int rows = gc_rows, groups = rows / kGcRows, cl = W / 128, most = gc_most;
    const size_t wrows = gc_wrows();
    int rc;
    void* const s_all = ctx->gc[slot].base;
    CUtensorMap tm_s{};
    if ((rc = make_tmap(ctx, &tm_s, d.dtype, s_all, static_cast<uint64_t>(Ts) * rows, W, W, kTileM))) return rc;
    const dim3 sgrid(static_cast<unsigned>(rows), static_cast<unsigned>((Ts + kCondSteps - 1) / kCondSteps));
    if (d.dtype == CSD_F16) cond_all_kernel<__half, 16><<<sgrid, 128, 0, st>>>(ws.cz, ws.te, static_cast<__half*>(s_all), R, cfg, W, rows, 0, Ts);
    else cond_all_kernel<__nv_bfloat16, 16><<<sgrid, 128, 0, st>>>(ws.cz, ws.te, static_cast<__nv_bfloat16*>(s_all), R, cfg, W, rows, 0, Ts);
    ctx->launches++;
    CSD_CUDA(ctx, cudaGetLastError());
    cudaStream_t gst = ctx->aux[slot];
    CSD_CUDA(ctx, cudaEventRecord(ctx->ev_prep[slot], st));
    CSD_CUDA(ctx, cudaStreamWaitEvent(gst, ctx->ev_prep[slot], 0));
    GcParams p{};
    p.R = R; p.cfg = cfg; p.W = W; p.L = L; p.C = d.C; p.T = Ts; p.rows = rows; p.sample_last = sample_last; p.cfg_scale = cfg_scale;
    p.maps = hd->d_gc_maps; p.c1 = hd->c1[0]; p.bsh = hd->bsh[0]; p.bsc = hd->bsc[0]; p.bg = hd->bg[0]; p.b1 = hd->b1[0]; p.b2 = hd->b2[0];
    p.bfsh = hd->bfsh; p.bfsc = hd->bfsc;
    p.win = hd->win; p.bin = hd->bin; p.wout_t = hd->wout_t; p.bout = hd->bout; p.x_T = x_T; p.eps = eps;
    p.x = ws.x; p.x0 = x0; p.mu1 = mu1; p.x1 = x1; p.traj_x = traj_x; p.traj_mu = traj_mu; p.err = ctx->d_err; p.status = ctx->d_err + 1;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeLaunchCompletionEvent;
    at[1].val.launchCompletionEvent.event = ctx->ev_on[slot]; at[1].val.launchCompletionEvent.flags = 0;
    cudaLaunchConfig_t lc{};
    lc.attrs = at;
    // Steps per chunk: a first chunk of a tile's width of rows, because nothing overlaps its products; then twice as many
    // each time, as far as the buffers go.
    int n = (256 + rows - 1) / rows;
    for (int t_hi = Ts, c = 0; t_hi >= 1; ++c, n *= 2) {
      if (n > most) n = most;
      if (n > t_hi) n = t_hi;
      const int t_lo = t_hi - n + 1, buf = c & 1;
      float4* mods = reinterpret_cast<float4*>(static_cast<char*>(ctx->gm[slot].base) + buf * gc_chunk_bytes(most));
      MgParams m{};
      m.nkb = W / kBlockK; m.tiles_n = (n * rows + 255) / 256; m.units = m.tiles_n * static_cast<int>(wrows / 256);
      m.wrow = hd->d_gc_rows + (gfold ? (3 * L + 2) * W / 256 : 0);
      m.s_row0 = (t_lo - 1) * rows; m.out = mods; m.err = ctx->d_err;
      if (c >= 2) CSD_CUDA(ctx, cudaStreamWaitEvent(gst, ctx->ev_read[slot][buf], 0));
      // Beside a running chain the products take the SMs it leaves, once it has its own: spread over the GPU first, their CTAs
      // leave some GPC without room for a cluster, which then waits for them (128 rows of 3 x 1024, T = 100: 2.76 against
      // 2.38 ms)
      if (c >= 1) CSD_CUDA(ctx, cudaStreamWaitEvent(gst, ctx->ev_on[slot], 0));
      int pairs = (c == 0 ? ctx->num_sms : ctx->num_sms - chains * groups * cl) / 2;
      if (pairs < 8) pairs = 8;
      if (pairs > m.units) pairs = m.units;
      lc.gridDim = dim3(static_cast<unsigned>(2 * pairs)); lc.blockDim = dim3(kMgThreads); lc.dynamicSmemBytes = kMgSmemBytes; lc.stream = gst;
      at[0].val.clusterDim.x = 2; lc.numAttrs = 1;
      if (d.dtype == CSD_F16) CSD_CUDA(ctx, cudaLaunchKernelEx(&lc, mods_gemm_kernel<0>, hd->Wrows, hd->Wx, tm_s, m));
      else CSD_CUDA(ctx, cudaLaunchKernelEx(&lc, mods_gemm_kernel<1>, hd->Wrows, hd->Wx, tm_s, m));
      CSD_CUDA(ctx, cudaEventRecord(ctx->ev_mods[slot][buf], gst));
      CSD_CUDA(ctx, cudaStreamWaitEvent(st, ctx->ev_mods[slot][buf], 0));
      p.t_hi = t_hi; p.t_lo = t_lo; p.mods = mods; p.nq = m.tiles_n * 64;
      for (int i = 0; i < n; ++i) { p.ca[i] = sc->a[t_lo - 1 + i]; p.cb[i] = sc->b[t_lo - 1 + i]; p.sigma[i] = sc->sigma[t_lo - 1 + i]; }
      lc.gridDim = dim3(static_cast<unsigned>(groups * cl)); lc.blockDim = dim3(kGcThreads); lc.dynamicSmemBytes = gc_layout(W).total + 1024; lc.stream = st;
      at[0].val.clusterDim.x = static_cast<unsigned>(cl); lc.numAttrs = 2;
      if (d.dtype == CSD_F16) CSD_CUDA(ctx, cudaLaunchKernelEx(&lc, gfold ? group_chain_kernel<__half, 0, true> : group_chain_kernel<__half, 0, false>, p));
      else CSD_CUDA(ctx, cudaLaunchKernelEx(&lc, gfold ? group_chain_kernel<__nv_bfloat16, 1, true> : group_chain_kernel<__nv_bfloat16, 1, false>, p));
      CSD_CUDA(ctx, cudaEventRecord(ctx->ev_read[slot][buf], st));
      ctx->launches += 2;
      t_hi = t_lo - 1;
    }
    return CSD_OK;
  }

  size_t wc_chunk_rows(int steps) const { return static_cast<size_t>(steps) * (wc.part < wc.slots ? wc.part : wc.slots) * kWcRows; }
  size_t wc_chunk_bytes(int steps) const { return wc_chunk_rows(steps) * (3 * L + 2) * W * 4; }
  size_t wc_step_bytes() const { return wc_chunk_rows(1) * W * 2 + 2 * wc_chunk_bytes(1); }

  // Bytes of the wide chain kernel's chunk buffer: by the steps that a call has and the limit, and not a whole number of its steps - of two calls
  // the one of fewer rows or blocks may have room for more steps, and must not have to replace what the other uses.  halvings: where
  // memory is short, shorter chunks (same bits), down to one step.
  size_t wc_need(int halvings) const {
    const size_t step = wc_step_bytes(), all = step * (Ts < kWcMaxSteps ? Ts : kWcMaxSteps), want = all < kWcBufferBytes ? all : kWcBufferBytes;
    return (want >> halvings) > step ? want >> halvings : step;
  }
  struct WxLayout { size_t stats, epart, xll, cnt, ticket, zeroed, u, v, hsum, total; };
  WxLayout wx_layout() const {
    const size_t rows = static_cast<size_t>(wc.nb) * kTileM, G = W / 128;
    size_t off = 0;
    auto take = [&](size_t bytes) { size_t o = off; off = align_up(off + bytes, 1024); return o; };
    WxLayout l{};
    l.stats = take(rows * G * 16); l.epart = take(rows * G * (lv_min ? kCPad2 : kCPad) * 8); l.xll = take(rows * kCPad * 8);
    l.cnt = take(static_cast<size_t>(wc.nb) * 512); l.ticket = take(2 * sizeof(int));
    l.zeroed = off;              // what precedes starts at zero
    l.u = take(rows * W * 2); l.v = take(rows * W * 2); l.hsum = take(lv_min ? rows * kCPad * 4 : 0);
    l.total = off;
    return l;
  }

  // The wide chain kernel, chunk by chunk of steps (launched with a chunk's first step) and part by part of the rows: s and the
  // condition products on the slot's own stream, ahead of the chain.
  int begin_wide_chain() {
    const csd_head_desc& d = hd->d;
    ChainWs& ws = ctx->ws[slot];
    const WxLayout l = wx_layout();
    char* const xb = static_cast<char*>(ctx->wx[slot].base);
    int rc;
    if ((rc = make_tmap(ctx, &wq.tm_s, d.dtype, ctx->gm[slot].base, wc_chunk_rows(wc_most), W, W, kTileM))) return rc;
    const uint64_t lines = static_cast<uint64_t>(wc.nb) * kTileM * W / 256;      // u, v as lines of 256 elements: 32 of them a k-block
    if ((rc = make_plain_tmap(ctx, &wq.tm_u, d.dtype, xb + l.u, lines)) || (rc = make_plain_tmap(ctx, &wq.tm_v, d.dtype, xb + l.v, lines))) return rc;
    CSD_CUDA(ctx, cudaMemsetAsync(xb, 0, l.zeroed, st));
    CSD_CUDA(ctx, cudaEventRecord(ctx->ev_prep[slot], st));
    CSD_CUDA(ctx, cudaStreamWaitEvent(ctx->aux[slot], ctx->ev_prep[slot], 0));
    WcParams& p = wq.p;
    p.R = R; p.cfg = cfg; p.W = W; p.L = L; p.C = d.C; p.T = Ts; p.sample_last = sample_last; p.cfg_scale = cfg_scale;
    p.maps = hd->d_wc_maps; p.b1 = hd->b1[0]; p.b2 = hd->b2[0]; p.win = hd->win; p.bin = hd->bin; p.wout_t = hd->wout_t; p.bout = hd->bout;
    p.x_T = x_T; p.eps = eps; p.x = ws.x; p.x0 = x0; p.mu1 = mu1; p.x1 = x1; p.traj_x = traj_x; p.traj_mu = traj_mu;
    p.u = xb + l.u; p.v = xb + l.v; p.stats = reinterpret_cast<ulonglong2*>(xb + l.stats); p.epart = reinterpret_cast<ulonglong2*>(xb + l.epart);
    p.xll = reinterpret_cast<ulonglong2*>(xb + l.xll); p.cnt = reinterpret_cast<unsigned*>(xb + l.cnt); p.hsum = reinterpret_cast<float*>(xb + l.hsum);
    p.lv1 = lv1; p.half_logdet = half_logdet; p.err = ctx->d_err; p.status = ctx->d_err + 1;
    wq.t_hi = Ts;
    return CSD_OK;
  }
  int launch_wide_chunk() {
    const csd_head_desc& d = hd->d;
    ChainWs& ws = ctx->ws[slot];
    const size_t chunk = wc_chunk_bytes(wc_most);
    void* const s_chunk = ctx->gm[slot].base;
    char* const gm = static_cast<char*>(s_chunk) + wc_chunk_rows(wc_most) * W * 2;
    int* const tickets = reinterpret_cast<int*>(static_cast<char*>(ctx->wx[slot].base) + wx_layout().ticket);
    const bool f16 = d.dtype == CSD_F16, lv = lv_min != nullptr;
    cudaStream_t gst = ctx->aux[slot];
    WcParams& p = wq.p;
    WmParams m{};
    m.nkb = W / kBlockK; m.nwt = (3 * L + 2) * W / 256; m.sb = 32; m.wrow = hd->d_wc_rows; m.bias = hd->d_wc_bias; m.err = ctx->d_err;
    cudaLaunchAttribute at[2];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2; at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
    at[1].id = cudaLaunchAttributeLaunchCompletionEvent;
    at[1].val.launchCompletionEvent.event = ctx->ev_on[slot]; at[1].val.launchCompletionEvent.flags = 0;
    // (Not a cooperative launch: only the CTAs of a row block, neighbours in the grid, wait for each other, so a launch of which some groups
    // have no SM yet gets on; and a cooperative one fails under the profiler.)
    cudaLaunchConfig_t lc{};
    lc.attrs = at;
    // Beside chains that leave most of the GPU free the products take only what is left, so that the next chunk's chain finds
    // its SMs; a chain that holds most of it takes turns with them.
    const int held = wc.ctas + beside, free_pairs = (held <= ctx->num_sms / 2 ? ctx->num_sms - held : ctx->num_sms) / 2;
    // Steps per chunk: one first, because nothing overlaps its products; then twice as many each time, as far as the buffers go.
    int& n = wq.n;
    const int t_hi = wq.t_hi;
    n = n ? 2 * n : 1;
    if (t_hi <= 4) n = t_hi;      // (short schedules)
    if (n > wc_most) n = wc_most;
    if (n > t_hi) n = t_hi;
    const int t_lo = t_hi - n + 1;
    for (int i = 0; i < n; ++i) {
      p.ca[i] = sc->a[t_lo - 1 + i]; p.cb[i] = sc->b[t_lo - 1 + i];
      p.s0[i] = lv ? lv_min[t_lo - 1 + i] : sc->sigma[t_lo - 1 + i]; p.s1[i] = lv ? lv_max[t_lo - 1 + i] : 0.0f;
    }
    for (int s0 = 0; s0 < wc.slots; s0 += wc.part, ++wq.launched) {
      const int slots = wc.slots - s0 < wc.part ? wc.slots - s0 : wc.part, rows = slots * kWcRows, c = wq.launched, buf = c & 1;
      float* const mods = reinterpret_cast<float*>(gm + buf * chunk);
      if (c >= 2) CSD_CUDA(ctx, cudaStreamWaitEvent(gst, ctx->ev_read[slot][buf], 0));
      if (c >= 1) CSD_CUDA(ctx, cudaStreamWaitEvent(gst, ctx->ev_on[slot], 0));
      CSD_CUDA(ctx, cudaMemsetAsync(tickets + buf, 0, sizeof(int), gst));
      const dim3 sgrid(static_cast<unsigned>(rows), static_cast<unsigned>((n + kCondSteps - 1) / kCondSteps));
      const float* te = ws.te + static_cast<size_t>(t_lo - 1) * W;
      if (f16) cond_all_kernel<__half, 128><<<sgrid, 128, 0, gst>>>(ws.cz, te, static_cast<__half*>(s_chunk), R, cfg, W, rows, s0 * kWcRows, n);
      else cond_all_kernel<__nv_bfloat16, 128><<<sgrid, 128, 0, gst>>>(ws.cz, te, static_cast<__nv_bfloat16*>(s_chunk), R, cfg, W, rows, s0 * kWcRows, n);
      CSD_CUDA(ctx, cudaGetLastError());
      m.nst = n * slots; m.ticket = tickets + buf; m.out = mods;
      int pairs = c == 0 ? ctx->num_sms / 2 : free_pairs;
      if (pairs > m.nst * m.nwt) pairs = m.nst * m.nwt;
      lc.gridDim = dim3(static_cast<unsigned>(2 * pairs)); lc.blockDim = dim3(kMgThreads); lc.dynamicSmemBytes = kMgSmemBytes; lc.stream = gst; lc.numAttrs = 1;
      if (f16) CSD_CUDA(ctx, cudaLaunchKernelEx(&lc, wide_mods_kernel<0>, hd->Wrows, wq.tm_s, m));
      else CSD_CUDA(ctx, cudaLaunchKernelEx(&lc, wide_mods_kernel<1>, hd->Wrows, wq.tm_s, m));
      CSD_CUDA(ctx, cudaEventRecord(ctx->ev_mods[slot][buf], gst));
      CSD_CUDA(ctx, cudaStreamWaitEvent(st, ctx->ev_mods[slot][buf], 0));
      p.t_hi = t_hi; p.t_lo = t_lo; p.slot0 = s0; p.slots = slots; p.mods = mods;
      lc.gridDim = dim3(static_cast<unsigned>((wc.halves == 2 ? slots : (slots + 1) / 2) * 2 * (W / 128))); lc.blockDim = dim3(kWcThreads);
      lc.dynamicSmemBytes = wc_layout(L, lv ? kCPad2 : kCPad, wc.halves).total + 1024; lc.stream = st; lc.numAttrs = 2;
      CSD_CUDA(ctx, cudaLaunchKernelEx(&lc, wide_kernel(d.dtype, lv, wc.halves), wq.tm_u, wq.tm_v, p));
      CSD_CUDA(ctx, cudaEventRecord(ctx->ev_read[slot][buf], st));
      ctx->launches += 3;
    }
    wq.t_hi = t_lo - 1;
    return CSD_OK;
  }

  int step(int t) {
    if (gck || fcg) return CSD_OK;   // already enqueued by begin()
    if (wck) return t == wq.t_hi ? launch_wide_chunk() : static_cast<int>(CSD_OK);
    const csd_head_desc& d = hd->d;
    ChainWs& ws = ctx->ws[slot];
    cur_t = t;
    const CUtensorMap& tm_s = tm_sb[t & 1];
    const float* sf = static_cast<const float*>(sbuf[t & 1]);
    const float* uf = static_cast<const float*>(ws.u);
    const float* vf = static_cast<const float*>(ws.v);
    const csd_head::TmSet& tmw = hd->tm[(tn == 64 || pair) ? 0 : 1];   // pairs load half of each B tile per CTA
    int rc = CSD_OK;
    for (int k = 0; k < L; ++k) {
      EpiParams e = ep;
      e.h = ws.h; e.stats = ws.stats;
      const bool folded_in = fold && k >= 1;        // the block's input is a' = h (1 + scale): no modulate kernel
      const bool folded_out = fold && k + 1 < L;    // the block's last kernel also forms a' of the next block
      if (folded_in) {
        if ((rc = launch_fold(FOLD_W1, k))) return rc;
        if (folded_out) rc = launch_fold(FOLD_GATE, k);
        if (rc) return rc;
        if (folded_out) continue;
      }
      // u = LN(h)(1 + scale) + shift
      e.bias0 = hd->bsh[k]; e.bias1 = hd->bsc[k]; e.out_act = ws.u;
      // s of the first step is written by the kernel right before the first modulate kernel; every later s is older
      const int dep_mod = (k == 0 && t == T) ? 0 : W;
      if (folded_in) rc = CSD_OK;
      else if (tc && mod64) rc = launch_tc<EPI_MOD, 1, 2>(ctx, d.dtype, 64, false, st, tm_s, hd->tm[0].Wss[k], tm_s, hd->tm[0].Wss[k], W, 0, dep_mod, W, e, &tm_u_out);
      else if (tc) rc = launch_tc<EPI_MOD, 1, 2>(ctx, d.dtype, tn, pair, st, tm_s, tmw.Wss[k], tm_s, tmw.Wss[k], W, 0, dep_mod, W, e, &tm_u_out);
      else rc = launch_simt<EPI_MOD, 1, 256>(ctx, st, sf, W, static_cast<const float*>(hd->Wss[k]), W, nullptr, 0,
                                             nullptr, 0, W, e);
      if (rc) return rc;
      // v = SiLU(W1 u + b1)
      e.bias0 = hd->b1[k]; e.bias1 = nullptr; e.out_act = ws.v;
      if (folded_in) rc = CSD_OK;
      else if (tc && pair && W % 256 == 0) {
        // CTA pairs over 256 x 256 tiles: per MMA byte the pair loads half as many operand bytes as with 256 x 128
        // tiles, and the first layer (one accumulator, K = W) is the kernel bound by that feed
        const CUtensorMap& w1 = hd->tm[1].W1[k];   // 128-row boxes: each CTA of the pair loads half of the 256 rows
        rc = d.dtype == CSD_F16 ? launch_tc_t<EPI_SILU_ACT, 1, 1, 256, __half, true>(ctx, st, tm_u, w1, tm_u, w1, W, 0, 0, W, e, &tm_v_out)
                                : launch_tc_t<EPI_SILU_ACT, 1, 1, 256, __nv_bfloat16, true>(ctx, st, tm_u, w1, tm_u, w1, W, 0, 0, W, e, &tm_v_out);
      }
      else if (tc && w1_wide) {
        const CUtensorMap& w1 = hd->W1_wide[k];
        rc = d.dtype == CSD_F16 ? launch_tc_t<EPI_SILU_ACT, 1, 1, 256, __half, false>(ctx, st, tm_u, w1, tm_u, w1, W, 0, 0, W, e, &tm_v_out)
                                : launch_tc_t<EPI_SILU_ACT, 1, 1, 256, __nv_bfloat16, false>(ctx, st, tm_u, w1, tm_u, w1, W, 0, 0, W, e, &tm_v_out);
      }
      else if (tc) rc = launch_tc<EPI_SILU_ACT, 1, 1>(ctx, d.dtype, tn, pair, st, tm_u, tmw.W1[k], tm_u, tmw.W1[k], W, 0, 0, W, e, &tm_v_out);
      else rc = launch_simt<EPI_SILU_ACT, 1, 128>(ctx, st, uf, W, static_cast<const float*>(hd->W1[k]), W, nullptr, 0,
                                                  nullptr, 0, W, e);
      if (rc) return rc;
      // h += gate * (W2 v + b2).  On the tensor-core path the gate product s Wg^T comes first: it does
      // not depend on the preceding kernel (which writes v) and overlaps with it.
      e.bias0 = hd->b2[k]; e.bias1 = hd->bg[k]; e.out_act = nullptr;
      if (folded_out) rc = launch_fold(FOLD_GATE, k);
      else if (tc) {
        EpiParams g = e;
        g.bias0 = hd->bg[k]; g.bias1 = hd->b2[k];
        rc = launch_tc<EPI_GATE_RES, 2, 1>(ctx, d.dtype, tn, pair, st, tm_s, tmw.Wg[k], tm_v, tmw.W2[k], W, W, W, W, g);
      }
      else rc = launch_simt<EPI_GATE_RES, 2, 128>(ctx, st, vf, W, static_cast<const float*>(hd->W2[k]), W, sf, W,
                                                  static_cast<const float*>(hd->Wg[k]), W, W, e);
      if (rc) return rc;
    }
    EpiParams e = ep;
    e.h = ws.h; e.stats = ws.stats; e.bias0 = hd->bfsh; e.bias1 = hd->bfsc; e.wout_t = hd->wout_t; e.epart = ws.epart;
    if (d.var_out) {   // 32 output columns: eps_hat | variance parameter
      if (tc && mod64) rc = launch_tc<EPI_MODF2, 1, 2>(ctx, d.dtype, 64, false, st, tm_s, hd->tm[0].Wfss, tm_s, hd->tm[0].Wfss, W, 0, W, W, e);
      else if (tc) rc = launch_tc<EPI_MODF2, 1, 2>(ctx, d.dtype, tn, pair, st, tm_s, tmw.Wfss, tm_s, tmw.Wfss, W, 0, W, W, e);
      else rc = launch_simt<EPI_MODF2, 1, 256>(ctx, st, sf, W, static_cast<const float*>(hd->Wfss), W, nullptr, 0, nullptr,
                                               0, W, e);
    }
    else if (tc && mod64) rc = launch_tc<EPI_MODF, 1, 2>(ctx, d.dtype, 64, false, st, tm_s, hd->tm[0].Wfss, tm_s, hd->tm[0].Wfss, W, 0, W, W, e);
    else if (tc) rc = launch_tc<EPI_MODF, 1, 2>(ctx, d.dtype, tn, pair, st, tm_s, tmw.Wfss, tm_s, tmw.Wfss, W, 0, W, W, e);
    else rc = launch_simt<EPI_MODF, 1, 256>(ctx, st, sf, W, static_cast<const float*>(hd->Wfss), W, nullptr, 0, nullptr,
                                            0, W, e);
    if (rc) return rc;
    if (batch_Rin) return launch_batch(1);
    if (traj_x) {   // slot j holds x_{T-j} and mu_{T-j}: this boundary produces x_{t-1} and mu_t
      sp.traj_x = traj_x + static_cast<size_t>(T - t + 1) * R * d.C;
      sp.traj_mu = traj_mu + static_cast<size_t>(T - t) * R * d.C;
    }
    sp.a = sc->a[t - 1]; sp.b = sc->b[t - 1];
    if (lv_min) { sp.sigma = 0.0f; sp.lv_min = lv_min[t - 1]; sp.lv_max = lv_max[t - 1]; }
    else sp.sigma = sc->sigma[t - 1];
    sp.eps_t = eps + static_cast<size_t>(t - 1) * R * d.C;
    // this boundary prepares h of step t - 1 and s of step t - 2
    sp.s = t >= 3 ? sbuf[(t - 2) & 1] : nullptr;
    if (t >= 3) sp.te_next = ws.te + static_cast<size_t>(t - 3) * W;
    sp.s_b = nullptr; sp.te_b = nullptr;
    return launch_step(t > 1 ? STEP_MID : STEP_LAST);
  }
};

// Buffers of one wide chain, or of the two of a round, which find their workspaces taken first.  Where memory is short the chunks of both
// get shorter; where not one step of each can be had both run the layer kernels (wc_most 0), so that equal heads of a round
// run equal kernels, and everything is given back.
int Chain::reserve_wide_chains(csd_ctx* ctx, Chain* const* c, int n) {
  int rc = CSD_OK;
  for (int i = 0; i < n; ++i) {
    Chain& a = *c[i];
    a.sizes();
    a.wc_asked = true; a.wc_most = 0;
    if (!a.wc.slots) a.wc = wide_cut_alone(ctx, a.hd->d, a.R, a.cfg);
    if ((rc = ensure_ws(ctx, ctx->ws[a.slot], a.hd->d, a.Rh, a.R, a.Ts))) return rc;
  }
  auto drop = [&](bool exchange) {       // (what a graph holds would not come back)
    rc = sync_streams(ctx);
    for (int i = 0; i < n && !rc; ++i) {
      if (!ctx->gm[c[i]->slot].in_graph) rc = give_up(ctx, ctx->gm[c[i]->slot]);
      if (!rc && exchange && !ctx->wx[c[i]->slot].in_graph) rc = give_up(ctx, ctx->wx[c[i]->slot]);
    }
  };
  bool tried = false;
  for (int h = 0;; ++h) {
    size_t need[2], grow = 0, back = 0, whole = 0, whole_back = 0;
    bool refused = false, least = h > 0;
    for (int i = 0; i < n; ++i) {
      const int slot = c[i]->slot;
      const HostIo* io[2] = {&ctx->gm[slot], &ctx->wx[slot]};
      need[i] = c[i]->wc_need(h);
      least = least && c[i]->wc_need(h - 1) == c[i]->wc_step_bytes();
      const size_t want[2] = {need[i], c[i]->wx_layout().total};
      for (int j = 0; j < 2; ++j) {
        const size_t own = io[j]->in_graph ? 0 : io[j]->cap;
        if (want[j] > io[j]->cap) { grow += want[j]; back += own; }
        if (want[j] > io[j]->cap || own) { whole += want[j]; whole_back += own; }
      }
      refused = refused || want[0] + want[1] >= ctx->wc_refused[slot];
    }
    if (least) {                                  // one step of each was not to be had
      if (tried) drop(true);
      return rc;
    }
    if (grow && refused) {
      if (capturing(ctx)) continue;
      if (!room_for(grow, back)) {                // perhaps what one chain has and does not need serves both
        if (!room_for(whole, whole_back)) continue;
        drop(true);
        if (rc) return rc;
      }
    }
    for (int i = 0; i < n && !rc; ++i) {
      tried = tried || grow;
      rc = ensure_buffer(ctx, ctx->wx[c[i]->slot], c[i]->wx_layout().total, "the chain's exchange buffers");
      if (!rc) rc = ensure_buffer(ctx, ctx->gm[c[i]->slot], need[i], "the condition products");
    }
    if (!rc) {
      for (int i = 0; i < n; ++i) {
        const int most = c[i]->Ts < kWcMaxSteps ? c[i]->Ts : kWcMaxSteps, fit = static_cast<int>(need[i] / c[i]->wc_step_bytes());
        c[i]->wc_most = fit < most ? fit : most;
      }
      return CSD_OK;
    }
    if (rc != CSD_ERR_WORKSPACE) return rc;
    rc = CSD_OK;
    ctx->err[0] = 0;
    for (int i = 0; i < n; ++i) {
      size_t& r = ctx->wc_refused[c[i]->slot];
      const size_t all = need[i] + c[i]->wx_layout().total;
      if (all < r) r = all;
    }
    drop(false);
    if (rc) return rc;
  }
}

// The two chains of a round in the wide chain kernel: side by side in the forms that take the least time by the model, as long as they
// leave some SMs to the condition products; else one after the other.
int place_wide_chains(Chain& a, Chain& b) {
  csd_ctx* ctx = a.ctx;
  if (!wide_takes(ctx, a.hd, a.R, a.cfg, a.slot, false) || !wide_takes(ctx, b.hd, b.R, b.cfg, b.slot, false)) return CSD_OK;
  const csd_head_desc &da = a.hd->d, &db = b.hd->d;
  double best = 0.0;
  for (int i = 0; i < 4; ++i) {
    const int ha = 1 + (i & 1), hb = 1 + (i >> 1);
    if ((ha == 2 && !wide_halves(da)) || (hb == 2 && !wide_halves(db))) continue;
    const WideCut ca = wide_cut(ctx, da, a.R, a.cfg, ha), cb = wide_cut(ctx, db, b.R, b.cfg, hb);
    const int held = ca.ctas + cb.ctas;
    if (ca.part < ca.slots || cb.part < cb.slots || held > ctx->num_sms - 18) continue;
    const double ta = wide_step_us(da, ha), tb = wide_step_us(db, hb);
    // Beside another chain and its products a step of two-slot groups takes a quarter longer: 1, 2, 4, 8 x 1024, 1024 rows of each chain, 49, 79,
    // 133, 241 us where the formula has 42, 64, 108, 196.
    const double la = ta * (ha == 1 ? 1.25 : 1.0), lb = tb * (hb == 1 ? 1.25 : 1.0);
    const double us = wide_us(ctx, la > lb ? la : lb, ta * ca.ctas + tb * cb.ctas, wide_mods_sm_us(da, ca.slots) + wide_mods_sm_us(db, cb.slots), held, 0.9);
    if (best > 0.0 && us >= best) continue;
    best = us;
    a.wc = ca; b.wc = cb; a.beside = cb.ctas; b.beside = ca.ctas;
  }
  Chain* const both[2] = {&b, &a};
  if (int rc = Chain::reserve_wide_chains(ctx, both, 2)) return rc;
  if (best <= 0.0 && b.wc_most > 0) a.st = b.st;
  return CSD_OK;
}

int run_chain(csd_ctx* ctx, int slot, cudaStream_t st, const csd_head* hd, const csd_schedule* sc, int R, int cfg,
              float cfg_scale, const float* z, const float* x_T, const float* eps, int sample_last, float* x0,
              float* mu1, float* x1) {
  Chain c{ctx, slot, st, hd, sc, R, cfg, cfg_scale, z, x_T, eps, sample_last, x0, mu1, x1};
  int rc = c.begin();
  for (int t = sc->T; t >= 1 && !rc; --t) rc = c.step(t);
  return rc;
}

int check_chain_args(csd_ctx* ctx, const csd_head* hd, const csd_schedule* sc, int R, int cfg, const void* z,
                     const void* x_T, const void* eps) {
  if (!hd) return fail(ctx, CSD_ERR_INVALID_ARG, "head is null");
  if (hd->ctx != ctx) return fail(ctx, CSD_ERR_INVALID_ARG, "head belongs to another context");
  if (hd->d.var_out) return fail(ctx, CSD_ERR_UNSUPPORTED, "this head predicts its variances (var_out = 1): use the _lv calls");
  int rc = check_sched(ctx, sc, true);
  if (rc) return rc;
  if (R < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "row count %d must be >= 1", R);
  if (cfg != 0 && cfg != 1) return fail(ctx, CSD_ERR_INVALID_ARG, "cfg must be 0 or 1");
  if (!z || !x_T || !eps) return fail(ctx, CSD_ERR_INVALID_ARG, "z / x_T / eps is null");
  return CSD_OK;
}

int check_lv_args(csd_ctx* ctx, const csd_head* hd, const csd_schedule_lv* sc, int R, int cfg, const void* z,
                  const void* x_T, const void* eps) {
  if (!hd) return fail(ctx, CSD_ERR_INVALID_ARG, "head is null");
  if (hd->ctx != ctx) return fail(ctx, CSD_ERR_INVALID_ARG, "head belongs to another context");
  if (!hd->d.var_out) return fail(ctx, CSD_ERR_UNSUPPORTED, "this head has a fixed variance (var_out = 0): use the calls without _lv");
  if (!sc) return fail(ctx, CSD_ERR_INVALID_ARG, "schedule is null");
  if (sc->T < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "schedule T = %d must be >= 1", sc->T);
  if (!sc->a || !sc->b || !sc->lv_min || !sc->lv_max || !sc->tfeat) return fail(ctx, CSD_ERR_INVALID_ARG, "schedule a / b / lv_min / lv_max / tfeat is null");
  for (int t = 0; t < sc->T; ++t)
    if (!(sc->lv_min[t] <= sc->lv_max[t]) || !std::isfinite(sc->lv_min[t]) || !std::isfinite(sc->lv_max[t]))
      return fail(ctx, CSD_ERR_INVALID_ARG, "schedule needs finite lv_min[%d] <= lv_max[%d]", t, t);
  if (R < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "row count %d must be >= 1", R);
  if (cfg != 0 && cfg != 1) return fail(ctx, CSD_ERR_INVALID_ARG, "cfg must be 0 or 1");
  if (!z || !x_T || !eps) return fail(ctx, CSD_ERR_INVALID_ARG, "z / x_T / eps is null");
  return CSD_OK;
}

// A learned-variance chain: the fixed-variance chain with the log-variance bounds in place of sigma.
Chain make_lv_chain(csd_ctx* ctx, int slot, cudaStream_t st, const csd_head* hd, const csd_schedule* view,
                    const csd_schedule_lv* sc, int R, int cfg, float cfg_scale, const float* z, const float* x_T,
                    const float* eps, int sample_last, float* x0, float* mu1, float* lv1, float* half_logdet, float* x1) {
  Chain c{ctx, slot, st, hd, view, R, cfg, cfg_scale, z, x_T, eps, sample_last, x0, mu1, x1};
  c.lv_min = sc->lv_min; c.lv_max = sc->lv_max; c.lv1 = lv1; c.half_logdet = half_logdet;
  return c;
}

int accept_scan_lv(csd_ctx* ctx, cudaStream_t st, int B, int gamma, int C, const float* x0, const float* mu_q,
                   const float* lv_q, const float* hld_q, const float* mu_p, const float* lv_p, const float* hld_p,
                   const float* u, float* logratio, float* log_sigma_rows, int32_t* n_accept, uint32_t* mask) {
  return launch_short(ctx, st, accept_scan_lv_kernel, (B + 3) / 4, 128, 0, B, gamma, C, x0, mu_q, lv_q, hld_q, mu_p, lv_p, hld_p,
                      u, logratio, log_sigma_rows, n_accept, mask);
}

// The word through which the blocks of a resampling launch count the sequences that reached the cap, or null, with cap_hits
// zeroed, where launches of this context may run side by side: a capturing stream (the graph's launches run whenever and
// wherever the caller says), the per-thread stream handle (one stream for every thread).
int cap_hits_tally(csd_ctx* ctx, cudaStream_t st, int32_t* cap_hits, unsigned long long** tally) {
  cudaStreamCaptureStatus capture = cudaStreamCaptureStatusNone;
  CSD_CUDA(ctx, cudaStreamIsCapturing(st, &capture));
  *tally = capture == cudaStreamCaptureStatusNone && st != cudaStreamPerThread ? ctx->tally() : nullptr;
  if (!*tally) CSD_CUDA(ctx, cudaMemsetAsync(cap_hits, 0, sizeof(int32_t), st));
  return CSD_OK;
}

template <bool LV>
int launch_resample(csd_ctx* ctx, cudaStream_t st, ResampleParams& p) {
  if (int rc = cap_hits_tally(ctx, st, p.cap_hits, &p.tally)) return rc;
  return launch_short(ctx, st, resample_kernel<LV>, (p.B + 3) / 4, 128, 0, p);
}

int resample_lv(csd_ctx* ctx, cudaStream_t st, int B, int gamma, int C, int cap, const float* log_sigma_rows,
                const int32_t* n_accept, const float* mu_p, const float* lv_p, const float* mu_q, const float* lv_q,
                const float* xi, const float* v, float* x_new, int32_t* n_prop, uint32_t* flags, int32_t* cap_hits) {
  ResampleParams p{};
  p.B = B; p.gamma = gamma; p.C = C; p.cap = cap; p.log_sigma_rows = log_sigma_rows; p.lv_p = lv_p; p.lv_q = lv_q;
  p.n_accept = n_accept; p.mu_p = mu_p; p.mu_q = mu_q; p.xi = xi; p.v = v; p.x_new = x_new; p.n_prop = n_prop; p.flags = flags;
  p.cap_hits = cap_hits;
  return launch_resample<true>(ctx, st, p);
}

double log_sigma_term(const csd_schedule* q, const csd_schedule* p, int C) {
  double acc = 0.0;
  for (int t = 1; t < q->T; ++t) acc += std::log(static_cast<double>(q->sigma[t])) - std::log(static_cast<double>(p->sigma[t]));
  return C * acc;
}

int accept_scan(csd_ctx* ctx, cudaStream_t st, int B, int gamma, int C, double log_sigma, float sp1, float sq1,
                const float* x0, const float* mu_q, const float* mu_p, const float* u, float* logratio,
                int32_t* n_accept, uint32_t* mask, const float* offset = nullptr) {
  const double lc = log_sigma + C * (std::log(static_cast<double>(sq1)) - std::log(static_cast<double>(sp1)));
  const float inv2vp = static_cast<float>(0.5 / (static_cast<double>(sp1) * sp1));
  const float inv2vq = static_cast<float>(0.5 / (static_cast<double>(sq1) * sq1));
  return launch_short(ctx, st, accept_scan_kernel, (B + 3) / 4, 128, 0, B, gamma, C, static_cast<float>(lc), inv2vp, inv2vq, x0,
                      mu_q, mu_p, u, logratio, n_accept, mask, offset);
}

int resample(csd_ctx* ctx, cudaStream_t st, int B, int gamma, int C, int cap, double log_sigma, float sp1, float sq1,
             const int32_t* n_accept, const float* mu_p, const float* mu_q, const float* xi, const float* v,
             float* x_new, int32_t* n_prop, uint32_t* flags, int32_t* cap_hits) {
  ResampleParams p{};
  p.B = B; p.gamma = gamma; p.C = C; p.cap = cap; p.log_sigma = static_cast<float>(log_sigma); p.sp1 = sp1; p.sq1 = sq1;
  p.log_sp1 = static_cast<float>(std::log(static_cast<double>(sp1))); p.log_sq1 = static_cast<float>(std::log(static_cast<double>(sq1)));
  p.n_accept = n_accept; p.mu_p = mu_p; p.mu_q = mu_q; p.xi = xi; p.v = v; p.x_new = x_new; p.n_prop = n_prop; p.flags = flags;
  p.cap_hits = cap_hits;
  return launch_resample<false>(ctx, st, p);
}

// Target chain over the R = B gamma verified positions with the B rows of position gamma + 1 appended (Alg. 1
// obtains p_{gamma+1} from the same parallel target pass): token rows [0, R) are the verified ones, [R, R + B) the
// bonus ones; with guidance the unconditional twins follow in the same order.  The side buffer holds the gathered
// inputs and the chain's last-step outputs for all R + B rows.
struct BonusBuf {
  float *z, *x_T, *eps, *mu1, *x0;
};

size_t bonus_buf_bytes(const csd_head_desc& d, int Rt, int cfg, int T) {
  const size_t m = cfg ? 2 : 1, rt = static_cast<size_t>(Rt);
  return align_up(rt * m * d.Dz * 4, 256) + align_up(rt * d.C * 4, 256) * 3 + align_up(static_cast<size_t>(T) * rt * d.C * 4, 256);
}

// Carves the (already large enough) side buffer and enqueues the gathering copies on `st`.
int gather_bonus_inputs(csd_ctx* ctx, cudaStream_t st, const csd_head_desc& d, int R, int B, int cfg, int T,
                        const float* z, const float* x_T, const float* eps, const float* z_next,
                        const float* x_T_next, const float* eps_next, BonusBuf& bb) {
  const size_t m = cfg ? 2 : 1, Rt = static_cast<size_t>(R) + B, C = d.C, Dz = d.Dz;
  char* p = static_cast<char*>(ctx->bn.base);
  bb.z = reinterpret_cast<float*>(p); p += align_up(Rt * m * Dz * 4, 256);
  bb.x_T = reinterpret_cast<float*>(p); p += align_up(Rt * C * 4, 256);
  bb.mu1 = reinterpret_cast<float*>(p); p += align_up(Rt * C * 4, 256);
  bb.x0 = reinterpret_cast<float*>(p); p += align_up(Rt * C * 4, 256);
  bb.eps = reinterpret_cast<float*>(p);
  for (size_t h = 0; h < m; ++h) {
    CSD_CUDA(ctx, cudaMemcpyAsync(bb.z + h * Rt * Dz, z + h * R * Dz, static_cast<size_t>(R) * Dz * 4, cudaMemcpyDeviceToDevice, st));
    CSD_CUDA(ctx, cudaMemcpyAsync(bb.z + (h * Rt + R) * Dz, z_next + h * B * Dz, static_cast<size_t>(B) * Dz * 4, cudaMemcpyDeviceToDevice, st));
  }
  CSD_CUDA(ctx, cudaMemcpyAsync(bb.x_T, x_T, static_cast<size_t>(R) * C * 4, cudaMemcpyDeviceToDevice, st));
  CSD_CUDA(ctx, cudaMemcpyAsync(bb.x_T + static_cast<size_t>(R) * C, x_T_next, static_cast<size_t>(B) * C * 4, cudaMemcpyDeviceToDevice, st));
  CSD_CUDA(ctx, cudaMemcpy2DAsync(bb.eps, Rt * C * 4, eps, static_cast<size_t>(R) * C * 4, static_cast<size_t>(R) * C * 4, T, cudaMemcpyDeviceToDevice, st));
  CSD_CUDA(ctx, cudaMemcpy2DAsync(bb.eps + static_cast<size_t>(R) * C, Rt * C * 4, eps_next, static_cast<size_t>(B) * C * 4, static_cast<size_t>(B) * C * 4, T, cudaMemcpyDeviceToDevice, st));
  return CSD_OK;
}

int check_verify_dims(csd_ctx* ctx, int B, int gamma, int C) {
  if (B < 1 || gamma < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "B = %d and gamma = %d must be >= 1", B, gamma);
  if (gamma > 32) return fail(ctx, CSD_ERR_UNSUPPORTED, "gamma = %d exceeds 32", gamma);
  if (C < 1 || C > kCPad) return fail(ctx, CSD_ERR_UNSUPPORTED, "token dim C = %d must be in [1, 16]", C);
  return CSD_OK;
}

}  // namespace

// ================================================================================== C ABI
extern "C" {

int csd_create(csd_ctx** out, int device, void* cuda_stream) {
  if (!out) return CSD_ERR_INVALID_ARG;
  *out = nullptr;
  int ndev = 0;
  if (cudaGetDeviceCount(&ndev) != cudaSuccess || device < 0 || device >= ndev) {
    cudaGetLastError();
    return CSD_ERR_CUDA;
  }
  if (device >= kMaxDevices) return CSD_ERR_UNSUPPORTED;
  DeviceGuard dg(device);   // the caller's current device is put back when this call returns
  if (!dg.ok) return CSD_ERR_CUDA;
  cudaDeviceProp prop;
  if (cudaGetDeviceProperties(&prop, device) != cudaSuccess) return CSD_ERR_CUDA;
  if (prop.major != 10) return CSD_ERR_UNSUPPORTED;  // kernels are built for sm_100a only
  csd_ctx* c = new (std::nothrow) csd_ctx();
  if (!c) return CSD_ERR_WORKSPACE;
  c->device = device;
  c->num_sms = prop.multiProcessorCount;
  c->stream = static_cast<cudaStream_t>(cuda_stream);
  bool ok = true;
  // side[1] outranks side[0]: csd_round puts the longer of its two chains there, so that the chain that decides
  // the round's duration gets free SMs first and the shorter one fills the gaps
  int prio_lo = 0, prio_hi = 0;
  cudaDeviceGetStreamPriorityRange(&prio_lo, &prio_hi);
  for (int i = 0; i < 2; ++i) {
    ok = ok && cudaStreamCreateWithPriority(&c->side[i], cudaStreamNonBlocking, i == 1 ? prio_hi : prio_lo) == cudaSuccess;
    ok = ok && cudaEventCreateWithFlags(&c->ev_done[i], cudaEventDisableTiming) == cudaSuccess;
    ok = ok && cudaStreamCreateWithPriority(&c->aux[i], cudaStreamNonBlocking, prio_lo) == cudaSuccess;
    ok = ok && cudaEventCreateWithFlags(&c->ev_prep[i], cudaEventDisableTiming) == cudaSuccess;
    ok = ok && cudaEventCreateWithFlags(&c->ev_on[i], cudaEventDisableTiming) == cudaSuccess;
    for (int j = 0; j < 2; ++j)
      ok = ok && cudaEventCreateWithFlags(&c->ev_mods[i][j], cudaEventDisableTiming) == cudaSuccess &&
           cudaEventCreateWithFlags(&c->ev_read[i][j], cudaEventDisableTiming) == cudaSuccess;
  }
  ok = ok && cudaEventCreateWithFlags(&c->ev_fork, cudaEventDisableTiming) == cudaSuccess;
  ok = ok && cudaMalloc(&c->d_err, 4 * sizeof(int)) == cudaSuccess;   // [0] first failed wait, [1] non-finite value seen, [2..3] tally_cap_hits
  ok = ok && cudaMemset(c->d_err, 0, 4 * sizeof(int)) == cudaSuccess;
  void* fn = nullptr;
  cudaDriverEntryPointQueryResult qres;
  ok = ok && cudaGetDriverEntryPoint("cuTensorMapEncodeTiled", &fn, cudaEnableDefault, &qres) == cudaSuccess &&
       qres == cudaDriverEntryPointSuccess && fn != nullptr;
  if (!ok) {
    cudaGetLastError();
    csd_destroy(c);
    return CSD_ERR_CUDA;
  }
  c->encode = reinterpret_cast<EncodeTiledFn>(fn);
  *out = c;
  return CSD_OK;
}

int csd_destroy(csd_ctx* c) {
  if (!c) return CSD_ERR_INVALID_ARG;
  DeviceGuard dg(c->device);
  cudaStreamSynchronize(c->stream);
  for (int i = 0; i < 2; ++i) {
    if (c->side[i]) { cudaStreamSynchronize(c->side[i]); cudaStreamDestroy(c->side[i]); }
    if (c->aux[i]) { cudaStreamSynchronize(c->aux[i]); cudaStreamDestroy(c->aux[i]); }
    if (c->ev_prep[i]) cudaEventDestroy(c->ev_prep[i]);
    if (c->ev_on[i]) cudaEventDestroy(c->ev_on[i]);
    for (int j = 0; j < 2; ++j) {
      if (c->ev_mods[i][j]) cudaEventDestroy(c->ev_mods[i][j]);
      if (c->ev_read[i][j]) cudaEventDestroy(c->ev_read[i][j]);
    }
    if (c->ev_done[i]) cudaEventDestroy(c->ev_done[i]);
  }
  for (ChainWs& w : c->ws)
    if (w.base && w.owned) cudaFree(w.base);
  for (cudaEvent_t e : c->ev_pool) cudaEventDestroy(e);
  if (c->ev_fork) cudaEventDestroy(c->ev_fork);
  for (void* b : c->in_graphs) cudaFree(b);
  if (c->io.base) cudaFree(c->io.base);
  if (c->sp.base) cudaFree(c->sp.base);
  if (c->un.base) cudaFree(c->un.base);
  if (c->bn.base) cudaFree(c->bn.base);
  for (HostIo& b : c->gc) if (b.base) cudaFree(b.base);
  for (HostIo& b : c->gm) if (b.base) cudaFree(b.base);
  for (HostIo& b : c->wx) if (b.base) cudaFree(b.base);
  if (c->d_err) cudaFree(c->d_err);
  cudaGetLastError();
  delete c;
  return CSD_OK;
}

const char* csd_last_error(const csd_ctx* c) { return c ? c->err : "null context"; }

int64_t csd_launch_count(const csd_ctx* c) { return c ? c->launches : 0; }

int csd_sync(csd_ctx* c) {
  if (!c) return CSD_ERR_INVALID_ARG;
  CSD_DEVICE(c);
  CSD_CUDA(c, cudaStreamSynchronize(c->stream));
  int e[2] = {0, 0};
  CSD_CUDA(c, cudaMemcpy(e, c->d_err, sizeof(e), cudaMemcpyDeviceToHost));
  if (e[0] != 0 || e[1] != 0) cudaMemset(c->d_err, 0, sizeof(e));
  if (e[0] != 0) {
    static const char* const roles[] = {"?", "TMA producer", "MMA issuer", "epilogue", "wait self-test"};
    const int role = e[0] & 0xf;
    return fail(c, CSD_ERR_TIMEOUT, "a device-side bounded wait gave up: %s (role %d), site %d, iteration %d, block %d",
                roles[role <= 4 ? role : 0], role, (e[0] >> 4) & 0xf, (e[0] >> 8) & 0xffff, (e[0] >> 24) & 0x7f);
  }
  if (e[1] != 0)
    return fail(c, CSD_ERR_NONFINITE, "a non-finite value reached a step update: an activation beyond the operand "
                "format's range (65504 for CSD_F16 heads: use CSD_BF16 or CSD_F32) or non-finite inputs");
  return CSD_OK;
}

int csd_set_wait_limit(csd_ctx* c, int64_t cycles) {
  if (!c) return CSD_ERR_INVALID_ARG;
  CSD_DEVICE(c);
  CSD_CUDA(c, cudaStreamSynchronize(c->stream));
  for (int i = 0; i < 2; ++i) CSD_CUDA(c, cudaStreamSynchronize(c->side[i]));
  const long long v = cycles > 0 ? static_cast<long long>(cycles) : 4000000000ll;
  CSD_CUDA(c, cudaMemcpyToSymbol(g_wait_limit_cycles, &v, sizeof(v)));
  return CSD_OK;
}

int csd_selftest_wait_timeout(csd_ctx* c) {
  if (!c) return CSD_ERR_INVALID_ARG;
  CSD_DEVICE(c);
  wait_timeout_selftest_kernel<<<1, 32, 0, c->stream>>>(c->d_err);
  c->launches++;
  CSD_CUDA(c, cudaGetLastError());
  return CSD_OK;
}

int csd_set_chain_mode(csd_ctx* c, int mode) {
  if (!c) return CSD_ERR_INVALID_ARG;
  if (mode != CSD_CHAIN_LAYERS && mode != CSD_CHAIN_LAYERS_PLAIN && mode != CSD_CHAIN_SMALL_BATCH && mode != CSD_CHAIN_LAYER_KERNELS) return fail(c, CSD_ERR_INVALID_ARG, "chain mode %d unknown", mode);
  c->chain_mode = mode;
  return CSD_OK;
}

int csd_profile(csd_ctx* c, int enable) {
  if (!c) return CSD_ERR_INVALID_ARG;
  CSD_DEVICE(c);
  CSD_CUDA(c, cudaStreamSynchronize(c->stream));
  c->prof_on = enable != 0;
  c->prof.clear();
  c->ev_used = 0;
  return CSD_OK;
}

int csd_profile_read(csd_ctx* c, int kernel_class, int64_t* launches, double* total_ms, double* total_flops) {
  if (!c) return CSD_ERR_INVALID_ARG;
  if (!launches || !total_ms || !total_flops) return fail(c, CSD_ERR_INVALID_ARG, "null output pointer");
  if (kernel_class < 0 || kernel_class > 6) return fail(c, CSD_ERR_INVALID_ARG, "kernel class %d not in [0, 6]", kernel_class);
  CSD_DEVICE(c);
  CSD_CUDA(c, cudaStreamSynchronize(c->stream));
  for (int i = 0; i < 2; ++i) CSD_CUDA(c, cudaStreamSynchronize(c->side[i]));
  *launches = 0; *total_ms = 0.0; *total_flops = 0.0;
  for (const ProfRec& r : c->prof) {
    if (r.cls != kernel_class) continue;
    float ms = 0.0f;
    CSD_CUDA(c, cudaEventElapsedTime(&ms, r.a, r.b));
    *launches += 1; *total_ms += ms; *total_flops += r.flops;
  }
  return CSD_OK;
}

int csd_schedule_ddpm(int T, const double* beta, double tau, float* a, float* b, float* sigma) {
  if (T < 1 || !beta || !a || !b || !sigma || !(tau > 0.0)) return CSD_ERR_INVALID_ARG;
  double abar = 1.0;
  for (int t = 0; t < T; ++t) {
    if (!(beta[t] > 0.0 && beta[t] < 1.0)) return CSD_ERR_INVALID_ARG;
    const double alpha = 1.0 - beta[t];
    abar *= alpha;
    a[t] = static_cast<float>(1.0 / std::sqrt(alpha));
    b[t] = static_cast<float>(beta[t] / (std::sqrt(alpha) * std::sqrt(1.0 - abar)));
    sigma[t] = static_cast<float>(tau * std::sqrt(beta[t]));
  }
  return CSD_OK;
}

int csd_schedule_ddim(int T_full, const double* beta_full, int n_steps, const int32_t* steps, double eta, float* a,
                      float* b, float* sigma) {
  if (T_full < 1 || n_steps < 1 || !beta_full || !steps || !a || !b || !sigma) return CSD_ERR_INVALID_ARG;
  if (!(eta > 0.0 && eta <= 1.0)) return CSD_ERR_INVALID_ARG;
  std::vector<double> abar(static_cast<size_t>(T_full));
  double acc = 1.0;
  for (int t = 0; t < T_full; ++t) {
    if (!(beta_full[t] > 0.0 && beta_full[t] < 1.0)) return CSD_ERR_INVALID_ARG;
    acc *= 1.0 - beta_full[t];
    abar[t] = acc;
  }
  for (int k = 0; k < n_steps; ++k) {
    if (steps[k] < 1 || steps[k] > T_full || (k > 0 && steps[k] <= steps[k - 1])) return CSD_ERR_INVALID_ARG;
    const double cur = abar[steps[k] - 1], prv = k > 0 ? abar[steps[k - 1] - 1] : 1.0;
    // variance of q_sigma(x_prev | x_t, x0_hat); the step to x_0 would have none (prv = 1): it gets the
    // variance of the chain's own forward step around the predicted x_0
    const double sg = k > 0 ? eta * std::sqrt((1.0 - prv) / (1.0 - cur)) * std::sqrt(1.0 - cur / prv) : eta * std::sqrt(1.0 - cur);
    const double keep = k > 0 ? std::sqrt(std::fmax(0.0, 1.0 - prv - sg * sg)) : 0.0;   // weight of eps_hat towards x_t
    const double scale = std::sqrt(prv / cur);
    a[k] = static_cast<float>(scale);
    b[k] = static_cast<float>(scale * std::sqrt(1.0 - cur) - keep);
    sigma[k] = static_cast<float>(sg);
  }
  return CSD_OK;
}

int csd_log_sigma_term(int T, const float* sigma_q, const float* sigma_p, int C, double* out) {
  if (T < 1 || C < 1 || !sigma_q || !sigma_p || !out) return CSD_ERR_INVALID_ARG;
  for (int t = 0; t < T; ++t)
    if (!(sigma_q[t] > 0.0f) || !(sigma_p[t] > 0.0f)) return CSD_ERR_INVALID_ARG;
  csd_schedule q{}, p{};
  q.T = T; q.sigma = sigma_q; p.T = T; p.sigma = sigma_p;
  *out = log_sigma_term(&q, &p, C);
  return CSD_OK;
}

int csd_head_create(csd_ctx* ctx, const csd_head_desc* desc, const csd_head_weights* w, csd_head** out) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  if (!desc || !w || !out) return fail(ctx, CSD_ERR_INVALID_ARG, "desc / weights / out is null");
  *out = nullptr;
  const csd_head_desc d = *desc;
  if (d.dtype != CSD_F32 && d.dtype != CSD_BF16 && d.dtype != CSD_F16) return fail(ctx, CSD_ERR_INVALID_ARG, "dtype %d unknown", d.dtype);
  if (d.C < 1 || d.W < 1 || d.L < 1 || d.Dz < 1 || d.F < 1)
    return fail(ctx, CSD_ERR_INVALID_ARG, "head dims must be positive (C=%d W=%d L=%d Dz=%d F=%d)", d.C, d.W, d.L, d.Dz, d.F);
  if (d.C > kCPad) return fail(ctx, CSD_ERR_UNSUPPORTED, "token dim C = %d exceeds 16", d.C);
  if (d.var_out != 0 && d.var_out != 1) return fail(ctx, CSD_ERR_INVALID_ARG, "var_out = %d must be 0 or 1", d.var_out);
  if (d.W % kTileN != 0) return fail(ctx, CSD_ERR_UNSUPPORTED, "width W = %d must be a multiple of 128", d.W);
  const int kmul = d.dtype != CSD_F32 ? kBlockK : kSimtBK;
  if (d.Dz % kmul != 0) return fail(ctx, CSD_ERR_UNSUPPORTED, "Dz = %d must be a multiple of %d", d.Dz, kmul);
  const float* const* ptrs = reinterpret_cast<const float* const*>(w);
  for (size_t i = 0; i < sizeof(csd_head_weights) / sizeof(float*); ++i)
    if (!ptrs[i]) return fail(ctx, CSD_ERR_INVALID_ARG, "weight pointer #%zu is null", i);
  CSD_DEVICE(ctx);

  csd_head* h = new (std::nothrow) csd_head();
  if (!h) return fail(ctx, CSD_ERR_WORKSPACE, "out of host memory");
  h->ctx = ctx; h->d = d; h->esz = d.dtype != CSD_F32 ? 2 : 4;
  const size_t W = d.W, L = d.L, Dz = d.Dz, F = d.F, C = d.C;

  // ---- GEMM weights, packed: Wz | per block (Wss, Wg, W1, W2) | Wfss
  const size_t n_gemm = W * Dz + L * (5 * W * W) + 2 * W * W;
  std::vector<float> stage;
  try { stage.resize(n_gemm); } catch (...) { delete h; return fail(ctx, CSD_ERR_WORKSPACE, "out of host memory"); }
  std::vector<size_t> o_wss(L), o_wg(L), o_w1(L), o_w2(L);
  size_t off = 0;
  const size_t o_wz = off; memcpy(&stage[off], w->Wz, W * Dz * 4); off += W * Dz;
  // AdaLN shift and scale rows interleaved in groups of 64: 64 shift rows | 64 scale rows | ...
  auto interleave = [&](const float* shift_rows, const float* scale_rows, float* dst) {
    for (size_t j = 0; j < W / kStatCols; ++j) {
      memcpy(dst + (2 * j) * kStatCols * W, shift_rows + j * kStatCols * W, kStatCols * W * 4);
      memcpy(dst + (2 * j + 1) * kStatCols * W, scale_rows + j * kStatCols * W, kStatCols * W * 4);
    }
  };
  for (size_t k = 0; k < L; ++k) {
    const float* ada = w->Wada + k * 3 * W * W;
    o_wss[k] = off; interleave(ada, ada + W * W, &stage[off]); off += 2 * W * W;
    o_wg[k] = off; memcpy(&stage[off], ada + 2 * W * W, W * W * 4); off += W * W;
    o_w1[k] = off; memcpy(&stage[off], w->W1 + k * W * W, W * W * 4); off += W * W;
    o_w2[k] = off; memcpy(&stage[off], w->W2 + k * W * W, W * W * 4); off += W * W;
  }
  const size_t o_wfss = off; interleave(w->Wfada, w->Wfada + W * W, &stage[off]); off += 2 * W * W;

  auto bail = [&](int code, const char* what) { csd_head_destroy(h); return fail(ctx, code, "%s", what); };
  if (cudaMalloc(&h->wblob, n_gemm * h->esz) != cudaSuccess) { cudaGetLastError(); return bail(CSD_ERR_WORKSPACE, "cannot allocate device memory for the weights"); }
  if (d.dtype != CSD_F32) {
    std::vector<uint16_t> hb;
    try { hb.resize(n_gemm); } catch (...) { return bail(CSD_ERR_WORKSPACE, "out of host memory"); }
    if (d.dtype == CSD_BF16) {
      for (size_t i = 0; i < n_gemm; ++i) hb[i] = f32_to_bf16_bits(stage[i]);
    } else {
      for (size_t i = 0; i < n_gemm; ++i) { const __half hv = __float2half_rn(stage[i]); memcpy(&hb[i], &hv, 2); }
    }
    if (cudaMemcpy(h->wblob, hb.data(), n_gemm * 2, cudaMemcpyHostToDevice) != cudaSuccess) return bail(CSD_ERR_CUDA, "weight upload failed");
  } else {
    if (cudaMemcpy(h->wblob, stage.data(), n_gemm * 4, cudaMemcpyHostToDevice) != cudaSuccess) return bail(CSD_ERR_CUDA, "weight upload failed");
  }
  auto wp = [&](size_t o) { return static_cast<void*>(static_cast<char*>(h->wblob) + o * h->esz); };
  h->Wz = wp(o_wz); h->Wfss = wp(o_wfss);
  h->Wss.resize(L); h->Wg.resize(L); h->W1.resize(L); h->W2.resize(L);
  for (size_t k = 0; k < L; ++k) { h->Wss[k] = wp(o_wss[k]); h->Wg[k] = wp(o_wg[k]); h->W1[k] = wp(o_w1[k]); h->W2[k] = wp(o_w2[k]); }

  // ---- fp32 side parameters
  std::vector<float> fs;
  auto put = [&](const float* src, size_t n) { size_t o = fs.size(); fs.insert(fs.end(), src, src + n); while (fs.size() % 4) fs.push_back(0.0f); return o; };
  const size_t f_bz = put(w->bz, W), f_wt1 = put(w->Wt1, W * F), f_bt1 = put(w->bt1, W), f_wt2 = put(w->Wt2, W * W),
               f_bt2 = put(w->bt2, W), f_bin = put(w->bin, W);
  // Wout transposed to [W, 16] (or [W, 32] for a head that also predicts its variances: columns 16.. hold the
  // variance rows C..2C of Wout), zero padded; the eps columns sit where they sit in a fixed-variance head
  const size_t epw = d.var_out ? kCPad2 : kCPad;
  std::vector<float> win_pad(W * kCPad, 0.0f), wout_t(W * epw, 0.0f), bout_pad(epw, 0.0f);
  for (size_t n = 0; n < W; ++n)
    for (size_t c = 0; c < C; ++c) {
      win_pad[n * kCPad + c] = w->Win[n * C + c];
      wout_t[n * epw + c] = w->Wout[c * W + n];
      if (d.var_out) wout_t[n * epw + kCPad + c] = w->Wout[(C + c) * W + n];
    }
  for (size_t c = 0; c < C; ++c) { bout_pad[c] = w->bout[c]; if (d.var_out) bout_pad[kCPad + c] = w->bout[C + c]; }
  const size_t f_win = put(win_pad.data(), win_pad.size()), f_wout = put(wout_t.data(), wout_t.size()),
               f_bout = put(bout_pad.data(), epw);
  // (block after block, then the final pair: f32_chain_kernel walks them with one stride, as it does the matrices above)
  std::vector<size_t> f_bsh(L), f_bsc(L), f_bg(L), f_b1(L), f_b2(L);
  for (size_t k = 0; k < L; ++k) {
    f_bsh[k] = put(w->bada + k * 3 * W, W); f_bsc[k] = put(w->bada + k * 3 * W + W, W);
    f_bg[k] = put(w->bada + k * 3 * W + 2 * W, W);
    f_b1[k] = put(w->b1 + k * W, W); f_b2[k] = put(w->b2 + k * W, W);
  }
  const size_t f_bfsh = put(w->bfada, W), f_bfsc = put(w->bfada + W, W);
  // folded blocks: c1_k = W1_k (1 + bscale_k), c2_k = W1_k bshift_k + b1_k  (double accumulation, rounded once)
  const bool folded = d.dtype != CSD_F32 && L >= 2;
  // the group chain kernel folds every block, the first included
  const bool gck = d.dtype != CSD_F32 && W % 512 == 0 && W <= static_cast<size_t>(kGcMaxW) && !d.var_out;
  const size_t kfold0 = gck ? 0 : 1;      // first block that has folded weights
  std::vector<size_t> f_c1(L, 0), f_c2(L, 0);
  if (folded || gck) {
    std::vector<float> v1(W), v2(W);
    for (size_t k = kfold0; k < L; ++k) {
      const float* W1k = w->W1 + k * W * W;
      const float* bsh = w->bada + k * 3 * W;
      const float* bsc = bsh + W;
      for (size_t n = 0; n < W; ++n) {
        double a1 = 0.0, a2 = 0.0;
        for (size_t j = 0; j < W; ++j) { a1 += static_cast<double>(W1k[n * W + j]) * (1.0 + bsc[j]); a2 += static_cast<double>(W1k[n * W + j]) * bsh[j]; }
        v1[n] = static_cast<float>(a1); v2[n] = static_cast<float>(a2 + w->b1[k * W + n]);
      }
      f_c1[k] = put(v1.data(), W); f_c2[k] = put(v2.data(), W);
    }
  }
  if (cudaMalloc(&h->fblob, fs.size() * 4) != cudaSuccess) { cudaGetLastError(); return bail(CSD_ERR_WORKSPACE, "cannot allocate device memory for the parameters"); }
  if (cudaMemcpy(h->fblob, fs.data(), fs.size() * 4, cudaMemcpyHostToDevice) != cudaSuccess) return bail(CSD_ERR_CUDA, "parameter upload failed");
  float* fb = h->fblob;
  h->bz = fb + f_bz; h->Wt1 = fb + f_wt1; h->bt1 = fb + f_bt1; h->Wt2 = fb + f_wt2; h->bt2 = fb + f_bt2;
  h->win = fb + f_win; h->bin = fb + f_bin; h->wout_t = fb + f_wout; h->bout = fb + f_bout;
  h->bfsh = fb + f_bfsh; h->bfsc = fb + f_bfsc;
  h->c1.assign(L, nullptr); h->c2.assign(L, nullptr);
  if (folded || gck) for (size_t k = kfold0; k < L; ++k) { h->c1[k] = fb + f_c1[k]; h->c2[k] = fb + f_c2[k]; }
  h->bsh.resize(L); h->bsc.resize(L); h->bg.resize(L); h->b1.resize(L); h->b2.resize(L);
  for (size_t k = 0; k < L; ++k) { h->bsh[k] = fb + f_bsh[k]; h->bsc[k] = fb + f_bsc[k]; h->bg[k] = fb + f_bg[k]; h->b1[k] = fb + f_b1[k]; h->b2[k] = fb + f_b2[k]; }

  if (d.dtype != CSD_F32) {
    int rc = CSD_OK;
    for (int i = 0; i < 2 && !rc; ++i) {
      const uint32_t tn = i == 0 ? 64 : 128;   // B box rows = MMA N: tn, or 2 tn for the interleaved shift | scale rows
      csd_head::TmSet& tm = h->tm[i];
      rc = make_tmap(ctx, &tm.Wz, d.dtype, h->Wz, W, Dz, Dz, tn);
      tm.Wss.resize(L); tm.Wg.resize(L); tm.W1.resize(L); tm.W2.resize(L);
      for (size_t k = 0; k < L && !rc; ++k) {
        rc = make_tmap(ctx, &tm.Wss[k], d.dtype, h->Wss[k], 2 * W, W, W, 2 * tn);
        if (!rc) rc = make_tmap(ctx, &tm.Wg[k], d.dtype, h->Wg[k], W, W, W, tn);
        if (!rc) rc = make_tmap(ctx, &tm.W1[k], d.dtype, h->W1[k], W, W, W, tn);
        if (!rc) rc = make_tmap(ctx, &tm.W2[k], d.dtype, h->W2[k], W, W, W, tn);
      }
      if (!rc) rc = make_tmap(ctx, &tm.Wfss, d.dtype, h->Wfss, 2 * W, W, W, 2 * tn);
    }
    if (!rc && (folded || gck)) {
      // xblob: Wgs_0 .. Wgs_{L-2} | Wf_1 .. Wf_{L-1} | Wf_0 (where block 0 is folded too), each [2 W, W] in operand format
      const size_t per = 2 * W * W, nx = (2 * (L - 1) + (gck ? 1 : 0)) * per;
      auto wf_slot = [&](size_t k) { return k == 0 ? 2 * (L - 1) : L - 1 + k - 1; };
      std::vector<float> xs;
      try { xs.resize(nx); } catch (...) { return bail(CSD_ERR_WORKSPACE, "out of host memory"); }
      float *dA = nullptr, *dB = nullptr, *dC = nullptr;
      std::vector<float> f1(W * W), f2(W * W);
      bool okx = cudaMalloc(&dA, W * W * 4) == cudaSuccess && cudaMalloc(&dB, W * W * 4) == cudaSuccess && cudaMalloc(&dC, W * W * 4) == cudaSuccess;
      for (size_t k = 0; k + 1 < L && okx; ++k)     // gate of block k | scale of block k + 1
        interleave(w->Wada + k * 3 * W * W + 2 * W * W, w->Wada + (k + 1) * 3 * W * W + W * W, &xs[k * per]);
      for (size_t k = kfold0; k < L && okx; ++k) {  // W1_k Wscale_k | W1_k Wshift_k
        const float* ada = w->Wada + k * 3 * W * W;
        const dim3 grid(static_cast<unsigned>(W / 32), static_cast<unsigned>(W / 32));
        okx = okx && cudaMemcpy(dA, w->W1 + k * W * W, W * W * 4, cudaMemcpyHostToDevice) == cudaSuccess;
        okx = okx && cudaMemcpy(dB, ada + W * W, W * W * 4, cudaMemcpyHostToDevice) == cudaSuccess;
        if (okx) square_matmul_kernel<<<grid, 256>>>(dA, dB, dC, static_cast<int>(W));
        okx = okx && cudaMemcpy(f1.data(), dC, W * W * 4, cudaMemcpyDeviceToHost) == cudaSuccess;
        okx = okx && cudaMemcpy(dB, ada, W * W * 4, cudaMemcpyHostToDevice) == cudaSuccess;
        if (okx) square_matmul_kernel<<<grid, 256>>>(dA, dB, dC, static_cast<int>(W));
        okx = okx && cudaMemcpy(f2.data(), dC, W * W * 4, cudaMemcpyDeviceToHost) == cudaSuccess;
        if (okx) interleave(f1.data(), f2.data(), &xs[wf_slot(k) * per]);
      }
      if (dA) cudaFree(dA);
      if (dB) cudaFree(dB);
      if (dC) cudaFree(dC);
      if (!okx) { cudaGetLastError(); return bail(CSD_ERR_CUDA, "fused weight products failed"); }
      std::vector<uint16_t> xb;
      try { xb.resize(nx); } catch (...) { return bail(CSD_ERR_WORKSPACE, "out of host memory"); }
      if (d.dtype == CSD_BF16) { for (size_t i = 0; i < nx; ++i) xb[i] = f32_to_bf16_bits(xs[i]); }
      else { for (size_t i = 0; i < nx; ++i) { const __half hv = __float2half_rn(xs[i]); memcpy(&xb[i], &hv, 2); } }
      if (cudaMalloc(&h->xblob, nx * 2) != cudaSuccess) { cudaGetLastError(); return bail(CSD_ERR_WORKSPACE, "cannot allocate device memory for the fused weights"); }
      if (cudaMemcpy(h->xblob, xb.data(), nx * 2, cudaMemcpyHostToDevice) != cudaSuccess) return bail(CSD_ERR_CUDA, "fused weight upload failed");
      h->Wgs.resize(L); h->Wf.resize(L); h->Wgs_half.resize(L); h->Wf_half.resize(L);
      char* xbase = static_cast<char*>(h->xblob);
      for (size_t k = 0; k + 1 < L && !rc; ++k) rc = make_tmap(ctx, &h->Wgs[k], d.dtype, xbase + k * per * 2, 2 * W, W, W, 256);
      for (size_t k = 1; k < L && !rc; ++k) rc = make_tmap(ctx, &h->Wf[k], d.dtype, xbase + wf_slot(k) * per * 2, 2 * W, W, W, 256);
      for (size_t k = 0; k + 1 < L && !rc; ++k) rc = make_tmap(ctx, &h->Wgs_half[k], d.dtype, xbase + k * per * 2, 2 * W, W, W, 128);
      for (size_t k = kfold0; k < L && !rc; ++k) rc = make_tmap(ctx, &h->Wf_half[k], d.dtype, xbase + wf_slot(k) * per * 2, 2 * W, W, W, 128);
    }
    if (!rc && W % 256 == 0) {
      h->W1_wide.resize(L);
      for (size_t k = 0; k < L && !rc; ++k) rc = make_tmap(ctx, &h->W1_wide[k], d.dtype, h->W1[k], W, W, W, 256);
    }
    if (rc) { csd_head_destroy(h); return rc; }
    if (gck) {
      // tables of the group chain kernel
      std::vector<CUtensorMap> maps;
      for (size_t k = 0; k < L; ++k) { maps.push_back(h->tm[1].W1[k]); maps.push_back(h->tm[1].W2[k]); }
      std::vector<int> rows;
      auto tiles = [&](size_t row, size_t n) { for (size_t r = 0; r < n; r += 256) rows.push_back(static_cast<int>(row + r)); };
      for (size_t k = 0; k < L; ++k) tiles(5 * k * W, 3 * W);
      tiles(5 * L * W, 2 * W);
      const size_t nx = (4 * L - 2) * W;                     // rows of xblob
      for (size_t r = 0; r < nx; r += 256) rows.push_back(~static_cast<int>(r));
      tiles(0, 2 * W); tiles((5 * (L - 1) + 2) * W, W); tiles(5 * L * W, 2 * W);
      if (cudaMalloc(&h->d_gc_rows, rows.size() * sizeof(int)) != cudaSuccess ||
          cudaMalloc(&h->d_gc_maps, maps.size() * sizeof(CUtensorMap)) != cudaSuccess) { cudaGetLastError(); return bail(CSD_ERR_WORKSPACE, "cannot allocate device memory for the group-chain tables"); }
      if (cudaMemcpy(h->d_gc_rows, rows.data(), rows.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess ||
          cudaMemcpy(h->d_gc_maps, maps.data(), maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice) != cudaSuccess) return bail(CSD_ERR_CUDA, "group-chain table upload failed");
      if ((rc = make_tmap(ctx, &h->Wrows, d.dtype, h->Wss[0], (5 * L + 2) * W, W, W, kTileM)) ||
          (rc = make_tmap(ctx, &h->Wx, d.dtype, h->xblob, nx, W, W, kTileM))) { csd_head_destroy(h); return rc; }
      h->gc_ready = true;
    }
    if (wide_width(d)) {
      std::vector<CUtensorMap> maps;
      for (size_t k = 0; k < L; ++k) { maps.push_back(h->tm[0].W1[k]); maps.push_back(h->tm[0].W2[k]); }
      std::vector<int> rows;
      std::vector<float> bias;
      auto pair_rows = [&](size_t row, const float* shift, const float* scale) {     // shift | scale rows, interleaved by 64
        for (size_t r = 0; r < 2 * W; r += 256) rows.push_back(static_cast<int>(row + r));
        for (size_t j = 0; j < W; j += kStatCols) { bias.insert(bias.end(), shift + j, shift + j + kStatCols); bias.insert(bias.end(), scale + j, scale + j + kStatCols); }
      };
      for (size_t k = 0; k < L; ++k) {
        const float* ba = w->bada + k * 3 * W;
        pair_rows(5 * k * W, ba, ba + W);
        for (size_t r = 0; r < W; r += 256) rows.push_back(~static_cast<int>((5 * k + 2) * W + r));
        bias.insert(bias.end(), ba + 2 * W, ba + 3 * W);
      }
      pair_rows(5 * L * W, w->bfada, w->bfada + W);
      if (cudaMalloc(&h->d_wc_rows, rows.size() * sizeof(int)) != cudaSuccess || cudaMalloc(&h->d_wc_bias, bias.size() * sizeof(float)) != cudaSuccess ||
          cudaMalloc(&h->d_wc_maps, maps.size() * sizeof(CUtensorMap)) != cudaSuccess) { cudaGetLastError(); return bail(CSD_ERR_WORKSPACE, "cannot allocate device memory for the wide-chain tables"); }
      if (cudaMemcpy(h->d_wc_rows, rows.data(), rows.size() * sizeof(int), cudaMemcpyHostToDevice) != cudaSuccess ||
          cudaMemcpy(h->d_wc_bias, bias.data(), bias.size() * sizeof(float), cudaMemcpyHostToDevice) != cudaSuccess ||
          cudaMemcpy(h->d_wc_maps, maps.data(), maps.size() * sizeof(CUtensorMap), cudaMemcpyHostToDevice) != cudaSuccess) return bail(CSD_ERR_CUDA, "wide-chain table upload failed");
      if ((rc = make_tmap(ctx, &h->Wrows, d.dtype, h->Wss[0], (5 * L + 2) * W, W, W, kTileM))) { csd_head_destroy(h); return rc; }
    }
  }
  *out = h;
  return CSD_OK;
}

int csd_head_destroy(csd_head* h) {
  if (!h) return CSD_ERR_INVALID_ARG;
  DeviceGuard dg(h->ctx ? h->ctx->device : 0);
  if (h->ctx) {
    cudaStreamSynchronize(h->ctx->stream);
    for (int i = 0; i < 2; ++i) cudaStreamSynchronize(h->ctx->side[i]);
  }
  if (h->wblob) cudaFree(h->wblob);
  if (h->fblob) cudaFree(h->fblob);
  if (h->xblob) cudaFree(h->xblob);
  if (h->d_gc_maps) cudaFree(h->d_gc_maps);
  if (h->d_gc_rows) cudaFree(h->d_gc_rows);
  if (h->d_wc_maps) cudaFree(h->d_wc_maps);
  if (h->d_wc_rows) cudaFree(h->d_wc_rows);
  if (h->d_wc_bias) cudaFree(h->d_wc_bias);
  cudaGetLastError();
  delete h;
  return CSD_OK;
}

int csd_draft_denoise(csd_ctx* ctx, const csd_head* head, const csd_schedule* sched, int R, int cfg, float cfg_scale,
                      const float* z, const float* x_T, const float* eps, float* x0, float* mu1, float* x1) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  int rc = check_chain_args(ctx, head, sched, R, cfg, z, x_T, eps);
  if (rc) return rc;
  if (!x0 || !mu1) return fail(ctx, CSD_ERR_INVALID_ARG, "x0 / mu1 is null");
  CSD_DEVICE(ctx);
  return run_chain(ctx, 0, ctx->stream, head, sched, R, cfg, cfg_scale, z, x_T, eps, 1, x0, mu1, x1);
}

// ---------------------------------------------------------------------------------------------
// csd_draft_denoise_static: the same kernels as csd_draft_denoise, but every intermediate buffer
// lives in this one file-scope device array instead of a cudaMalloc'ed workspace.
constexpr size_t kStaticScratchBytes = size_t(8) << 20;
static __device__ __align__(256) unsigned char g_static_scratch[kStaticScratchBytes];
static void* g_static_scratch_addr[kMaxDevices] = {nullptr};   // device address of the array, per device ordinal

int csd_draft_denoise_static(csd_ctx* ctx, const csd_head* head, const csd_schedule* sched, int R, int cfg,
                             float cfg_scale, const float* z, const float* x_T, const float* eps, float* x0,
                             float* mu1, float* x1) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  int rc = check_chain_args(ctx, head, sched, R, cfg, z, x_T, eps);
  if (rc) return rc;
  if (!x0 || !mu1) return fail(ctx, CSD_ERR_INVALID_ARG, "x0 / mu1 is null");
  if (ctx->prof_on) return fail(ctx, CSD_ERR_INVALID_ARG, "csd_draft_denoise_static: switch csd_profile off first (recording creates CUDA events)");
  CSD_DEVICE(ctx);
  // Bytes the chain's intermediates need: the same layout function the growable workspaces use.  Reject before
  // anything is enqueued.
  const csd_head_desc& d = head->d;
  const size_t need = ws_layout(d, R * (cfg ? 2 : 1), R, sched->T).total;
  if (need > kStaticScratchBytes)
    return fail(ctx, CSD_ERR_WORKSPACE,
                "csd_draft_denoise_static: this call needs %zu bytes of scratch but the built-in array holds %zu "
                "(rows R=%d%s, width %d, T=%d); use csd_draft_denoise or fewer rows", need, kStaticScratchBytes, R,
                cfg ? " doubled by guidance" : "", d.W, sched->T);
  // First call on this device: look up the device address of the array (the symbol's name is only a
  // host-side stand-in and must never be handed to a kernel).
  if (!g_static_scratch_addr[ctx->device]) {
    void* p = nullptr;
    const cudaError_t e = cudaGetSymbolAddress(&p, g_static_scratch);
    if (e != cudaSuccess || !p) {
      cudaGetLastError();
      return fail(ctx, CSD_ERR_CUDA, "cudaGetSymbolAddress(static scratch) failed: %s", cudaGetErrorString(e));
    }
    g_static_scratch_addr[ctx->device] = p;
  }
  ChainWs& ws = ctx->ws[2];
  ws.base = g_static_scratch_addr[ctx->device];
  ws.cap = kStaticScratchBytes;
  ws.owned = false;                      // never freed or grown: a call that does not fit is an error
  return run_chain(ctx, 2, ctx->stream, head, sched, R, cfg, cfg_scale, z, x_T, eps, 1, x0, mu1, x1);
}

int csd_accept_scan(csd_ctx* ctx, int B, int gamma, int C, double log_sigma_term_, float sigma1_p, float sigma1_q,
                    const float* x0_q, const float* mu1_q, const float* mu1_p, const float* u, float* logratio,
                    int32_t* n_accept, uint32_t* accept_mask) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  int rc = check_verify_dims(ctx, B, gamma, C);
  if (rc) return rc;
  if (!x0_q || !mu1_q || !mu1_p || !u || !logratio || !n_accept) return fail(ctx, CSD_ERR_INVALID_ARG, "null array argument");
  if (!(sigma1_p > 0.0f) || !(sigma1_q > 0.0f)) return fail(ctx, CSD_ERR_INVALID_ARG, "sigma1 must be > 0");
  CSD_DEVICE(ctx);
  return accept_scan(ctx, ctx->stream, B, gamma, C, log_sigma_term_, sigma1_p, sigma1_q, x0_q, mu1_q, mu1_p, u, logratio,
                     n_accept, accept_mask);
}

static int verify_impl(csd_ctx* ctx, const csd_head* head_p, const csd_schedule* sched_p, const csd_schedule* sched_q,
                       int B, int gamma, int cfg, float cfg_scale, const float* z_p, const float* x_T, const float* eps,
                       const float* x0_q, const float* mu1_q, const float* u, float* logratio, int32_t* n_accept,
                       uint32_t* accept_mask, float* mu1_p, bool bonus, const float* z_next, const float* x_T_next,
                       const float* eps_next, float* x_bonus, uint32_t* taken) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  if (B < 1 || gamma < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "B = %d and gamma = %d must be >= 1", B, gamma);
  int rc = check_chain_args(ctx, head_p, sched_p, B * gamma, cfg, z_p, x_T, eps);
  if (rc) return rc;
  if ((rc = check_sched(ctx, sched_q, false))) return rc;
  if (sched_q->T != sched_p->T) return fail(ctx, CSD_ERR_SHAPE, "draft T = %d and target T = %d differ", sched_q->T, sched_p->T);
  if ((rc = check_verify_dims(ctx, B, gamma, head_p->d.C))) return rc;
  if (!x0_q || !mu1_q || !u || !logratio || !n_accept || !mu1_p) return fail(ctx, CSD_ERR_INVALID_ARG, "null array argument");
  if (bonus && (!z_next || !x_T_next || !eps_next || !x_bonus)) return fail(ctx, CSD_ERR_INVALID_ARG, "z_next / x_T_next / eps_next / x_bonus is null");
  CSD_DEVICE(ctx);
  const int R = B * gamma, C = head_p->d.C, T = sched_p->T;
  BonusBuf bb{};
  if (bonus) {
    if ((rc = ensure_buffer(ctx, ctx->bn, bonus_buf_bytes(head_p->d, R + B, cfg, T), "the bonus rows"))) return rc;
    if ((rc = gather_bonus_inputs(ctx, ctx->stream, head_p->d, R, B, cfg, T, z_p, x_T, eps, z_next, x_T_next, eps_next, bb))) return rc;
    // every row samples at the last step; only the bonus rows' samples are used
    rc = run_chain(ctx, 1, ctx->stream, head_p, sched_p, R + B, cfg, cfg_scale, bb.z, bb.x_T, bb.eps, 1, bb.x0, bb.mu1, nullptr);
    if (rc) return rc;
    CSD_CUDA(ctx, cudaMemcpyAsync(mu1_p, bb.mu1, static_cast<size_t>(R) * C * 4, cudaMemcpyDeviceToDevice, ctx->stream));
  } else {
    rc = run_chain(ctx, 1, ctx->stream, head_p, sched_p, R, cfg, cfg_scale, z_p, x_T, eps, 0, nullptr, mu1_p, nullptr);
    if (rc) return rc;
  }
  rc = accept_scan(ctx, ctx->stream, B, gamma, C, log_sigma_term(sched_q, sched_p, C), sched_p->sigma[0],
                   sched_q->sigma[0], x0_q, mu1_q, mu1_p, u, logratio, n_accept, accept_mask);
  if (rc || !bonus) return rc;
  bonus_select_kernel<<<(B * C + 255) / 256, 256, 0, ctx->stream>>>(B, C, gamma, n_accept, bb.x0 + static_cast<size_t>(R) * C, x_bonus, taken);
  ctx->launches++;
  CSD_CUDA(ctx, cudaGetLastError());
  return CSD_OK;
}

int csd_verify(csd_ctx* ctx, const csd_head* head_p, const csd_schedule* sched_p, const csd_schedule* sched_q, int B,
               int gamma, int cfg, float cfg_scale, const float* z_p, const float* x_T, const float* eps,
               const float* x0_q, const float* mu1_q, const float* u, float* logratio, int32_t* n_accept,
               uint32_t* accept_mask, float* mu1_p) {
  return verify_impl(ctx, head_p, sched_p, sched_q, B, gamma, cfg, cfg_scale, z_p, x_T, eps, x0_q, mu1_q, u, logratio,
                     n_accept, accept_mask, mu1_p, false, nullptr, nullptr, nullptr, nullptr, nullptr);
}

int csd_verify_bonus(csd_ctx* ctx, const csd_head* head_p, const csd_schedule* sched_p, const csd_schedule* sched_q, int B,
                     int gamma, int cfg, float cfg_scale, const float* z_p, const float* x_T, const float* eps,
                     const float* x0_q, const float* mu1_q, const float* u, const float* z_next, const float* x_T_next,
                     const float* eps_next, float* logratio, int32_t* n_accept, uint32_t* accept_mask, float* mu1_p,
                     float* x_bonus, uint32_t* taken) {
  return verify_impl(ctx, head_p, sched_p, sched_q, B, gamma, cfg, cfg_scale, z_p, x_T, eps, x0_q, mu1_q, u, logratio,
                     n_accept, accept_mask, mu1_p, true, z_next, x_T_next, eps_next, x_bonus, taken);
}

int csd_verify_unaligned(csd_ctx* ctx, const csd_head* head_p, const csd_schedule* sched_p, const csd_schedule* sched_q,
                         int B, int gamma, int cfg, float cfg_scale, const float* z_p, const float* x_T,
                         const float* eps_p, const float* eps_q, const float* x0_q, const float* mu1_q, const float* u,
                         float* logratio, int32_t* n_accept, uint32_t* accept_mask, float* mu1_p) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  if (B < 1 || gamma < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "B = %d and gamma = %d must be >= 1", B, gamma);
  int rc = check_chain_args(ctx, head_p, sched_p, B * gamma, cfg, z_p, x_T, eps_p);
  if (rc) return rc;
  if ((rc = check_sched(ctx, sched_q, false))) return rc;
  if (sched_q->T != sched_p->T) return fail(ctx, CSD_ERR_SHAPE, "draft T = %d and target T = %d differ", sched_q->T, sched_p->T);
  if ((rc = check_verify_dims(ctx, B, gamma, head_p->d.C))) return rc;
  if (!eps_q || !x0_q || !mu1_q || !u || !logratio || !n_accept || !mu1_p) return fail(ctx, CSD_ERR_INVALID_ARG, "null array argument");
  CSD_DEVICE(ctx);
  const int R = B * gamma, C = head_p->d.C, T = sched_p->T;
  const size_t need = static_cast<size_t>(R) * 4;
  if ((rc = ensure_buffer(ctx, ctx->un, need, "the noise terms"))) return rc;
  float* d_off = static_cast<float*>(ctx->un.base);
  rc = run_chain(ctx, 1, ctx->stream, head_p, sched_p, R, cfg, cfg_scale, z_p, x_T, eps_p, 0, nullptr, mu1_p, nullptr);
  if (rc) return rc;
  noise_norm_term_kernel<<<(R + 127) / 128, 128, 0, ctx->stream>>>(R, C, T, eps_q, eps_p, d_off);
  ctx->launches++;
  CSD_CUDA(ctx, cudaGetLastError());
  return accept_scan(ctx, ctx->stream, B, gamma, C, log_sigma_term(sched_q, sched_p, C), sched_p->sigma[0],
                     sched_q->sigma[0], x0_q, mu1_q, mu1_p, u, logratio, n_accept, accept_mask, d_off);
}

int csd_bonus_token(csd_ctx* ctx, const csd_head* head_p, const csd_schedule* sched_p, int B, int gamma, int cfg,
                    float cfg_scale, const float* z_next, const float* x_T_next, const float* eps_next,
                    const int32_t* n_accept, float* x_bonus, uint32_t* taken) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  if (gamma < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "gamma = %d must be >= 1", gamma);
  int rc = check_chain_args(ctx, head_p, sched_p, B, cfg, z_next, x_T_next, eps_next);
  if (rc) return rc;
  if (!n_accept || !x_bonus) return fail(ctx, CSD_ERR_INVALID_ARG, "n_accept / x_bonus is null");
  CSD_DEVICE(ctx);
  const int C = head_p->d.C;
  if ((rc = ensure_buffer(ctx, ctx->bn, static_cast<size_t>(2) * B * C * 4, "the bonus samples"))) return rc;
  float* d_x0 = static_cast<float*>(ctx->bn.base);
  float* d_mu = d_x0 + static_cast<size_t>(B) * C;
  // the masks live on the device, so every sequence is sampled and the selection is a kernel: no host round trip
  rc = run_chain(ctx, 1, ctx->stream, head_p, sched_p, B, cfg, cfg_scale, z_next, x_T_next, eps_next, 1, d_x0, d_mu, nullptr);
  if (rc) return rc;
  bonus_select_kernel<<<(B * C + 255) / 256, 256, 0, ctx->stream>>>(B, C, gamma, n_accept, d_x0, x_bonus, taken);
  ctx->launches++;
  CSD_CUDA(ctx, cudaGetLastError());
  return CSD_OK;
}

int csd_draft_denoise_traj(csd_ctx* ctx, const csd_head* head, const csd_schedule* sched, int R, int cfg,
                           float cfg_scale, const float* z, const float* x_T, const float* eps, float* traj_x,
                           float* traj_mu) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  int rc = check_chain_args(ctx, head, sched, R, cfg, z, x_T, eps);
  if (rc) return rc;
  if (!traj_x || !traj_mu) return fail(ctx, CSD_ERR_INVALID_ARG, "traj_x / traj_mu is null");
  CSD_DEVICE(ctx);
  const size_t slot = static_cast<size_t>(R) * head->d.C;
  const int T = sched->T;
  // the last boundary writes x_0 and mu_1 through the chain's ordinary outputs, which are the last slots
  Chain c{ctx, 0, ctx->stream, head, sched, R, cfg, cfg_scale, z, x_T, eps, 1, traj_x + T * slot,
          traj_mu + (T - 1) * slot, nullptr};
  c.traj_x = traj_x; c.traj_mu = traj_mu;
  rc = c.begin();
  for (int t = T; t >= 1 && !rc; --t) rc = c.step(t);
  return rc;
}

int csd_verify_single_path(csd_ctx* ctx, const csd_head* head_p, const csd_schedule* sched_p,
                           const csd_schedule* sched_q, int B, int gamma, int cfg, float cfg_scale, const float* z_p,
                           const float* traj_x, const float* traj_mu_q, const float* u, int steps_per_pass,
                           float* logratio, int32_t* n_accept, uint32_t* accept_mask, float* mu_p_traj) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  if (B < 1 || gamma < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "B = %d and gamma = %d must be >= 1", B, gamma);
  if (static_cast<int64_t>(B) * gamma > (1 << 24)) return fail(ctx, CSD_ERR_UNSUPPORTED, "B * gamma exceeds 2^24 rows");
  const int R = B * gamma;
  if (!traj_x || !traj_mu_q) return fail(ctx, CSD_ERR_INVALID_ARG, "traj_x / traj_mu_q is null");
  int rc = check_chain_args(ctx, head_p, sched_p, R, cfg, z_p, traj_x, traj_mu_q);
  if (rc) return rc;
  if ((rc = check_sched(ctx, sched_q, false))) return rc;
  if (sched_q->T != sched_p->T) return fail(ctx, CSD_ERR_SHAPE, "draft T = %d and target T = %d differ", sched_q->T, sched_p->T);
  if ((rc = check_verify_dims(ctx, B, gamma, head_p->d.C))) return rc;
  if (!u || !logratio || !n_accept) return fail(ctx, CSD_ERR_INVALID_ARG, "null array argument");
  if (steps_per_pass < 0) return fail(ctx, CSD_ERR_INVALID_ARG, "steps_per_pass = %d must be >= 0", steps_per_pass);
  CSD_DEVICE(ctx);
  const int T = sched_p->T, C = head_p->d.C, Rh1 = R * (cfg ? 2 : 1);
  // steps per pass: enough head rows to fill the GPU several times over, few enough to keep the workspace
  // (about 16 W bytes per head row) modest
  constexpr int kRowsPerPass = 32768;
  int tb = steps_per_pass ? steps_per_pass : (kRowsPerPass + Rh1 - 1) / Rh1;
  if (tb > T) tb = T;
  if (static_cast<int64_t>(tb) * Rh1 > (int64_t(1) << 26)) return fail(ctx, CSD_ERR_UNSUPPORTED, "pass of %d steps has too many rows", tb);
  // device side buffer: [5, T] constants | mu^p of a pass [tb R, C] | per-step terms [T, R]
  const size_t o_mu = align_up(static_cast<size_t>(5) * T * 4, 256);
  const size_t o_acc = align_up(o_mu + static_cast<size_t>(tb) * R * C * 4, 256);
  const size_t need = o_acc + static_cast<size_t>(T) * R * 4;
  cudaStream_t st = ctx->stream;
  if ((rc = ensure_buffer(ctx, ctx->sp, need, "the single-path buffers"))) return rc;
  char* base = static_cast<char*>(ctx->sp.base);
  float* d_sched = reinterpret_cast<float*>(base);
  float* d_mu = reinterpret_cast<float*>(base + o_mu);
  float* d_terms = reinterpret_cast<float*>(base + o_acc);
  {
    // per step: a_t, b_t of the target, C (log sigma_q,t - log sigma_p,t), 1 / (2 sigma_p,t^2), 1 / (2 sigma_q,t^2)
    std::vector<float> hs(static_cast<size_t>(5) * T);
    for (int t = 0; t < T; ++t) {
      const double sp = sched_p->sigma[t], sq = sched_q->sigma[t];
      hs[t] = sched_p->a[t]; hs[T + t] = sched_p->b[t];
      hs[2 * T + t] = static_cast<float>(C * (std::log(sq) - std::log(sp)));
      hs[3 * T + t] = static_cast<float>(0.5 / (sp * sp));
      hs[4 * T + t] = static_cast<float>(0.5 / (sq * sq));
    }
    // pageable source: the runtime stages it before the call returns
    CSD_CUDA(ctx, cudaMemcpyAsync(d_sched, hs.data(), hs.size() * 4, cudaMemcpyHostToDevice, st));
  }
  for (int j0 = 0; j0 < T; j0 += tb) {
    const int n = T - j0 < tb ? T - j0 : tb;
    Chain c{ctx, 1, st, head_p, sched_p, n * R, cfg, cfg_scale, z_p, nullptr, nullptr, 0, nullptr, nullptr, nullptr};
    // the target's means of this pass: into the caller's [T, R, C] array (slot j0 onwards) when it wants them
    float* pass_mu = mu_p_traj ? mu_p_traj + static_cast<size_t>(j0) * R * C : d_mu;
    c.batch_Rin = R; c.batch_j0 = j0; c.batch_traj = traj_x; c.batch_sched = d_sched; c.batch_mu = pass_mu;
    c.ws_steps = tb; c.batch_reuse = j0 > 0;
    if ((rc = c.begin())) return rc;
    if ((rc = c.step(1))) return rc;
    single_path_terms_kernel<<<(n * R + 127) / 128, 128, 0, st>>>(R, C, T, j0, n, d_sched, traj_x, traj_mu_q, pass_mu, d_terms);
    ctx->launches++;
    CSD_CUDA(ctx, cudaGetLastError());
  }
  single_path_accept_kernel<<<(B + 3) / 4, 128, 0, st>>>(B, gamma, T, d_terms, u, logratio, n_accept, accept_mask);
  ctx->launches++;
  CSD_CUDA(ctx, cudaGetLastError());
  return CSD_OK;
}

int csd_resample(csd_ctx* ctx, int B, int gamma, int C, int cap, double log_sigma_term_, float sigma1_p, float sigma1_q,
                 const int32_t* n_accept, const float* mu1_p, const float* mu1_q, const float* xi, const float* v,
                 float* x_new, int32_t* n_prop, uint32_t* flags, int32_t* cap_hits) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  int rc = check_verify_dims(ctx, B, gamma, C);
  if (rc) return rc;
  if (cap < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "cap = %d must be >= 1", cap);
  if (!n_accept || !mu1_p || !mu1_q || !xi || !v || !x_new || !n_prop || !flags || !cap_hits)
    return fail(ctx, CSD_ERR_INVALID_ARG, "null array argument");
  if (!(sigma1_p > 0.0f) || !(sigma1_q > 0.0f)) return fail(ctx, CSD_ERR_INVALID_ARG, "sigma1 must be > 0");
  CSD_DEVICE(ctx);
  return resample(ctx, ctx->stream, B, gamma, C, cap, log_sigma_term_, sigma1_p, sigma1_q, n_accept, mu1_p, mu1_q, xi, v,
                  x_new, n_prop, flags, cap_hits);
}

static int round_impl(csd_ctx* ctx, const csd_head* head_q, const csd_head* head_p, const csd_schedule* sched_q,
                      const csd_schedule* sched_p, int B, int gamma, int cfg, float cfg_scale, int cap, const float* z_q,
                      const float* z_p, const float* x_T, const float* eps, const float* u, const float* xi,
                      const float* v, float* x0, float* mu1_q, float* mu1_p, float* logratio, int32_t* n_accept,
                      uint32_t* accept_mask, float* x_new, int32_t* n_prop, uint32_t* flags, int32_t* cap_hits,
                      bool bonus, const float* z_next, const float* x_T_next, const float* eps_next, float* x_bonus,
                      uint32_t* taken) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  if (B < 1 || gamma < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "B = %d and gamma = %d must be >= 1", B, gamma);
  const int R = B * gamma;
  int rc = check_chain_args(ctx, head_q, sched_q, R, cfg, z_q, x_T, eps);
  if (rc) return rc;
  if ((rc = check_chain_args(ctx, head_p, sched_p, R, cfg, z_p, x_T, eps))) return rc;
  if (sched_q->T != sched_p->T) return fail(ctx, CSD_ERR_SHAPE, "draft T = %d and target T = %d differ", sched_q->T, sched_p->T);
  if (head_q->d.C != head_p->d.C) return fail(ctx, CSD_ERR_SHAPE, "draft C = %d and target C = %d differ", head_q->d.C, head_p->d.C);
  const int C = head_p->d.C, T = sched_p->T;
  if ((rc = check_verify_dims(ctx, B, gamma, C))) return rc;
  if (cap < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "cap = %d must be >= 1", cap);
  if (!u || !xi || !v || !x0 || !mu1_q || !mu1_p || !logratio || !n_accept || !x_new || !n_prop || !flags || !cap_hits)
    return fail(ctx, CSD_ERR_INVALID_ARG, "null array argument");
  if (bonus && (!z_next || !x_T_next || !eps_next || !x_bonus)) return fail(ctx, CSD_ERR_INVALID_ARG, "z_next / x_T_next / eps_next / x_bonus is null");
  CSD_DEVICE(ctx);
  const int Rp = bonus ? R + B : R;    // token rows of the target chain
  // workspaces first (growing one synchronises), then fork the two chains
  if ((rc = ensure_ws(ctx, ctx->ws[0], head_q->d, R * (cfg ? 2 : 1), R, sched_q->T))) return rc;
  if ((rc = ensure_ws(ctx, ctx->ws[1], head_p->d, Rp * (cfg ? 2 : 1), Rp, sched_p->T))) return rc;
  if (bonus && (rc = ensure_buffer(ctx, ctx->bn, bonus_buf_bytes(head_p->d, Rp, cfg, T), "the bonus rows"))) return rc;
  CSD_CUDA(ctx, cudaEventRecord(ctx->ev_fork, ctx->stream));
  for (int i = 0; i < 2; ++i) CSD_CUDA(ctx, cudaStreamWaitEvent(ctx->side[i], ctx->ev_fork, 0));
  // the two chains' launches are interleaved step by step so that neither stream starves
  // the chain with more work per row goes to the higher-priority stream
  const double wq = static_cast<double>(head_q->d.L) * head_q->d.W * head_q->d.W, wp = static_cast<double>(head_p->d.L) * head_p->d.W * head_p->d.W;
  const int sq = wq > wp ? 1 : 0;
  cudaStream_t st_q = ctx->side[sq], st_p = ctx->side[1 - sq];
  BonusBuf bb{};
  if (bonus && (rc = gather_bonus_inputs(ctx, st_p, head_p->d, R, B, cfg, T, z_p, x_T, eps, z_next, x_T_next, eps_next, bb))) return rc;
  Chain cq{ctx, 0, st_q, head_q, sched_q, R, cfg, cfg_scale, z_q, x_T, eps, 1, x0, mu1_q, nullptr};
  Chain cp = bonus ? Chain{ctx, 1, st_p, head_p, sched_p, Rp, cfg, cfg_scale, bb.z, bb.x_T, bb.eps, 1, bb.x0, bb.mu1, nullptr}
                   : Chain{ctx, 1, st_p, head_p, sched_p, R, cfg, cfg_scale, z_p, x_T, eps, 0, nullptr, mu1_p, nullptr};
  cq.chains = cp.chains = 2;
  if ((rc = place_wide_chains(cq, cp))) return rc;
  rc = cp.begin();
  int rc2 = cq.begin();
  for (int t = sched_p->T; t >= 1 && !rc && !rc2; --t) {
    rc = cp.step(t);
    if (!rc) rc2 = cq.step(t);
  }
  if (bonus && !rc) CSD_CUDA(ctx, cudaMemcpyAsync(mu1_p, bb.mu1, static_cast<size_t>(R) * C * 4, cudaMemcpyDeviceToDevice, st_p));
  for (int i = 0; i < 2; ++i) {
    CSD_CUDA(ctx, cudaEventRecord(ctx->ev_done[i], ctx->side[i]));
    CSD_CUDA(ctx, cudaStreamWaitEvent(ctx->stream, ctx->ev_done[i], 0));
  }
  if (rc) return rc;
  if (rc2) return rc2;
  const double ls = log_sigma_term(sched_q, sched_p, C);
  rc = accept_scan(ctx, ctx->stream, B, gamma, C, ls, sched_p->sigma[0], sched_q->sigma[0], x0, mu1_q, mu1_p, u, logratio,
                   n_accept, accept_mask);
  if (rc) return rc;
  if (bonus) {
    bonus_select_kernel<<<(B * C + 255) / 256, 256, 0, ctx->stream>>>(B, C, gamma, n_accept, bb.x0 + static_cast<size_t>(R) * C, x_bonus, taken);
    ctx->launches++;
    CSD_CUDA(ctx, cudaGetLastError());
  }
  return resample(ctx, ctx->stream, B, gamma, C, cap, ls, sched_p->sigma[0], sched_q->sigma[0], n_accept, mu1_p, mu1_q, xi,
                  v, x_new, n_prop, flags, cap_hits);
}

int csd_round(csd_ctx* ctx, const csd_head* head_q, const csd_head* head_p, const csd_schedule* sched_q,
              const csd_schedule* sched_p, int B, int gamma, int cfg, float cfg_scale, int cap, const float* z_q,
              const float* z_p, const float* x_T, const float* eps, const float* u, const float* xi, const float* v,
              float* x0, float* mu1_q, float* mu1_p, float* logratio, int32_t* n_accept, uint32_t* accept_mask,
              float* x_new, int32_t* n_prop, uint32_t* flags, int32_t* cap_hits) {
  return round_impl(ctx, head_q, head_p, sched_q, sched_p, B, gamma, cfg, cfg_scale, cap, z_q, z_p, x_T, eps, u, xi, v, x0,
                    mu1_q, mu1_p, logratio, n_accept, accept_mask, x_new, n_prop, flags, cap_hits, false, nullptr, nullptr,
                    nullptr, nullptr, nullptr);
}

int csd_round_bonus(csd_ctx* ctx, const csd_head* head_q, const csd_head* head_p, const csd_schedule* sched_q,
                    const csd_schedule* sched_p, int B, int gamma, int cfg, float cfg_scale, int cap, const float* z_q,
                    const float* z_p, const float* x_T, const float* eps, const float* u, const float* xi, const float* v,
                    const float* z_next, const float* x_T_next, const float* eps_next, float* x0, float* mu1_q,
                    float* mu1_p, float* logratio, int32_t* n_accept, uint32_t* accept_mask, float* x_new,
                    int32_t* n_prop, uint32_t* flags, int32_t* cap_hits, float* x_bonus, uint32_t* taken) {
  return round_impl(ctx, head_q, head_p, sched_q, sched_p, B, gamma, cfg, cfg_scale, cap, z_q, z_p, x_T, eps, u, xi, v, x0,
                    mu1_q, mu1_p, logratio, n_accept, accept_mask, x_new, n_prop, flags, cap_hits, true, z_next, x_T_next,
                    eps_next, x_bonus, taken);
}

// ------------------------------------------------------------------ heads that predict their variances
int csd_schedule_lv_ddpm(int T, const double* beta, double tau, float* a, float* b, float* lv_min, float* lv_max) {
  if (T < 1 || !beta || !a || !b || !lv_min || !lv_max || !(tau > 0.0)) return CSD_ERR_INVALID_ARG;
  double abar = 1.0, abar_prev = 1.0;
  for (int t = 0; t < T; ++t) {
    if (!(beta[t] > 0.0 && beta[t] < 1.0)) return CSD_ERR_INVALID_ARG;
    const double alpha = 1.0 - beta[t];
    abar_prev = abar;
    abar *= alpha;
    a[t] = static_cast<float>(1.0 / std::sqrt(alpha));
    b[t] = static_cast<float>(beta[t] / (std::sqrt(alpha) * std::sqrt(1.0 - abar)));
    lv_max[t] = static_cast<float>(std::log(beta[t]) + 2.0 * std::log(tau));
    // posterior variance beta_t (1 - abar_{t-1}) / (1 - abar_t); zero at t = 1, which borrows the value of t = 2 below
    if (t > 0) lv_min[t] = static_cast<float>(std::log(beta[t] * (1.0 - abar_prev) / (1.0 - abar)) + 2.0 * std::log(tau));
  }
  lv_min[0] = T > 1 ? lv_min[1] : lv_max[0];
  return CSD_OK;
}

int csd_draft_denoise_lv(csd_ctx* ctx, const csd_head* head, const csd_schedule_lv* sched, int R, int cfg,
                         float cfg_scale, const float* z, const float* x_T, const float* eps, float* x0, float* mu1,
                         float* lv1, float* half_logdet, float* x1) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  int rc = check_lv_args(ctx, head, sched, R, cfg, z, x_T, eps);
  if (rc) return rc;
  if (!x0 || !mu1 || !lv1 || !half_logdet) return fail(ctx, CSD_ERR_INVALID_ARG, "x0 / mu1 / lv1 / half_logdet is null");
  CSD_DEVICE(ctx);
  csd_schedule view{sched->T, sched->a, sched->b, nullptr, sched->tfeat};
  Chain c = make_lv_chain(ctx, 0, ctx->stream, head, &view, sched, R, cfg, cfg_scale, z, x_T, eps, 1, x0, mu1, lv1,
                          half_logdet, x1);
  rc = c.begin();
  for (int t = sched->T; t >= 1 && !rc; --t) rc = c.step(t);
  return rc;
}

int csd_verify_lv(csd_ctx* ctx, const csd_head* head_p, const csd_schedule_lv* sched_p, int B, int gamma, int cfg,
                  float cfg_scale, const float* z_p, const float* x_T, const float* eps, const float* x0_q,
                  const float* mu1_q, const float* lv1_q, const float* half_logdet_q, const float* u, float* logratio,
                  int32_t* n_accept, uint32_t* accept_mask, float* mu1_p, float* lv1_p, float* half_logdet_p,
                  float* log_sigma_rows) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  if (B < 1 || gamma < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "B = %d and gamma = %d must be >= 1", B, gamma);
  int rc = check_lv_args(ctx, head_p, sched_p, B * gamma, cfg, z_p, x_T, eps);
  if (rc) return rc;
  if ((rc = check_verify_dims(ctx, B, gamma, head_p->d.C))) return rc;
  if (!x0_q || !mu1_q || !lv1_q || !half_logdet_q || !u || !logratio || !n_accept || !mu1_p || !lv1_p || !half_logdet_p ||
      !log_sigma_rows)
    return fail(ctx, CSD_ERR_INVALID_ARG, "null array argument");
  CSD_DEVICE(ctx);
  csd_schedule view{sched_p->T, sched_p->a, sched_p->b, nullptr, sched_p->tfeat};
  Chain c = make_lv_chain(ctx, 1, ctx->stream, head_p, &view, sched_p, B * gamma, cfg, cfg_scale, z_p, x_T, eps, 0,
                          nullptr, mu1_p, lv1_p, half_logdet_p, nullptr);
  rc = c.begin();
  for (int t = sched_p->T; t >= 1 && !rc; --t) rc = c.step(t);
  if (rc) return rc;
  return accept_scan_lv(ctx, ctx->stream, B, gamma, head_p->d.C, x0_q, mu1_q, lv1_q, half_logdet_q, mu1_p, lv1_p,
                        half_logdet_p, u, logratio, log_sigma_rows, n_accept, accept_mask);
}

int csd_resample_lv(csd_ctx* ctx, int B, int gamma, int C, int cap, const float* log_sigma_rows, const int32_t* n_accept,
                    const float* mu1_p, const float* lv1_p, const float* mu1_q, const float* lv1_q, const float* xi,
                    const float* v, float* x_new, int32_t* n_prop, uint32_t* flags, int32_t* cap_hits) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  int rc = check_verify_dims(ctx, B, gamma, C);
  if (rc) return rc;
  if (cap < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "cap = %d must be >= 1", cap);
  if (!log_sigma_rows || !n_accept || !mu1_p || !lv1_p || !mu1_q || !lv1_q || !xi || !v || !x_new || !n_prop || !flags || !cap_hits)
    return fail(ctx, CSD_ERR_INVALID_ARG, "null array argument");
  CSD_DEVICE(ctx);
  return resample_lv(ctx, ctx->stream, B, gamma, C, cap, log_sigma_rows, n_accept, mu1_p, lv1_p, mu1_q, lv1_q, xi, v, x_new,
                     n_prop, flags, cap_hits);
}

int csd_round_lv(csd_ctx* ctx, const csd_head* head_q, const csd_head* head_p, const csd_schedule_lv* sched_q,
                 const csd_schedule_lv* sched_p, int B, int gamma, int cfg, float cfg_scale, int cap, const float* z_q,
                 const float* z_p, const float* x_T, const float* eps, const float* u, const float* xi, const float* v,
                 float* x0, float* mu1_q, float* lv1_q, float* half_logdet_q, float* mu1_p, float* lv1_p,
                 float* half_logdet_p, float* log_sigma_rows, float* logratio, int32_t* n_accept, uint32_t* accept_mask,
                 float* x_new, int32_t* n_prop, uint32_t* flags, int32_t* cap_hits) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  if (B < 1 || gamma < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "B = %d and gamma = %d must be >= 1", B, gamma);
  const int R = B * gamma;
  int rc = check_lv_args(ctx, head_q, sched_q, R, cfg, z_q, x_T, eps);
  if (rc) return rc;
  if ((rc = check_lv_args(ctx, head_p, sched_p, R, cfg, z_p, x_T, eps))) return rc;
  if (sched_q->T != sched_p->T) return fail(ctx, CSD_ERR_SHAPE, "draft T = %d and target T = %d differ", sched_q->T, sched_p->T);
  if (head_q->d.C != head_p->d.C) return fail(ctx, CSD_ERR_SHAPE, "draft C = %d and target C = %d differ", head_q->d.C, head_p->d.C);
  const int C = head_p->d.C;
  if ((rc = check_verify_dims(ctx, B, gamma, C))) return rc;
  if (cap < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "cap = %d must be >= 1", cap);
  if (!u || !xi || !v || !x0 || !mu1_q || !lv1_q || !half_logdet_q || !mu1_p || !lv1_p || !half_logdet_p || !log_sigma_rows ||
      !logratio || !n_accept || !x_new || !n_prop || !flags || !cap_hits)
    return fail(ctx, CSD_ERR_INVALID_ARG, "null array argument");
  CSD_DEVICE(ctx);
  if ((rc = ensure_ws(ctx, ctx->ws[0], head_q->d, R * (cfg ? 2 : 1), R, sched_q->T))) return rc;
  if ((rc = ensure_ws(ctx, ctx->ws[1], head_p->d, R * (cfg ? 2 : 1), R, sched_p->T))) return rc;
  CSD_CUDA(ctx, cudaEventRecord(ctx->ev_fork, ctx->stream));
  for (int i = 0; i < 2; ++i) CSD_CUDA(ctx, cudaStreamWaitEvent(ctx->side[i], ctx->ev_fork, 0));
  const double wq = static_cast<double>(head_q->d.L) * head_q->d.W * head_q->d.W, wp = static_cast<double>(head_p->d.L) * head_p->d.W * head_p->d.W;
  const int sq = wq > wp ? 1 : 0;
  csd_schedule vq{sched_q->T, sched_q->a, sched_q->b, nullptr, sched_q->tfeat}, vp{sched_p->T, sched_p->a, sched_p->b, nullptr, sched_p->tfeat};
  Chain cq = make_lv_chain(ctx, 0, ctx->side[sq], head_q, &vq, sched_q, R, cfg, cfg_scale, z_q, x_T, eps, 1, x0, mu1_q, lv1_q,
                           half_logdet_q, nullptr);
  Chain cp = make_lv_chain(ctx, 1, ctx->side[1 - sq], head_p, &vp, sched_p, R, cfg, cfg_scale, z_p, x_T, eps, 0, nullptr, mu1_p,
                           lv1_p, half_logdet_p, nullptr);
  cq.chains = cp.chains = 2;
  if ((rc = place_wide_chains(cq, cp))) return rc;
  rc = cp.begin();
  int rc2 = cq.begin();
  for (int t = sched_p->T; t >= 1 && !rc && !rc2; --t) {
    rc = cp.step(t);
    if (!rc) rc2 = cq.step(t);
  }
  for (int i = 0; i < 2; ++i) {
    CSD_CUDA(ctx, cudaEventRecord(ctx->ev_done[i], ctx->side[i]));
    CSD_CUDA(ctx, cudaStreamWaitEvent(ctx->stream, ctx->ev_done[i], 0));
  }
  if (rc) return rc;
  if (rc2) return rc2;
  rc = accept_scan_lv(ctx, ctx->stream, B, gamma, C, x0, mu1_q, lv1_q, half_logdet_q, mu1_p, lv1_p, half_logdet_p, u, logratio,
                      log_sigma_rows, n_accept, accept_mask);
  if (rc) return rc;
  return resample_lv(ctx, ctx->stream, B, gamma, C, cap, log_sigma_rows, n_accept, mu1_p, lv1_p, mu1_q, lv1_q, xi, v, x_new,
                     n_prop, flags, cap_hits);
}

// ------------------------------------------------------------------ explicit Gaussian-mixture heads
static int check_gmm(csd_ctx* ctx, const csd_gmm* m, const char* what) {
  if (!m || !m->logw || !m->mu || !m->log_sigma) return fail(ctx, CSD_ERR_INVALID_ARG, "%s mixture or one of its arrays is null", what);
  if (m->K < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "%s mixture has K = %d components", what, m->K);
  return CSD_OK;
}
static GmmView gmm_view(const csd_gmm* m) { return GmmView{m->K, m->logw, m->mu, m->log_sigma}; }

int csd_gmm_draft_sample(csd_ctx* ctx, int R, int C, const csd_gmm* q, const float* u_comp, const float* noise, float* x,
                         int32_t* comp) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  int rc = check_gmm(ctx, q, "draft");
  if (rc) return rc;
  if (R < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "row count %d must be >= 1", R);
  if (C < 1 || C > 32) return fail(ctx, CSD_ERR_UNSUPPORTED, "token dim C = %d must be in [1, 32]", C);
  if (!u_comp || !noise || !x) return fail(ctx, CSD_ERR_INVALID_ARG, "null array argument");
  CSD_DEVICE(ctx);
  return launch_short(ctx, ctx->stream, gmm_sample_kernel, (R + 3) / 4, 128, 0, R, C, gmm_view(q), u_comp, noise, x, comp);
}

int csd_gmm_verify(csd_ctx* ctx, int B, int gamma, int C, const csd_gmm* q, const csd_gmm* p, const float* x,
                   const float* u, float* logratio, int32_t* n_accept, uint32_t* accept_mask) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  int rc = check_gmm(ctx, q, "draft");
  if (rc || (rc = check_gmm(ctx, p, "target"))) return rc;
  if (B < 1 || gamma < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "B = %d and gamma = %d must be >= 1", B, gamma);
  if (gamma > 32) return fail(ctx, CSD_ERR_UNSUPPORTED, "gamma = %d exceeds 32", gamma);
  if (C < 1 || C > 32) return fail(ctx, CSD_ERR_UNSUPPORTED, "token dim C = %d must be in [1, 32]", C);
  if (!x || !u || !logratio || !n_accept) return fail(ctx, CSD_ERR_INVALID_ARG, "null array argument");
  CSD_DEVICE(ctx);
  auto kern = C <= 16 ? gmm_verify_kernel<16> : gmm_verify_kernel<32>;
  return launch_short(ctx, ctx->stream, kern, B, 32 * gamma, 0, B, gamma, C, gmm_view(q), gmm_view(p), x, u, logratio, n_accept,
                      accept_mask);
}

int csd_gmm_resample(csd_ctx* ctx, int B, int gamma, int C, int cap, const csd_gmm* q, const csd_gmm* p,
                     const int32_t* n_accept, const float* w, const float* xi, const float* v, float* x_new,
                     int32_t* n_prop, uint32_t* flags, int32_t* cap_hits) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  int rc = check_gmm(ctx, q, "draft");
  if (rc || (rc = check_gmm(ctx, p, "target"))) return rc;
  if (B < 1 || gamma < 1 || gamma > 32) return fail(ctx, B < 1 || gamma < 1 ? CSD_ERR_INVALID_ARG : CSD_ERR_UNSUPPORTED, "B = %d, gamma = %d: need B >= 1 and 1 <= gamma <= 32", B, gamma);
  if (C < 1 || C > 32) return fail(ctx, CSD_ERR_UNSUPPORTED, "token dim C = %d must be in [1, 32]", C);
  if (cap < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "cap = %d must be >= 1", cap);
  if (!n_accept || !w || !xi || !v || !x_new || !n_prop || !flags || !cap_hits) return fail(ctx, CSD_ERR_INVALID_ARG, "null array argument");
  CSD_DEVICE(ctx);
  GmmResampleParams r{B, gamma, C, cap, gmm_view(q), gmm_view(p), n_accept, w, xi, v, x_new, n_prop, flags, cap_hits, nullptr};
  if ((rc = cap_hits_tally(ctx, ctx->stream, cap_hits, &r.tally))) return rc;
  const size_t smem = gmm_resample_smem_floats(q->K, p->K, C) * 4;
  const bool fits = smem <= 48 * 1024;
  auto kern = C <= 16 ? (fits ? gmm_resample_kernel<16, true> : gmm_resample_kernel<16, false>)
                      : (fits ? gmm_resample_kernel<32, true> : gmm_resample_kernel<32, false>);
  return launch_short(ctx, ctx->stream, kern, B, 128, fits ? smem : 0, r);
}

int csd_round_host(csd_ctx* ctx, const csd_head* head_q, const csd_head* head_p, const csd_schedule* sched_q,
                   const csd_schedule* sched_p, int B, int gamma, int cfg, float cfg_scale, int cap, const float* z_q,
                   const float* z_p, const float* x_T, const float* eps, const float* u, const float* xi,
                   const float* v, float* x0, float* mu1_q, float* mu1_p, float* logratio, int32_t* n_accept,
                   uint32_t* accept_mask, float* x_new, int32_t* n_prop, uint32_t* flags, int32_t* cap_hits) {
  if (!ctx) return CSD_ERR_INVALID_ARG;
  if (!head_q || !head_p || !sched_q || !sched_p) return fail(ctx, CSD_ERR_INVALID_ARG, "head / schedule is null");
  if (B < 1 || gamma < 1 || cap < 1) return fail(ctx, CSD_ERR_INVALID_ARG, "B, gamma, cap must be >= 1");
  if (!z_q || !z_p || !x_T || !eps || !u || !xi || !v || !x0 || !mu1_q || !mu1_p || !logratio || !n_accept || !x_new ||
      !n_prop || !flags || !cap_hits)
    return fail(ctx, CSD_ERR_INVALID_ARG, "null array argument");
  if (sched_q->T < 1 || sched_q->T != sched_p->T) return fail(ctx, CSD_ERR_SHAPE, "schedules disagree on T");
  CSD_DEVICE(ctx);
  const size_t R = static_cast<size_t>(B) * gamma, Rh = R * (cfg ? 2 : 1), C = head_p->d.C, T = sched_p->T;
  struct Item { const void* src; void* dst; size_t bytes; size_t off; bool in; };
  Item items[] = {
      {z_q, nullptr, Rh * head_q->d.Dz * 4, 0, true}, {z_p, nullptr, Rh * head_p->d.Dz * 4, 0, true},
      {x_T, nullptr, R * C * 4, 0, true},             {eps, nullptr, T * R * C * 4, 0, true},
      {u, nullptr, R * 4, 0, true},                   {xi, nullptr, static_cast<size_t>(B) * cap * C * 4, 0, true},
      {v, nullptr, static_cast<size_t>(B) * cap * 4, 0, true},
      {nullptr, x0, R * C * 4, 0, false},             {nullptr, mu1_q, R * C * 4, 0, false},
      {nullptr, mu1_p, R * C * 4, 0, false},          {nullptr, logratio, R * 4, 0, false},
      {nullptr, n_accept, static_cast<size_t>(B) * 4, 0, false},
      {nullptr, accept_mask, static_cast<size_t>(B) * 4, 0, false},
      {nullptr, x_new, static_cast<size_t>(B) * C * 4, 0, false},
      {nullptr, n_prop, static_cast<size_t>(B) * 4, 0, false}, {nullptr, flags, static_cast<size_t>(B) * 4, 0, false},
      {nullptr, cap_hits, 4, 0, false}};
  size_t total = 0;
  for (Item& it : items) { it.off = total; total = align_up(total + it.bytes, 256); }
  if (int rc = ensure_buffer(ctx, ctx->io, total, "the host-call mirrors")) return rc;
  char* base = static_cast<char*>(ctx->io.base);
  auto dp = [&](int i) { return base + items[i].off; };
  for (int i = 0; i < 7; ++i) CSD_CUDA(ctx, cudaMemcpyAsync(dp(i), items[i].src, items[i].bytes, cudaMemcpyHostToDevice, ctx->stream));
  CSD_CUDA(ctx, cudaMemsetAsync(dp(13), 0, items[13].bytes, ctx->stream));  // x_new: rows that are not resampled read 0
  int rc = csd_round(ctx, head_q, head_p, sched_q, sched_p, B, gamma, cfg, cfg_scale, cap, (const float*)dp(0),
                     (const float*)dp(1), (const float*)dp(2), (const float*)dp(3), (const float*)dp(4),
                     (const float*)dp(5), (const float*)dp(6), (float*)dp(7), (float*)dp(8), (float*)dp(9), (float*)dp(10),
                     (int32_t*)dp(11), (uint32_t*)dp(12), (float*)dp(13), (int32_t*)dp(14), (uint32_t*)dp(15),
                     (int32_t*)dp(16));
  if (rc) return rc;
  for (int i = 7; i < 17; ++i)
    if (items[i].dst) CSD_CUDA(ctx, cudaMemcpyAsync(items[i].dst, dp(i), items[i].bytes, cudaMemcpyDeviceToHost, ctx->stream));
  return csd_sync(ctx);
}

}  // extern "C"
