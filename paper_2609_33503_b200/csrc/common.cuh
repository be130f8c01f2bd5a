// Shared host/device helpers of the RelaxKV CUDA library (sm_100a).
#pragma once

#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <atomic>
#ifdef RELAXKV_NVTX
#include <nvtx3/nvToolsExt.h>
#endif

#include "relaxkv.h"

namespace relaxkv {

// ---- device status word -----------------------------------------------------------------
// One int4 per device: {status, kernel id, block, value}.  Kernels record the first problem they
// see with an atomic compare-and-swap and carry on without touching the offending data.
struct DeviceStatus {
  int status;
  int kernel;
  int block;
  int v0;
  int v1;
};

// Per-device values that are looked up once (defined in api.cu).  The lookups are idempotent, so the caches are
// plain atomics: two host threads that race on a first call both store the same value.
constexpr int kMaxDevices = 64;
DeviceStatus* status_word();             // device address of the status word of the current device; NULL on error
int sm_count_of_current_device();        // multiprocessors of the current device; 0 on error

// Optional NVTX ranges, one per C-ABI call and per kernel launch, so that a timeline taken of a caller's process
// can be attributed to the steps of Algorithm 1.  Compiled in with -DRELAXKV_NVTX (build.py: RELAXKV_NVTX=1).
#ifdef RELAXKV_NVTX
struct NvtxRange {
  explicit NvtxRange(const char* name) { nvtxRangePushA(name); }
  ~NvtxRange() { nvtxRangePop(); }
};
#define RELAXKV_RANGE_CAT2(a, b) a##b
#define RELAXKV_RANGE_CAT(a, b) RELAXKV_RANGE_CAT2(a, b)
#define RELAXKV_RANGE(name) ::relaxkv::NvtxRange RELAXKV_RANGE_CAT(relaxkv_nvtx_range_, __LINE__)(name)
#else
#define RELAXKV_RANGE(name) do { } while (0)
#endif

enum KernelId : int {
  KID_SETS = 1, KID_SELECT = 2, KID_SCORE = 3, KID_GATHER = 4, KID_SCATTER = 5,
  KID_ATTN_SIMT = 6, KID_ATTN_SM100 = 7, KID_SCORE_SM100 = 8, KID_GEMM_SM100 = 9, KID_DENSE = 10
};

__device__ __forceinline__ void report(DeviceStatus* st, int status, int kernel, int v0, int v1) {
  if (atomicCAS(&st->status, 0, status) == 0) {
    st->kernel = kernel;
    st->block = (int)blockIdx.x;
    st->v0 = v0;
    st->v1 = v1;
  }
}

// ---- host-side checks -------------------------------------------------------------------
inline bool aligned16(const void* p) { return (reinterpret_cast<uintptr_t>(p) & 15u) == 0; }

inline relaxkv_status check_shape(const relaxkv_shape* s) {
  if (!s || !s->h_ctx_len) return RELAXKV_ERR_INVALID_ARG;
  if (s->n_req < 1 || s->n_q_heads < 1 || s->n_kv_heads < 1) return RELAXKV_ERR_INVALID_ARG;
  if (s->n_q_heads % s->n_kv_heads != 0) return RELAXKV_ERR_INVALID_ARG;
  if (s->head_dim != 64 && s->head_dim != 128) return RELAXKV_ERR_UNSUPPORTED_SHAPE;
  if (s->n_q_heads / s->n_kv_heads > 16) return RELAXKV_ERR_UNSUPPORTED_SHAPE;
  if (s->n_req > 64) return RELAXKV_ERR_UNSUPPORTED_SHAPE;   // per-request scalars travel by value
  for (int b = 0; b < s->n_req; ++b)
    if (s->h_ctx_len[b] < 1) return RELAXKV_ERR_INVALID_ARG;
  if (!(s->softmax_scale > 0.f)) return RELAXKV_ERR_INVALID_ARG;
  return RELAXKV_OK;
}

inline relaxkv_status check_cache(const relaxkv_shape* s, const relaxkv_cache_view* c, bool need_v) {
  if (!c || !c->k || (need_v && !c->v) || !c->h_req_token_offset) return RELAXKV_ERR_INVALID_ARG;
  if (!aligned16(c->k) || (need_v && !aligned16(c->v))) return RELAXKV_ERR_INVALID_ARG;
  if (c->token_stride < s->head_dim || c->head_stride < s->head_dim) return RELAXKV_ERR_INVALID_ARG;
  if ((c->token_stride % 8) || (c->head_stride % 8)) return RELAXKV_ERR_INVALID_ARG;
  for (int b = 0; b < s->n_req; ++b)
    if (c->h_req_token_offset[b] < 0) return RELAXKV_ERR_INVALID_ARG;
  return RELAXKV_OK;
}

inline relaxkv_status cuda_ok(cudaError_t e) { return e == cudaSuccess ? RELAXKV_OK : RELAXKV_ERR_CUDA; }
inline relaxkv_status launch_ok() { return cuda_ok(cudaGetLastError()); }

inline size_t align_up(size_t x, size_t a) { return (x + a - 1) / a * a; }

// ---- chained launches (programmatic dependent launch) ------------------------------------
// The kernels of this library follow one another on a stream, many of them a few microseconds long, and between two of
// them the device drains, launches and ramps up again: 1.5 to 2.5 us each (8 layers of a query pass over 8K of context, 13
// launches per layer: 1609 us with plain launches of more than eight rows, 1539 us chained; the schedule of a repair and
// the loop around it 1 to 3 %).  Launched with the programmatic-serialization attribute, the next
// kernel's blocks become resident as soon as every block of the current one has called griddep_launch(); they may do
// whatever does not depend on earlier kernels (set-up, prefetching their weights into L2) and then block in griddep_wait()
// until the earlier kernels have completed and their writes are visible.  Rules kept by every kernel that is launched
// this way: nothing written by another kernel is read, and nothing at all is written, before griddep_wait(); everything
// read from global memory, index lists and data alike, is read through plain pointers (no const __restrict__, no __ldg: the
// compiler may move a read-only load up past the wait, which orders ordinary memory accesses alone); every
// block executes griddep_wait() (so a kernel never completes before its predecessors).  A kernel that takes tensor memory
// calls griddep_launch() only after it has got it: every block then holds its share before a later kernel's block can ask
// for some on the same SM.  Short kernels of a few blocks call griddep_launch() first thing, the tensor-core kernels of many blocks when
// a block is through with its work, behind a block barrier: the first thread that calls it speaks for its block, and with the
// call in front of the barrier the warps that had nothing to do let the next kernels come at once.  Their blocks then crowd onto the SMs that
// the first finished blocks leave (40 requests of up to 5 K, gather and attention 49.7 us, now 39; scoring one 16 K layer
// 65.9 / 62.9, a query pass over 8 K 1383 / 1336).
// Both instructions do nothing in a kernel that was launched the plain way.
__device__ __forceinline__ void griddep_wait() { asm volatile("griddepcontrol.wait;" ::: "memory"); }
__device__ __forceinline__ void griddep_launch() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }

bool chained_launch_enabled();           // process-wide switch (relaxkv_set_chained_launch), on by default

// cluster > 1: the grid's x dimension is made of clusters of that many blocks (grid.x is a multiple of it).
template <typename... KArgs, typename... Args>
inline cudaError_t launch_chained_clusters(int cluster, void (*kernel)(KArgs...), dim3 grid, dim3 block,
                                           size_t smem, cudaStream_t stream, Args&&... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = grid;
  cfg.blockDim = block;
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = chained_launch_enabled() ? 1 : 0;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = (unsigned)cluster; attr[1].val.clusterDim.y = 1; attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cluster > 1 ? 2 : 1;
  const cudaError_t e = cudaLaunchKernelEx(&cfg, kernel, static_cast<KArgs>(args)...);
  if (e != cudaSuccess) (void)cudaGetLastError();      // reported by the return value: not a second time by a later call's launch_ok()
  return e;
}

template <typename... KArgs, typename... Args>
inline cudaError_t launch_chained(void (*kernel)(KArgs...), dim3 grid, dim3 block, size_t smem, cudaStream_t stream,
                                  Args&&... args) {
  return launch_chained_clusters(1, kernel, grid, block, smem, stream, static_cast<Args&&>(args)...);
}

// Up to this many requests have their per-request scalars passed by value in kernel parameters.
constexpr int kMaxReqInline = 64;

// Per-request scalars a kernel needs, by value (small batches) - avoids any host->device copy.
struct ReqTable {
  int n_req;
  int ctx_len[kMaxReqInline];
  int q_len[kMaxReqInline];
  int q_cu[kMaxReqInline + 1];      // prefix of q_len
  long long ctx_cu[kMaxReqInline + 1];  // prefix of ctx_len
  long long tok_off[kMaxReqInline];     // cache token offset
  int k[kMaxReqInline];
  int k_cu[kMaxReqInline + 1];
  int bound_a[kMaxReqInline];       // call-specific host bound (e.g. max targets)
  int bound_b[kMaxReqInline];       // call-specific host bound (e.g. max ctx)
  int tile_cu[kMaxReqInline + 1];   // call-specific prefix (e.g. q tiles)
};

// Fills the shape-derived fields of a ReqTable (host).
inline void fill_req_table(ReqTable& t, const relaxkv_shape* s, const relaxkv_cache_view* c, const int32_t* h_k) {
  t.n_req = s->n_req;
  t.q_cu[0] = 0; t.ctx_cu[0] = 0; t.k_cu[0] = 0; t.tile_cu[0] = 0;
  for (int b = 0; b < s->n_req; ++b) {
    t.ctx_len[b] = s->h_ctx_len[b];
    t.q_len[b] = s->h_q_len ? s->h_q_len[b] : 0;
    t.q_cu[b + 1] = t.q_cu[b] + t.q_len[b];
    t.ctx_cu[b + 1] = t.ctx_cu[b] + t.ctx_len[b];
    t.tok_off[b] = c ? c->h_req_token_offset[b] : 0;
    t.k[b] = h_k ? h_k[b] : 0;
    t.k_cu[b + 1] = t.k_cu[b] + t.k[b];
    t.bound_a[b] = 0; t.bound_b[b] = 0; t.tile_cu[b + 1] = 0;
  }
}

// ---- workspace layout -------------------------------------------------------------------
// Calls are stream-ordered, so the regions of different calls overlap.
constexpr int kScoreSplitsMax = 64;   // key-range splits of the scoring passes (grid.z), at most
constexpr int kScoreSms = 148;        // SMs the splits are chosen for (a workspace size does not depend on the device asked)
constexpr int kScoreCtasMax = 32 * kScoreSms;   // CTAs of a scoring pass up to which its key range is split further
constexpr int kScoreMaxRows = 640;    // query rows (token x head-in-group) resident per scoring CTA
constexpr int kScoreTokBox = 8;       // query tokens per TMA box of the scoring kernel
constexpr int kCtxPadRows = 128;      // zero rows after the materialised context
// (target rows) x (context splits) the split workspace holds: 2048, and with few heads as many as 32 MB take, twice the context at most.
constexpr int kSplitRowsCap = 2048;
inline long long split_rows_cap(const relaxkv_shape* s) {
  long long sum_t = 0;
  for (int b = 0; b < s->n_req; ++b) sum_t += s->h_ctx_len[b];
  const long long fit = (32ll << 20) / ((long long)s->n_q_heads * s->head_dim * 4), twice = 2 * sum_t;
  const long long rows = fit < twice ? fit : twice;
  return rows > kSplitRowsCap ? rows : kSplitRowsCap;
}
constexpr int kMaxCtxSplits = 32;

constexpr int kScoreLayersPerLaunch = 48;   // layers scored by one launch (their tensor maps travel as parameters)

// Query-row blocks a request needs so that each block's rows fit resident (scoring kernel).
inline int score_blocks(int q_len, int group) {
  const int max_tok = kScoreMaxRows / group / kScoreTokBox * kScoreTokBox;
  return q_len > 0 ? (q_len + max_tok - 1) / max_tok : 0;
}

// Most key-range splits a launch of `layers` layers may take, by the query rows alone (the choice itself is not monotone in
// the context).  A workspace has room for that many, so a shorter context never needs more workspace than a longer one.
inline int score_splits_most(long long units_times_heads, int layers) {
  const long long per = units_times_heads * layers, most = per > 0 ? kScoreCtasMax / per : 1;
  return most < 1 ? 1 : (most > kScoreSplitsMax ? kScoreSplitsMax : (int)most);
}

// Key-range splits for a launch that scores `layers` layers at once (one CTA per SM): the count with the least rounds x longest
// CTA.  A CTA takes start + 128-key tiles x 128-row chunks of a tile x item, start and item being what it spends before its first
// product and per product of 128 x 128 (about 4 and 0.75 us, here in quarters of a us); a round is the time of the longest CTA on
// all SMs, and the rounds are those that all CTAs' time fills.  With at least two
// waves whatever the size, a 16K layer of 256 rows ran in 1.7 waves of four tiles per CTA: its scoring and schedule took 76 us,
// 70 in one wave; the 32K pass of a query of 128 rows 60 us per layer, now 57.
inline int score_splits(const relaxkv_shape* s, int layers) {
  const int group = s->n_q_heads / s->n_kv_heads;
  struct { int blocks, tiles, chunks; } req[kMaxReqInline];
  int n = 0, tiles = 1;
  long long units = 0;
  for (int b = 0; b < s->n_req; ++b) {
    const int q = s->h_q_len ? s->h_q_len[b] : 0, nb = score_blocks(q, group);
    if (nb == 0) continue;
    units += nb;
    const int tok = ((q + nb - 1) / nb + kScoreTokBox - 1) / kScoreTokBox * kScoreTokBox;
    req[n].blocks = nb;
    req[n].chunks = ((tok < q ? tok : q) * group + 127) / 128;
    req[n].tiles = (s->h_ctx_len[b] + 127) / 128;
    if (req[n].tiles > tiles) tiles = req[n].tiles;
    ++n;
  }
  const long long copies = (long long)s->n_kv_heads * layers;
  int best = 1;
  long long best_cost = 0;
  const int most = units > 0 ? score_splits_most(units * s->n_kv_heads, layers) : 1;
  for (int ns = 1; ns <= most && ns <= tiles; ++ns) {
    long long all = 0, longest = 1;
    const double inv = 1.0 / ns;                             // (a division per request and count was most of this function's time)
    for (int i = 0; i < n; ++i) {
      const int per = (int)((req[i].tiles + ns - 1) * inv + 1e-6);
      const long long cta = 16 + 3ll * req[i].chunks * per;
      all += cta * (req[i].tiles < ns ? req[i].tiles : ns) * req[i].blocks;      // the other splits of a short request are empty
      if (cta > longest) longest = cta;
    }
    const long long round = kScoreSms * longest, cost = (all * copies + round - 1) / round * longest;
    if (ns == 1 || cost < best_cost) { best_cost = cost; best = ns; }
  }
  return best;
}

struct WsLayout {
  // attention: materialised mixed context K~ / V~  [ctx_rows_cap, H_kv, D] bf16
  size_t kctx, vctx; long long ctx_rows_cap;
  // explicit-list attention: limit [sumT] i32 | fresh_row [sumT] i32
  size_t list_limit, list_fresh;
  // context split across blocks (few targets): partial O [split_rows_cap, H, D] f32 | partial lse [split_rows_cap, H] f32
  size_t split_o, split_lse;
  size_t refused;           // [kMaxReqInline] i32: requests that the attention kernel refuses
  // scoring (per launch of Lc <= kScoreLayersPerLaunch layers): lse [Lc, H, sumQ] f32 |
  // part [Lc, 2*n_splits, H, sumQ] float2 | colpart [Lc, 2*H_kv*max_blocks, sumT] f32
  size_t lse, part, colpart;
  // sets: counts [B + L*B] i32
  size_t counts;
  size_t total;
};

inline WsLayout ws_layout(const relaxkv_shape* s, int n_layers) {
  WsLayout w{};
  long long sum_t = 0, sum_q = 0;
  for (int b = 0; b < s->n_req; ++b) { sum_t += s->h_ctx_len[b]; sum_q += s->h_q_len ? s->h_q_len[b] : 0; }
  const size_t row_bytes = (size_t)s->n_kv_heads * s->head_dim * 2;
  w.ctx_rows_cap = sum_t + kCtxPadRows;
  size_t a = 0;
  w.kctx = a; a = align_up(a + (size_t)w.ctx_rows_cap * row_bytes, 1024);
  w.vctx = a; a = align_up(a + (size_t)w.ctx_rows_cap * row_bytes, 1024);
  w.list_limit = a; a = align_up(a + (size_t)sum_t * 4, 256);
  w.list_fresh = a; a = align_up(a + (size_t)sum_t * 4, 256);
  w.split_o = a; a = align_up(a + (size_t)split_rows_cap(s) * s->n_q_heads * s->head_dim * 4, 256);
  w.split_lse = a; a = align_up(a + (size_t)split_rows_cap(s) * s->n_q_heads * 4, 256);
  w.refused = a; a = align_up(a + kMaxReqInline * 4, 256);
  size_t attn_total = a;
  a = 0;
  const int lc_max = n_layers < kScoreLayersPerLaunch ? n_layers : kScoreLayersPerLaunch;
  w.lse = a; a = align_up(a + (size_t)lc_max * s->n_q_heads * sum_q * 4, 256);
  int max_blocks = 1, tiles = 1;
  long long units = 0;
  for (int b = 0; b < s->n_req; ++b) {
    const int nb = score_blocks(s->h_q_len ? s->h_q_len[b] : 0, s->n_q_heads / s->n_kv_heads);
    units += nb;
    if (nb > max_blocks) max_blocks = nb;
    if ((s->h_ctx_len[b] + 127) / 128 > tiles) tiles = (s->h_ctx_len[b] + 127) / 128;
  }
  // layers x splits of a launch, at most, over the launches of 1 to lc_max layers: min(splits x lc, max(lc, CTAs / units))
  const long long by_ctas = kScoreCtasMax / (units > 0 ? units * s->n_kv_heads : 1);
  const long long by_splits = (long long)(tiles < kScoreSplitsMax ? tiles : kScoreSplitsMax) * lc_max;
  const long long fit = by_ctas < by_splits ? by_ctas : by_splits;
  const long long part_slots = 2 * (fit > lc_max ? fit : lc_max);
  w.part = a; a = align_up(a + (size_t)part_slots * s->n_q_heads * sum_q * 8, 256);
  w.colpart = a; a = align_up(a + (size_t)lc_max * 2 * s->n_kv_heads * max_blocks * sum_t * 4, 256);
  size_t score_total = a;
  w.counts = 0;
  size_t sets_total = align_up((size_t)(s->n_req + (size_t)n_layers * s->n_req + 2) * 4, 256);
  w.total = attn_total > score_total ? attn_total : score_total;
  if (sets_total > w.total) w.total = sets_total;
  return w;
}

// ---- small device helpers -----------------------------------------------------------------
__device__ __forceinline__ float bf16_bits_to_float(uint16_t b) { return __uint_as_float(((uint32_t)b) << 16); }

__device__ __forceinline__ int warp_reduce_sum(int v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_reduce_sum(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}
__device__ __forceinline__ float warp_reduce_max(float v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// Find the request that owns global tile/row index x given an inclusive-exclusive prefix array.
__device__ __forceinline__ int find_segment(const int* cu, int n, int x) {
  int b = 0;
  while (b + 1 < n && x >= cu[b + 1]) ++b;
  return b;
}

}  // namespace relaxkv
