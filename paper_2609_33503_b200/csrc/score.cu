// Query-attention scoring (Section 3.2, score equation): two passes over the cached keys.
//   pass 1: log-normaliser of every query row's softmax over the context (skipped if supplied)
//   pass 2: column sums of exp(s - lse) over all query rows of a KV head, then the mean over heads
// followed by the segmented top-k (select.cu).  The two passes run on the tensor cores
// (score_sm100.cu); this file holds the entry point and the small kernels that combine their partial
// results in a fixed order, so results are bit-reproducible from run to run.
#include "attention_common.cuh"
#include "common.cuh"
#include "score_sm100.cuh"
#include "select.cuh"
#include <algorithm>

namespace relaxkv {

constexpr float kLn2 = 0.6931471805599453f;

// lse[layer, h, row] = ln sum over the partial (max, sum) pairs (log2 units in, natural log out).
// A block takes 32 consecutive rows, each warp every eighth partial of them (so that a warp reads 256 consecutive bytes; one
// warp per row, its lanes on the partials, fetched 8 bytes of every 32-byte sector: 68 us for 205 K rows of 12 partials,
// now 13 us behind the pass); a row's sums are added in a fixed order.  part is [layer][n_part][H*sum_q].  Rows of layers whose
// log-normalisers were supplied have only empty partials and are never read afterwards.
__global__ void __launch_bounds__(256) combine_lse_kernel(long long n_rows_total, long long n_rows, int n_part, const float2* part, float* lse) {
  __shared__ float s_m[8][32], s_z[8][32];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  const long long gidx = (long long)blockIdx.x * 32 + lane;
  griddep_launch();
  griddep_wait();
  const long long layer = min(gidx, n_rows_total - 1) / n_rows, idx = min(gidx, n_rows_total - 1) - layer * n_rows;
  const float2* pl = part + layer * n_part * n_rows + idx;
  float M = -INFINITY;
#pragma unroll 4
  for (int s = warp; s < n_part; s += 8) {
    const float2 p = pl[(long long)s * n_rows];
    if (p.y > 0.f) M = fmaxf(M, p.x);
  }
  s_m[warp][lane] = M;
  __syncthreads();
#pragma unroll
  for (int w = 0; w < 8; ++w) M = fmaxf(M, s_m[w][lane]);
  // 32 running sums per row, four of them in this warp; added up as a tree over the distances 16, 8, 4, 2, 1
  float v[4] = {0.f, 0.f, 0.f, 0.f};
  for (int s = warp; s < n_part; s += 32) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if (s + 8 * q < n_part) {
        const float2 p = pl[(long long)(s + 8 * q) * n_rows];
        if (p.y > 0.f) v[q] += p.y * exp2f(p.x - M);
      }
    }
  }
  s_z[warp][lane] = (v[0] + v[2]) + (v[1] + v[3]);
  __syncthreads();
  if (warp == 0 && gidx < n_rows_total) {
    const float u0 = (s_z[0][lane] + s_z[4][lane]) + (s_z[2][lane] + s_z[6][lane]);
    const float u1 = (s_z[1][lane] + s_z[5][lane]) + (s_z[3][lane] + s_z[7][lane]);
    lse[gidx] = (M + log2f(u0 + u1)) * kLn2;
  }
}

cudaError_t launch_combine_lse(int n_layers, int H, int sum_q, int n_part, const float2* part, float* lse, cudaStream_t stream) {
  const long long n_rows = (long long)H * sum_q, total = n_rows * n_layers;
  return launch_chained(combine_lse_kernel, (unsigned)((total + 31) / 32), 256, 0, stream, total, n_rows, n_part, part, lse);
}

// raw[layer, i] = (sum of the partial column sums in a fixed order: KV head, query-row block, warpgroup) / (H * Q_b)
// rt.tile_cu = prefix of the query-row blocks per request; colpart is [layer][2*Hkv*max_super][sum_t].
__global__ void finalize_raw_kernel(ReqTable rt, int n_layers, int H, int Hkv, int max_super,
                                    const float* colpart, float* raw) {
  griddep_launch();
  griddep_wait();
  const long long sum_t = rt.ctx_cu[rt.n_req];
  const long long gi = (long long)blockIdx.x * blockDim.x + threadIdx.x;
  if (gi >= sum_t * n_layers) return;
  const long long layer = n_layers == 1 ? 0 : gi / sum_t, i = gi - layer * sum_t;
  int b = 0;
  while (b + 1 < rt.n_req && i >= rt.ctx_cu[b + 1]) ++b;
  const int n_super = rt.tile_cu[b + 1] - rt.tile_cu[b];
  const float* cp = colpart + layer * (2 * Hkv * max_super) * sum_t;
  float s = 0.f;
  const int per_head = 2 * n_super, n_part = Hkv * per_head;
  // One behind the other, sixteen in flight: scores and top-k of one 16 K layer 61.2 us (eight) / 60.7, replayed from a graph 50.0 / 49.0.
  if (n_super == max_super) {
    cp += i;
#pragma unroll 16
    for (int m = 0; m < n_part; ++m) s += cp[(long long)m * sum_t];
  } else {
#pragma unroll 8
    for (int m = 0; m < n_part; ++m) {             // one loop, so that eight loads are in flight
      const int g = m / per_head;
      s += cp[(long long)(g * 2 * max_super + (m - g * per_head)) * sum_t + i];
    }
  }
  raw[gi] = s / ((float)H * (float)rt.q_len[b]);
}

template <int D>
static relaxkv_status score_layers(const relaxkv_shape* shape, ReqTable rt, const ScorePlan& plan, int n_layers,
                                   const void* const* q_layers, const relaxkv_cache_view* cache_layers,
                                   const float* const* lse_given, float* raw, char* workspace, const WsLayout& ws,
                                   cudaStream_t stream) {
  const int B = shape->n_req, H = shape->n_q_heads, Hkv = shape->n_kv_heads;
  float* lse_ws = reinterpret_cast<float*>(workspace + ws.lse);
  float2* part = reinterpret_cast<float2*>(workspace + ws.part);
  float* colpart = reinterpret_cast<float*>(workspace + ws.colpart);
  relaxkv_status rc = launch_score_sm100<D>(shape, rt, plan, n_layers, q_layers, cache_layers, lse_given, lse_ws, part,
                                            colpart, stream);
  if (rc != RELAXKV_OK) return rc;
  for (int b = 0; b < B; ++b) rt.tile_cu[b + 1] = rt.tile_cu[b] + plan.n_super[b];
  const long long total = rt.ctx_cu[B] * n_layers;
  return cuda_ok(launch_chained(finalize_raw_kernel, (unsigned)((total + 255) / 256), 256, 0, stream, rt, n_layers, H, Hkv, plan.max_super, colpart, raw));
}

}  // namespace relaxkv

using namespace relaxkv;

extern "C" relaxkv_status relaxkv_score_select(
    const relaxkv_shape* shape, int32_t n_layers,
    const void* const* q_layers, const relaxkv_cache_view* cache_layers,
    const float* const* row_lse_layers, const int32_t* h_k,
    float* raw_scores_out, float* norm_scores_out, int32_t* anchors_out,
    void* workspace, size_t workspace_bytes, relaxkv_stream stream_) {
  RELAXKV_RANGE("relaxkv_score_select");
  relaxkv_status rc = check_shape(shape);
  if (rc != RELAXKV_OK) return rc;
  if (n_layers < 1 || !q_layers || !cache_layers || !h_k || !raw_scores_out || !workspace || !shape->h_q_len)
    return RELAXKV_ERR_INVALID_ARG;
  for (int b = 0; b < shape->n_req; ++b) {
    if (shape->h_q_len[b] < 1) return RELAXKV_ERR_INVALID_ARG;
    if (h_k[b] < 1 || h_k[b] > shape->h_ctx_len[b]) return RELAXKV_ERR_INVALID_ARG;
  }
  for (int l = 0; l < n_layers; ++l) {
    if (!q_layers[l] || !aligned16(q_layers[l])) return RELAXKV_ERR_INVALID_ARG;
    if ((rc = check_cache(shape, &cache_layers[l], false)) != RELAXKV_OK) return rc;
  }
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return RELAXKV_ERR_INVALID_ARG;
  const WsLayout ws = ws_layout(shape, n_layers);
  if (workspace_bytes < ws.total) return RELAXKV_ERR_WORKSPACE_TOO_SMALL;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  long long sum_t = 0;
  for (int b = 0; b < shape->n_req; ++b) sum_t += shape->h_ctx_len[b];

  const ScorePlan plan = plan_score(shape);
  // Layers are scored in groups: one launch per pass covers up to kScoreLayersPerLaunch consecutive layers whose
  // cache views place the requests at the same token offsets (the usual case: all of them).
  for (int l0 = 0; l0 < n_layers;) {
    int l1 = l0 + 1;
    while (l1 < n_layers && l1 - l0 < kScoreLayersPerLaunch) {
      bool same = true;
      for (int b = 0; b < shape->n_req; ++b)
        same = same && cache_layers[l1].h_req_token_offset[b] == cache_layers[l0].h_req_token_offset[b];
      if (!same) break;
      ++l1;
    }
    ReqTable rt;
    fill_req_table(rt, shape, &cache_layers[l0], h_k);
    const float* const* lse = row_lse_layers ? row_lse_layers + l0 : nullptr;
    float* raw = raw_scores_out + (long long)l0 * sum_t;
    if (shape->head_dim == 128)
      rc = score_layers<128>(shape, rt, plan, l1 - l0, q_layers + l0, cache_layers + l0, lse, raw, static_cast<char*>(workspace), ws, stream);
    else
      rc = score_layers<64>(shape, rt, plan, l1 - l0, q_layers + l0, cache_layers + l0, lse, raw, static_cast<char*>(workspace), ws, stream);
    if (rc != RELAXKV_OK) return rc;
    l0 = l1;
  }
  if (!anchors_out) return RELAXKV_OK;      // scoring only: the caller reduces the scores first (head-sharded serving)
  ReqTable rt;
  fill_req_table(rt, shape, nullptr, h_k);
  return launch_select(rt, n_layers, raw_scores_out, norm_scores_out, anchors_out, stream);
}

// The query's own causal attention over [context, query] with the context scores taken from the same pass: the
// attention call leaves every row's log-normaliser, the column-sum pass of the scoring kernel then reads the context
// keys once more with those normalisers.  The statistics pass of relaxkv_score_select never runs.
extern "C" relaxkv_status relaxkv_query_prefill_attention(
    const relaxkv_shape* shape, const relaxkv_cache_view* cache, const void* q, void* out, float* lse_out,
    float* raw_scores_out, void* workspace, size_t workspace_bytes, relaxkv_stream stream_) {
  RELAXKV_RANGE("relaxkv_query_prefill_attention");
  relaxkv_status rc = check_shape(shape);
  if (rc != RELAXKV_OK) return rc;
  if ((rc = check_cache(shape, cache, true)) != RELAXKV_OK) return rc;
  if (!q || !out || !lse_out || !workspace || !shape->h_q_len || !aligned16(q) || !aligned16(out))
    return RELAXKV_ERR_INVALID_ARG;
  if ((reinterpret_cast<uintptr_t>(workspace) & 255u) != 0) return RELAXKV_ERR_INVALID_ARG;
  const int B = shape->n_req;
  int32_t ext_len[kMaxReqInline], q_len[kMaxReqInline];
  long long sum_q = 0;
  for (int b = 0; b < B; ++b) {
    if (shape->h_q_len[b] < 1) return RELAXKV_ERR_INVALID_ARG;
    const long long e = (long long)shape->h_ctx_len[b] + shape->h_q_len[b];
    if (e > 0x7fffffffLL) return RELAXKV_ERR_UNSUPPORTED_SHAPE;
    ext_len[b] = (int32_t)e;
    q_len[b] = shape->h_q_len[b];
    sum_q += q_len[b];
  }
  if (sum_q > 0x7fffffffLL) return RELAXKV_ERR_UNSUPPORTED_SHAPE;
  relaxkv_shape ext = *shape;                       // the same batch with the query's tokens counted into the cache rows
  ext.h_ctx_len = ext_len;
  // the context's own layout, which the scores take, needs no more than the one of context and query
  const WsLayout ws = ws_layout(&ext, 1), ws_sc = ws_layout(shape, 1);
  if (workspace_bytes < ws.total || workspace_bytes < ws_sc.total) return RELAXKV_ERR_WORKSPACE_TOO_SMALL;
  cudaStream_t stream = static_cast<cudaStream_t>(stream_);
  char* base = static_cast<char*>(workspace);
  ReqTable rt;
  fill_req_table(rt, shape, cache, nullptr);
  rc = cache_attention(&ext, cache, q, nullptr, nullptr, sum_q, q_len, out, lse_out, workspace, workspace_bytes, stream);
  if (rc != RELAXKV_OK || !raw_scores_out) return rc;
  // column sums over the CONTEXT keys with the rows' normalisers from the attention above
  const ScorePlan plan = plan_score(shape);
  const void* q_arr[1] = {q};
  const float* lse_arr[1] = {lse_out};
  if (shape->head_dim == 128)
    return score_layers<128>(shape, rt, plan, 1, q_arr, cache, lse_arr, raw_scores_out, base, ws_sc, stream);
  return score_layers<64>(shape, rt, plan, 1, q_arr, cache, lse_arr, raw_scores_out, base, ws_sc, stream);
}
