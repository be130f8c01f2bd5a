// Internal: launcher of the mixed-context gather, shared by the attention entry points.
#pragma once
#include "common.cuh"

namespace relaxkv {

// Materialises rows [0, rows_to_cover) of the context (rows past the true total are zero-filled for
// kCtxPadRows rows, the rest left alone) into k_out / v_out [ctx_rows, H_kv, D].  fresh_row (may be NULL):
// per context row, the row of k_new/v_new that replaces it (-1: read the cache) - used by the explicit-list path
// instead of looking the entry up in r_rank; only its first fresh_map_rows entries are valid.  n_new_rows: rows of
// k_new / v_new (a fresh-row index past it is reported in the status word and the row zero-filled).  work_counter (may be
// NULL): an int the kernel sets to zero for the kernel behind it.  refused: for an attention kernel behind
// it, which refuses requests of more targets or context entries than the host's bounds or with rows past n_new_rows: flag (NULL: none is
// wanted) says which, and their rows are marked in its first partial log-sum-exps, part_lse [part_rows, H].  all_fresh (0: never): a call of one request whose lists may turn out to hold
// that many entries both, so that the context is k_new / v_new row by row (all_rows_fresh): then nothing is copied, and the kernel behind
// reads those.
struct RefusedRows {
  int* flag;
  float* part_lse;
  long long part_rows;
  int H;
  const int *bound_targets, *bound_ctx;      // host [n_req]
};
relaxkv_status launch_gather(const relaxkv_shape* shape, int mode, const relaxkv_cache_view* cache,
                             const void* k_new, const void* v_new, const int32_t* u_pos, const int32_t* u_cu,
                             const int32_t* r_rank, const int32_t* r_cu_layer, const int32_t* fresh_row,
                             long long fresh_map_rows, long long n_new_rows, long long rows_to_cover, void* k_out, void* v_out, long long ctx_rows,
                             int* work_counter, const RefusedRows& refused, int all_fresh, cudaStream_t stream);

// A row of which there are no partial results to merge: its log-sum-exp of the first split is +inf, which no computation returns (a row that
// saw an infinite score has a sum of NaN, and -inf).
constexpr unsigned kRefusedLse = 0x7f800000;

// One request: |R_l| = |U| = the n rows of k_new (R_l is a subset of U in the same order, so its ranks are 0, 1, ... n - 1).
__device__ __forceinline__ bool all_rows_fresh(int n, const int* u_cu, const int* r_cu) {
  return n > 0 && u_cu[0] == 0 && u_cu[1] == n && r_cu[1] - r_cu[0] == n;
}

}  // namespace relaxkv
