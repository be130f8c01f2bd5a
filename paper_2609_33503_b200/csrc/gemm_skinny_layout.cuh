// Internal: shared memory of the projections of a few rows (gemm_skinny_sm100.cu): the ring of weight and x tiles, and the partial tiles that
// take its place at the end (no CUDA beyond the qualifiers).
#pragma once
#ifdef __CUDACC__
#define RELAXKV_SK_HD __host__ __device__
#else
#define RELAXKV_SK_HD
#endif

namespace relaxkv {

constexpr int kSkinnyMaxRows = 128;
constexpr int kSkFeat = 128, kSkBK = 64, kSkStagesMax = 7;
constexpr int kSkWBytes = kSkFeat * kSkBK * 2;                             // weights of a stage: 16 KB, as two 64-row boxes
constexpr int kSkRing2 = 108 * 1024, kSkRing1 = 192 * 1024;                // two blocks, one block per SM
constexpr int kSkCols2 = 64;                                               // widest MMA that always takes the two-block form
constexpr int sk_stage_bytes(int n_cols) { return kSkWBytes + n_cols * kSkBK * 2; }
constexpr int sk_stages(int n_cols, bool whole_sm) {
  const int n = (whole_sm ? kSkRing1 : kSkRing2) / sk_stage_bytes(n_cols);
  return n < kSkStagesMax ? n : kSkStagesMax;
}

// The partial tile of a block: parts of K times rows of x, 128 features, fp32.
RELAXKV_SK_HD constexpr int sk_part_bytes(int rows) { return rows * kSkFeat * 4; }

// The tile's features in groups of four (gate and up rows count once): block r of a cluster of S adds up groups [sk_quad(r), sk_quad(r + 1)).
RELAXKV_SK_HD constexpr int sk_quads(bool swiglu) { return (swiglu ? kSkFeat / 2 : kSkFeat) / 4; }
RELAXKV_SK_HD constexpr int sk_quad(int r, int S, bool swiglu) { return r * sk_quads(swiglu) / S; }

// A block's own partial tile and, behind it, a slot for each block of the cluster, as large as the groups that this block adds up: with S that
// does not divide the groups, more than as much again (seven blocks, gate/up: 21 slots of 16 groups' worth).
constexpr int sk_exchange_bytes(int S, int parts, int rows, bool swiglu) {
  const int groups = (sk_quads(swiglu) + S - 1) / S;
  return sk_part_bytes(parts * rows) + (S > 1 ? S * groups * parts * rows * (swiglu ? 2 : 1) * 16 : 0);
}
constexpr bool sk_exchange_fits(int S, int parts, int rows, bool swiglu, int n_cols, int n_stages) {
  return sk_exchange_bytes(S, parts, rows, swiglu) <= n_stages * sk_stage_bytes(n_cols);
}

}  // namespace relaxkv
