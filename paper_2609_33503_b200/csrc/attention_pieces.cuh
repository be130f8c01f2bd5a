// Internal: how an attention call over lists cuts the contexts of its longest tile pairs into pieces (no CUDA beyond the qualifiers).
#pragma once
#include <algorithm>
#ifdef __CUDACC__
#define RELAXKV_HD __host__ __device__ __forceinline__
#else
#define RELAXKV_HD inline
#endif

namespace relaxkv {

constexpr int kMaxPieceReqs = 64;

// Of request b the `long_pairs[b]` pairs with the longest contexts are cut into `pieces[b]` equal pieces each; their partial results lie in
// slots [slot_cu[b], slot_cu[b + 1]) (target rows, the longest pair first).  most = 0: no pair is cut.
struct PieceTable {
  int most;                                // pieces of a pair, at most
  int pieces[kMaxPieceReqs], long_pairs[kMaxPieceReqs], bound[kMaxPieceReqs];
  int slot_cu[kMaxPieceReqs + 1];
};

// Unit u of the n_units of a request: its piece of which of the pairs, counted from the longest (p_rev), or a whole pair (returns -1).  Pieces,
// longest pair first, and whole pairs, longest first, are spread evenly through one another: both get shorter, and the blocks start in this order.
RELAXKV_HD int unit_piece(int u, int n_units, int pieces, int long_pairs, int* p_rev) {
  const int n_cut = long_pairs * pieces;
  const int cut = (int)((long long)u * n_cut / n_units), cut_next = (int)((long long)(u + 1) * n_cut / n_units);
  if (cut_next == cut) { *p_rev = long_pairs + u - cut; return -1; }
  *p_rev = cut / pieces;
  return cut % pieces;
}

constexpr double kPieceStepUs = 1.65;      // a step of a pair: 128 keys against both tiles
constexpr double kPieceMergeSteps = 3.0;   // launch and latencies of the merge, in steps
constexpr double kPieceTurnSteps = 2.5;    // what a block's start costs beyond an item of the persistent form
constexpr double kPieceBytesPerStep = 3.0e6 * kPieceStepUs;      // partial results written and read again, at 3 TB/s beside the steps

// Targets spread along the context: pair p of n sees about (p + 1) / n of it.  A call of few pairs is as long as its longest one (160 pairs of up
// to 52 steps on 148 SMs: 89 us, where blocks all alike would take 50), so where that sets its time the pairs longer than 1/S of the
// longest are cut into up to S pieces, S by the least estimated time: the steps of an SM, a quarter of a piece for the blocks' uneven end, the
// blocks' starts, the merge and its traffic.  Calls of 6400 entries, whole / cut, and the steps estimated: 1229 targets of 8 / 2 heads 95 us (50
// steps) / 47 (26, four pieces), 4000 of 4 / 1 heads of dim 64 87 (50) / 50 (25, three), 600 of 32 / 8 heads 98 (50) / 78 (34, two); 1229 of 32 / 8 heads 104 (50) /
// 113 (52, two) and 5000 of 8 / 2 heads 96 (50) / 100 (51, two) stay whole: what is merged is too much.  tiles[b], pairs[b]: context tiles and pairs of
// a request; uncut: steps of the call without pieces; cap: target rows x pieces that the workspace holds.
inline PieceTable plan_pieces(const int* tiles, const int* pairs, const int* bound, int n_req, int pair_targets, int n_kv_heads, long long row_bytes,
                              long long cap, int sms, double uncut) {
  PieceTable best{};
  double all = 0.0, best_cost = 0.9 * uncut;
  int longest = 1;
  for (int b = 0; b < n_req; ++b) {
    if (pairs[b] > 0) longest = std::max(longest, tiles[b]);
    all += 0.5 * tiles[b] * (pairs[b] + 1) * (pairs[b] > 0);
  }
  const double per_sm = all * n_kv_heads / sms;
  for (int s = 2; s <= 8 && 2 * s <= longest; ++s) {
    const int piece = (longest + s - 1) / s;
    PieceTable t{};
    double units = 0.0, bytes = 0.0;
    for (int b = 0; b < n_req; ++b) {
      t.bound[b] = bound[b];
      t.pieces[b] = std::max(1, (tiles[b] + piece - 1) / piece);
      t.long_pairs[b] = t.pieces[b] > 1 ? pairs[b] - (int)((long long)piece * pairs[b] / tiles[b]) : 0;
      t.slot_cu[b + 1] = t.slot_cu[b] + t.long_pairs[b] * pair_targets;
      if (t.long_pairs[b] > 0) t.most = std::max(t.most, t.pieces[b]);
      units += t.long_pairs[b] * (t.pieces[b] - 1) + pairs[b];
      bytes += 2.0 * t.long_pairs[b] * pair_targets * t.pieces[b] * row_bytes;
    }
    if (t.most < 2 || (long long)t.slot_cu[n_req] * t.most > cap) continue;
    const double cost = std::max((double)piece, per_sm + 0.25 * piece) + kPieceMergeSteps + bytes / kPieceBytesPerStep +
                        kPieceTurnSteps * std::max(0.0, units * n_kv_heads / sms - 1.0);
    if (cost < best_cost) { best_cost = cost; best = t; }
  }
  return best;
}

}  // namespace relaxkv
