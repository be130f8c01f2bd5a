// Internal: how the one-token attention splits the contexts of a batch over blocks (host only, no CUDA).
#pragma once
#include <algorithm>

namespace relaxkv {

constexpr int kDecStartTiles = 6;      // start and merge of a block, in key tiles (about 9 us against 1.4 us per tile)

// Key tiles per block for contexts of n_tiles[0 .. n_req) tiles and room for `slots` blocks per KV head at once.
// The fewest, at least two, for which all blocks are resident at once.  With more than half as many requests as room that leaves
// long requests whole beside short ones (18 requests of 1 K tokens and one of 64 K: one block of 512 tiles, 340 us): there
// the fewest tiles are taken for which all blocks, started one after the other, end with the longest one - where that makes the
// longest block less than half as long, so that not even a second round of blocks could be slower.
inline int decode_tiles_per_block(const int* n_tiles, int n_req, int slots) {
  int most = 2;
  long long all = 0;
  for (int b = 0; b < n_req; ++b) { most = std::max(most, n_tiles[b]); all += n_tiles[b]; }
  auto blocks = [&](int p) { long long n = 0; for (int b = 0; b < n_req; ++b) n += (n_tiles[b] + p - 1) / p; return n; };
  auto fewest = [&](auto fits) {       // fits(p) stays true once it is; fits(most) need not be asked
    int lo = 2, hi = most;
    while (lo < hi) { const int mid = lo + (hi - lo) / 2; if (fits(mid)) hi = mid; else lo = mid + 1; }
    return lo;
  };
  const int at_once = fewest([&](int p) { return blocks(p) <= std::max(slots, n_req); });
  if (2 * n_req <= slots) return at_once;
  const int in_turn = fewest([&](int p) { return blocks(p) * kDecStartTiles + all <= (long long)slots * (kDecStartTiles + p); });
  return 2 * (kDecStartTiles + in_turn) <= kDecStartTiles + at_once ? in_turn : at_once;
}

// Blocks of a request of n tiles, at least two tiles each.
inline int decode_blocks(int n, int tiles_per_block) {
  return std::max(1, std::min((n + tiles_per_block - 1) / tiles_per_block, n / 2));
}

}  // namespace relaxkv
