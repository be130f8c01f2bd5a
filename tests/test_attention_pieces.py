"""How an attention call over lists cuts its longest tile pairs into pieces: the host's rule and the order of the blocks (attention_pieces.cuh),
compiled by themselves."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_33503_b200", "csrc")
MAIN = r"""
#include "attention_pieces.cuh"
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
using namespace relaxkv;
int main() {
  std::mt19937 r(1);
  int cut_calls = 0;
  for (int it = 0; it < 40000; ++it) {
    const int n_req = 1 + (it % 3 ? 0 : r() % 8), hkv = 1 << (r() % 4), targets = 256 / (1 + r() % 8);
    const long long row_bytes = 512ll * hkv * (1 + r() % 8), cap = 2048 << (r() % 4);
    std::vector<int> tiles(n_req), pairs(n_req), bound(n_req);
    double longest = 0;
    for (int b = 0; b < n_req; ++b) {
      const int ctx = (int)std::pow(2.0, std::uniform_real_distribution<>(0, 16)(r));
      bound[b] = r() % (ctx + 1);
      tiles[b] = (ctx + 127) / 128;
      pairs[b] = (bound[b] + targets - 1) / targets;
      if (pairs[b]) longest = std::max(longest, (double)tiles[b]);
    }
    const PieceTable t = plan_pieces(tiles.data(), pairs.data(), bound.data(), n_req, targets, hkv, row_bytes, cap, 148, longest);
    if (t.most == 0) continue;
    ++cut_calls;
    if (t.most < 2 || t.most > 8 || (long long)t.slot_cu[n_req] * t.most > cap) { std::printf("slots\n"); return 1; }
    for (int b = 0; b < n_req; ++b) {
      const int L = t.long_pairs[b], S = t.pieces[b], n = pairs[b] + L * (S - 1);
      if (L < 0 || L > pairs[b] || S < 1 || S > 8 || t.slot_cu[b + 1] - t.slot_cu[b] != L * targets) { std::printf("table\n"); return 1; }
      std::vector<int> seen(pairs[b], 0);
      int last_cut = 0, last_whole = L;
      for (int u = 0; u < n; ++u) {
        int p = -1;
        const int piece = unit_piece(u, n, S, L, &p);
        if (p < 0 || p >= pairs[b] || (piece >= 0) != (p < L)) { std::printf("unit %d of %d: pair %d of %d\n", u, n, p, pairs[b]); return 1; }
        if (piece >= 0 ? (piece != seen[p] || p < last_cut) : p < last_whole) { std::printf("order\n"); return 1; }
        (piece >= 0 ? last_cut : last_whole) = p;
        ++seen[p];
      }
      for (int p = 0; p < pairs[b]; ++p)
        if (seen[p] != (p < L ? S : 1)) { std::printf("pair %d: %d blocks\n", p, seen[p]); return 1; }
    }
  }
  std::printf("%d\n", cut_calls);
  return 0;
}
"""


def test_every_piece_has_one_block_and_room_for_its_rows(tmp_path):
    """40000 calls of one to eight requests with up to 64 K entries: every piece of every pair is one block's, pieces and whole pairs
    start from the longest, and the partial rows fit the workspace."""
    (tmp_path / "main.cpp").write_text(MAIN)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", CSRC, str(tmp_path / "main.cpp"), "-o", str(tmp_path / "main")])
    r = subprocess.run([str(tmp_path / "main")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 2000
