"""Shared memory of the projections of a few rows (gemm_skinny_layout.cuh), compiled by itself: what the blocks of a cluster stage and receive
lies inside the ring that they reuse, in every launch that the guard lets through, and the guard lets through what is launched."""
import os
import subprocess

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_33503_b200", "csrc")
MAIN = r"""
#include "gemm_skinny_layout.cuh"
#include <algorithm>
#include <cstdio>
using namespace relaxkv;
int main() {
  int close = 0;
  for (int whole = 0; whole < 2; ++whole)
    for (int rows = 2; rows <= kSkinnyMaxRows; ++rows)
      for (int swiglu = 0; swiglu < 2; ++swiglu)
        for (int S = 1; S <= 8; ++S)
          for (int parts = 1; parts <= 8; parts *= 2) {
            if (parts > 1 && (S * parts != 8 || rows > 4 || swiglu)) continue;      // up to four rows: eight parts of K in all
            const int n_cols = (rows + 15) & ~15, n_stages = sk_stages(n_cols, whole), ring = n_stages * sk_stage_bytes(n_cols);
            if (n_stages < 1 || n_stages > kSkStagesMax) { std::printf("stages\n"); return 1; }
            // as the kernel lays them out: the own tile, then the slot of each block src at sk_part_bytes + src * (what this block adds up)
            const int per = parts * rows * (swiglu ? 2 : 1) * 16;
            int end = 0, staged = 0;
            for (int r = 0; r < S; ++r) {
              const int mine = sk_quad(r + 1, S, swiglu) - sk_quad(r, S, swiglu);
              if (mine < 1) { std::printf("a block of %d adds nothing\n", S); return 1; }
              staged += mine * per;
              for (int src = 0; src < S && S > 1; ++src) end = std::max(end, sk_part_bytes(parts * rows) + (src + 1) * mine * per);
            }
            if (staged != sk_part_bytes(parts * rows)) { std::printf("the staged tile has %d bytes\n", staged); return 1; }
            end = std::max(end, staged);
            const bool fits = sk_exchange_fits(S, parts, rows, swiglu, n_cols, n_stages);
            if (fits && end > ring) { std::printf("%d rows, %d blocks, gate/up %d, whole SM %d: %d bytes in a ring of %d\n", rows, S, swiglu, whole, end, ring); return 1; }
            // clusters are launched with a whole SM, and with half of one up to kSkCols2 columns (wider ones have more tiles than clusters)
            if (!fits && (whole || n_cols <= kSkCols2)) { std::printf("%d rows, %d blocks, gate/up %d, whole SM %d: refused\n", rows, S, swiglu, whole); return 1; }
            close += !fits;
          }
  std::printf("%d\n", close);
  return 0;
}
"""


def test_partial_tiles_lie_inside_the_ring(tmp_path):
    (tmp_path / "main.cpp").write_text(MAIN)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", CSRC, str(tmp_path / "main.cpp"), "-o", str(tmp_path / "main")])
    r = subprocess.run([str(tmp_path / "main")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    assert int(r.stdout) > 100
