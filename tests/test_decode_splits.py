"""How the one-token attention splits the contexts of a batch over blocks: the host's rule (decode_splits.cuh), compiled by itself."""
import os
import subprocess

import pytest

CSRC = os.path.join(os.path.dirname(os.path.dirname(os.path.abspath(__file__))), "paper_2609_33503_b200", "csrc")
MAIN = r"""
#include "decode_splits.cuh"
#include <chrono>
#include <cmath>
#include <cstdio>
#include <random>
#include <vector>
int main() {
  std::mt19937 r(1);
  double worst = 0;
  for (int it = 0; it < 60000; ++it) {
    const int rooms[] = {18, 9, 148, 37, 74};
    const int n_req = 1 + r() % 64, slots = rooms[r() % 5];
    std::vector<int> n(n_req);
    for (int& x : n) x = (int)std::pow(2.0, std::uniform_real_distribution<>(0, it % 2 ? 13 : 9)(r));
    const int per = relaxkv::decode_tiles_per_block(n.data(), n_req, slots);
    long long all = 0, blocks = 0;
    int longest = 0;
    for (int x : n) {
      const int ns = relaxkv::decode_blocks(x, per), share = (x + ns - 1) / ns;
      if (ns < 1 || (ns > 1 && x / ns < 2)) { std::printf("a block of less than two tiles: %d tiles, %d blocks\n", x, ns); return 1; }
      all += x; blocks += ns;
      if (share > longest) longest = share;
    }
    if (2 * n_req <= slots && blocks > slots) { std::printf("%lld blocks, room for %d\n", blocks, slots); return 1; }
    const double best = std::max(2.0, (all + (double)relaxkv::kDecStartTiles * n_req) / slots) + relaxkv::kDecStartTiles;
    worst = std::max(worst, (relaxkv::kDecStartTiles + longest) / best);
  }
  std::vector<int> n(64, 8);
  n[0] = 7812;                                             // one context of 1 M tokens beside 63 of 1 K
  const auto t = std::chrono::steady_clock::now();
  volatile int sink = 0;
  for (int i = 0; i < 200; ++i) sink += relaxkv::decode_tiles_per_block(n.data(), 64, 18);
  std::printf("%.3f %.3f\n", worst, std::chrono::duration<double>(std::chrono::steady_clock::now() - t).count() / 200 * 1e6);
  return 0;
}
"""


@pytest.fixture(scope="module")
def result(tmp_path_factory):
    d = tmp_path_factory.mktemp("splits")
    (d / "main.cpp").write_text(MAIN)
    subprocess.check_call(["g++", "-O2", "-std=c++17", "-I", CSRC, str(d / "main.cpp"), "-o", str(d / "main")])
    r = subprocess.run([str(d / "main")], capture_output=True, text=True)
    assert r.returncode == 0, r.stdout
    return [float(x) for x in r.stdout.split()]


def test_no_block_is_much_longer_than_the_average(result):
    """Over 60000 batches of 1 to 64 requests with contexts of 1 to 8192 tiles: at least two tiles per block, all blocks resident at
    once while the requests are at most half the room, and the longest block's time (start included) at most twice an even share:
    a block longer than that is split where that halves it."""
    assert result[0] <= 2.0 + 1e-9


def test_the_rule_takes_a_few_microseconds(result):
    """64 requests, one of 1 M tokens: a search in halves.  (Step by step from the even share it took 2 ms per call.)"""
    assert result[1] < 200.0
