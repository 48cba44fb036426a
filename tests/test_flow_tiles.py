"""The tile list of the FP64 window factorisation, as its kernel computes it, against plain loops (host code only)."""
from _native import compile_program, run_program

PROGRAM = r"""
#include <cstdio>
#include <algorithm>
#include <random>
#include <vector>
#include "lma_f64.cuh"
using namespace lma::f64;
int main() {
  std::mt19937 rng(7);
  auto draw = [&](int lo, int hi) { return std::uniform_int_distribution<int>(lo, hi)(rng); };
  for (int trial = 0; trial < 400; ++trial) {
    const int nw = trial < 40 ? 1 : draw(1, 64), nchain = draw(1, nw);
    std::vector<FlowWin> f(nw);
    int maxpan = 0;
    for (FlowWin& w : f) {
      w = FlowWin{};
      w.npan = trial % 5 == 0 ? draw(1, 4) : draw(1, 40);
      w.nrt = w.npan + draw(1, 20);
      maxpan = std::max(maxpan, w.npan);
    }
    // rounds of nchain windows, column by column; what the chain's panel needs ahead of the tiles that need the panel
    std::vector<int4> want;
    for (int w0 = 0; w0 < nw; w0 += nchain)
      for (int j = 0; j < maxpan; ++j)
        for (int w = w0; w < std::min(nw, w0 + nchain); ++w) {
          if (j >= f[w].npan) continue;
          if (j > 0 && j + 1 < f[w].npan) {
            want.push_back(make_int4(w, j + 1, j, 0));
            want.push_back(make_int4(w, j + 1, j + 1, 0));
          }
          for (int i = std::min(j + 2, f[w].npan); i < f[w].nrt; ++i) want.push_back(make_int4(w, i, j, 0));
        }
    int64_t total = 0;
    for (const FlowWin& w : f) total += flow_columns(w.npan, w.nrt, w.npan);
    std::vector<int4> got((size_t)total, make_int4(-1, -1, -1, -1));
    for (int w = 0; w < nw; ++w)
      for (int j = 0; j < f[w].npan; ++j) {
        int64_t at = 0;
        for (int v = 0; v < nw; ++v) at += flow_ahead(f[v], v, w, j, nchain);
        for (int q = 0; q < flow_column(f[w].npan, f[w].nrt, j); ++q) {
          if (at + q < 0 || at + q >= total) return printf("out of the list: trial %d\n", trial), 1;
          got[(size_t)(at + q)] = flow_tile(f[w].npan, w, j, q);
        }
      }
    if (total != (int64_t)want.size()) return printf("size: trial %d\n", trial), 1;
    for (size_t t = 0; t < want.size(); ++t)
      if (want[t].x != got[t].x || want[t].y != got[t].y || want[t].z != got[t].z)
        return printf("trial %d tile %zu\n", trial, t), 1;
  }
  printf("ok\n");
  return 0;
}
"""


def test_tile_list_matches_plain_loops(tmp_path):
    assert run_program(compile_program(PROGRAM, tmp_path)).strip() == "ok"
