"""CPU check of the tiled form's item order when the last wave's pairs are cut
finer (split_tail in csrc/tiled_schedule.h, compiled with the host C++ compiler):
for every pair count up to a few waves of several grids, one- and two-stage nets
of both image sides, every warp task of every pair is in exactly one item, every
stage-1 item comes after its pair's stage-0 items, and every wait for a slot is
for an earlier item (so a queue that is worked off in order ends)."""

import os
import shutil
import subprocess

import pytest

HERE = os.path.dirname(os.path.abspath(__file__))
CSRC = os.path.join(os.path.dirname(HERE), "paper_2303_05420_gb300", "csrc")

PROGRAM = r"""
#include <cstdio>
#include <vector>
#include "tiled_schedule.h"
using namespace nkf::sched;
struct Q {
  int n, R[8], nt0[8], split[8], wn[8];
  int64_t p0[8], g0[9], f0[9], G, G64, T0, LAG;
  int S[2];
};
static int cuts = 0;
static int check(int side, int wt, int rounds, int64_t pairs, int grid, bool two) {
  Q q = {};
  q.n = 1;
  q.R[0] = side;
  q.nt0[0] = tasks_per_pair(side);
  q.split[0] = 1;
  q.wn[0] = wt;
  q.G = q.g0[1] = pairs;
  q.T0 = q.f0[1] = pairs * q.nt0[0];
  q.G64 = side == 64 ? pairs : 0;
  const int whole = q.nt0[0];
  int64_t np[8] = {pairs};
  const bool cut = split_tail(q, np, grid, rounds);
  cuts += cut;
  int64_t total = 0;
  for (int b = 0; b < q.n; ++b) {
    total += np[b];
    // the parts share a task's warp tasks, each warp the same number of them
    if (q.split[b] * q.wn[b] != wt || q.wn[b] % (wt / rounds) || q.nt0[b] != whole * q.split[b]) return 1;
    if (q.g0[b + 1] - q.g0[b] != np[b] || q.p0[b] != q.g0[b] || np[b] < 1) return 2;
  }
  if (total != pairs || q.f0[q.n] != q.T0) return 3;
  const Plan p = make_plan(two, q.R, np, q.n, grid);
  q.LAG = p.LAG;
  q.S[0] = p.S[0];
  q.S[1] = p.S[1];
  const int64_t items = q.T0 + (two ? q.G : 0);
  std::vector<int> done((size_t)pairs * whole * wt, 0), st1(pairs, 0);
  std::vector<int64_t> first(pairs, -1), last(pairs, -1), pos1(pairs, -1);
  for (int64_t m = 0; m < items; ++m) {
    int64_t k;
    if (decode(q, two, m, &k)) {
      if (k < 0 || k >= pairs || st1[k]++) return 4;
      pos1[k] = m;
      continue;
    }
    int b, sub;
    int64_t g;
    if (k < 0 || k >= q.T0) return 5;
    stage0_of(q, k, &b, &g, &sub);
    if (g < q.g0[b] || g >= q.g0[b + 1]) return 6;
    const int t = sub / q.split[b], w0 = (sub - t * q.split[b]) * q.wn[b];
    for (int w = w0; w < w0 + q.wn[b]; ++w)
      if (t >= whole || w >= wt || done[(g * whole + t) * wt + w]++) return 7;
    if (first[g] < 0) first[g] = m;
    last[g] = m;
  }
  for (int v : done)
    if (v != 1) return 8;
  if (!two) return 0;
  for (int64_t g = 0; g < pairs; ++g) {
    if (st1[g] != 1 || pos1[g] <= last[g]) return 9;
    int ring;
    int64_t prev;
    const int64_t s = slot(q, block_of_pair(q, g), g, &ring, &prev);
    if (s < 0 || s >= q.S[ring]) return 10;
    if (prev >= 0 && pos1[prev] >= first[g]) return 11;
  }
  return 0;
}
int main() {
  // (side, warp tasks of a task, of a warp): 32x32 on 8 and on 16 warps, 64x64
  const int shapes[][3] = {{32, 32, 4}, {32, 32, 2}, {64, 64, 4}};
  for (auto& s : shapes)
    for (int grid : {1, 3, 7, 152, 304})
      for (int64_t pairs = 1; pairs <= (grid < 100 ? 60 : 140); ++pairs)
        for (bool two : {false, true}) {
          const int e = check(s[0], s[1], s[2], pairs, grid, two);
          if (e) {
            std::printf("FAIL %d: side %d rounds %d pairs %lld grid %d two %d\n", e, s[0], s[2], (long long)pairs, grid, two);
            return 1;
          }
        }
  std::printf(cuts > 100 ? "ok\n" : "FAIL: nothing was cut\n");
  return 0;
}
"""


def test_items_of_cut_waves(tmp_path):
    cxx = shutil.which("g++") or shutil.which("c++")
    if cxx is None:
        pytest.skip("no host C++ compiler")
    src, exe = tmp_path / "split.cpp", str(tmp_path / "split")
    src.write_text(PROGRAM)
    subprocess.run([cxx, "-O2", "-std=c++17", "-I", CSRC, str(src), "-o", exe], check=True)
    out = subprocess.run([exe], capture_output=True, text=True, timeout=300)
    assert out.returncode == 0 and out.stdout.strip() == "ok", out.stdout + out.stderr
