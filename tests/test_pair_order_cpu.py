"""The waits of the two-step kernel (csrc/pair_order.h), checked on the host.

The rules are compiled into a small model of one block: four warps in each of
the four groups, barriers that count four arrivals a phase.  What a warp may
do depends only on arrivals that are never taken back, so for each event the
furthest that everything else can get without it is one fixed point, and
"without this event that one does not happen" is an exact answer.  Checked
for bands of every height that the rules can tell apart:
  - no barrier completes the phase after the awaited one while a warp still
    waits (it would then test the wrong parity and wait for ever);
  - no warp reaches a wait two phases early (the parity would pass it);
  - B pulls a row only after the seven rows of A it reads, A stores a row only
    after B has read what that replaces and after the rows that were in its
    place;
  - every band comes to its end."""
import os
import subprocess

import pytest

ROOT = os.path.dirname(os.path.dirname(os.path.abspath(__file__)))

MODEL = r"""
#include <cstdio>
#include <vector>
#include "pair_order.h"
using namespace lbm;

enum Kind { STORED, PULLED };
struct Op { bool arrive; Kind kind; int row; };  // a wait for, or an arrival for, the row
struct Warp { std::vector<Op> ops; };

static std::vector<Warp> block(int rows) {
  std::vector<Warp> w;
  for (int group = 0; group < 4; ++group)
    for (int k = 0; k < 4; ++k) {
      Warp v;
      if (group < 2) {
        for (int t = group; t < rows + 6; t += 2) {
          if (pair_a_pulled(t) >= 0) v.ops.push_back({false, PULLED, pair_a_pulled(t)});
          if (pair_a_stored(t) >= 0) v.ops.push_back({false, STORED, pair_a_stored(t)});
          v.ops.push_back({true, STORED, t});  // row t is written just before this
        }
      } else {
        for (int q = group - 2; q < rows; q += 2) {
          for (int n = pair_b_begin(q); n <= pair_b_end(q); ++n) v.ops.push_back({false, STORED, n});
          v.ops.push_back({true, PULLED, q});  // row q is read just before this
        }
      }
      w.push_back(v);
    }
  return w;
}

struct Reach {
  std::vector<int> at;           // next operation of each warp
  std::vector<int> count[2][8];  // arrivals per phase of each barrier
  int done(Kind k, int bar) const {  // completed phases
    int n = 0;
    for (int c : count[k][bar]) {
      if (c < 4) break;
      ++n;
    }
    return n;
  }
};

// the furthest that the block gets while warp `held` does not do operation `op`
static Reach run(const std::vector<Warp>& w, int held, int op) {
  Reach r;
  r.at.assign(w.size(), 0);
  for (auto& kind : r.count)
    for (auto& bar : kind) bar.assign(64, 0);
  for (bool moved = true; moved;) {
    moved = false;
    for (size_t i = 0; i < w.size(); ++i)
      while (r.at[i] < (int)w[i].ops.size() && !((int)i == held && r.at[i] == op)) {
        const Op& o = w[i].ops[r.at[i]];
        if (o.arrive) ++r.count[o.kind][o.row % kPairBars][o.row / kPairBars];
        else if (r.done(o.kind, o.row % kPairBars) <= o.row / kPairBars) break;
        ++r.at[i];
        moved = true;
      }
  }
  return r;
}

#define CHECK(cond, ...) \
  if (!(cond)) { std::printf(__VA_ARGS__); return 1; }

int main() {
  for (int rows = 1; rows <= 40; ++rows) {
    const auto w = block(rows);
    const Reach all = run(w, -1, 0);
    for (size_t i = 0; i < w.size(); ++i)
      CHECK(all.at[i] == (int)w[i].ops.size(), "%d rows: warp %zu stops at operation %d\n", rows, i, all.at[i])
    for (size_t i = 0; i < w.size(); i += 4)  // the warps of a group are alike
      for (int op = 0; op < (int)w[i].ops.size(); ++op) {
        const Op o = w[i].ops[op];
        const Reach r = run(w, (int)i, op);
        if (!o.arrive) {
          CHECK(o.row >= 0 && r.done(o.kind, o.row % kPairBars) <= o.row / kPairBars + 1,
                "%d rows: warp %zu can miss the phase of row %d (kind %d)\n", rows, i, o.row, o.kind)
          continue;
        }
        for (size_t v = 0; v < w.size(); ++v) {
          if (v == i) continue;
          for (int k = 0; k < (int)w[v].ops.size() && k <= r.at[v]; ++k) {
            const Op x = w[v].ops[k];
            // reached without the arrival of a phase earlier: its parity would pass
            CHECK(x.arrive || x.kind != o.kind || x.row != o.row + kPairBars,
                  "%d rows: warp %zu can wait for row %d before row %d\n", rows, v, x.row, o.row)
            if (!x.arrive) continue;
            // v can be writing (reading) row x.row although o has not happened
            if (o.kind == STORED && x.kind == PULLED)
              CHECK(o.row < x.row || o.row > x.row + 6, "%d rows: row %d pulled before row %d is stored\n", rows, x.row, o.row)
            if (o.kind == PULLED && x.kind == STORED)
              CHECK(o.row != x.row - 8, "%d rows: row %d stored before row %d is pulled\n", rows, x.row, o.row)
            if (o.kind == STORED && x.kind == STORED)  // (a thread's own rows are in order)
              CHECK((x.row - o.row) % 2 == 0 || x.row - o.row < 2 || x.row - o.row > 8,
                    "%d rows: row %d stored before row %d\n", rows, x.row, o.row)
          }
        }
      }
  }
  return 0;
}
"""


def test_no_wait_misses_its_phase_and_no_row_is_used_early(tmp_path):
    src, exe = tmp_path / "model.cpp", tmp_path / "model"
    src.write_text(MODEL)
    inc = os.path.join(ROOT, "paper_1608_06345_gb300", "csrc")
    p = subprocess.run([os.environ.get("CXX", "g++"), "-O2", "-std=c++17", "-I", inc, str(src), "-o", str(exe)],
                       capture_output=True, text=True)
    assert p.returncode == 0, p.stderr
    p = subprocess.run([str(exe)], capture_output=True, text=True, timeout=120)
    if p.returncode:
        pytest.fail(p.stdout)
