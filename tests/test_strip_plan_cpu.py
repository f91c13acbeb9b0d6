"""Strip heights of the tensor-core launches (csrc/strip_plan.h) against a plain search."""
import os
import random
import subprocess

from paper_2305_11566_gb300 import build

MAIN = r"""
#include <cstdio>
#include "strip_plan.h"
int main() {  // lines: lanes, extra, number of columns' heights, the heights; output: groups, strip rows
  int lanes, n;
  double extra;
  while (scanf("%d %lf %d", &lanes, &extra, &n) == 3) {
    std::vector<sv::StripCols> g;
    for (int i = 0, h; i < n; ++i) {
      if (scanf("%d", &h) != 1) return 1;
      sv::add_cols(g, h, 1 + i % 3);
    }
    printf("%zu %d\n", g.size(), sv::pick_strip_rows(g, lanes, extra));
  }
}
"""


def plain(lanes, extra, cols):
    """Lowest modelled time over the candidate heights, whole columns among them; the lowest wins ties."""
    top = max(h for h, _ in cols)
    hs, cand = min(2, top), []
    while hs < top:
        cand.append(hs)
        hs += 1 if hs < 64 else hs // 8
    cand.append(top)
    best = None
    for hs in cand:
        parts = [(h, -(-h // hs), c) for h, c in cols]
        rounds = -(-sum(m * c for _, m, c in parts) // lanes)
        cost = rounds * (max(-(-h // m) for h, m, _ in parts) + extra)
        if best is None or cost < best[0] - 1e-9:
            best = (cost, hs)
    return best[1]


def test_strip_rows_equal_the_plain_search(tmp_path):
    rng = random.Random(4)
    calls = [(152, 1.5, [188] * 40), (152, 0.5, [1]), (1, 1.5, [8192, 8191]), (152, 0.5, [94, 93, 92, 93] * 16)]
    for _ in range(300):
        kinds = [rng.randint(1, rng.choice([8, 64, 300, 8192])) for _ in range(rng.choice([1, 1, 4, 20]))]
        calls.append((rng.choice([1, 4, 38, 152, 304, 456]), rng.choice([0.5, 1.5]),
                      [kinds[i % len(kinds)] for i in range(rng.randint(1, 80))]))
    src, exe = tmp_path / "plan.cpp", tmp_path / "plan"
    src.write_text(MAIN)
    subprocess.check_call(["g++", "-std=c++17", "-O1", "-I", build.CSRC, "-o", str(exe), str(src)])
    text = "\n".join(f"{l} {e} {len(h)} {' '.join(map(str, h))}" for l, e, h in calls)
    out = subprocess.run([str(exe)], input=text, capture_output=True, text=True, check=True).stdout.split("\n")
    for (lanes, extra, heights), line in zip(calls, out):
        groups, rows = map(int, line.split())
        if len(set(heights)) <= 16:
            assert groups == len(set(heights))  # a candidate costs one step per distinct height
        want = plain(lanes, extra, [(h, 1 + i % 3) for i, h in enumerate(heights)])
        assert rows == want, (lanes, extra, heights, rows, want)
