// strip_plan.h -- how the columns of a tensor-core launch are cut into strips (host code).
#pragma once

#include <algorithm>
#include <vector>

namespace sv {

// The columns of a launch that are Hu rows tall.
struct StripCols { int Hu; long long cols; };

// Columns of equal height are one group where the height is among the first kHeights (a search over more
// costs more than it saves).
constexpr int kHeights = 16;
inline void add_cols(std::vector<StripCols>& groups, int Hu, long long cols) {
  for (int i = 0; i < (int)groups.size() && i < kHeights; ++i)
    if (groups[i].Hu == Hu) {
      groups[i].cols += cols;
      return;
    }
  groups.push_back({Hu, cols});
}

// Strip height of a launch: `lanes` CTAs take the strips in turn, a CTA's time is its strips' rows plus
// `extra` rows' worth per strip (halo, ring restart), and the launch lasts as long as its busiest CTA.
// Every column of Hu rows is cut into equal strips, so candidates differ in how many rounds of
// strips there are and how much of the last round idles.  Four strips per CTA of whatever height, the last
// one of a column short, left 25-40 % of a launch in its tail (64 pairs of 1242 x 375: enc2 188 us against 137 at
// 32 rows, dec1 489 against 305 at 4).
// Calls that are not replayed search on every call, so equal columns are one group and a candidate's
// strip heights are worked out only as far as they can matter.  Seven layers of 64 pairs on one host core:
// 166 -> 8 us for four sizes in turn (grouped only where neighbours were equal), 165 -> 75 us for 60 sizes.
inline int pick_strip_rows(const std::vector<StripCols>& groups, int lanes, double extra) {
  const int n = (int)groups.size();
  std::vector<float> top(n);  // Hu - 0.5: ceil(Hu / hs) = int(top / hs) + 1, far enough from whole numbers for FP32
  std::vector<int> cols(n);
  int maxHu = 1;
  for (int i = 0; i < n; ++i) {
    top[i] = (float)groups[i].Hu - 0.5f;
    cols[i] = (int)groups[i].cols;
    maxHu = std::max(maxHu, groups[i].Hu);
  }
  int best = maxHu;
  double best_cost = 1e300;
  auto consider = [&](int hs) {  // true: one round of strips, taller ones only last longer
    const float inv = 1.0f / (float)hs;
    long long strips = 0;
    for (int i = 0; i < n; ++i) strips += (long long)((int)(top[i] * inv) + 1) * cols[i];
    const long long rounds = (strips + lanes - 1) / lanes;
    const int m0 = (maxHu + hs - 1) / hs;
    int tall = (maxHu + m0 - 1) / m0;
    if ((double)rounds * (tall + extra) >= best_cost - 1e-9) return rounds == 1;
    for (int i = 0; i < n && tall < hs; ++i) {
      const int m = (groups[i].Hu + hs - 1) / hs;
      tall = std::max(tall, (groups[i].Hu + m - 1) / m);
    }
    const double cost = (double)rounds * (tall + extra);
    if (cost < best_cost - 1e-9) {
      best_cost = cost;
      best = hs;
    }
    return rounds == 1;
  };
  for (int hs = std::min(2, maxHu); hs < maxHu; hs += hs < 64 ? 1 : hs / 8)
    if (consider(hs)) return best;
  consider(maxHu);  // whole columns
  return best;
}

// The strips of one column: equal heights, or (fixed) hs rows and a shorter last one.
template <typename F>
void cut_column(int Hu, int hs, bool fixed, F&& f) {
  const int m = (Hu + hs - 1) / hs;
  for (int t = 0; t < m; ++t) {
    const int i0 = fixed ? t * hs : (int)((long long)Hu * t / m), i1 = fixed ? std::min(Hu, i0 + hs) : (int)((long long)Hu * (t + 1) / m);
    f(i0, i1 - i0);
  }
}

}  // namespace sv
