// How many workers a launch of the tensor-core attention kernel takes, and who joins the parts of cut units.  Plain host code
// (no CUDA), so that the rule can be walked over many batches without a device.
#pragma once

#include <algorithm>

constexpr int REKV_MAX_PARTS_INSIDE = 4;  // parts of a unit that the attention kernel joins itself

struct AttendPlan {
  int workers;        // each takes a contiguous range of the launch's chunks, equal to one chunk
  bool merge_inside;  // cut units are joined by the worker that finishes the last part, else by a merge launch
};

// total: chunks of all units; max_ch: of the longest unit; equal: every unit has max_ch; max_w: workers that can run at once;
// may_merge: a merge launch may follow.
inline AttendPlan rekv_attend_plan(int total, int units, int max_ch, bool equal, int max_w, bool may_merge) {
  // Long ranges: all workers there are, ranges cut where they fall.  A launch of few units (one layer) is a trade
  // between chunks one after the other (0.8 us each), a range with parts of two units (a second Q, result and pipeline start:
  // whole workers per unit avoid it), and joining parts.  The merge launch costs such a launch about 2 us, a join inside the
  // kernel 4 to 6 (fence, counter and the parts' latency, one after the other, at its very end).  28 layers one at a time,
  // 113 chunks, 4 units (us): 1 worker per unit 3268, 2, 3, 4 joined inside 2096, 1672, 1490, 6, 9, 18 with the merge launch
  // 1112, 978, 918; 11 chunks, 8 units, 9 layers: 322, 300, 288, 295, 255, 264.
  AttendPlan p;
  p.workers = std::min(max_w, total);
  auto joins = [&] { return (max_ch - 1) / std::max(1, total / p.workers) + 2 <= REKV_MAX_PARTS_INSIDE; };  // parts of a unit, at most
  p.merge_inside = joins();
  float best = 0.8f * (float)((total + p.workers - 1) / p.workers) + (units % p.workers ? 9.f : 0.f);
  // (k: two chunks at least in the longest unit's ranges; where the others are much shorter, units * k can exceed all chunks)
  for (int k = 1; (k == 1 || k < max_ch) && units * k <= std::min(max_w, total); ++k) {
    const float t = 0.8f * (float)((max_ch + k - 1) / k) + (k == 1 ? 0.f : 2.f + 0.05f * (float)k);
    if (t < best) {
      best = t;
      p.workers = units * k;
      p.merge_inside = k == 1 && equal;
    }
  }
  if (!may_merge && !p.merge_inside) {
    // Fewer workers: whole units each where all are equally long; where one is much longer than the rest, ranges of more than
    // a third of it, so that it falls into four at most.
    const int range = (max_ch - 1) / (REKV_MAX_PARTS_INSIDE - 1) + 1;
    p.workers = std::min({p.workers, units, total / range});
    p.merge_inside = true;
  }
  return p;
}
