// How many workers a launch of the tensor-core attention kernel takes, who joins the parts of cut units, and who puts out the
// results.  Plain host code (no CUDA), so that the rules can be walked over many batches without a device.
#pragma once

#include <algorithm>
#include <numeric>

constexpr int REKV_MAX_PARTS_INSIDE = 4;  // parts of a unit that the attention kernel joins itself

struct AttendPlan {
  int workers;        // each takes a contiguous range of the launch's chunks, equal to one chunk
  bool merge_inside;  // cut units are joined by the worker that finishes the last part, else by a merge launch
  int parts;          // of a unit, at most (equal units: the most that one has)
};

// total: chunks of all units; max_ch: of the longest unit; equal: every unit has max_ch; max_w: workers that can run at once;
// may_merge: a merge launch may follow; pairs: workers are CTA pairs.
//
// What a number of workers costs (us), from launches of 1 to 28 layers: 0.75 for each chunk of a range -- 1 on single CTAs, which
// bring whole tiles -- one after the other; 8 for each segment of a range (the part of a unit in it: Q, the pipeline's start, the result); 4 for each end of a range
// that cuts a unit (partials written and joined inside, at the end of the segment), or 2 for the merge launch and 0.15 for each
// part.  The longest range decides, so that a few workers less can be faster: equal units per worker have no cuts, and ranges
// of 4/3 units touch two units each where 1.3 units touch three.  One B200, all workers (74 pairs) against this choice, us:
//   12 layers of 144 units of 50 chunks   151 -> 142 (72 workers)     8 layers, 96 units of 50     112 -> 104 (72)
//   encoding step, 192 units of 15        102 -> 94 (64)              12 layers, 48 units of 113   120 -> 115 (72)
//   (single CTAs, 28 layers, 112 units of 113: 148 workers 164, 140 workers 169)
//   28 layers one at a time, 4 units of 113: 1 worker per unit 3268, 2, 3, 4 joined inside 2096, 1672, 1490, 6, 9, 18 with the
//   merge launch 1112, 978, 918; 8 units of 11, 9 layers: 322, 300, 288, 295, 255, 264.
inline AttendPlan rekv_attend_plan(int total, int units, int max_ch, bool equal, int max_w, bool may_merge,
                                    bool pairs) {
  const float CHUNK = pairs ? 0.75f : 1.f;
  constexpr float SEGMENT = 8.f, CUT = 4.f, MERGE = 2.f, MERGE_PART = 0.15f;
  const int most = std::min(max_w, total);
  AttendPlan best = {0, true, 1};
  float best_cost = 0.f;
  for (int w = most; w >= 1 && (3 * w >= most || best.workers == 0); --w) {
    // the most segments of a range, partial segments of a range and parts of a unit.  Equal units, units / w = p / q in lowest
    // terms: ranges start at multiples of 1 / q of a unit (rounded up to a chunk, which cuts no further unit).
    int segments = units / w + 2, cuts = 2, parts = (max_ch - 1) / (total / w) + 2;
    bool even = false;  // q whole workers for each unit
    if (equal) {
      const int g = std::gcd(units, w), p = units / g, q = w / g;
      segments = (p - 1 + q - 1) / q + 1;
      parts = (q - 1 + p - 1) / p + 1;
      cuts = q == 1 ? 0 : p == 1 || q == 2 ? 1 : 2;
      even = p == 1;
    }
    const bool inside = parts <= REKV_MAX_PARTS_INSIDE;
    if (!inside && !may_merge) continue;
    const bool by_merge = !inside || (even && cuts > 0 && may_merge);
    const float join = by_merge ? MERGE + MERGE_PART * (float)parts
                                : CUT * (float)cuts + (equal && !even && parts > 2 ? CUT * (float)(parts - 2) : 0.f);
    const float cost = CHUNK * (float)((total + w - 1) / w) + SEGMENT * (float)segments + join;
    if (best.workers == 0 || cost < best_cost) {
      best = {w, !by_merge, parts};
      best_cost = cost;
    }
  }
  return best;
}

// Whether four warps of their own put out the segments' results while the softmax warps go on with the next segment.  They take
// registers from the softmax warps (216 -> 176 a thread: two loads of a row instead of one, and spills in the pair), which a
// range of one segment or of short ones does not get back, and pairs never do: their softmax warps are the pace.  One B200, us
// without / with, the same contexts in turn (a library against itself: within 1 %):
//   pairs   28 layers of 4 KV heads, 64 tokens, 19, 63, 113 chunks  107 / 118, 262 / 276, 444 / 456; 32 tokens, 113 chunks 232 / 236
//           40 layers of 8 KV heads, 32 tokens, 63 chunks 388 / 411; 16 questions, 63 chunks 3050 / 3108
//           (in runs of seconds, at the power limit: 1800-frame question 261 / 265, 16 questions 3187 / 3232)
//   single  40 layers of 8 KV heads, 16 tokens, 13, 32, 63, 113 chunks  84.7 / 85.8, 159 / 154, 251 / 248, 450 / 432;
//           5 tokens, 13, 32, 44, 113 chunks  77 / 80, 139 / 141, 170 / 170, 396 / 381; 28 layers of 4 KV heads, 3 questions of
//           12 tokens, 13, 32, 113 chunks  87 / 91, 151 / 148, 458 / 446
inline bool rekv_attend_output_warps(int workers, int units, int max_ch, bool pairs) {
  constexpr int MIN_CHUNKS = 32;
  return !pairs && workers < units && max_ch >= MIN_CHUNKS;
}

// Parts that a thread of the merge launch (two threads for a row's column quad, a block for 128 rows of 32 quads) has in flight.  More
// of them are fewer rounds of loads but more registers, and a grid that is not resident at once pays a second start: 4, 8 or 10 in
// flight (48, 73, 94 registers) let 5, 3 or 2 blocks be resident on an SM.  So 4 where 8 would not be resident, 10 only where it is
// and saves a round.  One B200, 12 layers one at a time, us with 4 / 8 / 10 (a library against itself: within 2 %):
//   320 blocks, 13 parts 268 / 258 / 270; 480, 7 parts 326 / 339 / 347; 512, 9 parts 400 / 414 / 422; 1024, 4 parts 417 / 441 / 465;
//   256 blocks, 18 parts 322 / 308 / 298; 64, 19 parts 221 / 221 / 216; 64, 27 parts 240 / 235 / 240; 192, 22 parts 304 / 297 / 305
inline int rekv_merge_ahead(int parts, long long blocks, int sms) {
  if (blocks > 3ll * sms) return 4;
  return parts > 16 && parts <= 20 && blocks <= 2ll * sms ? 10 : 8;
}
