// The decode-shaped attention kernel of step 5 (Eq. 3): the launch parameters and the decoding of a unit index.  A unit is
// (layer, kv head, question); a launch covers units * steps steps -- a step is one or several context frames, or a tile of X's
// tokens -- cut into contiguous ranges of `per` steps per CTA.
#pragma once

#include "ptx_helpers.cuh"
#include "rekv_internal.cuh"

namespace rekv_att {

struct TcParams {
  const __nv_bfloat16* q;
  __nv_bfloat16* out;
  char* const* tbl;
  // Eq. 3 in full: the own K/V of X, [L][sum_Ns][H_kv][128] as the caller passes them, and their lengths (nQ = 0: none)
  const __nv_bfloat16* k_self;
  const __nv_bfloat16* v_self;
  QBatch sb;
  // rotary embedding: (cos, sin) per [position][64], or null; context token j is at position j when rot_ctx is set (else it
  // is not rotated), token s of X at pos_x + s
  const float2* tab;
  const float2* tab_c;   // the same, ordered by 16-byte chunks (rope_table_kernel)
  int n_pos, pos_x, rot_ctx;
  float* part_o;
  float* part_ml;
  int* unit_cnt;     // per unit: parts finished so far (the last part merges; self-resetting)
  int* status;
  QBatch qb;
  int Hq, Hkv, G, Nf, Npad, ncf, MP, layer0;
  int early;         // the context table and its pages are complete whatever the kernels just before this launch do
  int F;             // frames of a step
  int fsteps;        // steps of a unit: its context frames, F at a time ...
  int steps;         // ... then tiles of F * N_pad tokens of X
  // test-only knobs (0 / -1 = off): iteration limit of the bounded waits, and the step (of one or several frames) whose copies CTA 0
  // leaves out so that a wait runs out
  unsigned wait_limit;
  int skip_copy_entry;
  int part_slots;    // capacity of part_o / part_ml in 16-row parts
  int per;           // steps per CTA, when parts == 0
  int parts;         // > 0: CTAs per unit (CTA k * units + u is part k of unit u); frame_parts of them share the unit's first
  int frame_parts;   // `split` steps evenly, the last part has the rest of its steps (alone, or besides its share)
  int split, units;
  long long total;   // units * steps
  float scale_log2;
};

struct UnitInfo {
  int l, g, qi, rows_q;
  long long q_row0;
};

__device__ __forceinline__ UnitInfo decode_unit(const TcParams& p, long long u) {
  UnitInfo ui;
  ui.qi = (int)(u % p.MP);
  const long long r = u / p.MP;
  ui.g = (int)(r % p.Hkv);
  ui.l = p.layer0 + (int)(r / p.Hkv);
  ui.rows_q = (p.qb.cu[ui.qi + 1] - p.qb.cu[ui.qi]) * p.G;
  ui.q_row0 = (long long)ui.l * p.qb.sumNq + p.qb.cu[ui.qi];
  return ui;
}

// k_attend_decode.cu: the load-bound kernel for questions of at most 16 rows per KV head
constexpr int DEC_THREADS = 256;
constexpr int DEC_WARPS = 8;
constexpr uint32_t DEC_SCRATCH = DEC_WARPS * 16 * (132 + 2) * 4;  // the warps' (O, max, sum) at the end of a range
}  // namespace rekv_att
