// Shared by the decode-shaped attention kernel of step 5 (Eq. 3) and its merge kernels: the launch parameters and the
// decoding of a unit index.  A unit is (layer, kv head, question); a launch covers units * ncf (unit, context frame)
// steps, cut into contiguous ranges of `per` steps per CTA.
#pragma once

#include "ptx_helpers.cuh"
#include "rekv_internal.cuh"

namespace rekv_att {

struct TcParams {
  const __nv_bfloat16* q;
  __nv_bfloat16* out;
  char* const* tbl;
  // Eq. 3 in full (FULL instantiation and the merge kernel only; null otherwise)
  char* const* tbl_k;      // per context slot: rotated copy of the page's K tiles, or null = K from the page
  const float* self_o;     // per output row: sum of p*v over the tokens of X the row sees, relative to self_ml[0]
  const float* self_ml;    // per output row: (max, sum) of that part, log2 domain
  float* part_o;
  float* part_ml;
  int* unit_cnt;     // per unit: parts finished so far (decode kernel: the last part merges; self-resetting)
  int* status;
  QBatch qb;
  int Hq, Hkv, G, Nf, Npad, ncf, MP, layer0;
  // test-only knobs (0 = off): iteration limit of the bounded waits, and the frame whose copy CTA 0 leaves out so that a
  // wait runs out with nothing in flight
  unsigned wait_limit;
  int skip_copy_entry;
  int per;          // (unit, frame) steps per CTA
  long long total;  // units * ncf
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
constexpr uint32_t DEC_SCRATCH = DEC_WARPS * 16 * (128 + 2) * 4;  // the warps' (O, max, sum) at the end of a range
__global__ void attend_decode_kernel(const TcParams p);
// k_attend_combine.cu: joins the (max, sum, O) partials of a unit's parts
__global__ void combine_tc5_kernel(const TcParams p);
__global__ void combine_many_kernel(const TcParams p);  // units of many parts (launches of few units)

}  // namespace rekv_att
