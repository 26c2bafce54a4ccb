// Step 5 (Eq. 3) on the 5th-generation tensor cores: GQA attention of the question tokens over the
// gathered context, read page by page through the context table, followed (Eq. 3 in full) by the tokens of X itself.
//
// What bounds it.  A question of 32 tokens at G = 7 brings 224 rows to every K/V byte: 196 FLOP/B, near the ridge of
// tensor rate and memory rate, with one exponential per logit besides.  One CTA with two 128-row tiles in tensor memory
// (O0 O1 S0 S1 = all 512 columns) ran each tile as the chain S -> softmax -> P V -> next S: 3950 cycles per chunk pair
// for 2800 of tensor work, 218 us = 0.58 of the copy rate.  Here a unit's 256 rows belong to a CLUSTER OF TWO CTAs that work
// on one product (tcgen05 cta_group::2): each CTA owns one 128-row tile and brings half of every K and V tile, so tensor
// memory holds O and THREE buffers of S (P over S) and the ring twice as many chunks.  S runs up to three chunks ahead,
// two softmax warpgroups take the chunks alternately, and neither waits for a product of its own chunk.
// 28 layers, 72 frames of 196 tokens, 32 query tokens: 218 -> 179 to 194 us at 1965 MHz, by box (0.65 to 0.70 of the copy rate; a chunk
// takes 1536 cycles, of which HBM alone needs 1476); in runs of seconds the card's 1000 W hold the whole question at 249 to 261 us,
// which is why fewer instructions and bytes are what counts.
//
// Work split ("stream-K" in chunks).  A unit is (layer, kv head, question, 128 or 256 rows), a row being (question
// token, query head of the KV group).  Eq. 3 without a positional term does not depend on the order or grouping of the
// context tokens, so a unit's context frames are ONE token stream cut into dense 128-token chunks that run across frame
// boundaries.  In the stream a frame takes N_s = N_f rounded up to a multiple of 8 rows, so that a token's row in a chunk
// tile has the swizzle phase (row & 7) it has in its page: a chunk tile is assembled in shared memory by contiguous bulk
// copies.  The gap rows' and the tail's logits are masked and their V rows zeroed.  X's tokens (staged in the page layout)
// follow at stream row ncf * N_s with a causal mask, as part of the same stream: no separate kernel, no extra merge.
// The chunks of all units are dealt to the workers (CTA pairs, or single CTAs) in contiguous ranges that differ by at
// most one chunk.
//
// Single CTAs (CG = 1) serve batches in which every question has at most 128 rows: the same kernel with whole K/V
// tiles per CTA.
//
// Warp roles of a CTA:
//   warp 0      K tiles (bulk copies, a piece per lane)
//   warp 1      tcgen05.mma issue, first CTA of a pair only: S(t) and, three chunks behind, O += P V
//   warp 2      V tiles; zeroes the V rows that carry no token
//   warp 3      second CTA of a pair: passes its tiles' arrivals on to the issuing CTA
//   warp 3 (warp 1 in a pair's second CTA)   the next segment's Q tile (cp.async, double-buffered)
//   warps 4-7, 8-11   softmax of the even / odd chunks, one thread per row (= TMEM lane), fp32
//   warps 12-15 (OUT)   the segments' results, so that the softmax warps go on with the next segment's chunks meanwhile: single
//                       CTAs with several long segments each (attend_plan.h); else the softmax warps put out the results
// After set-up the service warpgroup shrinks to 72 (56 with output warps) registers per thread and the softmax warpgroups grow to
// 216 (176) (setmaxnreg), so that a softmax thread holds a whole S row chunk: one or two TMEM loads and two TMEM stores per
// chunk (a warp's tcgen05.ld/st cost about 90 cycles each whatever their width).
//
// The exponentials of a segment (the part of a unit in one range) take the row maximum of its first chunk as their
// reference m: a softmax does not depend on m, and 2^(x - m) far above 1 loses nothing in fp32 or in bf16's exponent.
// Only a chunk whose row sum leaves [0, 2^60) needs a higher one; as both softmax warpgroups and O share m, such a segment is
// marked, put out no result, and is run again at the end of the CTA's range chunk by chunk, with O rescaled when the
// maximum is raised (never with ordinary inputs).
//
// A segment that is not a whole unit is a part of it, (max, sum, O) per row.  Up to four parts per unit are joined by the
// worker that completes the last one: if every other part is counted when its own is done, straight from its O
// registers.  Nobody waits for anybody.  Else merge_tc5_kernel joins them
// (attend_plan.h says when).
// Every wait is bounded: on expiry the status word is set and the CTA leaves.
#include <algorithm>
#include <type_traits>

#include "attend_common.cuh"
#include "attend_plan.h"

using namespace rekv_ptx;
using namespace rekv_att;

namespace {

constexpr int SM_WARP0 = 4, OUT_WARP0 = 12;            // first softmax warp, first output warp
// OUT: four more warps put out the segments' results, else the softmax warps do it themselves (rekv_attend_output_warps).
// Registers per thread: 128 * service + 256 * softmax (+ 128 * output) <= threads * those at launch
template <bool OUT>
struct Warps {
  static constexpr int THREADS = OUT ? 512 : 384;
  static constexpr int REGS_SERVICE = OUT ? 56 : 72, REGS_SOFTMAX = OUT ? 176 : 216, REGS_OUT = 104;
  static constexpr int OUT_WARPS = OUT ? 4 : 8, COLUMNS = OUT ? 128 : 64;   // columns of a row that an output thread puts out
};
constexpr int CHUNK = 128;                             // stream rows per chunk
constexpr int S_BUFS = 3;                              // S/P buffers in tensor memory
constexpr uint32_t TMEM_COLS = 512;                    // O [0,128), S/P [128,512)
constexpr uint32_t Q_TILE_BYTES = 128 * 256;           // 128 rows x 128 dims bf16
constexpr uint32_t RING_BYTES = 160 * 1024;            // K and V tiles in flight
constexpr float RESCALE_SUM_LIMIT = 1.152921504606846976e18f;  // 2^60
constexpr int MAX_PARTS_INSIDE = REKV_MAX_PARTS_INSIDE;
constexpr uint32_t WAIT_LIMIT = 1u << 22;
// P is cut (not rounded) to bf16: a value with mantissa m in [1, 2) loses u * 2^-7 / m of itself, u uniform in [0, 1).
// The mantissa of 2^x is log-uniform, E[1/m] = 1 / (2 ln 2), so the mean loss is 0.7213 * 2^-8 of the value, and scaling
// by 1 + 0.7213 * 2^-8 beforehand makes the cut value right on average (its spread equals that of rounding to
// nearest).  log2 of that factor, and its inverse for the row sum:
constexpr float TRUNC_GAIN_LOG2 = 0.0040592f;
constexpr float TRUNC_GAIN_INV = 0.99719028f;

template <int CG>
struct Ring {  // K and V rings of one CTA: half tiles in a pair, whole tiles alone
  static constexpr uint32_t TILE = 32768 / CG;
  static constexpr int KB = CG == 2 ? 5 : 2, VB = CG == 2 ? 5 : 3;
  static constexpr int K_ROWS = CHUNK / CG;        // tokens of a K tile in this CTA (both 64-dim halves)
  static constexpr uint32_t K_HALF = K_ROWS * 128; // one 64-dim half of a K tile; a V half has CHUNK rows
  static_assert((KB + VB) * TILE == RING_BYTES, "ring plan");
};
constexpr uint32_t V_HALF = CHUNK * 128;

// barrier slots (8 bytes each)
constexpr int B_KFULL = 0, B_KEMPTY = 5, B_VFULL = 10, B_VEMPTY = 15, B_SFULL = 20, B_PREADY = 23, B_QFULL = 26,
              B_QFREE = 28, B_OFULL = 30, B_OFREE = 31, B_MREADY = 32, B_LREADY = 34, B_LFREE = 36, B_COUNT = 38;
// small shared state after the barriers (bytes)
constexpr uint32_t OFF_M = 8 * B_COUNT;               // float [2 parity][128]: the segment's reference maxima
constexpr uint32_t OFF_L = OFF_M + 1024;              // float [2 parity][128]: row sums
constexpr uint32_t OFF_REDO = OFF_L + 1024;           // u64: segments to run again
constexpr uint32_t OFF_WORDS = OFF_REDO + 8;          // u32: tmem slot, abort, overflow marks [2], fast, last, again
constexpr uint32_t SMALL_BYTES = OFF_WORDS + 32;
constexpr size_t TC_SMEM = 2 * Q_TILE_BYTES + RING_BYTES + SMALL_BYTES;  // (the dynamic segment is 1024-byte aligned)
static_assert(TC_SMEM <= 227 * 1024, "shared-memory plan of the attention kernel");

struct Tc5Params {
  const __nv_bfloat16* q;
  __nv_bfloat16* out;
  char* const* tbl;
  char* const* tbl_k;      // per context slot: rotated copy of the page's K tiles, or null = K from the page
  const char* x_kv;        // X's K/V in the page layout (stage_x_kernel), or null = no X
  long long x_rows;        // its rows per (layer, kv head, K/V, half)
  float4* part_o;          // [slot][CTA of the pair][32 column quads][128 rows]
  float2* part_ml;         // [slot][CTA of the pair][128 rows] (max, sum)
  int* unit_cnt;           // per worker and CTA of the pair: finished parts of the cut unit that starts in its range
  int* status;
  QBatch qb;
  QBatch sb;               // X's lengths (nQ = 0: none)
  int Hq, Hkv, G, Nf, Ns, ncf, layer0, nl;
  int W;                   // workers
  int total;               // chunks of all units
  int per_lh;              // chunks of one (layer, kv head)
  int merge_inside;        // cut units are joined by the worker that finishes the last part
  int early_q;             // Q does not depend on the kernels just before this launch
  int split_rem;           // see row_blocks
  int second;              // the second launch of two that run side by side: it starts once the first one's CTAs have all seen
                           // their predecessors' results, and waits for the first launch only at its end
  unsigned wait_limit;     // test-only knobs (0 / -1 = off), see rekv_test_set_wait_limit
  int skip_copy_entry;
  int part_slots;          // capacity of part_o / part_ml in 128-row slots (checks build)
  float scale_log2;
};

__host__ __device__ __forceinline__ int x_len(const Tc5Params& p, int qi) {
  return p.sb.nQ ? p.sb.cu[qi + 1] - p.sb.cu[qi] : 0;
}
__host__ __device__ __forceinline__ int stream_rows(const Tc5Params& p, int nx) {
  return nx > 0 ? p.ncf * p.Ns + nx : (p.ncf - 1) * p.Ns + p.Nf;
}
__host__ __device__ __forceinline__ int stream_chunks(const Tc5Params& p, int qi) {
  return (stream_rows(p, x_len(p, qi)) + CHUNK - 1) / CHUNK;
}
// Units of a question in this launch, and the first row of unit mp.  A question's rows are taken 256 at a time by CTA pairs;
// with split_rem a remainder of at most 128 rows goes to a launch of single CTAs instead of filling half a pair.
template <int CG>
__host__ __device__ __forceinline__ int row_blocks(const Tc5Params& p, int qi) {
  const int rows = (p.qb.cu[qi + 1] - p.qb.cu[qi]) * p.G;
  if (!p.split_rem) return (rows + 128 * CG - 1) / (128 * CG);
  return CG == 2 ? (rows + 127) >> 8 : ((rows - 1) & 255) < 128 ? 1 : 0;
}
template <int CG>
__host__ __device__ __forceinline__ int block_row0(const Tc5Params& p, int rows_q, int mp) {
  return CG == 1 && p.split_rem ? (rows_q - 1) & ~255 : mp * 128 * CG;
}

// A segment: the chunks [I0, I1) of one unit that lie in a worker's range.
struct Seg {
  int l, g, qi, m0, rows_q, nq, nx;
  int I0, I1, nch;
  int uc0;             // global index of the unit's first chunk
  long long q_row0;    // row of the question's first token in q / out, in tokens
};

template <int CG>
__device__ __forceinline__ Seg decode_seg(const Tc5Params& p, int pos, int end) {
  Seg s;
  const int lh = pos / p.per_lh;
  int rem = pos - lh * p.per_lh;
  s.g = lh % p.Hkv;
  s.l = p.layer0 + lh / p.Hkv;
  int qi = 0, nch = stream_chunks(p, 0);
  for (; qi < p.qb.nQ - 1; ++qi) {
    const int tot = row_blocks<CG>(p, qi) * nch;
    if (rem < tot) break;
    rem -= tot;
    nch = stream_chunks(p, qi + 1);
  }
  const int mp = rem / nch;
  s.qi = qi;
  s.nch = nch;
  s.nq = p.qb.cu[qi + 1] - p.qb.cu[qi];
  s.nx = x_len(p, qi);
  s.rows_q = s.nq * p.G;
  s.m0 = block_row0<CG>(p, s.rows_q, mp);
  s.I0 = rem - mp * nch;
  s.I1 = min(nch, s.I0 + (end - pos));
  s.uc0 = pos - s.I0;
  s.q_row0 = (long long)s.l * p.qb.sumNq + p.qb.cu[qi];
  return s;
}
__device__ __forceinline__ int worker_of(const Tc5Params& p, int c) {
  return (int)((long long)c * p.W / p.total);
}

__device__ __forceinline__ float max3(float a, float b, float c) {
  float r;
  asm("max.f32 %0, %1, %2, %3;" : "=f"(r) : "f"(a), "f"(b), "f"(c));
  return r;
}

__device__ __forceinline__ void store_row_part(__nv_bfloat16* dst, const float* o, float inv) {  // 32 columns of a row
#pragma unroll
  for (int v = 0; v < 4; ++v) {
    uint4 x;
    x.x = pack_bf16(o[8 * v] * inv, o[8 * v + 1] * inv);
    x.y = pack_bf16(o[8 * v + 2] * inv, o[8 * v + 3] * inv);
    x.z = pack_bf16(o[8 * v + 4] * inv, o[8 * v + 5] * inv);
    x.w = pack_bf16(o[8 * v + 6] * inv, o[8 * v + 7] * inv);
    *reinterpret_cast<uint4*>(dst + 8 * v) = x;
  }
}

// the output warps meet; the conjunction of their values
template <int THREADS>
__device__ __forceinline__ bool out_and(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "barrier.cta.red.and.pred q, 1, %2, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v), "n"(THREADS)
      : "memory");
  return r != 0;
}

template <int CG, bool OUT>
__global__ void __launch_bounds__(Warps<OUT>::THREADS, 1) attend_tc5_kernel(const __grid_constant__ Tc5Params p) {
  using R = Ring<CG>;
  using WP = Warps<OUT>;
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = smem_raw;
  const uint32_t s_q = smem_u32(smem);                  // two Q tiles
  if (s_q & 1023u) {  // (the declared alignment: cannot happen; the swizzled tiles would be misread)
    if (threadIdx.x == 0) atomicExch(p.status, -2034);
    return;
  }
  const uint32_t s_k = s_q + 2 * Q_TILE_BYTES;          // K ring
  const uint32_t s_v = s_k + R::KB * R::TILE;           // V ring
  const uint32_t s_bar = s_q + 2 * Q_TILE_BYTES + RING_BYTES;
  unsigned char* small = smem + 2 * Q_TILE_BYTES + RING_BYTES;
  volatile float* s_m = reinterpret_cast<volatile float*>(small + OFF_M);
  float* s_l = reinterpret_cast<float*>(small + OFF_L);
  unsigned long long* s_redo = reinterpret_cast<unsigned long long*>(small + OFF_REDO);
  volatile uint32_t* s_words = reinterpret_cast<volatile uint32_t*>(small + OFF_WORDS);
  volatile uint32_t* s_tmem_slot = s_words;
  volatile uint32_t* s_abort = s_words + 1;
  volatile uint32_t* s_over = s_words + 2;   // [2] by segment parity: number (+ 1) of the last segment with an overflow
  volatile uint32_t* s_fast = s_words + 4;   // every other part of the unit is in place
  volatile uint32_t* s_last = s_words + 5;
  volatile uint32_t* s_again = s_words + 6;  // segments are run again

  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const uint32_t rank = CG == 2 ? cluster_ctarank() : 0u;
  const bool leader = rank == 0;
  const int worker = (int)blockIdx.x / CG;
  auto bar = [&](int b) { return s_bar + 8u * (uint32_t)b; };
  auto lead_bar = [&](int b) { return CG == 2 ? mapa(s_bar + 8u * (uint32_t)b, 0) : s_bar + 8u * (uint32_t)b; };
  auto arrive_lead = [&](int b) {  // an arrival at the issuing CTA's barrier
    if constexpr (CG == 2)
      mbar_arrive_cluster(lead_bar(b));
    else
      mbar_arrive(bar(b));
  };

  // ---- one-time set-up -------------------------------------------------------------------------
  if (tid == 0) {
    const int peer = CG == 2 && leader ? 1 : 0;  // the other CTA's tiles are announced by its warp 3
    for (int i = 0; i < R::KB; ++i) {
      mbar_init(bar(B_KFULL + i), 1 + peer);
      mbar_init(bar(B_KEMPTY + i), 1);
    }
    for (int i = 0; i < R::VB; ++i) {
      mbar_init(bar(B_VFULL + i), 2 + peer);   // the copies' bytes (with their arrival) and the zeroed rows
      mbar_init(bar(B_VEMPTY + i), 1);
    }
    for (int i = 0; i < S_BUFS; ++i) {
      mbar_init(bar(B_SFULL + i), 1);
      mbar_init(bar(B_PREADY + i), 4 * CG);    // one arrival per softmax warp of the chunk's warpgroup(s)
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(B_QFULL + i), 8 + peer);   // eight softmax warps (first segment), or the Q warp eight at once
      mbar_init(bar(B_QFREE + i), 1);
    }
    mbar_init(bar(B_OFULL), 1);
    mbar_init(bar(B_OFREE), WP::OUT_WARPS * CG);
    for (int i = 0; i < 2; ++i) {
      mbar_init(bar(B_MREADY + i), 4);
      mbar_init(bar(B_LREADY + i), 8);
      mbar_init(bar(B_LFREE + i), WP::OUT_WARPS);
    }
    for (int i = 1; i < 7; ++i) s_words[i] = 0;
    *s_redo = 0ull;
    fence_barrier_init();
  }
  if (warp == 0) {
    tmem_alloc<CG>(smem_u32((const void*)s_tmem_slot), TMEM_COLS);
    tmem_relinquish<CG>();
  }
  fence_proxy_async();
  tc_fence_before();
  __syncthreads();
  if constexpr (CG == 2) cluster_sync_all();  // the peer's barriers are initialised before anything arrives there
  tc_fence_after();
  const uint32_t tmem = *s_tmem_slot;
  // (With early_q the softmax warps load the first Q tile before their wait.)  No warp releases the next launch before its own
  // wait: one thread's release counts for its CTA, and the next launch may take what this one's predecessors wrote as complete.
  const bool loads_q = warp >= SM_WARP0 && warp < OUT_WARP0;
  // The service warps wait where they first need what this launch's predecessors wrote: their index work comes before that.
  const bool waits_later = p.early_q && loads_q;
  auto depend = [&]() {
    if (!p.second) grid_dep_wait();
    grid_dep_launch();
  };
  if (!waits_later && warp >= SM_WARP0) depend();

  const uint32_t wait_limit = p.wait_limit ? p.wait_limit : WAIT_LIMIT;
  auto try_wait = [&](int b, uint32_t parity) -> bool {
    return mbar_try_wait(bar(b), parity);
  };
  auto wait = [&](int b, uint32_t parity) -> bool {
    for (uint32_t it = 0; it < wait_limit; ++it) {
      if (try_wait(b, parity)) return true;
      if (*s_abort) return false;
      if (it > 2048) __nanosleep(64);
    }
    *s_abort = 1;
    atomicExch(p.status, REKV_ERR_TIMEOUT);
    return false;
  };

  const int range0 = (int)(((long long)worker * p.total + p.W - 1) / p.W);
  const int range1 = (int)(((long long)(worker + 1) * p.total + p.W - 1) / p.W);
  const int Rc = p.ncf * p.Ns;                              // stream rows of the context
  const uint32_t page_half = (uint32_t)p.Nf * 128u;         // one 64-dim half of a head tile in a page
  // the bit of a segment in the run-again mask: the first and the last segment of a range (the only ones that can be
  // parts of a unit) have one of their own
  auto redo_bit = [&](int si, const Seg& s, int pos) -> unsigned long long {
    const bool last = pos + (s.I1 - s.I0) >= range1;
    return 1ull << (si == 0 ? 0 : last ? 1 : 2 + si % 62);
  };

  auto redo_mask = [&](bool either) -> unsigned long long {  // of this CTA, or of either CTA of the pair
    unsigned long long m = *reinterpret_cast<volatile unsigned long long*>(s_redo);
    if (CG == 2 && either) m |= ld_cluster_u64(mapa(smem_u32(s_redo), rank ^ 1u));
    return m;
  };

  // Q rows [r0, r0 + 2 * pairs) of a segment -> the swizzled K-major operand layout, two rows per instruction (16 lanes of 16
  // bytes each)
  auto load_q = [&](const Seg& s, uint32_t par, int r0, auto pairs) {
    const uint32_t dst = s_q + par * Q_TILE_BYTES + (uint32_t)((lane & 15) >> 3) * (Q_TILE_BYTES / 2);
    const int c = lane & 7;
    const __nv_bfloat16* src = p.q + (s.q_row0 * p.Hq + s.g * p.G) * 128 + (lane & 15) * 8;
#pragma unroll 8
    for (int k = 0; k < decltype(pairs)::value; ++k) {
      const int row = r0 + 2 * k + (lane >> 4);
      const int rr = s.m0 + (int)rank * 128 + row;
      const bool valid = rr < s.rows_q;
      const int n = rr / p.G, j = rr - n * p.G;
      cp_async16(dst + row * 128 + ((c ^ (row & 7)) << 4), src + (valid ? ((long long)n * p.Hq + j) * 128 : 0),
                 valid ? 16u : 0u);
    }
    cp_async_wait_all();
    fence_proxy_async();
    __syncwarp();
  };

  if (loads_q) {  // the first segment's Q
    load_q(decode_seg<CG>(p, range0, range1), 0, (warp - SM_WARP0) * 16, std::integral_constant<int, 8>{});
    if (lane == 0) mbar_arrive(bar(B_QFULL));
    if (waits_later) depend();
  }

  auto hand_back_o = [&]() {  // O has been read: the next segment's first P V may overwrite it
    tc_fence_before();
    __syncwarp();
    if (lane == 0) arrive_lead(B_OFREE);
  };
  // ================= a segment's result, one thread per row (and half of its columns without output warps) =================
  // With output warps (OUT) the softmax warps go on with the next segment's chunks meanwhile.
  auto result = [&](const Seg& s, int si, int pos, uint32_t segn, bool safe, bool& ok, int part) {
    const uint32_t par = segn & 1u;
    int row = ((warp & 3) << 5) | lane;
    if constexpr (!OUT) asm volatile("" : "+r"(row));   // (see the call)
    const int rr = s.m0 + (int)rank * 128 + row;
    const bool valid = rr < s.rows_q;
    const bool warp_idle = s.m0 + (int)rank * 128 + ((warp & 3) << 5) >= s.rows_q;
    const int n = rr / p.G, j = rr - n * p.G;
    const bool cut = s.I0 != 0 || s.I1 != s.nch;
    const bool boss = warp == (OUT ? OUT_WARP0 : SM_WARP0) && lane == 0;
    const int w_first = cut ? worker_of(p, s.uc0) : worker;
    const int n_parts = cut ? worker_of(p, s.uc0 + s.nch - 1) - w_first + 1 : 1;
    int* cnt = p.unit_cnt + w_first * CG + (int)rank;
    if (ok) ok = wait(B_LREADY + par, (segn >> 1) & 1u);
    const float m_own = s_m[par * 128 + row], l_own = s_l[par * 128 + row] * TRUNC_GAIN_INV;  // (the sums are of scaled values)
    const bool over = s_over[par] == segn + 1;
    if (boss && cut && p.merge_inside) *s_fast = __ldcg(cnt) == n_parts - 1;
    __syncwarp();
    if (OUT && lane == 0) mbar_arrive(bar(B_LFREE + par));
    if (ok) ok = wait(B_OFULL, segn & 1u);
    // (a wait that ran out ran out for all warps that meet below)
    if (OUT || (cut && p.merge_inside)) ok = out_and<32 * WP::OUT_WARPS>(ok);
    bool put = ok;
    if (ok && !safe && over) {
      put = false;
      if (boss) {
        atomicOr(s_redo, redo_bit(si, s, pos));
        if (CG == 2) fence_cluster();  // (the barrier at the end of the pass does not publish it)
      }
    }
    if (safe && !(redo_mask(false) & redo_bit(si, s, pos))) put = false;  // (the pair's other CTA asked for it)
    // O, 32 of the row's columns at a time.  The next segment's first P V waits until it has been read.  The range's last segment has
    // none behind it, and a pair hands nothing back: nobody would wait for the other CTA's arrival before the issuing one's shared memory
    // is given away.  (Waiting for it at the kernel's end: 28 layers, 64 tokens, 12 frames 107 -> 110 us, encoding step 239 -> 250.)
    const bool last = CG == 2 && !safe && pos + (s.I1 - s.I0) >= range1;
    const uint32_t t_o = tmem + ((uint32_t)((warp & 3) << 5) << 16);
    const int col0 = part * WP::COLUMNS;
    auto load_o = [&](int c0, float (&o)[32]) {
      uint32_t ou[32];
      tmem_ld32(t_o + (uint32_t)c0, ou);
      tmem_wait_ld32(ou);
#pragma unroll
      for (int i = 0; i < 32; ++i) o[i] = __uint_as_float(ou[i]);
    };
    auto o_free = [&]() {
      if (!last) hand_back_o();
    };
    if (put) tc_fence_after();
    __nv_bfloat16* dst = p.out + ((s.q_row0 + (valid ? n : 0)) * p.Hq + s.g * p.G + (valid ? j : 0)) * 128;
    if (!cut) {
      if (put && !warp_idle) {
        const float inv = l_own > 0.f ? 1.f / l_own : 0.f;
#pragma unroll 1
        for (int c0 = col0; c0 < col0 + WP::COLUMNS; c0 += 32) {
          float o[32];
          load_o(c0, o);
          if (valid) store_row_part(dst + c0, o, inv);
        }
      }
      o_free();
    } else {
      // a part of a unit: slot 2 w + 1 for a unit that starts in worker w's range, 2 w for one that started before
      const int slot = (2 * worker + (s.I0 == 0 ? 1 : 0)) * CG + (int)rank;
      const bool slot_ok = REKV_CHECK(slot >= 0 && slot < p.part_slots, p.status, 32);  // (checks build)
      const bool fast = p.merge_inside && *s_fast != 0;  // every other part is counted: no partial of its own
      bool finish = fast;
      if (!fast) {
        if (put && !warp_idle) {
#pragma unroll 1
          for (int c0 = col0; c0 < col0 + WP::COLUMNS; c0 += 32) {
            float o[32];
            load_o(c0, o);
            float4* po = p.part_o + ((long long)slot * 32 + (c0 >> 2)) * 128 + row;
            if (valid && slot_ok) {
#pragma unroll
              for (int v = 0; v < 8; ++v)
                po[(long long)v * 128] = make_float4(o[4 * v], o[4 * v + 1], o[4 * v + 2], o[4 * v + 3]);
            }
          }
          if (part == 0 && valid && slot_ok) p.part_ml[(long long)slot * 128 + row] = make_float2(m_own, l_own);
        }
        o_free();
        if (p.merge_inside) {  // publish, count, and join the parts if this one was the last
          __threadfence();
          out_and<32 * WP::OUT_WARPS>(true);
          if (boss) *s_last = put && atomicAdd(cnt, 1) == n_parts - 1;
          out_and<32 * WP::OUT_WARPS>(true);
          finish = *s_last != 0;
        }
      }
      // every part is counted: nobody else touches the counter in this launch, and the next one finds it at zero (a CTA
      // whose rows all lie beyond the unit's counts like any other)
      if (finish && put && boss) *cnt = 0;
      if (finish && put && !warp_idle) {
        __threadfence();
        // M = the maximum over the parts, weights 2^(m_k - M), numerators and denominator accumulated in part order: the
        // same arithmetic whichever worker came last
        const int own = fast ? worker - w_first : -1;  // (its own partial, where it wrote one, is read like the others)
        float2 ml[MAX_PARTS_INSIDE];
        float M = -1e30f;
#pragma unroll
        for (int k = 0; k < MAX_PARTS_INSIDE; ++k) {
          ml[k] = make_float2(-INFINITY, 0.f);
          if (k < n_parts) {
            const int sk = (2 * (w_first + k) + (k == 0 ? 1 : 0)) * CG + (int)rank;
            ml[k] = k == own ? make_float2(m_own, l_own) : __ldcg(p.part_ml + (long long)sk * 128 + row);
            M = fmaxf(M, ml[k].x);
          }
        }
        float den = 0.f;
#pragma unroll
        for (int k = 0; k < MAX_PARTS_INSIDE; ++k) {
          ml[k].x = ex2(ml[k].x - M);
          den = fmaf(ml[k].x, ml[k].y, den);
        }
        const float inv = den > 0.f ? 1.f / den : 0.f;
#pragma unroll 1
        for (int c0 = col0; c0 < col0 + WP::COLUMNS; c0 += 32) {
          float acc[32];
#pragma unroll
          for (int i = 0; i < 32; ++i) acc[i] = 0.f;
#pragma unroll
          for (int k = 0; k < MAX_PARTS_INSIDE; ++k)
            if (k < n_parts) {
              const float w = ml[k].x;
              if (k == own) {
                float o[32];
                load_o(c0, o);
#pragma unroll
                for (int i = 0; i < 32; ++i) acc[i] = fmaf(w, o[i], acc[i]);
              } else {
                const int sk = (2 * (w_first + k) + (k == 0 ? 1 : 0)) * CG + (int)rank;
                const float4* po = p.part_o + ((long long)sk * 32 + (c0 >> 2)) * 128 + row;
                float4 x[8];
#pragma unroll
                for (int v = 0; v < 8; ++v) x[v] = __ldcg(po + (long long)v * 128);
#pragma unroll
                for (int v = 0; v < 8; ++v) {
                  acc[4 * v] = fmaf(w, x[v].x, acc[4 * v]);
                  acc[4 * v + 1] = fmaf(w, x[v].y, acc[4 * v + 1]);
                  acc[4 * v + 2] = fmaf(w, x[v].z, acc[4 * v + 2]);
                  acc[4 * v + 3] = fmaf(w, x[v].w, acc[4 * v + 3]);
                }
              }
            }
          if (valid) store_row_part(dst + c0, acc, inv);
        }
      }
      if (fast) o_free();
      if (p.merge_inside) out_and<32 * WP::OUT_WARPS>(true);  // (s_fast and s_last have been read)
    }
  };

  // The roles run the same range loop with the role as a compile-time constant, so that each side of the register
  // reallocation below is compiled against its own register budget.  Pass 0 runs the whole range; pass 1, only
  // if some row's reference maximum was too low, runs the marked segments again.
  auto run = [&](auto role) {
    constexpr int ROLE = decltype(role)::value;  // 0: copies and products, 1: softmax, 2: output
    uint32_t t = 0;        // chunks so far (both passes): ring slots and barrier phases follow from it
    uint32_t segn = 0;     // segments so far
    uint32_t issued = 0, phase = 0;  // producers: tiles whose copies are on their way; parity of the ring's current round
    int slot = 0;                    // ... and their next ring entry
    bool ok = true;
#pragma unroll 1
    for (int pass = 0; pass < 2; ++pass) {
      const bool safe = pass == 1;
      const uint32_t ahead = safe ? 1u : (uint32_t)S_BUFS;  // S runs this many chunks before P V
      uint32_t t_base = t;                                  // first chunk of the pass
      uint32_t pend0 = 0, pend1 = 0, pend2 = 0;             // MMA issuer: P V of the chunks t-3, t-2, t-1
      int pos = range0;
      // (without output warps the softmax warps meet at the cut segments of launches that join them: a warp whose wait ran out goes
      // through the rest of the range without waiting, so that it is missing at no such meeting)
      const bool meets = ROLE == 1 && !OUT && p.merge_inside != 0;
#pragma unroll 1
      for (int si = 0; pos < range1 && (ok || meets); ++si) {
        const Seg s = decode_seg<CG>(p, pos, range1);
        const int nseg = s.I1 - s.I0;
        if (safe && !(redo_mask(true) & redo_bit(si, s, pos))) {
          pos += nseg;
          continue;
        }
        const uint32_t par = segn & 1u;
        const int R_end = stream_rows(p, s.nx);
        const int x_off = s.nx ? ((p.sb.cu[s.qi] + 7) & ~7) + 8 * s.qi : 0;  // X's first staged row

        if constexpr (ROLE == 0) {
          auto produce = [&](auto which) {
            // ================= producers =================
            constexpr int kv = decltype(which)::value;
            char* const* pages = p.tbl + ((long long)s.l * p.qb.nQ + s.qi) * p.ncf;
            if (kv == 0 && p.tbl_k) pages = p.tbl_k + ((long long)s.l * p.qb.nQ + s.qi) * p.ncf;
            // offset of this tile (of its first half) in a page; rotated copies hold the K tiles alone
            const long long tile_off = kv == 0 ? (p.tbl_k ? (long long)s.g * 2 * page_half : (long long)s.g * 4 * page_half)
                                               : (long long)s.g * 4 * page_half + 2 * page_half;
            const char* xt = p.x_kv ? p.x_kv + (((long long)(s.l * p.Hkv + s.g) * 2 + kv) * 2 * p.x_rows + x_off) * 128 : nullptr;
            // Everything per chunk is stepped, not divided: this loop's length is prefetch depth lost (at 1400 cycles per chunk
            // for V it was the whole kernel's pace).
            constexpr int nb = kv == 0 ? R::KB : R::VB;
            constexpr int halves = kv == 0 || CG == 1 ? 2 : 1;   // 64-dim halves of the tile in this CTA: both, except a pair's V
            const uint32_t ring0 = kv == 0 ? s_k : s_v;
            constexpr uint32_t dst_half = kv == 0 ? R::K_HALF : V_HALF;
            constexpr int width = kv == 0 ? R::K_ROWS : CHUNK;   // stream rows of this CTA's part of the tile: a pair's CTA r takes
            const int shift = kv == 0 ? (int)rank * R::K_ROWS : 0;  // tokens [64 r, 64 r + 64) of K, and V's 64-dim half r
            const long long src_half = lane == 31 ? p.x_rows * 128 : (long long)page_half;
            const long long src_off = (lane == 31 ? 0ll : tile_off) + (kv == 1 && CG == 2 ? (long long)rank * src_half : 0ll);
            int a = s.I0 * CHUNK + shift;
            int f_lo = a / p.Ns, pos_a = a - f_lo * p.Ns;    // row a is row pos_a of frame f_lo
            int fb = -64;                                    // a lane holds the page pointer of frame fb + lane
            const char* my_page = nullptr;
            if (issued == 0) depend();
#pragma unroll 1
            for (int I = s.I0; I < s.I1 && ok; ++I) {
              if (f_lo < p.ncf && f_lo + 17 >= fb + 32) {
                fb = f_lo;
                my_page = reinterpret_cast<const char*>(
                    __ldcg(reinterpret_cast<const unsigned long long*>(pages) + min(fb + lane, p.ncf - 1)));
              }
              // lane i < 31: the piece of frame f_lo + i; lane 31: the piece of X.  rel: its first row, from a
              const char* page = reinterpret_cast<const char*>(__shfl_sync(
                  0xffffffffu, reinterpret_cast<unsigned long long>(my_page), (f_lo - fb + lane) & 31));
              const int rows = min(width, R_end - a);
              const int rel = lane == 31 ? Rc - a : lane * p.Ns - pos_a;
              const bool real = lane == 31 ? s.nx > 0 : f_lo + lane < p.ncf;
              const int ta = max(0, -rel), tb = min(lane == 31 ? s.nx : p.Nf, rows - rel);
              const uint32_t n_bytes = real && tb > ta ? (uint32_t)(tb - ta) * 128u : 0u;
              const char* src = (lane == 31 ? xt : page) + src_off + (long long)ta * 128;
              const uint32_t dst0 = ring0 + (uint32_t)slot * R::TILE;
              const uint32_t dst = dst0 + (uint32_t)(rel + ta) * 128u;
              const uint32_t sum = __reduce_add_sync(0xffffffffu, n_bytes) * (uint32_t)halves;
              if (issued >= (uint32_t)nb && !wait((kv == 0 ? B_KEMPTY : B_VEMPTY) + slot, phase ^ 1u)) {
                ok = false;
                break;
              }
              const int full = (kv == 0 ? B_KFULL : B_VFULL) + slot;
              const bool skip = p.skip_copy_entry >= 0 && blockIdx.x == 0 && (int)(2 * issued) + kv == p.skip_copy_entry;  // test-only
              if (!skip) {
                if (lane == 0) mbar_expect_tx(bar(full), sum);
                __syncwarp();
                // (checks build) a piece must lie inside its tile half and start on 16 bytes at both ends; one that does
                // not is left out, and the wait for the tile then runs out and reports it
                if (n_bytes && REKV_CHECK(src != nullptr && (reinterpret_cast<uintptr_t>(src) & 15) == 0 && rel + ta >= 0 &&
                                              dst + n_bytes <= dst0 + dst_half && dst >= dst0,
                                          p.status, 31)) {
                  bulk_g2s(dst, src, n_bytes, bar(full));
                  if (halves == 2) bulk_g2s(dst + dst_half, src + src_half, n_bytes, bar(full));
                }
              }
              if constexpr (kv == 1) {
                // V rows without a token -- the frames' gap rows, and the rows after the stream's end up to the products'
                // depth (lane 30's piece) -- are zeroed behind the tile's second arrival; the copies do not touch them
                const int N = (rows + 15) & ~15;
                const int z0 = lane == 30 ? rows : max(0, rel + p.Nf);
                const int z1 = lane == 30 ? N : lane < 30 && real ? min(rows, rel + p.Ns) : 0;
                uint32_t gaps = __ballot_sync(0xffffffffu, z1 > z0);
                if (gaps) {
                  unsigned char* tile = smem + (dst0 - s_q) + (lane & 7) * 16;
                  while (gaps) {
                    const int l = __ffs(gaps) - 1;
                    gaps &= gaps - 1;
                    const int g0 = __shfl_sync(0xffffffffu, z0, l), g1 = __shfl_sync(0xffffffffu, z1, l);
                    for (int r = g0 + (lane >> 3); r < g1; r += 4) {
                      *reinterpret_cast<uint4*>(tile + r * 128) = make_uint4(0, 0, 0, 0);
                      if (CG == 1) *reinterpret_cast<uint4*>(tile + r * 128 + V_HALF) = make_uint4(0, 0, 0, 0);
                    }
                  }
                  fence_proxy_async();
                  __syncwarp();
                }
                if (lane == 0 && !skip) mbar_arrive(bar(full));
              }
              ++issued;
              if (++slot == nb) {
                slot = 0;
                phase ^= 1u;
              }
              a += CHUNK;
              pos_a += CHUNK;
              while (pos_a >= p.Ns) {
                pos_a -= p.Ns;
                ++f_lo;
              }
            }
          };
          if (warp == 0) {
            produce(std::integral_constant<int, 0>{});
          } else if (warp == 2) {
            produce(std::integral_constant<int, 1>{});
          } else if (warp == 1 && leader) {
            // ================= MMA issuer =================
            // S of chunk t, then P V of chunk t - ahead.  Descriptors are built once; per instruction only the 14-bit
            // start-address field advances.
            const uint32_t desc_hi = (1024u >> 4) | (1u << 14) | (2u << 29);  // SBO = 1024 B, version, SWIZZLE_128B
            const uint32_t lbo_v = ((V_HALF >> 4) & 0x3FFFu) << 16;           // pitch of V's two 64-dim blocks (CG = 1)
            const uint32_t lbo_k = 1u << 16;                                  // unused for K-major operands
            const uint32_t idesc_s = idesc_bf16(128 * CG, CHUNK, 0), idesc_pv = idesc_bf16(128 * CG, 128, 1);
            auto desc = [&](uint32_t lo) { return ((uint64_t)desc_hi << 32) | (uint64_t)lo; };
            // a pending P V: bits 0-3 depth in 16-token steps, bit 4 first of its segment, bit 5 last, bits 6.. segment
            auto issue_pv = [&](uint32_t tt, uint32_t d) {
              const uint32_t slot = tt % R::VB;
              const uint32_t sg = d >> 6;
              if (ok) ok = wait(B_VFULL + slot, (tt / R::VB) & 1u);
              if (ok && (d & 16u) && sg > 0) ok = wait(B_OFREE, (sg - 1) & 1u);
              if (ok) ok = wait(B_PREADY + tt % S_BUFS, (tt / S_BUFS) & 1u);
              if (!ok) return;
              tc_fence_after();
              const uint32_t v_lo = ((s_v + slot * R::TILE) >> 4) | lbo_v;
              const uint32_t a_ = tmem + 128u + (tt % S_BUFS) * 128u;
              const int nk = (int)(d & 15u);
              if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < 8; ++kk)
                  if (kk < nk) mma_ts<CG>(tmem, a_ + 8 * kk, desc(v_lo + 128 * kk), idesc_pv, !(d & 16u) || kk > 0);
                tc_commit<CG>(bar(B_VEMPTY + slot));
                if (d & 32u) tc_commit<CG>(bar(B_OFULL));
              }
              __syncwarp();
            };
#pragma unroll 1
            for (int I = s.I0; I < s.I1 && ok; ++I) {
              const uint32_t tt = t + (uint32_t)(I - s.I0);
              if (tt - t_base >= ahead) {
                issue_pv(tt - ahead, safe ? pend2 : pend0);
                if (!ok) break;
              }
              if (I == s.I0) {
                ok = wait(B_QFULL + par, (segn >> 1) & 1u);
                fence_proxy_async();  // (the Q rows came through generic-proxy copies)
              }
              const uint32_t slot = tt % R::KB;
              if (ok) ok = wait(B_KFULL + slot, (tt / R::KB) & 1u);
              if (!ok) break;
              tc_fence_after();
              const uint32_t k_lo = ((s_k + slot * R::TILE) >> 4) | lbo_k;
              const uint32_t q_lo = ((s_q + par * Q_TILE_BYTES) >> 4) | lbo_k;
              const uint32_t d_ = tmem + 128u + (tt % S_BUFS) * 128u;
              if (elect_one()) {
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                  mma_ss<CG>(d_, desc(q_lo + 2 * kk), desc(k_lo + 2 * kk), idesc_s, kk > 0);
#pragma unroll
                for (int kk = 0; kk < 4; ++kk)
                  mma_ss<CG>(d_, desc(q_lo + (Q_TILE_BYTES / 32) + 2 * kk), desc(k_lo + (R::K_HALF >> 4) + 2 * kk), idesc_s, 1);
                tc_commit<CG>(bar(B_SFULL + tt % S_BUFS));
                tc_commit<CG>(bar(B_KEMPTY + slot));
                if (I == s.I1 - 1) tc_commit<CG>(bar(B_QFREE + par));
              }
              __syncwarp();
              const uint32_t nk = (uint32_t)(min(CHUNK, R_end - I * CHUNK) + 15) >> 4;
              pend0 = pend1;
              pend1 = pend2;
              pend2 = nk | (I == s.I0 ? 16u : 0u) | (I == s.I1 - 1 ? 32u : 0u) | (segn << 6);
            }
            // end of the pass: the P V still outstanding
            if (ok && pos + nseg >= range1 && !safe) {
              const uint32_t t1 = t + (uint32_t)nseg;
              const uint32_t n = min((uint32_t)S_BUFS, t1 - t_base);
              if (n >= 3) issue_pv(t1 - 3, pend0);
              if (n >= 2 && ok) issue_pv(t1 - 2, pend1);
              if (n >= 1 && ok) issue_pv(t1 - 1, pend2);
            }
            if (ok && safe) {  // a segment that is run again is finished before the next
              issue_pv(t + (uint32_t)nseg - 1, pend2);
              t_base = t + (uint32_t)nseg;
            }
          } else if (CG == 2 && warp == 3 && !leader) {
            // ================= relay: this CTA's tiles, announced to the issuing CTA in the order it waits for them =====
            auto pass_on = [&](int b, uint32_t parity) {
              if (ok) ok = wait(b, parity);
              if (ok && lane == 0) arrive_lead(b);
              __syncwarp();
            };
#pragma unroll 1
            for (int I = s.I0; I < s.I1 && ok; ++I) {
              const uint32_t tt = t + (uint32_t)(I - s.I0);
              if (tt - t_base >= ahead) pass_on(B_VFULL + (tt - ahead) % R::VB, ((tt - ahead) / R::VB) & 1u);
              if (I == s.I0) {
                if (ok) ok = wait(B_QFULL + par, (segn >> 1) & 1u);
                fence_proxy_async();
                if (ok && lane == 0) arrive_lead(B_QFULL + par);
                __syncwarp();
              }
              pass_on(B_KFULL + tt % R::KB, (tt / R::KB) & 1u);
            }
            const uint32_t t1 = t + (uint32_t)nseg;
            if (safe || pos + nseg >= range1) {
              for (uint32_t n = min(ahead, t1 - t_base); n > 0; --n) pass_on(B_VFULL + (t1 - n) % R::VB, ((t1 - n) / R::VB) & 1u);
              t_base = t1;
            }
          } else if (segn > 0) {
            // ================= Q of the segments after the first, behind the current one's work =================
            // (the first segment's rows are loaded by the eight softmax warps, which have nothing else to do yet: by one
            // warp they took 5 us)
            if (segn == 1) depend();
            if (segn >= 2) ok = wait(B_QFREE + par, ((segn >> 1) - 1) & 1u);
            if (ok) {
              load_q(s, par, 0, std::integral_constant<int, 64>{});
              if (lane == 0) mbar_arrive_n(bar(B_QFULL + par), 8);
            }
          }
        } else if constexpr (ROLE == 1) {
          // ================= softmax, one thread per row =================
          const int wg = (warp - SM_WARP0) >> 2;           // this warpgroup takes the chunks with t % 2 == wg
          const uint32_t lane_base = (uint32_t)((warp & 3) << 5) << 16;
          const int row = ((warp & 3) << 5) | lane;
          // a warp whose 32 rows all lie beyond the unit's rows only keeps the barriers moving
          const bool warp_idle = s.m0 + (int)rank * 128 + ((warp & 3) << 5) >= s.rows_q;
          // last stream row this row sees among X's tokens
          const int lim = Rc + (s.nx - s.nq) + (s.m0 + (int)rank * 128 + row) / p.G;
          const int first_wg = safe ? 0 : (int)(t & 1u);
          const int rows_in = s.nx ? Rc : R_end;           // chunks that end at or before this row need no tail mask
          const uint32_t gap_bits = p.Ns != p.Nf ? (0xFFu << (p.Nf & 7)) & 0xFFu : 0u;  // gap columns of an 8-row group
          float m_used = 0.f, l_sum = 0.f;
          bool over = false, have_m = false;
          // the state of the segment before the last has been read: its places and barriers are this one's
          // (without output warps this warpgroup has read it itself, after the other one was done with it)
          if (OUT && segn >= 2) ok = wait(B_LFREE + par, ((segn >> 1) - 1) & 1u);
          int i0 = wg ^ first_wg;
          if (safe && wg != 0) i0 = nseg;
          const int istep = safe ? 1 : 2;
          int pos0 = (int)(((long long)(s.I0 + i0) * CHUNK) % p.Ns);
          const int pstep = (istep * CHUNK) % p.Ns;
#pragma unroll 1
          for (int i = i0; i < nseg && ok; i += istep) {
            const uint32_t c = t + (uint32_t)i;
            const uint32_t buf = c % S_BUFS;
            const uint32_t t_s = tmem + lane_base + 128u + buf * 128u;
            const int row0 = (s.I0 + i) * CHUNK;
            const int p0 = pos0;
            pos0 += pstep;
            if (pos0 >= p.Ns) pos0 -= p.Ns;
            if (!wait(B_SFULL + buf, (c / S_BUFS) & 1u)) {
              ok = false;
              break;
            }
            tc_fence_after();
            if (warp_idle) {  // no valid row in this warp's 32 lanes: their P and O rows are never read back
              tc_fence_before();
              __syncwarp();
              if (lane == 0) {
                if (i == 0) mbar_arrive(bar(B_MREADY + par));
                arrive_lead(B_PREADY + buf);
              }
              continue;
            }
            const float NEG_INF = -INFINITY;
            uint32_t sv[128];
            if constexpr (OUT) {  // (an instruction's registers must fit those at launch)
              tmem_ld64<0>(t_s, sv);
              tmem_ld64<64>(t_s + 64, sv);
            } else {
              tmem_ld128(t_s, sv);
            }
            tmem_wait_ld128(sv);
            // Columns without a token.  N_s is a multiple of 8 and so is every frame's start, so a frame's gap is the end
            // of one aligned 8-column group, with the same bits in every frame: the groups that have one are found by
            // stepping over the frames, each masked behind a warp-uniform switch.
            if (row0 + CHUNK <= rows_in) {
              if (gap_bits) {
#pragma unroll 1
                for (int e = p.Ns - p0; e <= CHUNK; e += p.Ns) {
#define REKV_MASK8(GI)                                                        \
  case GI:                                                                    \
    _Pragma("unroll") for (int jj = 1; jj < 8; ++jj)                          \
      if ((gap_bits >> jj) & 1u) sv[8 * (GI) + jj] = __float_as_uint(NEG_INF); \
    break;
                  switch ((e >> 3) - 1) {
                    REKV_MASK8(0) REKV_MASK8(1) REKV_MASK8(2) REKV_MASK8(3) REKV_MASK8(4) REKV_MASK8(5) REKV_MASK8(6)
                    REKV_MASK8(7) REKV_MASK8(8) REKV_MASK8(9) REKV_MASK8(10) REKV_MASK8(11) REKV_MASK8(12) REKV_MASK8(13)
                    REKV_MASK8(14) REKV_MASK8(15)
                    default: break;
                  }
#undef REKV_MASK8
                }
              }
            } else {  // the stream's last chunks: gaps, the end, and X's causal limit
              uint32_t mk[4];
#pragma unroll
              for (int k = 0; k < 4; ++k) {
                const int col = lane + 32 * k;
                const bool gap = row0 + col < Rc && (p0 + col) % p.Ns >= p.Nf;
                mk[k] = __ballot_sync(0xffffffffu, row0 + col >= R_end || gap);
                if (s.nx) {
                  const int x = lim - row0 - 32 * k;  // last visible column of these 32
                  mk[k] |= x >= 31 ? 0u : x < 0 ? 0xffffffffu : 0xfffffffeu << x;
                }
              }
#pragma unroll
              for (int jj = 0; jj < 128; ++jj)
                if ((mk[jj >> 5] >> (jj & 31)) & 1u) sv[jj] = __float_as_uint(NEG_INF);
            }
            auto row_max = [&]() -> float {  // of the chunk's logits, in log2 units
              float gmx[8];
#pragma unroll
              for (int a8 = 0; a8 < 8; ++a8)
                gmx[a8] = max3(__uint_as_float(sv[a8]), __uint_as_float(sv[8 + a8]), __uint_as_float(sv[16 + a8]));
#pragma unroll
              for (int cc = 24; cc + 16 <= 128; cc += 16)
#pragma unroll
                for (int a8 = 0; a8 < 8; ++a8)
                  gmx[a8] = max3(gmx[a8], __uint_as_float(sv[cc + a8]), __uint_as_float(sv[cc + 8 + a8]));
#pragma unroll
              for (int a8 = 0; a8 < 8; ++a8) gmx[a8] = fmaxf(gmx[a8], __uint_as_float(sv[120 + a8]));
              return max3(max3(gmx[0], gmx[1], gmx[2]), max3(gmx[3], gmx[4], gmx[5]), fmaxf(gmx[6], gmx[7])) * p.scale_log2;
            };
            // P = 2^(S*scale - m) as bf16 pairs over the front of S (two stores of 32 columns); returns the row sum.
            // The conversion instruction shares the transcendental unit with ex2 (a quarter-rate pipe), so P is cut to
            // bf16 by taking the upper halves (one byte permute per pair) of 2^(x - m) * (1 + TRUNC_GAIN), the factor
            // that makes the cut value equal to 2^(x - m) on average over the mantissa -- folded into the exponent,
            // and taken out of the row sum once at the end.  All 128 columns are done whatever the chunk's width
            // (masked columns give exactly 0): one straight run of code keeps the transcendental unit fed.  Scaling and
            // summing take two columns per instruction: a long launch runs at the card's power limit, where fewer
            // instructions are time (1800-frame question 279 -> 271 us, 16-question batch 3440 -> 3343).
            auto exp_pass = [&]() -> float {
              const float neg_m = TRUNC_GAIN_LOG2 - m_used;
              float ps0 = 0.f, ps1 = 0.f, ps2 = 0.f, ps3 = 0.f;
#pragma unroll
              for (int hf = 0; hf < 2; ++hf) {
                uint32_t pk[32];
#pragma unroll
                for (int jj = 0; jj < 32; jj += 2) {
                  const uint32_t* v = sv + 64 * hf;
                  float e0 = __uint_as_float(v[2 * jj]), e1 = __uint_as_float(v[2 * jj + 1]);
                  float e2 = __uint_as_float(v[2 * jj + 2]), e3 = __uint_as_float(v[2 * jj + 3]);
                  fma_f32x2(e0, e1, p.scale_log2, neg_m);
                  fma_f32x2(e2, e3, p.scale_log2, neg_m);
                  e0 = ex2(e0);
                  e1 = ex2(e1);
                  e2 = ex2(e2);
                  e3 = ex2(e3);
                  add_f32x2(ps0, ps1, e0, e1);
                  add_f32x2(ps2, ps3, e2, e3);
                  pk[jj] = __byte_perm(__float_as_uint(e0), __float_as_uint(e1), 0x7632);
                  pk[jj + 1] = __byte_perm(__float_as_uint(e2), __float_as_uint(e3), 0x7632);
                }
                tmem_st32(t_s + 32 * hf, pk);
              }
              return (ps0 + ps1) + (ps2 + ps3);
            };
            if (i == 0) {  // the segment's first chunk: its row maximum becomes the reference of both warpgroups
              m_used = fmaxf(row_max(), -1e30f);  // (a row that sees nothing keeps a finite reference)
              have_m = true;
              s_m[par * 128 + row] = m_used;
              s_l[par * 128 + row] = 0.f;
              __syncwarp();
              if (lane == 0) mbar_arrive(bar(B_MREADY + par));
            } else if (!have_m) {
              if (!wait(B_MREADY + par, (segn >> 1) & 1u)) {
                ok = false;
                break;
              }
              m_used = s_m[par * 128 + row];
              have_m = true;
            }
            if (safe && i > 0) {
              // run again, chunk by chunk: a row whose maximum lies above the reference raises it, and O and the row sum
              // shrink by 2^(old - new).  Every earlier P V is complete (this chunk's S was issued after it).
              const float gm = row_max();
              const bool need = gm > m_used + 8.f;
              if (__any_sync(0xffffffffu, need)) {
                const float alpha = need ? ex2(m_used - gm) : 1.f;
                if (need) m_used = gm;
                l_sum *= alpha;
#pragma unroll 1
                for (int pc = 0; pc < 8; ++pc) {
                  uint32_t o[16];
                  tmem_ld16(tmem + lane_base + pc * 16, o);
                  tmem_wait_ld16(o);
#pragma unroll
                  for (int e = 0; e < 16; ++e) o[e] = __float_as_uint(__uint_as_float(o[e]) * alpha);
                  tmem_st16(tmem + lane_base + pc * 16, o);
                }
              }
            }
            const float cs = exp_pass();
            // (a logit more than 60 octaves above the reference: the segment has to be run again)
            if (__any_sync(0xffffffffu, !(cs < RESCALE_SUM_LIMIT))) over = true;
            l_sum += cs;
            tmem_wait_st();
            tc_fence_before();
            __syncwarp();
            if (lane == 0) arrive_lead(B_PREADY + buf);
          }

          // the row's sum and reference for the output warps (two addends, whose order does not matter; a segment that is run
          // again is warpgroup 0's alone)
          if (!warp_idle) {
            if (safe && wg == 0) {
              s_l[par * 128 + row] = l_sum;
              s_m[par * 128 + row] = m_used;
            } else if (have_m) {
              atomicAdd(s_l + par * 128 + row, l_sum);
            }
            if (over) s_over[par] = segn + 1;
          }
          __syncwarp();
          if (lane == 0) mbar_arrive(bar(B_LREADY + par));
          if constexpr (!OUT) {
            // (worked out again, from values the compiler cannot trace back, instead of being held in registers -- or in local
            // memory -- through the chunk loop, as everything that is constant over the segments otherwise would be)
            int pos_e = pos, wg_e = wg;
            asm volatile("" : "+r"(pos_e), "+r"(wg_e));
            result(decode_seg<CG>(p, pos_e, range1), si, pos_e, segn, safe, ok, wg_e);
          }
        } else {
          result(s, si, pos, segn, safe, ok, 0);
        }
        t += (uint32_t)nseg;
        ++segn;
        pos += nseg;
      }
      if (pass == 0) {
        // every role and both CTAs of a pair have finished the range: is there anything to run again?
        __syncwarp();
        if constexpr (CG == 2)
          cluster_sync_relaxed();
        else
          __syncthreads();
        if (redo_mask(true) == 0ull || *s_abort) break;
        if constexpr (CG == 2) {
          *s_again = 1;
          if constexpr (ROLE == (OUT ? 2 : 1)) hand_back_o();   // the last segment's, after all
        }
      }
    }
    if constexpr (ROLE == 0) {
      // A CTA that gives up must not return while copies into its shared memory are still on their way: the producers
      // wait (bounded) for the tiles they have issued and nobody consumed -- at most the rings' depth.
      if (*s_abort && (warp == 0 || warp == 2)) {
        const uint32_t nb = warp == 0 ? R::KB : R::VB;
        for (uint32_t r = issued > nb ? issued - nb : 0; r < issued; ++r)
          for (uint32_t it = 0; it < wait_limit && !try_wait((warp == 0 ? B_KFULL : B_VFULL) + (int)(r % nb), (r / nb) & 1u); ++it)
            __nanosleep(64);
      }
    }
  };
  if (warp < SM_WARP0) {
    reg_dealloc<WP::REGS_SERVICE>();
    run(std::integral_constant<int, 0>{});
  } else if (warp < OUT_WARP0) {
    reg_alloc<WP::REGS_SOFTMAX>();
    run(std::integral_constant<int, 1>{});
  } else {
    if constexpr (OUT) {
      reg_dealloc<WP::REGS_OUT>();
      run(std::integral_constant<int, 2>{});
    }
  }

  __syncwarp();
  tc_fence_before();
  if constexpr (CG == 2) {
    // (a pair that gave up, or ran segments again, has not waited for all of each other's arrivals: the barrier orders them)
    if (__any_sync(0xffffffffu, (*s_abort | *s_again) != 0))
      cluster_sync_all();
    else
      cluster_sync_relaxed();
  } else {
    __syncthreads();
  }
  if (p.second) grid_dep_wait();
  if (warp == 0) tmem_dealloc<CG>(tmem, TMEM_COLS);
}

// Joins the parts of units where the attention kernel does not (launches of few units, such as one layer: several whole workers
// each; units of more than MAX_PARTS_INSIDE parts).
// grid = (units, CTAs of a pair, 32 column quads), 256 threads: a thread per (row, every second part), consecutive threads on
// consecutive rows, so that a part is read in 2 KB runs and up to 20 parts are one round of loads: MERGE_AHEAD in flight per thread
// (rekv_merge_ahead); the two groups' results meet in shared memory.  (Four groups instead of two, eight in flight: 962 us against 946
// for 28 layers of 28 heads, 72 frames, one at a time.)
constexpr int MERGE_GROUPS = 2;
template <int CG, int MERGE_AHEAD>
__global__ void __launch_bounds__(128 * MERGE_GROUPS, MERGE_AHEAD <= 4 ? 5 : MERGE_AHEAD <= 8 ? 3 : 2) merge_tc5_kernel(const __grid_constant__ Tc5Params p) {
  const int lh = (int)blockIdx.x / p.W, rank = blockIdx.y;  // blockIdx.x counts (layer, kv head) x row blocks; W = row blocks
  int mp = (int)blockIdx.x - lh * p.W, qi = 0, c0 = lh * p.per_lh;
  for (; qi < p.qb.nQ - 1; ++qi) {
    const int nb = row_blocks<CG>(p, qi);
    if (mp < nb) break;
    mp -= nb;
    c0 += nb * stream_chunks(p, qi);
  }
  const int nch = stream_chunks(p, qi);
  c0 += mp * nch;
  const int W = p.merge_inside;  // (this kernel's copy of the parameters: the attention launch's workers)
  auto worker_at = [&](int c) { return (int)((long long)c * W / p.total); };
  const int w0 = worker_at(c0), n_parts = worker_at(c0 + nch - 1) - w0 + 1;
  const int row = threadIdx.x & 127, grp = threadIdx.x >> 7, quad = blockIdx.z;
  const int rows_q = (p.qb.cu[qi + 1] - p.qb.cu[qi]) * p.G;
  const int row_b = block_row0<CG>(p, rows_q, mp) + rank * 128;
  const int rr = row_b + row;
  __shared__ float4 s_o[MERGE_GROUPS][128];
  __shared__ float2 s_ml[MERGE_GROUPS][128];
  grid_dep_wait();
  grid_dep_launch();
  if (n_parts <= 1 || row_b >= rows_q) return;  // (the whole block)
  float M = -1e30f, den = 0.f;
  float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
  if (rr < rows_q) {
#pragma unroll 1
    for (int k0 = grp; k0 < n_parts; k0 += MERGE_AHEAD * MERGE_GROUPS) {
      float2 ml[MERGE_AHEAD];
      float4 o[MERGE_AHEAD];
#pragma unroll
      for (int i = 0; i < MERGE_AHEAD; ++i) {
        const int k = k0 + i * MERGE_GROUPS;
        ml[i] = make_float2(-INFINITY, 0.f);
        o[i] = make_float4(0.f, 0.f, 0.f, 0.f);
        if (k < n_parts) {
          const long long sk = (long long)(2 * (w0 + k) + (k == 0 ? 1 : 0)) * CG + rank;
          ml[i] = p.part_ml[sk * 128 + row];
          o[i] = p.part_o[(sk * 32 + quad) * 128 + row];
        }
      }
      float Mn = M;
#pragma unroll
      for (int i = 0; i < MERGE_AHEAD; ++i) Mn = fmaxf(Mn, ml[i].x);
      const float a = ex2(M - Mn);
      M = Mn;
      den *= a;
      acc.x *= a;
      acc.y *= a;
      acc.z *= a;
      acc.w *= a;
#pragma unroll
      for (int i = 0; i < MERGE_AHEAD; ++i) {
        const float w = ex2(ml[i].x - M);
        den = fmaf(w, ml[i].y, den);
        acc.x = fmaf(w, o[i].x, acc.x);
        acc.y = fmaf(w, o[i].y, acc.y);
        acc.z = fmaf(w, o[i].z, acc.z);
        acc.w = fmaf(w, o[i].w, acc.w);
      }
    }
  }
  s_o[grp][row] = acc;
  s_ml[grp][row] = make_float2(M, den);
  __syncthreads();
  if (grp != 0 || rr >= rows_q) return;
  float Mx = M;
#pragma unroll
  for (int i = 1; i < MERGE_GROUPS; ++i) Mx = fmaxf(Mx, s_ml[i][row].x);
  acc = make_float4(0.f, 0.f, 0.f, 0.f);
  den = 0.f;
#pragma unroll
  for (int i = 0; i < MERGE_GROUPS; ++i) {
    const float w = ex2(s_ml[i][row].x - Mx);
    const float4 o = s_o[i][row];
    den = fmaf(w, s_ml[i][row].y, den);
    acc.x = fmaf(w, o.x, acc.x);
    acc.y = fmaf(w, o.y, acc.y);
    acc.z = fmaf(w, o.z, acc.z);
    acc.w = fmaf(w, o.w, acc.w);
  }
  const float inv = den > 0.f ? 1.f / den : 0.f;
  const int n = rr / p.G, j = rr - n * p.G;
  const int g = lh % p.Hkv, l = p.layer0 + lh / p.Hkv;
  uint2 packed;
  packed.x = pack_bf16(acc.x * inv, acc.y * inv);
  packed.y = pack_bf16(acc.z * inv, acc.w * inv);
  *reinterpret_cast<uint2*>(p.out + ((((long long)l * p.qb.sumNq + p.qb.cu[qi] + n) * p.Hq + g * p.G + j) * 128 + quad * 4)) = packed;
}

template <int CG, bool OUT>
cudaError_t prepare_tc5() {  // the kernel's shared-memory limit, once per device
  static PerDeviceOnce attr;
  return attr.run([] {
    return cudaFuncSetAttribute(attend_tc5_kernel<CG, OUT>, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)TC_SMEM);
  });
}

// workers that can run at once: CTA pairs (clusters of two), or CTAs
template <int CG>
int max_workers() {
  static int known[REKV_MAX_DEVICES] = {};
  int dev = 0;
  if (cudaGetDevice(&dev) != cudaSuccess) return 1;
  const bool cacheable = dev >= 0 && dev < REKV_MAX_DEVICES;
  if (cacheable && known[dev] > 0) return known[dev];
  int n = rekv_sm_count() / CG;
  if (CG == 2) {
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(2 * n);
    cfg.blockDim = dim3(Warps<false>::THREADS);
    cfg.dynamicSmemBytes = TC_SMEM;
    cudaLaunchAttribute at[1];
    at[0].id = cudaLaunchAttributeClusterDimension;
    at[0].val.clusterDim.x = 2;
    at[0].val.clusterDim.y = at[0].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 1;
    int m = 0;
    if (prepare_tc5<CG, false>() == cudaSuccess && cudaOccupancyMaxActiveClusters(&m, attend_tc5_kernel<CG, false>, &cfg) == cudaSuccess && m > 0)
      n = std::min(n, m);
    else
      cudaGetLastError();
  }
  if (cacheable) known[dev] = n;
  return n;
}

template <int CG>
cudaError_t launch_tc5(rekv_ctx* c, Tc5Params& p, cudaStream_t st, bool timed) {
  p.per_lh = 0;
  int blocks = 0, max_ch = 1;
  bool equal = true;  // every unit has max_ch chunks
  for (int i = 0; i < p.qb.nQ; ++i) {
    const int nb = row_blocks<CG>(p, i), nc = stream_chunks(p, i);
    p.per_lh += nb * nc;
    blocks += nb;
    equal = equal && (nb == 0 || blocks == nb || nc == max_ch);
    if (nb > 0) max_ch = std::max(max_ch, nc);
  }
  const long long total = (long long)p.per_lh * p.Hkv * p.nl;
  if (total > 0x7fffffff / 2) return cudaErrorInvalidValue;
  p.total = (int)total;
  // (split launches: no merge launch between or after the two)
  const int units = p.nl * p.Hkv * blocks;
  const AttendPlan plan = rekv_attend_plan(p.total, units, max_ch, equal, max_workers<CG>(), !p.split_rem, CG == 2);
  p.W = plan.workers;
  p.merge_inside = plan.merge_inside;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)(p.W * CG));
  bool out = false;
  if constexpr (CG == 1) out = rekv_attend_output_warps(p.W, units, max_ch, false);   // (pairs are not compiled with output warps)
  cfg.blockDim = dim3(out ? Warps<true>::THREADS : Warps<false>::THREADS);
  cfg.dynamicSmemBytes = TC_SMEM;
  cfg.stream = st;
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  at[1].id = cudaLaunchAttributeClusterDimension;
  at[1].val.clusterDim.x = CG;
  at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
  cfg.attrs = at;
  cfg.numAttrs = 2;
  if (timed && !p.second) cudaEventRecord(c->ev_t0, st);
  auto launch = [&](auto with_out) {
    constexpr bool OUT = decltype(with_out)::value;
    const cudaError_t ep = prepare_tc5<CG, OUT>();
    return ep == cudaSuccess ? cudaLaunchKernelEx(&cfg, attend_tc5_kernel<CG, OUT>, p) : ep;
  };
  cudaError_t e;
  if constexpr (CG == 1)
    e = out ? launch(std::true_type{}) : launch(std::false_type{});
  else
    e = launch(std::false_type{});
  if (e != cudaSuccess) return e;
  c->launches += 1;
  if (timed) {
    cudaEventRecord(c->ev_t1, st);
    c->timing_valid = true;
    c->merge_timed = false;
  }
  if (!p.merge_inside) {
    Tc5Params m = p;
    m.merge_inside = p.W;
    m.W = blocks;
    long long tiles = 0;   // of 128 rows: a block without rows leaves at once
    for (int i = 0; i < p.qb.nQ; ++i) tiles += ((p.qb.cu[i + 1] - p.qb.cu[i]) * p.G + 127) / 128;
    const int ahead = rekv_merge_ahead(plan.parts, tiles * p.nl * p.Hkv * 32, rekv_sm_count());
    const auto merge = ahead == 4 ? merge_tc5_kernel<CG, 4> : ahead == 8 ? merge_tc5_kernel<CG, 8> : merge_tc5_kernel<CG, 10>;
    e = rekv_launch_pdl(merge, dim3((unsigned)units, CG, 32), dim3(128 * MERGE_GROUPS), 0, st, m);
    if (e != cudaSuccess) return e;
    c->launches += 1;
    if (timed) {
      cudaEventRecord(c->ev_t2, st);
      c->merge_timed = true;
    }
  }
  return cudaGetLastError();
}

}  // namespace

cudaError_t rekv_launch_attend_tc5(rekv_ctx* c, const void* q, const QBatch& qb, int ncf, int layer0, int layer1,
                                   void* out, cudaStream_t st, bool timed, const AttendFullArgs* full) {
  const StoreView& s = c->sv;
  if (rekv_decode_shaped(c, qb, ncf, layer1 - layer0))
    return rekv_launch_attend_decode(c, q, qb, ncf, layer0, layer1, out, st, timed, full);
  Tc5Params p;
  p.q = (const __nv_bfloat16*)q;
  p.out = (__nv_bfloat16*)out;
  p.tbl = c->ctx_tbl;
  p.tbl_k = full ? full->tbl_k : nullptr;
  p.x_kv = full ? full->x_kv : nullptr;
  p.x_rows = full ? full->x_rows : 0;
  p.part_o = (float4*)c->part_o;
  p.part_ml = (float2*)c->part_ml;
  p.unit_cnt = c->unit_cnt;
  p.status = c->status;
  p.qb = qb;
  p.sb.nQ = 0;
  if (full) p.sb = *full->sb;
  p.Hq = s.Hq;
  p.Hkv = s.Hkv;
  p.G = s.G;
  p.Nf = s.Nf;
  p.Ns = (s.Nf + 7) & ~7;
  p.ncf = ncf;
  p.layer0 = layer0;
  p.nl = layer1 - layer0;
  p.early_q = c->q_early_ok && !full;
  p.wait_limit = c->test_wait_limit;
  p.skip_copy_entry = c->test_skip_copy_entry;
  p.part_slots = (int)c->part_units;
  p.scale_log2 = 1.4426950408889634f / sqrtf(128.f);
  // Pairs as soon as a question has a second row tile; batches of one-tile questions would leave the pair's second CTA idle.
  // A remainder of at most 128 rows beside full pairs gets a launch of single CTAs of its own when the pairs' ranges are long
  // (MIN_SPLIT chunks): in a pair it costs as much as 256 rows, but a launch costs about ten chunks' time.
  constexpr int MIN_SPLIT = 64;
  bool two_tiles = false, rest = false;
  long long pair_chunks = 0;
  for (int i = 0; i < qb.nQ; ++i) {
    const int rows = (qb.cu[i + 1] - qb.cu[i]) * s.G;
    two_tiles = two_tiles || rows > 128;
    rest = rest || ((rows - 1) & 255) < 128;
    pair_chunks += (long long)((rows + 255) / 256) * stream_chunks(p, i);
  }
  p.split_rem = 0;
  p.second = 0;
  if (!two_tiles) return launch_tc5<1>(c, p, st, timed);
  if (!rest || pair_chunks * p.nl * p.Hkv < (long long)MIN_SPLIT * max_workers<2>()) return launch_tc5<2>(c, p, st, timed);
  p.split_rem = 1;
  p.early_q = 0;  // (the second launch's start tells that the selection is complete)
  Tc5Params r = p;
  cudaError_t e = launch_tc5<2>(c, p, st, timed);
  if (e != cudaSuccess) return e;
  // its own partial slots and counters: at most four slots and two counters per worker of the first launch
  const int off = 4 * max_workers<2>();
  r.part_o += (long long)off * 32 * 128;
  r.part_ml += (long long)off * 128;
  r.part_slots -= off;
  r.unit_cnt += off;
  r.second = 1;
  return launch_tc5<1>(c, r, st, timed);
}
