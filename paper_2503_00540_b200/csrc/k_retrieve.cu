// Steps 2-3: question vector, cosine scores against every frame representative (Eq. 2, tau = 1),
// and the exact top-r selection, per layer and per question.
#include "ptx_helpers.cuh"
#include "rekv_internal.cuh"

namespace {

// The arithmetic of the scores, for the three launches and the one-launch form alike: a score has the same bits whichever
// of them a call takes (a layer at a time or all layers, and rekv_score_frames_static), and so has the selection.  Fixed
// orders, and no product left to the compiler to contract:
//   question vector  64 partial sums, row r of the question in sum r mod 64, joined pairwise as a binary tree
//   its square norm  32-dim blocks by butterflies, four of them per KV group, groups in order
//   dot, row norm    per lane float4 by float4, then a butterfly over the lanes
constexpr int Q_SLOTS = 64;
__device__ __forceinline__ float add_dot4(float acc, const float4& a, const float4& b) {
  return __fadd_rn(acc, __fmaf_rn(a.w, b.w, __fmaf_rn(a.z, b.z, __fmaf_rn(a.y, b.y, __fmul_rn(a.x, b.x)))));
}
__device__ __forceinline__ float square_norm_of_warp(float a) {  // of the warp's 32 dims
  float sq = __fmul_rn(a, a);
  for (int o = 16; o; o >>= 1) sq = __fadd_rn(sq, __shfl_xor_sync(0xffffffffu, sq, o));
  return sq;
}

// ---- question vector: mean over the question's tokens and over the G query heads of each KV group
// grid = (nQ, layers, H_kv), layer = layer0 + blockIdx.y; 1024 threads = 64 row slots x 16 lanes of 16 bytes, U rows
// per thread in flight.  Latency is all this kernel has: with U = 4 a question of 36 tokens at G = 7 is one round of loads deep,
// and a block has an SM for itself (46 registers); launches of more blocks than SMs take U = 2 and two blocks per SM.
// Writes the group's 128 dims of the question vector and its partial sum of squares (the score kernel adds the H_kv partials).
constexpr int QM_THREADS = 1024;
template <int U>
__global__ void __launch_bounds__(QM_THREADS, U <= 2 ? 2 : 1)
    qmean_kernel(const uint4* __restrict__ q, QBatch qb, int Hq, int Hkv, int G, float* __restrict__ qa, float* __restrict__ qsq,
                 int maxQ, int layer0) {
  // launched with programmatic stream serialisation: its blocks are resident when the kernel before it ends (the
  // caller's, which wrote the queries, or the library's own), and wait here for that kernel's results
  rekv_ptx::grid_dep_wait();
  rekv_ptx::grid_dep_launch();
  const int qi = blockIdx.x, l = layer0 + blockIdx.y, g = blockIdx.z;
  const int n0 = qb.cu[qi], rows = (qb.cu[qi + 1] - n0) * G;
  const int c = threadIdx.x & 15, slot = threadIdx.x >> 4, lane = threadIdx.x & 31;
  const uint4* base = q + (((long long)l * qb.sumNq + n0) * Hq + g * G) * 16 + c;
  float acc[8];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] = 0.f;
  for (int m0 = slot; m0 < rows; m0 += U * Q_SLOTS) {
    uint4 x[U];
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const int m = m0 + Q_SLOTS * u, n = m / G;
      x[u] = m < rows ? __ldg(base + ((long long)n * Hq + (m - n * G)) * 16) : make_uint4(0, 0, 0, 0);
    }
#pragma unroll
    for (int u = 0; u < U; ++u) {
      const uint32_t v[4] = {x[u].x, x[u].y, x[u].z, x[u].w};
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        acc[2 * i] += __uint_as_float(v[i] << 16);
        acc[2 * i + 1] += __uint_as_float(v[i] & 0xFFFF0000u);
      }
    }
  }
  __shared__ float part[32][128];
  __shared__ float part2[8][128];
  __shared__ float red[4];
#pragma unroll
  for (int i = 0; i < 8; ++i) acc[i] += __shfl_xor_sync(0xffffffffu, acc[i], 16);
  if (lane < 16) {
    float4* dst = reinterpret_cast<float4*>(&part[threadIdx.x >> 5][c * 8]);
    dst[0] = make_float4(acc[0], acc[1], acc[2], acc[3]);
    dst[1] = make_float4(acc[4], acc[5], acc[6], acc[7]);
  }
  __syncthreads();
  const int d = threadIdx.x & 127, k = threadIdx.x >> 7;
  part2[k][d] = (part[4 * k][d] + part[4 * k + 1][d]) + (part[4 * k + 2][d] + part[4 * k + 3][d]);
  __syncthreads();
  if (threadIdx.x < 128) {
    float a = ((part2[0][d] + part2[1][d]) + (part2[2][d] + part2[3][d])) +
              ((part2[4][d] + part2[5][d]) + (part2[6][d] + part2[7][d]));
    a = __fdiv_rn(a, (float)rows);
    qa[((long long)l * maxQ + qi) * (Hkv * 128) + g * 128 + d] = a;
    const float sq = square_norm_of_warp(a);
    if (lane == 0) red[threadIdx.x >> 5] = sq;
  }
  __syncthreads();
  if (threadIdx.x == 0) qsq[((long long)l * maxQ + qi) * Hkv + g] = (red[0] + red[1]) + (red[2] + red[3]);
}

// ---- cosine scores.  grid = (item chunks, L); an item is a frame, or with block retrieval a block of
// `block` consecutive frames whose vector is the mean of their representatives.  One warp per item: the
// representative rows are read once (float4 per lane, coalesced), the norm and the dot product with
// every question of the batch come from the same registers, reduced with warp shuffles.  The table is
// read once per batch.  n_visible counts items here.
// SCORE_MAX_V4 = float4 per lane (4: D' <= 512, 8: D' <= 1024); fpc = frames per CTA (a multiple of 16), chosen by
// the launcher so that the whole grid is resident at once (no second, mostly empty wave).
template <int SCORE_MAX_V4>
__global__ void __launch_bounds__(256, SCORE_MAX_V4 <= 4 ? 3 : 2)
    score_kernel(const float* __restrict__ reps, const float* __restrict__ qa, const float* __restrict__ qsq, int nQ,
                 int maxQ, int Dp, int Hkv, int max_frames, int n_visible, int q_group, float* __restrict__ scores,
                 int block, int layer0, int fpc, int* __restrict__ status) {
  extern __shared__ float4 s_q[];  // [q_group][Dp/4]
  __shared__ float s_qn[REKV_MAX_QUESTIONS];
  const int l = layer0 + blockIdx.y;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int f0 = blockIdx.x * fpc;
  const int f1 = min(f0 + fpc, n_visible);
  const int nv4 = Dp / 128;  // float4 per lane
  const float eps = 1e-8f;
  // (past L1: a CTA may start while kernels that use the table's addresses otherwise are still running)
  float4 r0[SCORE_MAX_V4], r1[SCORE_MAX_V4];
  auto load_rows = [&](int f) {
    const float4* row0 = reinterpret_cast<const float4*>(reps + ((long long)l * max_frames + (long long)f * block) * Dp);
    const float4* row1 = row0 + (f + 1 < f1 ? (long long)block * (Dp / 4) : 0);
#pragma unroll
    for (int i = 0; i < SCORE_MAX_V4; ++i)
      if (i < nv4) {
        r0[i] = __ldcg(row0 + i * 32 + lane);
        r1[i] = __ldcg(row1 + i * 32 + lane);
      }
  };
  auto in_table = [&](int f) {
    return REKV_CHECK((long long)(f + (f + 1 < f1 ? 2 : 1)) * block <= max_frames && f >= 0, status, 11);
  };
  // The first rows are asked for before the question vectors are there: the table was complete before the question-vector kernel
  // released this launch (every kernel here releases the next one only after its own wait).  28 layers of 1800 frames one at a time
  // 887 -> 870 us, all at once 260 -> 256; 12 layers of blocks of 4 frames, 8 KV heads 67 -> 63.
  int have = -1;
  if (f0 + warp * 2 < f1 && in_table(f0 + warp * 2)) load_rows(have = f0 + warp * 2);
  rekv_ptx::grid_dep_wait();
  rekv_ptx::grid_dep_launch();
  if (threadIdx.x < nQ) {
    float sq = 0.f;
    for (int g = 0; g < Hkv; ++g) sq += qsq[((long long)l * maxQ + threadIdx.x) * Hkv + g];
    s_qn[threadIdx.x] = fmaxf(__fsqrt_rn(sq), eps);
  }

  for (int qg0 = 0; qg0 < nQ; qg0 += q_group) {
    const int qn = min(q_group, nQ - qg0);
    __syncthreads();
    const float4* src = reinterpret_cast<const float4*>(qa + ((long long)l * maxQ + qg0) * Dp);
    for (int i = threadIdx.x; i < qn * (Dp / 4); i += blockDim.x) s_q[i] = src[i];
    __syncthreads();
    // two frames per iteration: twice the loads in flight per warp
    for (int f = f0 + warp * 2; f < f1; f += 16) {
      const bool two = f + 1 < f1;
      if (!in_table(f)) continue;
      if (f != have) load_rows(f);
      have = -1;   // (block means are formed in place)
      if (block > 1) {  // block vector = mean of the block's frame vectors
        const float4* row0 = reinterpret_cast<const float4*>(reps + ((long long)l * max_frames + (long long)f * block) * Dp);
        const float4* row1 = row0 + (two ? (long long)block * (Dp / 4) : 0);
        for (int j = 1; j < block; ++j) {
#pragma unroll
          for (int i = 0; i < SCORE_MAX_V4; ++i)
            if (i < nv4) {
              const float4 a = __ldg(row0 + (long long)j * (Dp / 4) + i * 32 + lane);
              const float4 b = __ldg(row1 + (long long)j * (Dp / 4) + i * 32 + lane);
              r0[i].x += a.x; r0[i].y += a.y; r0[i].z += a.z; r0[i].w += a.w;
              r1[i].x += b.x; r1[i].y += b.y; r1[i].z += b.z; r1[i].w += b.w;
            }
        }
        const float fb = (float)block;
#pragma unroll
        for (int i = 0; i < SCORE_MAX_V4; ++i)
          if (i < nv4) {
            r0[i].x = __fdiv_rn(r0[i].x, fb); r0[i].y = __fdiv_rn(r0[i].y, fb);
            r0[i].z = __fdiv_rn(r0[i].z, fb); r0[i].w = __fdiv_rn(r0[i].w, fb);
            r1[i].x = __fdiv_rn(r1[i].x, fb); r1[i].y = __fdiv_rn(r1[i].y, fb);
            r1[i].z = __fdiv_rn(r1[i].z, fb); r1[i].w = __fdiv_rn(r1[i].w, fb);
          }
      }
      float n0 = 0.f, n1 = 0.f;
#pragma unroll
      for (int i = 0; i < SCORE_MAX_V4; ++i)
        if (i < nv4) {
          n0 = add_dot4(n0, r0[i], r0[i]);
          n1 = add_dot4(n1, r1[i], r1[i]);
        }
      for (int o = 16; o; o >>= 1) {
        n0 += __shfl_xor_sync(0xffffffffu, n0, o);
        n1 += __shfl_xor_sync(0xffffffffu, n1, o);
      }
      n0 = fmaxf(__fsqrt_rn(n0), eps);
      n1 = fmaxf(__fsqrt_rn(n1), eps);
      // Eight questions' dot products with both items are reduced together: at every step a lane hands over the half of its
      // sums that the other lane keeps, 16 shuffles for 16 sums instead of 80.
      int q0 = 0;
      for (; q0 + 4 <= qn; q0 += 8) {
        float d[16];  // [item][question]
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          d[j] = d[8 + j] = 0.f;
          if (q0 + j < qn) {
#pragma unroll
            for (int i = 0; i < SCORE_MAX_V4; ++i)
              if (i < nv4) {
                const float4 a = s_q[(q0 + j) * (Dp / 4) + i * 32 + lane];
                d[j] = add_dot4(d[j], r0[i], a);
                d[8 + j] = add_dot4(d[8 + j], r1[i], a);
              }
          }
        }
#pragma unroll
        for (int n = 8, o = 16; n >= 1; n >>= 1, o >>= 1) {
          const bool up = (lane & o) != 0;
#pragma unroll
          for (int i = 0; i < n; ++i) {
            const float send = up ? d[i] : d[i + n], keep = up ? d[i + n] : d[i];
            d[i] = keep + __shfl_xor_sync(0xffffffffu, send, o);
          }
        }
        const float sum = d[0] + __shfl_xor_sync(0xffffffffu, d[0], 1);
        const int item = lane >> 4, j = q0 + ((lane >> 1) & 7);  // lane bits 4..1 are the sum's index
        if (!(lane & 1) && j < qn && (item == 0 || two))
          scores[((long long)l * nQ + qg0 + j) * n_visible + f + item] = __fdiv_rn(sum, s_qn[qg0 + j] * (item ? n1 : n0));
      }
      for (int qi = q0; qi < qn; ++qi) {
        float d0 = 0.f, d1 = 0.f;
#pragma unroll
        for (int i = 0; i < SCORE_MAX_V4; ++i)
          if (i < nv4) {
            const float4 a = s_q[qi * (Dp / 4) + i * 32 + lane];
            d0 = add_dot4(d0, r0[i], a);
            d1 = add_dot4(d1, r1[i], a);
          }
        for (int o = 16; o; o >>= 1) {
          d0 += __shfl_xor_sync(0xffffffffu, d0, o);
          d1 += __shfl_xor_sync(0xffffffffu, d1, o);
        }
        if (lane == 0) {
          const float qn_ = s_qn[qg0 + qi];
          float* dst = scores + ((long long)l * nQ + qg0 + qi) * n_visible + f;
          dst[0] = __fdiv_rn(d0, qn_ * n0);
          if (two) dst[1] = __fdiv_rn(d1, qn_ * n1);
        }
      }
    }
  }
}

// ---- exact top-k by radix select on the score keys (score order, then lower index first).
// Order-preserving 32-bit image of a score: larger score <=> larger key; NaN ranks as -inf, -0 == +0.
__device__ __forceinline__ unsigned score_key(float s) {
  unsigned u = __float_as_uint(s);
  if (s != s) u = 0xFF800000u;
  if (s == 0.f) u = 0u;
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

// grid = (nQ, L), 512 threads.  Candidates are frames [0, n_cand).  Up to 2048 of them keep their keys in registers, and one
// histogram over 2048 equal steps between the smallest and the largest score finds the step that holds the k-th largest:
// every candidate in a higher step is selected, and the few in that step are ranked exactly against each other (score, then
// lower index).  Otherwise -- more candidates, a NaN among them, a step with more than TK_LIST members -- four 8-bit radix
// passes over the score keys find the k-th largest key T exactly, with the number of candidates above it; one ordered
// compaction then emits, in ascending frame index, every frame above T and the lowest-index frames equal to T that are
// still needed (ties go to the lower index).  Latency is all: the radix passes took 4.3 us per launch of 1792 candidates
// (their first pass puts all cosines into a few bins, whose atomics queue).
// With block retrieval the candidates are blocks; a selected block b_i is written as its `block` frames
// b_i*block .. b_i*block + block-1 (k_eff counts items, top_k counts output slots).
// With tbl != null (cache all in HBM) the block also writes the context table of its (layer, question) -- the
// selected frames' pages then the trailing frames' pages, as the gather kernel would -- so that no further
// launch stands between the selection and the attention.
struct TopkTable {
  char** tbl;            // [L][nQ][ncf] page pointers, or null
  char* hbm;
  long long page_bytes;
  int L, ncf, n_vis_frames;
};
constexpr int TK_BINS = 2048, TK_LIST = 64;
// s: the question's scores (global or shared memory), complete for the calling block of 512 threads
__device__ __forceinline__ void select_topk(const float* s, int qi, int l, int nQ, int n_cand, int top_k, int k_eff,
                                            int32_t* __restrict__ idx_out, int block, const TopkTable& tt, int copies,
                                            int* __restrict__ status) {
  int32_t* out = idx_out + ((long long)l * nQ + qi) * top_k;
  __shared__ __align__(16) unsigned hist[TK_BINS];  // (the radix passes use its front)
  __shared__ unsigned s_prefix;
  __shared__ int s_krem;
  __shared__ int warp_gt[16], warp_eq[16];
  __shared__ int s_base_gt, s_base_eq;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;

  // entry `at` of the selection, and with it the page of that context slot; `copies` layers get the same selection
  char** row = tt.tbl ? tt.tbl + ((long long)l * nQ + qi) * tt.ncf : nullptr;
  auto page_of = [&](int frame) { return tt.hbm + ((long long)frame * tt.L + l) * tt.page_bytes; };
  auto emit_item = [&](int at, int frame) {
    for (int r = 0; r < copies; ++r) out[(long long)r * nQ * top_k + at] = frame;
    if (row) row[at] = page_of(frame);
  };
  const int k_frames = k_eff > 0 ? k_eff * block : 0;
  for (int j = k_frames + threadIdx.x; j < top_k; j += blockDim.x)
    for (int r = 0; r < copies; ++r) out[(long long)r * nQ * top_k + j] = -1;
  if (row)  // the trailing frames
    for (int j = k_frames + threadIdx.x; j < tt.ncf; j += blockDim.x) row[j] = page_of(tt.n_vis_frames - tt.ncf + j);
  if (k_eff <= 0) return;
  // up to TK_CACHE * 512 candidates keep their keys in registers: one read of the scores instead of five.  A thread
  // holds TK_CACHE consecutive candidates, so that the ordered compaction at the end is one scan over the threads.
  constexpr int TK_CACHE = 4;
  const bool cached = n_cand <= TK_CACHE * 512;
  unsigned kc[TK_CACHE];
#pragma unroll
  for (int j = 0; j < TK_CACHE; ++j) {
    const int i = threadIdx.x * TK_CACHE + j;
    kc[j] = (cached && i < n_cand) ? score_key(s[i]) : 0u;
  }
  if (threadIdx.x == 0) {
    s_prefix = 0u;
    s_krem = k_eff;
    s_base_gt = 0;
    s_base_eq = 0;
  }
  *reinterpret_cast<uint4*>(hist + 4 * threadIdx.x) = make_uint4(0, 0, 0, 0);
  if (cached) {
    __shared__ unsigned w_lo[16], w_hi[16], w_cnt[16];
    __shared__ unsigned l_key[TK_LIST];
    __shared__ int l_idx[TK_LIST];
    __shared__ int s_bin, s_need, s_members, s_n;
    unsigned k_lo = 0xFFFFFFFFu, k_hi = 0u;
#pragma unroll
    for (int j = 0; j < TK_CACHE; ++j)
      if ((int)threadIdx.x * TK_CACHE + j < n_cand) {
        k_lo = min(k_lo, kc[j]);
        k_hi = max(k_hi, kc[j]);
      }
    k_lo = __reduce_min_sync(0xffffffffu, k_lo);
    k_hi = __reduce_max_sync(0xffffffffu, k_hi);
    if (lane == 0) {
      w_lo[warp] = k_lo;
      w_hi[warp] = k_hi;
    }
    if (threadIdx.x == 0) s_n = 0;
    __syncthreads();
    k_lo = __reduce_min_sync(0xffffffffu, w_lo[lane & 15]);
    k_hi = __reduce_max_sync(0xffffffffu, w_hi[lane & 15]);
    auto value = [](unsigned k) { return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k); };
    const float lo = value(k_lo), width = value(k_hi) - lo;
    // (an infinite or NaN score, equal scores, or a width that overflows: the radix passes)
    if (width > 0.f && width < 3.0e38f) {
      const float scale = (float)TK_BINS / width;
      int bin[TK_CACHE];
#pragma unroll
      for (int j = 0; j < TK_CACHE; ++j) {  // monotone in the score
        bin[j] = -1;
        if ((int)threadIdx.x * TK_CACHE + j < n_cand) {
          bin[j] = min((int)((value(kc[j]) - lo) * scale), TK_BINS - 1);
          atomicAdd(&hist[bin[j]], 1u);
        }
      }
      __syncthreads();
      // thread t holds bins [4t, 4t + 4); inclusive suffix sums over the block
      const uint4 h = *reinterpret_cast<const uint4*>(hist + 4 * threadIdx.x);
      const int tot = (int)(h.x + h.y + h.z + h.w);
      int suf = tot;
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_down_sync(0xffffffffu, suf, o);
        if (lane + o < 32) suf += v;
      }
      if (lane == 0) w_cnt[warp] = suf;
      __syncthreads();
      suf += __reduce_add_sync(0xffffffffu, lane < 16 && lane > warp ? (int)w_cnt[lane & 15] : 0);
      if (suf >= k_eff && suf - tot < k_eff) {  // the k-th largest lies in this thread's bins
        int above = suf - tot, d = 3;
        const int b[4] = {(int)h.x, (int)h.y, (int)h.z, (int)h.w};
        for (; d > 0 && above + b[d] < k_eff; --d) above += b[d];
        s_bin = 4 * threadIdx.x + d;
        s_need = k_eff - above;
        s_members = b[d];
      }
      __syncthreads();
      const int at = s_bin, need = s_need, members = s_members;
      if (members <= TK_LIST) {  // (uniform)
        bool sel[TK_CACHE];
#pragma unroll
        for (int j = 0; j < TK_CACHE; ++j) {
          sel[j] = bin[j] > at || (bin[j] == at && need == members);
          if (need != members && bin[j] == at) {
            const int n = atomicAdd(&s_n, 1);
            l_key[n] = kc[j];
            l_idx[n] = threadIdx.x * TK_CACHE + j;
          }
        }
        if (need != members) {
          __syncthreads();
#pragma unroll
          for (int j = 0; j < TK_CACHE; ++j)
            if (bin[j] == at) {
              const int i = threadIdx.x * TK_CACHE + j;
              int before = 0;
              for (int n = 0; n < members; ++n) before += l_key[n] > kc[j] || (l_key[n] == kc[j] && l_idx[n] < i);
              sel[j] = before < need;
            }
        }
        // ordered compaction: an exclusive scan over the threads
        int cnt = 0;
#pragma unroll
        for (int j = 0; j < TK_CACHE; ++j) cnt += sel[j];
        int sc = cnt;
        for (int o = 1; o < 32; o <<= 1) {
          const int v = __shfl_up_sync(0xffffffffu, sc, o);
          if (lane >= o) sc += v;
        }
        if (lane == 31) warp_gt[warp] = sc;
        __syncthreads();
        int pos = sc - cnt + __reduce_add_sync(0xffffffffu, lane < warp ? warp_gt[lane & 15] : 0);
#pragma unroll
        for (int j = 0; j < TK_CACHE; ++j)
          if (sel[j]) {
            const int i = threadIdx.x * TK_CACHE + j;
            if (REKV_CHECK(pos < k_eff && i < n_cand, status, 21))
              for (int jj = 0; jj < block; ++jj) emit_item(pos * block + jj, i * block + jj);
            ++pos;
          }
        return;
      }
      __syncthreads();
      *reinterpret_cast<uint4*>(hist + 4 * threadIdx.x) = make_uint4(0, 0, 0, 0);
    }
  }
  __syncthreads();
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
    unsigned* h = hist + 256 * pass;
    const unsigned prefix = s_prefix;
    const unsigned mask = pass == 0 ? 0u : (0xFFFFFFFFu << (shift + 8));
    if (cached) {
#pragma unroll
      for (int j = 0; j < TK_CACHE; ++j)
        if ((int)threadIdx.x * TK_CACHE + j < n_cand && (kc[j] & mask) == prefix) atomicAdd(&h[(kc[j] >> shift) & 255u], 1u);
    } else {
      for (int i = threadIdx.x; i < n_cand; i += blockDim.x) {
        const unsigned key = score_key(s[i]);
        if ((key & mask) == prefix) atomicAdd(&h[(key >> shift) & 255u], 1u);
      }
    }
    __syncthreads();
    if (warp == 0) {
      // lane owns bins [8*lane, 8*lane+8); suffix sums over lanes locate the bin of the k-th largest
      unsigned b[8], tot = 0;
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        b[j] = h[lane * 8 + j];
        tot += b[j];
      }
      unsigned suf = tot;  // inclusive suffix sum over lanes >= this one
      for (int o = 1; o < 32; o <<= 1) {
        unsigned v = __shfl_down_sync(0xffffffffu, suf, o);
        if (lane + o < 32) suf += v;
      }
      const int krem = s_krem;
      const unsigned ball = __ballot_sync(0xffffffffu, (int)suf >= krem);
      const int owner = 31 - __clz(ball);  // highest lane whose suffix still reaches krem
      if (lane == owner) {
        int above = (int)(suf - tot);  // candidates in higher lanes' bins
        int d = 7;
        for (; d > 0; --d) {
          if (above + (int)b[d] >= krem) break;
          above += (int)b[d];
        }
        s_krem = krem - above;
        s_prefix = prefix | ((unsigned)(lane * 8 + d) << shift);
      }
    }
    __syncthreads();
  }
  const unsigned thr = s_prefix;  // key of the k_eff-th largest score
  const int need_eq = s_krem;     // how many candidates equal to it are selected (lowest indices first)
  // Ordered compaction of a stretch of blockDim.x * TK_CACHE candidates starting at i0, thread t holding candidates
  // i0 + t * TK_CACHE + j: counts of "greater" and "equal" per thread, an exclusive scan over the block (shuffles
  // inside a warp, the warps' totals through shared memory), then
  // output position = selected frames before this one = (greater before) + min(equal before, need_eq).
  auto emit = [&](const int i0, const unsigned (&key_in)[TK_CACHE]) {
    int cg = 0, ce = 0;
#pragma unroll
    for (int j = 0; j < TK_CACHE; ++j) {
      const int i = i0 + threadIdx.x * TK_CACHE + j;
      cg += i < n_cand && key_in[j] > thr;
      ce += i < n_cand && key_in[j] == thr;
    }
    int sg = cg, se = ce;  // inclusive scans over the warp
    for (int o = 1; o < 32; o <<= 1) {
      const int vg = __shfl_up_sync(0xffffffffu, sg, o), ve = __shfl_up_sync(0xffffffffu, se, o);
      if (lane >= o) {
        sg += vg;
        se += ve;
      }
    }
    if (lane == 31) {
      warp_gt[warp] = sg;
      warp_eq[warp] = se;
    }
    __syncthreads();
    int og = s_base_gt + sg - cg, oe = s_base_eq + se - ce;  // greater / equal candidates before this thread's
    {
      const int wg = lane < 16 ? warp_gt[lane] : 0, we = lane < 16 ? warp_eq[lane] : 0;
      const unsigned below = lane < warp ? 0xffffffffu : 0u;
      int ag = wg & (int)below, ae = we & (int)below;  // totals of the warps before this one
      for (int o = 16; o; o >>= 1) {
        ag += __shfl_xor_sync(0xffffffffu, ag, o);
        ae += __shfl_xor_sync(0xffffffffu, ae, o);
      }
      og += ag;
      oe += ae;
    }
#pragma unroll
    for (int j = 0; j < TK_CACHE; ++j) {
      const int i = i0 + threadIdx.x * TK_CACHE + j;
      const bool gt = i < n_cand && key_in[j] > thr, eq = i < n_cand && key_in[j] == thr;
      int pos = -1;
      if (gt) pos = og + min(oe, need_eq);
      if (eq && oe < need_eq) pos = og + oe;
      if (pos >= 0 && REKV_CHECK(pos < k_eff && i < n_cand, status, 21))
        for (int jj = 0; jj < block; ++jj) emit_item(pos * block + jj, i * block + jj);
      og += gt;
      oe += eq;
    }
  };
  if (cached) {
    emit(0, kc);
  } else {
    for (int i0 = 0; i0 < n_cand; i0 += blockDim.x * TK_CACHE) {
      unsigned key[TK_CACHE];
#pragma unroll
      for (int j = 0; j < TK_CACHE; ++j) {
        const int i = i0 + threadIdx.x * TK_CACHE + j;
        key[j] = i < n_cand ? score_key(s[i]) : 0u;
      }
      emit(i0, key);
      __syncthreads();  // everybody has read the warps' totals
      if (threadIdx.x == 0) {
        int tg = 0, te = 0;
        for (int w = 0; w < 16; ++w) {
          tg += warp_gt[w];
          te += warp_eq[w];
        }
        s_base_gt += tg;
        s_base_eq += te;
      }
      __syncthreads();
    }
  }
}

__global__ void __launch_bounds__(512) topk_kernel(const float* __restrict__ scores, int nQ, int n_visible,
                                                   int n_cand, int top_k, int k_eff, int32_t* __restrict__ idx_out,
                                                   int block, int layer0, TopkTable tt, int copies, int* __restrict__ status) {
  const int qi = blockIdx.x, l = layer0 + blockIdx.y;
  rekv_ptx::grid_dep_wait();
  rekv_ptx::grid_dep_launch();
  select_topk(scores + ((long long)l * nQ + qi) * n_visible, qi, l, nQ, n_cand, top_k, k_eff, idx_out, block, tt, copies, status);
}

// ---- steps 2-3 of a layer in one launch: question vectors, scores and selection by one cluster per layer.  Three launches
// pass 4 us from one to the next, whatever little they do; here the CTAs exchange what they have through distributed shared
// memory: every CTA sums a share of the query rows and sends its partial sum to all, scores a share of the items -- whose
// first rows are on their way while the sums are exchanged -- and sends the scores to the CTA that selects for the question.
// grid = (CTAs per cluster, layers), 512 threads; RB rows of float4 x V4 per lane are in flight per warp; CPG CTAs (1, 2, 4, 8) sum
// the rows of one KV group.
constexpr int RK_MAX_Q = 4;          // questions
constexpr int RK_MAX_SMEM = 64 * 1024;
constexpr int RK_MAX_ITEMS = 2048;   // items scored (the selection's histogram path)
struct RetrieveArgs {
  const uint4* q;
  const float* reps;
  float* scores;                     // [L][nQ][n_scored], or null
  int32_t* idx_out;
  int* status;
  TopkTable tt;
  int Hq, Hkv, max_frames, n_scored, n_cand, top_k, k_eff, block, layer0, CL;
  unsigned wait_limit;               // test-only knobs (0 = off), see rekv_test_set_wait_limit, rekv_test_set_retrieve
  int test;
  QBatch qb;
};
// A wait ran out (the status word says so).  No selection, but a list and a table that are safe to follow: what comes next in the
// stream reads them before anyone has read the status.  (Out of line: the launch fetches its code anew every time.)
__device__ __noinline__ void retrieve_failed(const RetrieveArgs& p, int qi, int l) {
  const long long row = (long long)l * p.qb.nQ + qi;
  for (int j = threadIdx.x; j < p.top_k; j += blockDim.x) p.idx_out[row * p.top_k + j] = -1;
  if (p.tt.tbl)
    for (int j = threadIdx.x; j < p.tt.ncf; j += blockDim.x) p.tt.tbl[row * p.tt.ncf + j] = p.tt.hbm + (long long)l * p.tt.page_bytes;  // frame 0
}
template <int V4, int RB, int CPG>
__global__ void __launch_bounds__(512, V4 * RB <= 8 ? 2 : 1) retrieve_kernel(const __grid_constant__ RetrieveArgs p) {
  using namespace rekv_ptx;
  extern __shared__ __align__(16) float rk_smem[];
  const int Dp = p.Hkv * 128, nQ = p.qb.nQ, CL = p.CL;
  float* s_vec = rk_smem;                                       // [nQ][Hkv][CPG][128] partial sums, from all CTAs
  float* s_q = s_vec + nQ * p.Hkv * CPG * 128;                  // [nQ][Dp] question vectors
  float* s_score = s_q + nQ * Dp;                               // [n_scored] of the question this CTA selects for
  __shared__ __align__(16) float s_part[Q_SLOTS / 2][128];
  __shared__ __align__(16) float s_red[RK_MAX_Q][32];            // square norms of the 32-dim blocks
  __shared__ __align__(8) unsigned long long s_bar[2];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  const int rank = (int)cluster_ctarank(), l = p.layer0 + blockIdx.y;
  const uint32_t bar_vec = smem_u32(&s_bar[0]), bar_score = smem_u32(&s_bar[1]);
  if (tid == 0) {
    mbar_init(bar_vec, 1);
    mbar_init(bar_score, 1);
    fence_barrier_init();
    mbar_expect_tx(bar_vec, (uint32_t)(nQ * p.Hkv * CPG * 512));
    if (rank < nQ) mbar_expect_tx(bar_score, (uint32_t)p.n_scored * 4u);
  }
  __syncthreads();
  cluster_sync_all();
  grid_dep_wait();
  grid_dep_launch();
  auto wait = [&](uint32_t bar) {
    if (mbar_wait_cluster_bounded(bar, 0, p.wait_limit ? p.wait_limit : 1u << 22)) return true;
    atomicExch(p.status, REKV_ERR_TIMEOUT);
    return false;
  };

  const int per = (p.n_scored + CL - 1) / CL;
  const int f0 = rank * per, f1 = min(f0 + per, p.n_scored);
  const float4* reps_l = reinterpret_cast<const float4*>(p.reps + (long long)l * p.max_frames * Dp) + lane;
  float4 r[RB][V4];
  auto load_rows = [&](int f) {
#pragma unroll
    for (int b = 0; b < RB; ++b) {
      const float4* row = reps_l + (long long)min(f + b, f1 - 1) * p.block * (Dp / 4);
#pragma unroll
      for (int i = 0; i < V4; ++i)
        if (i < p.Hkv) r[b][i] = __ldg(row + i * 32);
    }
  };
  int f = f0 + warp * RB;

  // ---- question vectors: mean over the question's tokens and the G query heads of each KV group
  // (each CTA of a group's CPG takes Q_SLOTS / CPG of the sums, a slot -- two with CPG = 1 -- per 16 lanes of 16 bytes)
  constexpr int slots = Q_SLOTS / CPG, TURNS = CPG == 1 ? 2 : 1;
  const int G = p.Hq / p.Hkv, g = rank / CPG;
  for (int qi = 0; qi < nQ; ++qi) {
    const int n0 = p.qb.cu[qi], rows = (p.qb.cu[qi + 1] - n0) * G;
    if (g < p.Hkv) {
      const int c = tid & 15;
      const uint4* base = p.q + (((long long)l * p.qb.sumNq + n0) * p.Hq + g * G) * 16 + c;
      const int sl = tid >> 4;
      if (sl < slots) {
        float acc[TURNS][8];
#pragma unroll
        for (int w = 0; w < TURNS; ++w)
#pragma unroll
          for (int i = 0; i < 8; ++i) acc[w][i] = 0.f;
        for (int m0 = (rank - g * CPG) * slots + sl; m0 < rows; m0 += 4 * Q_SLOTS) {
          uint4 x[TURNS][4];
#pragma unroll
          for (int w = 0; w < TURNS; ++w)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const int m = m0 + 32 * w + u * Q_SLOTS, n = m / G;
              x[w][u] = m < rows ? __ldg(base + ((long long)n * p.Hq + (m - n * G)) * 16) : make_uint4(0, 0, 0, 0);
            }
#pragma unroll
          for (int w = 0; w < TURNS; ++w)
#pragma unroll
            for (int u = 0; u < 4; ++u) {
              const uint32_t v[4] = {x[w][u].x, x[w][u].y, x[w][u].z, x[w][u].w};
#pragma unroll
              for (int i = 0; i < 4; ++i) {
                acc[w][2 * i] += __uint_as_float(v[i] << 16);
                acc[w][2 * i + 1] += __uint_as_float(v[i] & 0xFFFF0000u);
              }
            }
        }
#pragma unroll
        for (int w = 0; w < TURNS; ++w) {
#pragma unroll
          for (int i = 0; i < 8; ++i) acc[w][i] += __shfl_xor_sync(0xffffffffu, acc[w][i], 16);
          if (lane < 16) {
            float4* dst = reinterpret_cast<float4*>(&s_part[warp + 16 * w][c * 8]);
            dst[0] = make_float4(acc[w][0], acc[w][1], acc[w][2], acc[w][3]);
            dst[1] = make_float4(acc[w][4], acc[w][5], acc[w][6], acc[w][7]);
          }
        }
      }
      __syncthreads();
      // thread t sends columns 4 (t & 31) .. of the CTA's sum to CTA t / 32 (every thread adds its columns up itself)
      if (warp < CL) {
        auto add4 = [](const float4& a, const float4& b) { return make_float4(a.x + b.x, a.y + b.y, a.z + b.z, a.w + b.w); };
        auto quad = [&](int k) {
          const float4* x = reinterpret_cast<const float4*>(&s_part[4 * k][lane * 4]);
          return add4(add4(x[0], x[32]), add4(x[64], x[96]));
        };
        float4 a = quad(0);
        if (CPG <= 4) a = add4(a, quad(1));
        if (CPG <= 2) a = add4(a, add4(quad(2), quad(3)));
        if (CPG <= 1) a = add4(a, add4(add4(quad(4), quad(5)), add4(quad(6), quad(7))));
        const uint32_t dst = smem_u32(s_vec + ((qi * p.Hkv * CPG + rank) * 128 + lane * 4));
        if (!((p.test & REKV_TEST_RETRIEVE_SKIP_SUM) && rank == 0 && blockIdx.y == 0))
          st_async_v4(mapa(dst, (uint32_t)warp), a, mapa(bar_vec, (uint32_t)warp));
      }
      __syncthreads();  // (s_part is written again for the next question)
    }
  }
  if (f < f1) load_rows(f);  // the first items' rows arrive while the sums are exchanged
  bool ok = wait(bar_vec);
  for (int qi = 0; qi < nQ; ++qi) {
    const float rows = (float)((p.qb.cu[qi + 1] - p.qb.cu[qi]) * G);
    for (int d = tid; d < Dp; d += 512) {
      const float* v = s_vec + (qi * p.Hkv + (d >> 7)) * CPG * 128 + (d & 127);
      float a = v[0];
      if (CPG >= 2) a += v[128];
      if (CPG >= 4) a += v[256] + v[384];
      if (CPG >= 8) a += (v[512] + v[640]) + (v[768] + v[896]);
      a = __fdiv_rn(a, rows);
      s_q[qi * Dp + d] = a;
      const float sq = square_norm_of_warp(a);
      if (lane == 0) s_red[qi][d >> 5] = sq;
    }
  }
  __syncthreads();

  // ---- scores: every lane holds its part of RB rows; dot products and norms by shuffles
  const float eps = 1e-8f;
  const float4* s_q4 = reinterpret_cast<const float4*>(s_q) + lane;
  while (f < f1) {
    if (p.block > 1) {  // block vector = mean of the block's frame vectors
      const float fb = (float)p.block;
#pragma unroll
      for (int b = 0; b < RB; ++b) {
        const float4* row = reps_l + (long long)min(f + b, f1 - 1) * p.block * (Dp / 4);
        for (int j = 1; j < p.block; ++j)
#pragma unroll
          for (int i = 0; i < V4; ++i)
            if (i < p.Hkv) {
              const float4 x = __ldg(row + (long long)j * (Dp / 4) + i * 32);
              r[b][i].x += x.x; r[b][i].y += x.y; r[b][i].z += x.z; r[b][i].w += x.w;
            }
#pragma unroll
        for (int i = 0; i < V4; ++i)
          if (i < p.Hkv) {
            r[b][i].x = __fdiv_rn(r[b][i].x, fb); r[b][i].y = __fdiv_rn(r[b][i].y, fb);
            r[b][i].z = __fdiv_rn(r[b][i].z, fb); r[b][i].w = __fdiv_rn(r[b][i].w, fb);
          }
      }
    }
    float rn[RB];
#pragma unroll
    for (int b = 0; b < RB; ++b) {
      float n = 0.f;
#pragma unroll
      for (int i = 0; i < V4; ++i)
        if (i < p.Hkv) n = add_dot4(n, r[b][i], r[b][i]);
      for (int o = 16; o; o >>= 1) n += __shfl_xor_sync(0xffffffffu, n, o);
      rn[b] = fmaxf(__fsqrt_rn(n), eps);
    }
    for (int qi = 0; qi < nQ; ++qi) {
      float qn = 0.f;
#pragma unroll
      for (int k = 0; k < V4; ++k)
        if (k < p.Hkv) {
          const float4 x = *reinterpret_cast<const float4*>(&s_red[qi][4 * k]);
          qn += (x.x + x.y) + (x.z + x.w);
        }
      qn = fmaxf(__fsqrt_rn(qn), eps);
      float d[RB];
#pragma unroll
      for (int b = 0; b < RB; ++b) d[b] = 0.f;
#pragma unroll
      for (int i = 0; i < V4; ++i)
        if (i < p.Hkv) {
          const float4 a = s_q4[qi * (Dp / 4) + i * 32];
#pragma unroll
          for (int b = 0; b < RB; ++b) d[b] = add_dot4(d[b], r[b][i], a);
        }
#pragma unroll
      for (int b = 0; b < RB; ++b) {
        for (int o = 16; o; o >>= 1) d[b] += __shfl_xor_sync(0xffffffffu, d[b], o);
        const float sc = __fdiv_rn(d[b], qn * rn[b]);
        if (lane == b && f + b < f1 && REKV_CHECK((long long)(f + b + 1) * p.block <= p.max_frames, p.status, 11)) {
          if (!((p.test & REKV_TEST_RETRIEVE_SKIP_SCORE) && f + b == 0 && blockIdx.y == 0))
            st_async_f32(mapa(smem_u32(s_score + f + b), (uint32_t)qi), sc, mapa(bar_score, (uint32_t)qi));
          if (p.scores) p.scores[((long long)l * nQ + qi) * p.n_scored + f + b] = sc;
        }
      }
    }
    f += 16 * RB;
    if (f < f1) load_rows(f);
  }
  // ---- selection: CTA qi for question qi
  if (rank < nQ) {
    ok = wait(bar_score) && ok;
    ok = __syncthreads_and(ok);
    if (ok) {
      select_topk(s_score, rank, l, nQ, p.n_cand, p.top_k, p.k_eff, p.idx_out, p.block, p.tt, 1, p.status);
      return;
    }
    retrieve_failed(p, rank, l);
  }
  // a thread whose wait ran out stays until the others are done or here too: they may still send into this CTA's shared memory
  if (!ok) cluster_sync_threads();
}

// ---- external retrieval (Eq. 2 with its temperature): cosine of each question embedding with every frame
// embedding (or with the mean of a block's frame embeddings), divided by tau.  grid = ceil(items / 8), 256
// threads, a warp per item: the item's vector is read once into registers (float4 per lane, coalesced) and
// scored against every question of the batch, whose embeddings sit in shared memory in groups.
constexpr int EXT_MAX_V4 = 16;  // float4 per lane: embedding dim <= 2048
__global__ void __launch_bounds__(256) ext_score_kernel(const float* __restrict__ embs, const float* __restrict__ q,
                                                        int nQ, int E, int n_items, int block, int q_group, float tau,
                                                        float* __restrict__ scores) {
  extern __shared__ float4 s_qe[];  // [q_group][E/4]
  __shared__ float s_qn[REKV_MAX_QUESTIONS];
  rekv_ptx::grid_dep_wait();
  rekv_ptx::grid_dep_launch();
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int item = blockIdx.x * 8 + warp;
  const int e4 = E / 4;
  const float eps = 1e-8f;
  float4 r[EXT_MAX_V4];
  float vn = 0.f;
  if (item < n_items) {
#pragma unroll
    for (int i = 0; i < EXT_MAX_V4; ++i)
      if (i * 32 + lane < e4) {
        const float4* row = reinterpret_cast<const float4*>(embs + (long long)item * block * E) + i * 32 + lane;
        float4 a = __ldg(row);
        for (int j = 1; j < block; ++j) {  // block vector = mean of the block's frame vectors
          const float4 b = __ldg(row + (long long)j * e4);
          a.x += b.x; a.y += b.y; a.z += b.z; a.w += b.w;
        }
        if (block > 1) {
          const float fb = (float)block;
          a.x = __fdiv_rn(a.x, fb); a.y = __fdiv_rn(a.y, fb); a.z = __fdiv_rn(a.z, fb); a.w = __fdiv_rn(a.w, fb);
        }
        r[i] = a;
        vn += a.x * a.x + a.y * a.y + a.z * a.z + a.w * a.w;
      }
    for (int o = 16; o; o >>= 1) vn += __shfl_xor_sync(0xffffffffu, vn, o);
    vn = fmaxf(__fsqrt_rn(vn), eps);
  }
  for (int qg0 = 0; qg0 < nQ; qg0 += q_group) {
    const int qn = min(q_group, nQ - qg0);
    __syncthreads();
    const float4* src = reinterpret_cast<const float4*>(q + (long long)qg0 * E);
    for (int i = threadIdx.x; i < qn * e4; i += 256) s_qe[i] = src[i];
    __syncthreads();
    for (int qi = warp; qi < qn; qi += 8) {  // the questions' norms
      float sq = 0.f;
      for (int i = lane; i < e4; i += 32) {
        const float4 a = s_qe[qi * e4 + i];
        sq += a.x * a.x + a.y * a.y + a.z * a.z + a.w * a.w;
      }
      for (int o = 16; o; o >>= 1) sq += __shfl_xor_sync(0xffffffffu, sq, o);
      if (lane == 0) s_qn[qi] = fmaxf(__fsqrt_rn(sq), eps);
    }
    __syncthreads();
    if (item < n_items) {
      for (int qi = 0; qi < qn; ++qi) {
        float d = 0.f;
#pragma unroll
        for (int i = 0; i < EXT_MAX_V4; ++i)
          if (i * 32 + lane < e4) {
            const float4 a = s_qe[qi * e4 + i * 32 + lane];
            d += r[i].x * a.x + r[i].y * a.y + r[i].z * a.z + r[i].w * a.w;
          }
        for (int o = 16; o; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
        if (lane == 0) scores[(long long)(qg0 + qi) * n_items + item] = __fdiv_rn(d, tau * s_qn[qi] * vn);
      }
    }
  }
}


// Launch of the score kernel over frames [0, n_scored) of nl layers.  Frames per CTA grow until the grid fits the
// device in one wave at the kernel's occupancy.
// What the score kernel needs besides the grid.
struct ScoreArgs {
  int nl, n_scored;
  const float* reps;
  const float* qa;
  const float* qsq;
  int nQ, maxQ, Dp, Hkv, max_frames;
  float* scores;
  int block, layer0;
  int* status;
};
template <int V4>
cudaError_t launch_score_v4(const ScoreArgs& a, bool pdl, cudaStream_t st) {
  int q_group = (int)((96 * 1024) / (a.Dp * sizeof(float)));
  if (q_group > a.nQ) q_group = a.nQ;
  const size_t smem = (size_t)q_group * a.Dp * sizeof(float);
  static PerDeviceOnce attr;
  cudaError_t e = attr.run([] {
    return cudaFuncSetAttribute(score_kernel<V4>, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
  });
  if (e != cudaSuccess) return e;
  // blocks per SM by the dynamic shared memory in KB (asking the runtime on every call costs as much as a launch)
  static int known[REKV_MAX_DEVICES][97] = {};
  int dev = 0, occ = 0;
  const int kb = (int)((smem + 1023) / 1024);
  const bool cacheable = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < REKV_MAX_DEVICES && kb <= 96;
  if (cacheable) occ = known[dev][kb];
  if (occ < 1) {
    if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, score_kernel<V4>, 256, smem) != cudaSuccess || occ < 1) occ = 1;
    if (cacheable) known[dev][kb] = occ;
  }
  int per_layer = (rekv_sm_count() * occ) / a.nl;
  if (per_layer < 1) per_layer = 1;
  int fpc = ((a.n_scored + per_layer - 1) / per_layer + 15) & ~15;
  if (fpc < 16) fpc = 16;
  const dim3 grid((a.n_scored + fpc - 1) / fpc, a.nl);
  if (pdl)
    return rekv_launch_pdl(score_kernel<V4>, grid, dim3(256), smem, st, a.reps, a.qa, a.qsq, a.nQ, a.maxQ, a.Dp, a.Hkv,
                           a.max_frames, a.n_scored, q_group, a.scores, a.block, a.layer0, fpc, a.status);
  score_kernel<V4><<<grid, 256, smem, st>>>(a.reps, a.qa, a.qsq, a.nQ, a.maxQ, a.Dp, a.Hkv, a.max_frames, a.n_scored, q_group,
                                            a.scores, a.block, a.layer0, fpc, a.status);
  return cudaGetLastError();
}
cudaError_t launch_score(const ScoreArgs& a, bool pdl, cudaStream_t st) {
  return a.Dp <= 512 ? launch_score_v4<4>(a, pdl, st) : launch_score_v4<8>(a, pdl, st);
}

template <int V4, int RB, int CPG>
cudaError_t prepare_retrieve_kernel() {  // once per device
  static PerDeviceOnce attr;
  return attr.run([] {
    cudaError_t e = cudaFuncSetAttribute(retrieve_kernel<V4, RB, CPG>, cudaFuncAttributeMaxDynamicSharedMemorySize, RK_MAX_SMEM);
    if (e != cudaSuccess) return e;
    return cudaFuncSetAttribute(retrieve_kernel<V4, RB, CPG>, cudaFuncAttributeNonPortableClusterSizeAllowed, 1);
  });
}
struct RetrieveLaunch {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  RetrieveLaunch(int cl, int nl, size_t smem, cudaStream_t st) {
    cfg.gridDim = dim3((unsigned)cl, (unsigned)nl);
    cfg.blockDim = dim3(512);
    cfg.dynamicSmemBytes = smem;
    cfg.stream = st;
    at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    at[0].val.programmaticStreamSerializationAllowed = 1;
    at[1].id = cudaLaunchAttributeClusterDimension;
    at[1].val.clusterDim.x = (unsigned)cl;
    at[1].val.clusterDim.y = at[1].val.clusterDim.z = 1;
    cfg.attrs = at;
    cfg.numAttrs = 2;
  }
};
// Clusters of CL CTAs that the device can hold at once, asked once per device.  16 CTAs are beyond the portable size, and a
// partition of the device may have no 16 SMs of one GPC: then 0.  (RB * V4 = 16: one CTA per SM, else two.)
template <int V4, int RB, int CPG, int CL>
int resident_retrieve_clusters() {
  static int known[REKV_MAX_DEVICES] = {};  // + 1
  int dev = 0, n = 0;
  const bool cacheable = cudaGetDevice(&dev) == cudaSuccess && dev >= 0 && dev < REKV_MAX_DEVICES;
  if (cacheable && known[dev]) return known[dev] - 1;
  RetrieveLaunch l(CL, 1, RK_MAX_SMEM, nullptr);
  if (prepare_retrieve_kernel<V4, RB, CPG>() != cudaSuccess ||
      cudaOccupancyMaxActiveClusters(&n, retrieve_kernel<V4, RB, CPG>, &l.cfg) != cudaSuccess) {
    cudaGetLastError();
    n = 0;
  }
  if (cacheable) known[dev] = n + 1;
  return n;
}

// CTAs per cluster of the one-launch retrieval, or 0 where the three launches are better.
// Every warp has to hold all of its rows at once (one round of loads): 28 layers of 1800 frames, 4 KV heads, one at a time: two
// rounds on 16 CTAs, 994 us against 919 with the scores spread over 113 blocks; 9 layers of 439 frames, 8 KV heads: 229 against 253.
// And all layers' clusters have to be resident at once: 16 CTAs with one per SM (7 layers), else 8 with two, less an eighth of the 33
// that the device reports (29), since the last ones start late.  20 retrievals in a graph, clusters against three launches, us
// each, 64 frames: 8 to 15 layers 5.9 against 8.8, 28 7.4 against 9.5, 30 7.5 against 9.6, 31 8.2 against 9.7, 32 10.1 against
// 9.6, 80 19.4 against 15.3; 9 layers of 1000 frames on 16 CTAs 14.7 against 11.1.
int retrieve_cluster(const QBatch& qb, const StoreView& s, int nl, int n_scored, int block, int top_k, int* rows) {
  if (qb.nQ > RK_MAX_Q || top_k <= 0 || n_scored <= 0 || (long long)qb.sumNq * s.Hq * 256 > (1 << 20)) return 0;
  const bool narrow = s.Hkv <= 4;
  int cl = 16;
  if (nl > (narrow ? resident_retrieve_clusters<4, 4, 4, 16>() : resident_retrieve_clusters<8, 2, 2, 16>())) {
    cl = 8;
    const int n8 = narrow ? resident_retrieve_clusters<4, 2, 2, 8>() : resident_retrieve_clusters<8, 1, 1, 8>();
    if (nl > n8 - n8 / 8) return 0;
  }
  const int most = cl / (narrow ? 4 : 8);  // up to 16 float4 per lane on 16 CTAs, 8 on 8
  const long long frames = (long long)n_scored * block;
  // the fewest rows per warp that do it: short code, which every launch fetches anew
  for (*rows = 1; *rows < most && frames > (long long)cl * 16 * *rows;) *rows *= 2;
  return n_scored <= RK_MAX_ITEMS && frames <= (long long)cl * 16 * *rows ? cl : 0;
}
template <int V4, int RB, int CPG>
cudaError_t launch_retrieve_kernel(const RetrieveArgs& a, int nl, cudaStream_t st) {
  const cudaError_t e = prepare_retrieve_kernel<V4, RB, CPG>();
  if (e != cudaSuccess) return e;
  RetrieveLaunch l(a.CL, nl, ((size_t)a.qb.nQ * (a.Hkv * CPG + a.Hkv) * 128 + a.n_scored) * sizeof(float), st);
  return cudaLaunchKernelEx(&l.cfg, retrieve_kernel<V4, RB, CPG>, a);
}
template <int V4, int CPG>
cudaError_t launch_retrieve_rows(const RetrieveArgs& a, int nl, int rows, cudaStream_t st) {
  if (V4 == 4 && rows == 4) return launch_retrieve_kernel<V4, V4 == 4 ? 4 : 2, CPG>(a, nl, st);
  return rows == 2 ? launch_retrieve_kernel<V4, 2, CPG>(a, nl, st) : launch_retrieve_kernel<V4, 1, CPG>(a, nl, st);
}

}  // namespace

cudaError_t rekv_launch_retrieve(rekv_ctx* c, const void* q, const QBatch& qb, int top_k, const CtxGeom& geom,
                                 int n_visible, int layer0, int layer1, int32_t* idx_out, float* scores, cudaStream_t st,
                                 bool write_table) {
  // q, idx_out and scores are indexed with the absolute layer by the kernels; a caller that holds one
  // layer's rows only passes pointers moved back by layer0 layers
  const StoreView& s = c->sv;
  const int maxQ = c->cfg.max_questions;
  const int nl = layer1 - layer0;
  // b = 1: every visible frame is scored (the window's scores are reported but not candidates);
  // b > 1: the complete candidate blocks are scored
  const int b = c->cfg.block_frames;
  const int n_scored = b == 1 ? n_visible : geom.n_items;
  TopkTable tt = {};
  if (write_table) {  // HBM-resident cache: the context table comes out of the same launch
    tt.tbl = c->ctx_tbl;
    tt.hbm = s.hbm;
    tt.page_bytes = s.page_bytes;
    tt.L = s.L;
    tt.ncf = geom.ncf;
    tt.n_vis_frames = n_visible;
  }
  int rk_rows = 0;
  const int cl = c->test_retrieve & REKV_TEST_RETRIEVE_NO_CLUSTER ? 0 : retrieve_cluster(qb, s, nl, n_scored, b, top_k, &rk_rows);
  if (cl) {
    RetrieveArgs a;
    a.q = (const uint4*)q;
    a.reps = s.reps;
    a.scores = scores == c->scores ? nullptr : scores;
    a.idx_out = idx_out;
    a.status = c->status;
    a.tt = tt;
    a.Hq = s.Hq;
    a.Hkv = s.Hkv;
    a.max_frames = s.max_frames;
    a.n_scored = n_scored;
    a.n_cand = geom.n_items;
    a.top_k = top_k;
    a.k_eff = geom.k_items;
    a.block = b;
    a.layer0 = layer0;
    a.qb = qb;
    a.CL = cl;
    a.wait_limit = c->test_wait_limit;
    a.test = c->test_retrieve;
    cudaError_t e;
    const int cpg = cl / s.Hkv >= 8 ? 8 : cl / s.Hkv >= 4 ? 4 : cl / s.Hkv >= 2 ? 2 : 1;
    if (s.Hkv <= 4)
      e = cpg == 8   ? launch_retrieve_rows<4, 8>(a, nl, rk_rows, st)
          : cpg == 4 ? launch_retrieve_rows<4, 4>(a, nl, rk_rows, st)
                     : launch_retrieve_rows<4, 2>(a, nl, rk_rows, st);
    else
      e = cpg == 2 ? launch_retrieve_rows<8, 2>(a, nl, rk_rows, st)
                   : launch_retrieve_rows<8, 1>(a, nl, rk_rows, st);
    if (e != cudaSuccess) return e;
    c->launches += 1;
    return cudaGetLastError();
  }
  if (n_scored > 0) {
    ScoreArgs a = {nl, n_scored, s.reps, c->qa, c->qnorm, qb.nQ, maxQ, s.Dp, s.Hkv, s.max_frames, scores, b, layer0, c->status};
    cudaError_t e;
    e = rekv_launch_pdl((long long)qb.nQ * nl * s.Hkv > rekv_sm_count() ? qmean_kernel<2> : qmean_kernel<4>, dim3(qb.nQ, nl, s.Hkv), dim3(QM_THREADS), 0, st, (const uint4*)q, qb, s.Hq,
                        s.Hkv, s.G, c->qa, c->qnorm, maxQ, layer0);
    if (e != cudaSuccess) return e;
    c->launches += 1;
    e = launch_score(a, true, st);
    if (e != cudaSuccess) return e;
    c->launches += 1;
  }
  if (top_k > 0) {
    cudaError_t e2 = rekv_launch_pdl(topk_kernel, dim3(qb.nQ, nl), dim3(512), 0, st, scores, qb.nQ, n_scored,
                                     geom.n_items, top_k, geom.k_items, idx_out, b, layer0, tt, 1, c->status);
    if (e2 != cudaSuccess) return e2;
    c->launches += 1;
  }
  return cudaGetLastError();
}

cudaError_t rekv_launch_retrieve_external(rekv_ctx* c, const float* q_emb, int nQ, int top_k, const CtxGeom& geom,
                                          int n_visible, float tau, int32_t* idx_out, float* scores, cudaStream_t st) {
  const StoreView& s = c->sv;
  const int E = c->cfg.ext_embed_dim, b = c->cfg.block_frames;
  const int n_scored = b == 1 ? n_visible : geom.n_items;
  int q_group = (int)((96 * 1024) / (E * sizeof(float)));
  if (q_group > nQ) q_group = nQ;
  static PerDeviceOnce attr;
  cudaError_t ea = attr.run([] {
    return cudaFuncSetAttribute(ext_score_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, 96 * 1024);
  });
  if (ea != cudaSuccess) return ea;
  if (n_scored > 0) {
    cudaError_t e1 = rekv_launch_pdl(ext_score_kernel, dim3((n_scored + 7) / 8), dim3(256), (size_t)q_group * E * sizeof(float),
                                     st, (const float*)c->ext_emb, q_emb, nQ, E, n_scored, b, q_group, tau, scores);
    if (e1 != cudaSuccess) return e1;
    c->launches += 1;
  }
  if (top_k > 0) {
    cudaError_t e2 = rekv_launch_pdl(topk_kernel, dim3(nQ, 1), dim3(512), 0, st, (const float*)scores, nQ, n_scored,
                                     geom.n_items, top_k, geom.k_items, idx_out, b, 0, TopkTable{}, s.L, c->status);
    if (e2 != cudaSuccess) return e2;
    c->launches += 1;
  }
  return cudaGetLastError();
}

// ---------------------------------------------------------------------------------------------
// rekv_score_frames_static: scoring without any allocation.
//
// Some hosts cannot let a library allocate device memory: a serving engine that has handed the whole
// GPU to its own memory pool, or a latency-critical thread for which the implicit device
// synchronisation of cudaMalloc/cudaFree is not acceptable.  For them this entry point runs the
// question-vector and cosine-score kernels of one layer with their intermediate (the fp32 question
// vectors and their partial squared norms) in a fixed array that is part of the library image, so
// nothing is allocated, here or in any routine it calls.
//
// The array lives in every GPU context that loads the library, for the life of the process.  All
// calls on a device share it: it is fully rewritten by each call (nothing in it has to start at
// zero), it keeps the last call's contents afterwards, and two calls whose kernels overlap on the
// GPU (different streams, no ordering between them) race on it.
// ---------------------------------------------------------------------------------------------
namespace {

constexpr int STATIC_MAX_QUESTIONS = 16;
constexpr int STATIC_MAX_DP = 1024;                       // H_kv * 128
constexpr int STATIC_QA_FLOATS = STATIC_MAX_QUESTIONS * STATIC_MAX_DP;
constexpr int STATIC_QSQ_FLOATS = STATIC_MAX_QUESTIONS * 8;
// 66 048 bytes: question vectors [16][1024] followed by partial squared norms [16][8]
static __device__ __align__(256) float g_static_scratch[STATIC_QA_FLOATS + STATIC_QSQ_FLOATS];

constexpr int STATIC_MAX_DEVICES = 64;
float* g_static_scratch_addr[STATIC_MAX_DEVICES] = {nullptr};  // device address of the array, per device

}  // namespace

extern "C" int rekv_score_frames_static(const void* q, const int32_t* cu_q, int nQ, int n_q_heads, int n_kv_heads,
                                        int head_dim, const float* reps, int n_frames, float* scores_out, void* stream) {
  if (!q || !cu_q || !reps || !scores_out) {
    rekv_set_error(nullptr, "rekv_score_frames_static: null pointer argument");
    return REKV_ERR_ARG;
  }
  if (head_dim != REKV_HEAD_DIM || n_kv_heads < 1 || n_kv_heads > 8 || n_q_heads < n_kv_heads ||
      n_q_heads % n_kv_heads) {
    rekv_set_error(nullptr, "rekv_score_frames_static: head_dim must be 128 and 1 <= H_kv <= 8 must divide H_q");
    return REKV_ERR_ARG;
  }
  if (nQ < 1 || nQ > STATIC_MAX_QUESTIONS) {
    rekv_set_error(nullptr, "rekv_score_frames_static: at most 16 questions per call (fixed scratch size)");
    return REKV_ERR_ARG;
  }
  if (n_frames < 1) {
    rekv_set_error(nullptr, "rekv_score_frames_static: no frames");
    return REKV_ERR_EMPTY;
  }
  QBatch qb;
  qb.nQ = nQ;
  if (cu_q[0] != 0) {
    rekv_set_error(nullptr, "rekv_score_frames_static: cu_q[0] must be 0");
    return REKV_ERR_ARG;
  }
  for (int i = 0; i < nQ; ++i) {
    if (cu_q[i + 1] <= cu_q[i]) {
      rekv_set_error(nullptr, "rekv_score_frames_static: a question has no tokens");
      return REKV_ERR_ARG;
    }
    qb.cu[i] = cu_q[i];
  }
  qb.cu[nQ] = qb.sumNq = cu_q[nQ];

  // Set-up, once per device, with that device current: in host code the array's name is only a
  // stand-in; the kernels need its device address, which the runtime resolves here.
  int dev = -1;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess || dev < 0 || dev >= STATIC_MAX_DEVICES) {
    rekv_set_error(nullptr, "rekv_score_frames_static: no current CUDA device (or ordinal >= 64)");
    cudaGetLastError();
    return REKV_ERR_CUDA;
  }
  if (!g_static_scratch_addr[dev]) {
    float* ptr = nullptr;
    e = cudaGetSymbolAddress((void**)&ptr, g_static_scratch);
    if (e != cudaSuccess || !ptr) {
      rekv_set_error(nullptr, "rekv_score_frames_static: cudaGetSymbolAddress failed for the scratch array");
      cudaGetLastError();
      return REKV_ERR_CUDA;
    }
    g_static_scratch_addr[dev] = ptr;
  }
  float* qa = g_static_scratch_addr[dev];
  float* qsq = qa + STATIC_QA_FLOATS;

  const int Dp = n_kv_heads * REKV_HEAD_DIM, G = n_q_heads / n_kv_heads;
  cudaStream_t st = (cudaStream_t)stream;
  qmean_kernel<4><<<dim3(nQ, 1, n_kv_heads), QM_THREADS, 0, st>>>((const uint4*)q, qb, n_q_heads, n_kv_heads, G, qa, qsq,
                                                         STATIC_MAX_QUESTIONS, 0);
  const ScoreArgs a = {1, n_frames, reps, qa, qsq, nQ, STATIC_MAX_QUESTIONS, Dp, n_kv_heads, n_frames, scores_out, 1, 0, nullptr};
  e = launch_score(a, false, st);
  if (e != cudaSuccess) {
    rekv_set_error(nullptr, cudaGetErrorString(e));
    return REKV_ERR_CUDA;
  }
  return REKV_OK;
}
