// Eq. 3 in full, the pieces around the attention kernel: O = Attn(W_Q X, [R_k, W_K X], [R_v, W_V X]).
//   - rotary position embedding ("Positional Encoding" paragraph): the retrieved tokens are taken as
//     consecutive tokens, so context token j has position j and token s of X has position n_ctx + s.
//     A table of (cos, sin) per (position, pair) is built once per context in double precision;
//     queries are rotated into a workspace, the context's K tiles into rotated copies (one extra pass
//     over K; the attention kernel then reads K from the copies and V from the pages).
//   - the tokens of X itself follow the context in the attention kernels' token stream, with a causal mask: for the
//     tensor-core kernel their K/V are staged in the pages' layout first; the decode-shaped kernel takes them, the queries
//     and the keys un-rotated and rotates in registers.
// Pairing of dimensions: i with i + 64 (head_dim 128), angle = position * theta^(-2i/128).
#include <algorithm>

#include "ptx_helpers.cuh"
#include "rekv_internal.cuh"

namespace {

using namespace rekv_ptx;

// Twice: in the order of the pairs, and for threads that take the eight pairs of a 16-byte chunk each, chunk c and float4 w of
// (cos, sin) at [position][w][c], so that eight threads read whole lines (four rows of a warp: 4 lines per load instead of 16).
__global__ void rope_table_kernel(float2* __restrict__ tab, float2* __restrict__ tab_c, int n_pos, double theta) {
  const int i = threadIdx.x & 63;
  const long long pos = (long long)blockIdx.x * (blockDim.x >> 6) + (threadIdx.x >> 6);
  if (pos >= n_pos) return;
  const double angle = (double)pos * pow(theta, -2.0 * (double)i / 128.0);
  double s, c;
  sincos(angle, &s, &c);
  tab[pos * 64 + i] = make_float2((float)c, (float)s);
  tab_c[pos * 64 + (((i >> 1) & 3) * 8 + (i >> 3)) * 2 + (i & 1)] = make_float2((float)c, (float)s);
}

// rotates the 8 pairs (lo[e], hi[e]) held as bf16 in two 16-byte chunks; cs: the pairs' (cos, sin),
// two pairs per float4
__device__ __forceinline__ void rotate_chunk(uint4& lo, uint4& hi, const float4 (&cs)[4]) {
  uint32_t* l = reinterpret_cast<uint32_t*>(&lo);
  uint32_t* h = reinterpret_cast<uint32_t*>(&hi);
#pragma unroll
  for (int w = 0; w < 4; ++w) rotate_pair(l[w], h[w], cs[w]);
}
// chunk c of position pos, from the table ordered by chunks
__device__ __forceinline__ void load_cs(float4 (&cs)[4], const float2* __restrict__ tab_c, long long pos, int c) {
  const float4* t = reinterpret_cast<const float4*>(tab_c + pos * 64) + c;
#pragma unroll
  for (int w = 0; w < 4; ++w) cs[w] = __ldg(t + 8 * w);
}
__device__ __forceinline__ void rotate_chunk(uint4& lo, uint4& hi, const float2* __restrict__ tab_c, long long pos, int c) {
  float4 cs[4];
  load_cs(cs, tab_c, pos, c);
  rotate_chunk(lo, hi, cs);
}

// Position of query row n (global row index in the packed batch): n_ctx + (N_s - N_q) + local index.
__device__ __forceinline__ int find_question(const QBatch& qb, int n) {
  int qi = 0;
  while (qi < qb.nQ - 1 && n >= qb.cu[qi + 1]) ++qi;
  return qi;
}

// Queries rotated into q_rot, and X's K/V into the pages' layout behind the context's token stream: per (layer, KV head,
// K/V, 64-dim half) x_rows rows of 128 bytes with the 16-byte chunks XOR-swizzled by (row & 7), question i's tokens from row
// round8(cu_self[i]) + 8 i on; K rotated on the way.  grid = (ceil(rows / 32), layers), 256 threads: 8 threads per row, one
// 16-byte chunk of each half per thread.  Rows: with rotary embedding the sum_Nq * H_q query rows, then (x_kv != null) the
// sum_Ns * H_kv rows of K and as many of V.
__global__ void __launch_bounds__(256) stage_x_kernel(const uint4* __restrict__ q, uint4* __restrict__ q_rot,
                                                      const uint4* __restrict__ k_self, const uint4* __restrict__ v_self,
                                                      char* __restrict__ x_kv, long long x_rows, QBatch qb, QBatch sb, int Hq,
                                                      int Hkv, int n_ctx_tokens, const float2* __restrict__ tab, int layer0) {
  grid_dep_wait();
  grid_dep_launch();
  const int l = layer0 + blockIdx.y;
  const int c = threadIdx.x & 7;
  int row = blockIdx.x * 32 + (threadIdx.x >> 3);
  const int q_rows = tab ? qb.sumNq * Hq : 0, x_n = x_kv ? sb.sumNq * Hkv : 0;
  if (row < q_rows) {
    const int n = row / Hq;
    const int qi = find_question(qb, n);
    const int nq = qb.cu[qi + 1] - qb.cu[qi], ns = sb.cu[qi + 1] - sb.cu[qi];
    const int pos = n_ctx_tokens + (ns - nq) + (n - qb.cu[qi]);
    const long long base = ((long long)l * qb.sumNq * Hq + row) * 16;  // 16 chunks of 16 bytes per row
    uint4 lo = q[base + c], hi = q[base + 8 + c];
    rotate_chunk(lo, hi, tab, pos, c);
    q_rot[base + c] = lo;
    q_rot[base + 8 + c] = hi;
    return;
  }
  row -= q_rows;
  const int kv = row >= x_n ? 1 : 0;
  row -= kv * x_n;
  if (row >= x_n) return;
  const int tok = row / Hkv, g = row - tok * Hkv;
  const int qi = find_question(sb, tok);
  const int s = tok - sb.cu[qi];
  const uint4* src = (kv ? v_self : k_self) + ((long long)l * sb.sumNq * Hkv + row) * 16;
  uint4 lo = src[c], hi = src[8 + c];
  if (!kv && tab) rotate_chunk(lo, hi, tab, n_ctx_tokens + s, c);
  const int r = ((sb.cu[qi] + 7) & ~7) + 8 * qi + s;
  char* dst = x_kv + (((long long)(l * Hkv + g) * 2 + kv) * 2 * x_rows + r) * 128 + ((c ^ (r & 7)) << 4);
  *reinterpret_cast<uint4*>(dst) = lo;
  *reinterpret_cast<uint4*>(dst + x_rows * 128) = hi;
}

// Rotated copies of the context's K tiles.  grid = (ncf * parts, nQ, L), 256 threads; a part of a page is a share of its rows (a
// block per page left most of the device idle where the context is a window: 28 layers of 8 frames 17.5 us, encoding step with
// parts 244 -> 241).  Long contexts are bound by HBM: 808 MB read and written at 72 frames, 132 us.  A K tile of one KV head is
// two 64-dim halves of [N_f rows][128 B] with 16-byte chunks XOR-swizzled by (row & 7): dimension pair
// (i, i + 64) sits at the same swizzled offset of the two halves, so a thread moves one chunk of each.
__global__ void __launch_bounds__(256) rope_stage_kernel(char* const* __restrict__ tbl, char** __restrict__ tbl_k,
                                                         char* __restrict__ k_rot, int nQ, int ncf, int Hkv, int Nf,
                                                         const float2* __restrict__ tab, int layer0, int parts) {
  grid_dep_wait();
  // (no divisions where a page is one block: 300 against 305 us for 12 tokens over 72 frames)
  const int slot = parts == 1 ? blockIdx.x : blockIdx.x / parts, part = blockIdx.x - slot * parts;
  const int qi = blockIdx.y, l = layer0 + blockIdx.z;
  const long long e = ((long long)l * nQ + qi) * ncf + slot;
  const char* page = tbl[e];
  const long long half_bytes = (long long)Nf * 128;
  char* dst = k_rot + e * Hkv * 2 * half_bytes;
  if (threadIdx.x == 0 && part == 0) tbl_k[e] = dst;
  // a thread takes (row, chunk) positions and walks the KV heads: the (cos, sin) of a position are loaded
  // once for all heads, and four heads' chunks are in flight before the first rotation
  constexpr int U = 4;
  const int rc1 = parts == 1 ? Nf * 8 : (part + 1) * Nf / parts * 8;
  for (int rc = (parts == 1 ? 0 : part * Nf / parts * 8) + threadIdx.x; rc < rc1; rc += 256) {
    const int c = rc & 7, r = rc >> 3;
    const long long off = (long long)r * 128 + ((c ^ (r & 7)) << 4);
    float4 cs[4];
    const float4* tr = reinterpret_cast<const float4*>(tab + ((long long)slot * Nf + r) * 64 + c * 8);
#pragma unroll
    for (int w = 0; w < 4; ++w) cs[w] = __ldg(tr + w);
    for (int g0 = 0; g0 < Hkv; g0 += U) {
      uint4 lo[U], hi[U];
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (g0 + u < Hkv) {
          const char* src = page + (long long)(g0 + u) * 4 * half_bytes + off;  // the page holds K then V of each KV head
          lo[u] = __ldcs(reinterpret_cast<const uint4*>(src));
          hi[u] = __ldcs(reinterpret_cast<const uint4*>(src + half_bytes));
        }
#pragma unroll
      for (int u = 0; u < U; ++u)
        if (g0 + u < Hkv) {
          rotate_chunk(lo[u], hi[u], cs);
          char* d = dst + (long long)(g0 + u) * 2 * half_bytes + off;
          *reinterpret_cast<uint4*>(d) = lo[u];
          *reinterpret_cast<uint4*>(d + half_bytes) = hi[u];
        }
    }
  }
}

}  // namespace

cudaError_t rekv_launch_rope_table(rekv_ctx* c, cudaStream_t st) {
  rope_table_kernel<<<(c->rope_positions + 3) / 4, 256, 0, st>>>(c->rope_tab, c->rope_tab_c, c->rope_positions,
                                                                (double)c->cfg.rope_theta);
  return cudaGetLastError();
}

// What the tensor-core kernel needs for Eq. 3 in full (the decode-shaped kernel takes everything as the caller passes it),
// in two halves.  Layers [layer0, layer1): q, k_self, v_self are indexed with the absolute layer (a caller that holds one
// layer's rows passes pointers moved back by layer0 layers), as the library's own buffers are.
// First half, independent of the retrieval: rotated queries (with rotary embedding), and X's K/V staged behind the
// context's token stream.
cudaError_t rekv_launch_attend_full_self(rekv_ctx* c, const void* q, const void* k_self, const void* v_self,
                                         const QBatch& qb, const QBatch& sb, int ncf, cudaStream_t st, int layer0,
                                         int layer1) {
  const StoreView& s = c->sv;
  const int nl = layer1 - layer0;
  if (rekv_decode_shaped(c, qb, ncf, nl)) return cudaSuccess;
  const bool rope = c->cfg.rope_theta > 0.f;
  const int rows = (rope ? qb.sumNq * s.Hq : 0) + 2 * sb.sumNq * s.Hkv;
  cudaError_t e = rekv_launch_pdl(stage_x_kernel, dim3((rows + 31) / 32, nl), dim3(256), 0, st, (const uint4*)q,
                                  (uint4*)c->q_rot, (const uint4*)k_self, (const uint4*)v_self, c->x_kv, c->x_rows, qb, sb,
                                  s.Hq, s.Hkv, rekv_pos_x(c, ncf), rope ? c->rope_tab_c : nullptr, layer0);
  if (e == cudaSuccess) c->launches += 1;
  return e;
}

// Second half, after the context table is there: rotated copies of the context's keys (consecutive positions).
cudaError_t rekv_launch_attend_full_ctx(rekv_ctx* c, const QBatch& qb, int ncf, cudaStream_t st, int layer0,
                                        int layer1) {
  const StoreView& s = c->sv;
  if (!rekv_rope_ctx(c) || ncf == 0 || rekv_decode_shaped(c, qb, ncf, layer1 - layer0)) return cudaSuccess;
  // a page's rows over several blocks while that makes at most sixteen blocks for each SM, and 32 rows for a block
  const long long pages = (long long)ncf * qb.nQ * (layer1 - layer0);
  const int parts = (int)std::max(1ll, std::min<long long>(s.Nf / 32, 16ll * rekv_sm_count() / pages));
  cudaError_t e = rekv_launch_pdl(rope_stage_kernel, dim3(ncf * parts, qb.nQ, layer1 - layer0), dim3(256), 0, st, c->ctx_tbl, c->tbl_k,
                                  c->k_rot, qb.nQ, ncf, s.Hkv, s.Nf, c->rope_tab, layer0, parts);
  if (e == cudaSuccess) c->launches += 1;
  return e;
}
