#include <algorithm>

#include "attend_common.cuh"

using namespace rekv_ptx;

namespace rekv_att {

// Step 5 (Eq. 3) for few query rows per KV head (decode steps: N_q * G <= 16): the step is bound by reading the
// context, not by the contraction (AI ~ G FLOP/B), so this kernel only has to keep the loads in flight, and does everything
// a step needs in ONE launch: a layer is 29 MB at most (4.5 us), as long as one or two launches.
// A frame's K and V tiles are double-buffered whole (two frames in flight per SM) and the 16-row tile is worked on by eight
// warps that split the frame's tokens among themselves with mma.sync (m16n8k16, ldmatrix straight from the swizzled
// tiles); their (max, sum, O) are merged through shared memory at the end of a range.
// Rotary embedding: the queries are rotated as they are loaded, and the keys in registers between ldmatrix and mma -- the
// dimensions i and i + 64 of a token lie in the same lane's fragments of k-blocks kb and kb + 4 -- with (cos, sin) from the
// table in L2, which cost less than half of the time that the pages take to arrive (a separate pass read and wrote every key
// of the context once more for each token).  Rotated values are rounded to bf16.
// The tokens of X (Eq. 3 in full) are further steps of the unit behind its frames, copied into a free stage by all threads.
// A unit cut into parts is merged by the CTA that finishes its last part, whatever the number of parts.

// Both products are taken transposed, S^T = K Q^T and O^T = V^T P^T, so that the query rows are the 8-wide side of
// m16n8k16: at most 8 rows (NT = 1: one token at G <= 8) need half the products and half the accumulators of a 16-row
// tile, and the registers hold a unit's (cos, sin) instead, asked for before the frame has arrived.

// Self-check of an address or index before it is used: a violation is recorded in the status word (read by
// rekv_check_status as error -(1000 + code)) and the access is skipped instead of faulting.
#define DEC_GUARD(cond, code) ((cond) ? true : (atomicExch(p.status, -(1000 + (code))), false))
template <int NT>
__global__ void __launch_bounds__(DEC_THREADS, 1) attend_decode_kernel(const __grid_constant__ TcParams p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t s_base = smem_u32(smem);
  const uint32_t tile_bytes = 2u * p.Npad * 128u;  // one K (or V) head tile: two 64-dim halves
  const uint32_t half_stride = p.Npad * 128u;
  const uint32_t ring_bytes = max(4u * tile_bytes, DEC_SCRATCH);  // the merge scratch reuses the ring
  const uint32_t bar0 = s_base + ring_bytes;  // full[stage]
  volatile uint32_t* s_abort = reinterpret_cast<volatile uint32_t*>(smem + ring_bytes + 16);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  auto zero_pads = [&]() {  // the pad rows [Nf, Npad) of every tile half; bulk copies never touch them
    const int pad_rows = p.Npad - p.Nf;
    const int n16 = 8 * pad_rows * 8;  // (stage, K/V, half) x rows x 16-byte chunks
    for (int i = tid; i < n16; i += DEC_THREADS) {
      const int c = i & 7, r = (i >> 3) % pad_rows, hh = (i >> 3) / pad_rows;
      *reinterpret_cast<uint4*>(smem + (hh >> 1) * tile_bytes + (hh & 1) * half_stride + (p.Nf + r) * 128 + c * 16) =
          make_uint4(0, 0, 0, 0);
    }
  };
  zero_pads();
  if (tid == 0) {
    mbar_init(bar0, 1);
    mbar_init(bar0 + 8, 1);
    *s_abort = 0;
    fence_barrier_init();
  }
  fence_proxy_async();
  __syncthreads();
  // The first frames of the CTA may be asked for before the kernels before this one are done when the context has been
  // read by an earlier attention launch (the table and its pages are then complete); everything else comes after the wait.
  if (!p.early) {
    grid_dep_wait();
    grid_dep_launch();
  }

  const uint32_t half_bytes = (uint32_t)p.Nf * 128u;
  const int lm = lane >> 3, lr = lane & 7;   // ldmatrix: matrix index and row within it
  const int lg = lane >> 2, lt = lane & 3;   // fragments: group and thread in group

  // The CTA's steps: whole ranges of one unit when every unit has `parts` CTAs of its own, else `per` steps of the launch's
  // sequence of (unit, step)
  long long pos, end;
  if (p.parts > 0) {
    const long long u = blockIdx.x / p.parts;
    const int k = (int)(blockIdx.x - u * p.parts);
    pos = u * p.steps + (long long)k * p.steps / p.parts;
    end = u * p.steps + (long long)(k + 1) * p.steps / p.parts;
  } else {
    pos = (long long)blockIdx.x * p.per;
    end = min(pos + (long long)p.per, p.total);
  }
  // where CTA c keeps its part of unit u (a CTA that works on two units has a part of each)
  auto part_of = [&](long long u, long long c) { return p.parts > 0 ? c : c + u; };
  uint32_t cnt = 0;  // frames consumed so far by this CTA: stage = cnt & 1, phase = (cnt >> 1) & 1
  uint32_t issued = 0;  // thread 0: frames whose copies have been issued (sequence numbers [0, issued))
  const uint32_t wait_limit = p.wait_limit ? p.wait_limit : (1u << 22);
  bool ok = true, waited = false;

  while (pos < end && ok) {
    const long long u = pos / p.steps;
    const int f0 = (int)(pos - u * p.steps);
    const int nst = (int)min((long long)(p.steps - f0), end - pos);   // steps of this segment
    const int nfr = max(0, min(p.ncf - f0, nst));                      // ... the first nfr of them frames
    const UnitInfo ui = decode_unit(p, u);
    char* const* pages = p.tbl + ((long long)ui.l * p.qb.nQ + ui.qi) * p.ncf + f0;
    const bool whole_unit = (nst == p.steps);
    const int ns = p.sb.nQ ? p.sb.cu[ui.qi + 1] - p.sb.cu[ui.qi] : 0;
    const int nq = p.qb.cu[ui.qi + 1] - p.qb.cu[ui.qi];
    auto issue = [&](int i) {  // frame i of this range into stage (cnt + i) & 1
      const uint32_t st = (cnt + i) & 1;
      const char* kt = reinterpret_cast<const char*>(__ldcg(reinterpret_cast<const unsigned long long*>(pages) + i)) +
                       (long long)(ui.g * 2) * p.Nf * 256;
      const uint32_t bar = bar0 + 8 * st;
      const uint32_t dst = s_base + st * 2u * tile_bytes;
      issued = cnt + i + 1;
      if (p.skip_copy_entry >= 0 && blockIdx.x == 0 && (int)(cnt + i) == p.skip_copy_entry) return;  // test-only
      if (!DEC_GUARD(kt != nullptr && (reinterpret_cast<uintptr_t>(kt) & 15) == 0 && (half_bytes & 15) == 0, 1)) return;
      if (!DEC_GUARD(dst + 2u * tile_bytes <= s_base + ring_bytes && (dst & 15) == 0 && (half_stride & 15) == 0, 2)) return;
      mbar_expect_tx(bar, 4u * half_bytes);
      bulk_g2s(dst, kt, half_bytes, bar);
      bulk_g2s(dst + half_stride, kt + half_bytes, half_bytes, bar);
      bulk_g2s(dst + tile_bytes, kt + 2 * half_bytes, half_bytes, bar);
      bulk_g2s(dst + tile_bytes + half_stride, kt + 3 * half_bytes, half_bytes, bar);
    };
    if (tid == 0) {
      if (nfr > 0) issue(0);
      if (nfr > 1) issue(1);
    }
    if (p.early && !waited) {
      grid_dep_wait();
      grid_dep_launch();
      waited = true;
    }
    // Q^T fragments (every warp holds the same rows): row 8 nt + lg, dims 16 kb + 2 lt (+ 8)
    auto row_index = [&](int r) {
      const int n = r / p.G, j = r - n * p.G;
      return (ui.q_row0 + n) * p.Hq + ui.g * p.G + j;
    };
    uint32_t qf[NT][8][2];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      const int r = 8 * nt + lg;
      const bool valid = r < ui.rows_q;
      const uint32_t* src = reinterpret_cast<const uint32_t*>(p.q + row_index(valid ? r : 0) * 128) + lt;
#pragma unroll
      for (int kb = 0; kb < 8; ++kb) {
        qf[nt][kb][0] = valid ? __ldg(src + kb * 8) : 0u;
        qf[nt][kb][1] = valid ? __ldg(src + kb * 8 + 4) : 0u;
      }
      if (p.tab) {  // token n of the question is token N_s - N_q + n of X
        const float2* t = p.tab + (long long)(p.pos_x + ns - nq + (valid ? r / p.G : 0)) * 64 + 2 * lt;
#pragma unroll
        for (int kb = 0; kb < 4; ++kb)
#pragma unroll
          for (int e = 0; e < 2; ++e)
            rotate_pair(qf[nt][kb][e], qf[nt][kb + 4][e], __ldg(reinterpret_cast<const float4*>(t + kb * 16 + e * 8)));
      }
    }
    float oacc[NT][8][4];      // O^T: dims 16 dm + lg (+ 8), rows 8 nt + 2 lt (+ 1)
    float m_r[NT][2], l_r[NT][2];
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
#pragma unroll
      for (int dm = 0; dm < 8; ++dm) oacc[nt][dm][0] = oacc[nt][dm][1] = oacc[nt][dm][2] = oacc[nt][dm][3] = 0.f;
      m_r[nt][0] = m_r[nt][1] = -INFINITY;
      l_r[nt][0] = l_r[nt][1] = 0.f;
    }

    for (int i = 0; i < nst; ++i) {
      const bool is_x = i >= nfr;
      const uint32_t st = is_x ? 0u : (cnt + i) & 1;
      const int x0 = is_x ? (f0 + i - p.ncf) * p.Npad : 0;             // a tile of X: its first token ...
      const int n_tok = is_x ? min(ns - x0, p.Npad) : p.Nf;            // tokens of the step (none: X of a shorter question)
      // this warp's tokens: whole 16-token units, spread as evenly as they go
      const int nu = (max(n_tok, 0) + 15) >> 4;
      const int u0 = warp * nu / DEC_WARPS, u1 = (warp + 1) * nu / DEC_WARPS;
      const bool rot = p.tab != nullptr && (is_x || p.rot_ctx);
      const int pos_t = is_x ? p.pos_x + x0 : (f0 + i) * p.Nf;         // position of the step's first token
      // (cos, sin) of a unit: tokens lg (+ 8), dims 16 kb + 2 lt (+ 8); asked for before the frame is waited for
      float4 cs[4][4];
      auto ask_cs = [&](int un) {
        const int at = pos_t + un * 16 + lg;
        const float2* t0 = p.tab + (long long)min(at, p.n_pos - 1) * 64 + 2 * lt;   // (pad rows: any position)
        const float2* t1 = p.tab + (long long)min(at + 8, p.n_pos - 1) * 64 + 2 * lt;
#pragma unroll
        for (int kb = 0; kb < 4; ++kb)
#pragma unroll
          for (int e = 0; e < 4; ++e)
            cs[kb][e] = __ldg(reinterpret_cast<const float4*>(((e & 1) ? t1 : t0) + kb * 16 + (e >> 1) * 8));
      };
      if (rot && u1 > u0) ask_cs(u0);
      if (is_x) {
        // both stages are free (the segment's frames are done): rows x0 .. of X in the pages' layout, zeros behind them up
        // to a whole 16-token unit
        for (int it = tid; it < nu * 16 * 32; it += DEC_THREADS) {
          const int c = it & 15, kv = (it >> 4) & 1, r = it >> 5;
          uint4 x = make_uint4(0, 0, 0, 0);
          if (r < n_tok)
            x = __ldg(reinterpret_cast<const uint4*>(kv ? p.v_self : p.k_self) +
                      (((long long)ui.l * p.sb.sumNq + p.sb.cu[ui.qi] + x0 + r) * p.Hkv + ui.g) * 16 + c);
          *reinterpret_cast<uint4*>(smem + kv * tile_bytes + (c >> 3) * half_stride + r * 128 + (((c & 7) ^ (r & 7)) << 4)) = x;
        }
        __syncthreads();
      } else {
        bool got = false;
        for (uint32_t it = 0; it < wait_limit; ++it) {
          if (mbar_try_wait(bar0 + 8 * st, ((cnt + i) >> 1) & 1)) {
            got = true;
            break;
          }
          if (*s_abort) break;
          if (it > 2048) __nanosleep(64);
        }
        if (!got) {
          *s_abort = 1;
          ok = false;
        }
      }
      const uint32_t sK = s_base + st * 2u * tile_bytes, sV = sK + tile_bytes;
      // last token of the step that a row sees: all of a frame, X up to the row's own token
      int last[NT][2];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int e = 0; e < 2; ++e) last[nt][e] = is_x ? ns - nq + (8 * nt + 2 * lt + e) / p.G - x0 : p.Nf - 1;
#pragma unroll 1
      for (int un = u0; un < u1 && ok; ++un) {
        const int t0 = un * 16;
        // S^T of the unit, two chains of four products.  K fragments: tokens lg (+ 8), dims 16 kb + 2 lt (+ 8); chunk
        // 2 kb + (lm >> 1) of the row, swizzled with row & 7 = lr, so that the k-block only flips address bits 5 and 6
        const uint32_t a0 = sK + (uint32_t)(t0 + (lm & 1) * 8 + lr) * 128u + (uint32_t)(((lm >> 1) ^ lr) << 4);
        float sacc[NT][4], s2[NT][4];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int e = 0; e < 4; ++e) sacc[nt][e] = s2[nt][e] = 0.f;
#pragma unroll
        for (int kb = 0; kb < 4; ++kb) {
          uint32_t a[4] = {0, 0, 0, 0}, b[4] = {0, 0, 0, 0};
          const uint32_t addr = a0 ^ (uint32_t)(kb << 5);
          if (DEC_GUARD(addr + half_stride + 16 <= s_base + ring_bytes && (addr & 15) == 0, 3)) {
            ldmatrix_x4(a[0], a[1], a[2], a[3], addr);
            ldmatrix_x4(b[0], b[1], b[2], b[3], addr + half_stride);
          }
          if (rot) {
#pragma unroll
            for (int e = 0; e < 4; ++e) rotate_pair(a[e], b[e], cs[kb][e]);
          }
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) {
            mma_bf16_16816(sacc[nt], a, qf[nt][kb][0], qf[nt][kb][1]);
            mma_bf16_16816(s2[nt], b, qf[nt][kb + 4][0], qf[nt][kb + 4][1]);
          }
        }
        if (rot && un + 1 < u1) ask_cs(un + 1);
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int e = 0; e < 4; ++e) sacc[nt][e] += s2[nt][e];
        uint32_t pf[NT][2];
#pragma unroll
        for (int nt = 0; nt < NT; ++nt) {
          float al[2];
#pragma unroll
          for (int e = 0; e < 2; ++e) {
            const float s0 = t0 + lg <= last[nt][e] ? sacc[nt][e] * p.scale_log2 : -INFINITY;
            const float s1 = t0 + lg + 8 <= last[nt][e] ? sacc[nt][2 + e] * p.scale_log2 : -INFINITY;
            float mx = fmaxf(s0, s1);
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 4));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 8));
            mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 16));
            const float mn = fmaxf(m_r[nt][e], mx);
            const float ref = mn == -INFINITY ? 0.f : mn;  // (a row that has seen nothing yet: its terms are 2^-inf = 0)
            al[e] = ex2(m_r[nt][e] - ref);
            m_r[nt][e] = mn;
            sacc[nt][e] = ex2(s0 - ref);
            sacc[nt][2 + e] = ex2(s1 - ref);
            l_r[nt][e] = l_r[nt][e] * al[e] + (sacc[nt][e] + sacc[nt][2 + e]);
          }
          if (__any_sync(0xffffffffu, al[0] != 1.f || al[1] != 1.f)) {
#pragma unroll
            for (int dm = 0; dm < 8; ++dm) {
              oacc[nt][dm][0] *= al[0];
              oacc[nt][dm][1] *= al[1];
              oacc[nt][dm][2] *= al[0];
              oacc[nt][dm][3] *= al[1];
            }
          }
          // P^T as the B operand: each 8x8 block (tokens x rows) transposed between the lanes
          pf[nt][0] = movmatrix_trans(pack_bf16(sacc[nt][0], sacc[nt][1]));
          pf[nt][1] = movmatrix_trans(pack_bf16(sacc[nt][2], sacc[nt][3]));
        }
        const uint32_t v0 = sV + (uint32_t)(t0 + (lm >> 1) * 8 + lr) * 128u + (uint32_t)(((lm & 1) ^ lr) << 4);
#pragma unroll
        for (int dm = 0; dm < 8; ++dm) {
          const uint32_t addr = (v0 ^ (uint32_t)((dm & 3) << 5)) + (dm >= 4 ? half_stride : 0u);
          uint32_t v[4] = {0, 0, 0, 0};
          if (DEC_GUARD(addr + 16 <= s_base + ring_bytes && (addr & 15) == 0, 4)) ldmatrix_x4_trans(v[0], v[1], v[2], v[3], addr);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(oacc[nt][dm], v, pf[nt][0], pf[nt][1]);
        }
      }
      __syncthreads();  // every warp is done with this stage
      if (*s_abort) ok = false;
      if (!ok) break;
      if (tid == 0 && i + 2 < nfr) issue(i + 2);
    }
    if (!ok) {
      // a copy never completed: record it and give the copies still in flight -- the last two frames issued, one
      // per stage -- a bounded chance to land before the CTA's shared memory is given up
      if (tid == 0) {
        atomicExch(p.status, REKV_ERR_TIMEOUT);
        for (uint32_t e = issued > 2 ? issued - 2 : 0; e < issued; ++e)
          for (uint32_t it = 0; it < wait_limit && !mbar_try_wait(bar0 + 8 * (e & 1), (e >> 1) & 1); ++it)
            __nanosleep(64);
      }
      __syncthreads();
      break;
    }
    cnt += nfr;

    // ---- merge the eight warps' parts through shared memory (no copy is in flight now) ----
    constexpr int ROW = 132;   // floats per row: lanes of a store (four rows, eight dims) fall into 32 banks
    float* sm_o = reinterpret_cast<float*>(smem);                      // [warp][8 NT rows][ROW]
    float2* sm_ml = reinterpret_cast<float2*>(sm_o + DEC_WARPS * 8 * NT * ROW);  // [warp][8 NT rows]
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {
      float* wo = sm_o + (warp * 8 * NT + 8 * nt + 2 * lt) * ROW + lg;
#pragma unroll
      for (int dm = 0; dm < 8; ++dm) {
        wo[dm * 16] = oacc[nt][dm][0];
        wo[ROW + dm * 16] = oacc[nt][dm][1];
        wo[dm * 16 + 8] = oacc[nt][dm][2];
        wo[ROW + dm * 16 + 8] = oacc[nt][dm][3];
      }
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        float l = l_r[nt][e];
        l += __shfl_xor_sync(0xffffffffu, l, 4);
        l += __shfl_xor_sync(0xffffffffu, l, 8);
        l += __shfl_xor_sync(0xffffffffu, l, 16);
        if (lg == 0) sm_ml[warp * 8 * NT + 8 * nt + 2 * lt + e] = make_float2(m_r[nt][e], l);
      }
    }
    __syncthreads();
#pragma unroll
    for (int nt = 0; nt < NT; ++nt) {  // a warp per row, a float4 of its 128 columns per lane
      const int r = 8 * nt + warp;
      if (r >= ui.rows_q || !DEC_GUARD(ui.rows_q <= 8 * NT && ui.qi < p.qb.nQ && ui.g < p.Hkv, 6)) continue;
      float M = -1e30f;  // (not -inf: the weight of a warp that saw nothing, m = -inf, is then a plain 0)
#pragma unroll
      for (int w = 0; w < DEC_WARPS; ++w) M = fmaxf(M, sm_ml[w * 8 * NT + r].x);
      float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
      float den = 0.f;
#pragma unroll
      for (int w = 0; w < DEC_WARPS; ++w) {
        const float2 ml = sm_ml[w * 8 * NT + r];
        const float wt = ex2(ml.x - M);
        const float4 x = *reinterpret_cast<const float4*>(sm_o + (w * 8 * NT + r) * ROW + lane * 4);
        den = fmaf(wt, ml.y, den);
        acc.x = fmaf(wt, x.x, acc.x);
        acc.y = fmaf(wt, x.y, acc.y);
        acc.z = fmaf(wt, x.z, acc.z);
        acc.w = fmaf(wt, x.w, acc.w);
      }
      if (whole_unit) {
        const float inv = den > 0.f ? 1.f / den : 0.f;
        *reinterpret_cast<uint2*>(p.out + row_index(r) * 128 + lane * 4) =
            make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
      } else if (DEC_GUARD((long long)blockIdx.x + u < p.part_slots, 5)) {
        const long long slot = part_of(u, blockIdx.x);  // a part: 16 rows
        __stcg(reinterpret_cast<float4*>(p.part_o + (slot * 16 + r) * 128) + lane, acc);
        if (lane == 0) __stcg(reinterpret_cast<float2*>(p.part_ml) + slot * 16 + r, make_float2(M, den));
      }
    }
    if (!whole_unit) {
      // The range covered a part of the unit.  The CTA that finishes a unit's last part merges all of them (no further
      // launch): parts are published with a fence, counted with an atomic, and the counter is left at zero for the next
      // launch.
      volatile int& s_last = *reinterpret_cast<volatile int*>(smem + ring_bytes + 24);  // beside the barriers
      const long long c_first = p.parts > 0 ? u * p.parts : (u * p.steps) / p.per;
      const int n_parts = p.parts > 0 ? p.parts : (int)(((u + 1) * p.steps - 1) / p.per - c_first + 1);
      __threadfence();
      __syncthreads();
      if (tid == 0) {
        const int prev = atomicAdd(p.unit_cnt + u, 1);
        s_last = prev == n_parts - 1 ? 1 : 0;
        if (s_last) p.unit_cnt[u] = 0;
      }
      __syncthreads();
      if (s_last) {
        __threadfence();
        // a warp per row, a float4 of its 128 columns per lane; a lane's (max, sum) are those of parts k0 + lane and
        // k0 + 32 + lane.  The rows of U parts are in flight (28 layers, 37 parts each: twelve 575 us, twenty 612, whose
        // registers spill).
        constexpr int U = 12;
        for (int r = warp; r < ui.rows_q; r += DEC_WARPS) {
          const float2* ml_r = reinterpret_cast<const float2*>(p.part_ml) + part_of(u, c_first) * 16 + r;
          const float4* o_r = reinterpret_cast<const float4*>(p.part_o + (part_of(u, c_first) * 16 + r) * 128) + lane;
          float M = -1e30f, den = 0.f;
          float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int k0 = 0; k0 < n_parts; k0 += 64) {
            const int kn = min(64, n_parts - k0);
            const float2 ml0 = lane < kn ? __ldcg(ml_r + (k0 + lane) * 16) : make_float2(-INFINITY, 0.f);
            const float2 ml1 = 32 + lane < kn ? __ldcg(ml_r + (k0 + 32 + lane) * 16) : make_float2(-INFINITY, 0.f);
            float4 x[U];
#pragma unroll
            for (int i = 0; i < U; ++i)
              if (i < kn) x[i] = __ldcg(o_r + (long long)(k0 + i) * 16 * 32);
            float Mn = fmaxf(M, fmaxf(ml0.x, ml1.x));
            for (int o = 16; o; o >>= 1) Mn = fmaxf(Mn, __shfl_xor_sync(0xffffffffu, Mn, o));
            const float a = ex2(M - Mn), w0 = ex2(ml0.x - Mn), w1 = ex2(ml1.x - Mn);
            M = Mn;
            float d = fmaf(w0, ml0.y, w1 * ml1.y);
            for (int o = 16; o; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            den = fmaf(den, a, d);
            acc = make_float4(acc.x * a, acc.y * a, acc.z * a, acc.w * a);
#pragma unroll 1
            for (int k1 = 0; k1 < kn; k1 += U) {  // added in part order
#pragma unroll
              for (int i = 0; i < U; ++i)
                if (k1 + i < kn) {
                  const int k = k1 + i;
                  const float wk = __shfl_sync(0xffffffffu, k < 32 ? w0 : w1, k & 31);
                  acc.x = fmaf(wk, x[i].x, acc.x);
                  acc.y = fmaf(wk, x[i].y, acc.y);
                  acc.z = fmaf(wk, x[i].z, acc.z);
                  acc.w = fmaf(wk, x[i].w, acc.w);
                }
#pragma unroll
              for (int i = 0; i < U; ++i)
                if (k1 + U + i < kn) x[i] = __ldcg(o_r + (long long)(k0 + k1 + U + i) * 16 * 32);
            }
          }
          const float inv = den > 0.f ? 1.f / den : 0.f;
          *reinterpret_cast<uint2*>(p.out + row_index(r) * 128 + lane * 4) =
              make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
        }
      }
    }
    __syncthreads();  // the scratch is a K tile again from here on
    if (p.Npad > p.Nf) zero_pads();   // the merge scratch (or a tile of X) covered pad rows
    fence_proxy_async();  // the next range's bulk copies land where these generic-proxy accesses were
    __syncthreads();
    pos += nst;
  }
}


}  // namespace rekv_att

namespace {
size_t decode_smem(int Nf) {
  const int npad = (Nf + 15) & ~15;
  return std::max((size_t)4 * 2 * npad * 128, (size_t)rekv_att::DEC_SCRATCH) + 64 + 1024;
}
}  // namespace

// Decode-shaped batches (at most 16 query rows per KV head in every question) take the kernel that is built around the
// loads; it needs two whole frames of one KV head in shared memory.
bool rekv_decode_shaped(const rekv_ctx* c, const QBatch& qb, int ncf, int nl) {
  for (int i = 0; i < qb.nQ; ++i)
    if ((qb.cu[i + 1] - qb.cu[i]) * c->sv.G > 16) return false;
  return ncf > 0 && decode_smem(c->sv.Nf) <= 227 * 1024 && (size_t)nl * c->sv.Hkv * qb.nQ <= c->cnt_units;
}

cudaError_t rekv_launch_attend_decode(rekv_ctx* c, const void* q, const QBatch& qb, int ncf, int layer0, int layer1,
                                      void* out, cudaStream_t st, bool timed, const AttendFullArgs* full) {
  using namespace rekv_att;
  const StoreView& s = c->sv;
  TcParams p;
  p.q = (const __nv_bfloat16*)(full ? full->q : q);
  p.out = (__nv_bfloat16*)out;
  p.tbl = c->ctx_tbl;
  p.k_self = full ? (const __nv_bfloat16*)full->k_self : nullptr;
  p.v_self = full ? (const __nv_bfloat16*)full->v_self : nullptr;
  p.sb.nQ = 0;
  if (full) p.sb = *full->sb;
  p.early = c->ctx_settled && c->ctx_stream == st;
  p.tab = full ? c->rope_tab : nullptr;
  p.n_pos = c->rope_positions;
  p.pos_x = rekv_pos_x(c, ncf);
  p.rot_ctx = rekv_rope_ctx(c);
  p.part_o = c->part_o;
  p.part_ml = c->part_ml;
  p.part_slots = (int)(c->part_units * 8);
  p.unit_cnt = c->unit_cnt;
  p.status = c->status;
  p.qb = qb;
  p.Hq = s.Hq;
  p.Hkv = s.Hkv;
  p.G = s.G;
  p.Nf = s.Nf;
  p.Npad = (s.Nf + 15) & ~15;
  p.wait_limit = c->test_wait_limit;
  p.skip_copy_entry = c->test_skip_copy_entry;
  p.ncf = ncf;
  p.layer0 = layer0;
  p.scale_log2 = 1.4426950408889634f / sqrtf(128.f);
  p.MP = qb.nQ;  // one unit per question
  int max_ns = 0;
  for (int i = 0; full && i < qb.nQ; ++i) max_ns = std::max(max_ns, full->sb->cu[i + 1] - full->sb->cu[i]);
  p.steps = ncf + (max_ns + p.Npad - 1) / p.Npad;
  const long long units = (long long)(layer1 - layer0) * s.Hkv * p.MP;
  p.total = units * p.steps;
  const int n_sm = rekv_sm_count();
  long long grid;
  p.parts = 0;
  // One layer: every unit gets CTAs of its own, since a CTA with parts of two units pays the end of a range twice.
  if (units * 4 <= n_sm && p.steps > 1) {
    // ... as few as the longest of them allows (24 steps on 18 CTAs are two steps each: twelve CTAs, twelve parts to join)
    p.parts = (int)std::min<long long>(n_sm / units, p.steps);
    const int longest = (p.steps + p.parts - 1) / p.parts;
    p.parts = (p.steps + longest - 1) / longest;
    p.per = p.steps;
    grid = units * p.parts;
  } else if (units >= 4 * n_sm || n_sm + units > p.part_slots) {
    grid = units;  // enough units to fill the machine: one whole unit per CTA, no partials
    p.per = p.steps;
  } else {
    grid = p.total < n_sm ? p.total : n_sm;
    p.per = (int)((p.total + grid - 1) / grid);
    grid = (p.total + p.per - 1) / p.per;
  }
  static PerDeviceOnce dec_attr;
  cudaError_t e = dec_attr.run([] {
    cudaError_t e1 = cudaFuncSetAttribute(attend_decode_kernel<1>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
    if (e1 != cudaSuccess) return e1;
    return cudaFuncSetAttribute(attend_decode_kernel<2>, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024);
  });
  if (e != cudaSuccess) return e;
  if (timed) cudaEventRecord(c->ev_t0, st);
  bool few = true;
  for (int i = 0; i < qb.nQ; ++i) few = few && (qb.cu[i + 1] - qb.cu[i]) * s.G <= 8;
  e = rekv_launch_pdl(few ? attend_decode_kernel<1> : attend_decode_kernel<2>, dim3((unsigned)grid), dim3(DEC_THREADS), decode_smem(s.Nf), st, p);
  if (e != cudaSuccess) return e;
  if (timed) {
    cudaEventRecord(c->ev_t1, st);
    c->timing_valid = true;
    c->merge_timed = false;
  }
  c->launches += 1;
  return cudaGetLastError();
}
