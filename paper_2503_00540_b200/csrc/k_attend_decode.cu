#include <algorithm>

#include "attend_common.cuh"

using namespace rekv_ptx;

namespace rekv_att {

// Step 5 (Eq. 3) for few query rows per KV head (decode steps: N_q * G <= 16): the step is bound by reading the
// context, not by the contraction (AI ~ G FLOP/B), so this kernel only has to keep the loads in flight, and does everything
// a step needs in ONE launch: a layer is 29 MB at most (4.5 us), as long as one or two launches.
// A step's K and V tiles -- a frame's, or several small frames' -- are double-buffered whole (two steps in flight per SM) and
// the 16-row tile is worked on by eight warps that split the step's tokens among themselves with mma.sync (m16n8k16, ldmatrix
// straight from the swizzled tiles); their (max, sum, O) are merged through shared memory at the end of a range.
// What bounds a layer of its own (28 layers one after the other, 72 frames of 196 tokens, rotary embedding): the chain behind the
// dependency wait, in us: Q 0.7, two frames 3.4, parts out 0.9, join 4; and the copies of the frames, 6.7 from a CTA's start, which
// can begin when the SM's CTA of the launch before has left.  So everything that does not depend on the launch before is done
// before the wait (the frames, their rotation), X is asked for right after it, and the join has all its loads in flight:
// 562 -> 391 us, 20 -> 14 a layer.
// Rotary embedding: the queries are rotated as they are loaded.  The keys of a CTA's first two steps are rotated in place in
// shared memory before the dependency wait (where the context is known to be complete), later ones in registers between ldmatrix
// and mma -- the dimensions i and i + 64 of a token lie in the same lane's fragments of k-blocks kb and kb + 4 -- with (cos, sin)
// from the table in L2 (a separate pass read and wrote every key of the context once more for each token).  Rotated values are
// rounded to bf16.
// The tokens of X (Eq. 3 in full) are further steps of the unit behind its frames, copied into a free stage by all threads.
// A unit cut into parts is merged by the CTA that finishes its last part, whatever the number of parts.

// Both products are taken transposed, S^T = K Q^T and O^T = V^T P^T, so that the query rows are the 8-wide side of
// m16n8k16: at most 8 rows (NT = 1: one token at G <= 8) need half the products and half the accumulators of a 16-row
// tile, and the registers hold a unit's (cos, sin) instead, asked for before the frame has arrived.

// Self-check of an address or index before it is used: a violation is recorded in the status word (read by
// rekv_check_status as error -(1000 + code)) and the access is skipped instead of faulting.
#define DEC_GUARD(cond, code) ((cond) ? true : (atomicExch(p.status, -(1000 + (code))), false))
template <int NT, bool ROPE>
__global__ void __launch_bounds__(DEC_THREADS, 1) attend_decode_kernel(const __grid_constant__ TcParams p) {
  extern __shared__ __align__(1024) unsigned char smem_raw[];
  unsigned char* smem = (unsigned char*)(((uintptr_t)smem_raw + 1023) & ~(uintptr_t)1023);
  const uint32_t s_base = smem_u32(smem);
  const int stage_rows = p.F * p.Npad;               // rows of a step: F frames of N_pad rows, or that many tokens of X
  const uint32_t half_stride = stage_rows * 128u;
  const uint32_t tile_bytes = 2u * half_stride;      // K (or V) of a step: two 64-dim halves
  const uint32_t ring_bytes = max(4u * tile_bytes, DEC_SCRATCH);  // the merge scratch reuses the ring
  const uint32_t bar0 = s_base + ring_bytes;  // full[stage]
  volatile uint32_t* s_abort = reinterpret_cast<volatile uint32_t*>(smem + ring_bytes + 16);
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;

  auto zero_pads = [&]() {  // the pad rows [Nf, Npad) of every frame in every tile half; bulk copies never touch them
    const int pad_rows = p.Npad - p.Nf;
    const int n16 = 8 * p.F * pad_rows * 8;  // (stage, K/V, half) x frames x rows x 16-byte chunks
    for (int i = tid; i < n16; i += DEC_THREADS) {
      const int c = i & 7, r = (i >> 3) % pad_rows, hf = (i >> 3) / pad_rows, f = hf % p.F, hh = hf / p.F;
      *reinterpret_cast<uint4*>(smem + hh * half_stride + (f * p.Npad + p.Nf + r) * 128 + c * 16) = make_uint4(0, 0, 0, 0);
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

  // The CTA's steps: a range of one unit when every unit has `parts` CTAs of its own -- frame_parts of them with even shares of
  // its first `split` steps, the last one with the rest -- else `per` steps of the launch's sequence of (unit, step)
  long long pos, end;
  if (p.parts > 0) {
    const int k = (int)(blockIdx.x / (unsigned)p.units), u = (int)blockIdx.x - k * p.units;
    pos = (long long)u * p.steps + k * p.split / p.frame_parts;
    end = (long long)u * p.steps + (k + 1 == p.parts ? p.steps : (k + 1) * p.split / p.frame_parts);
  } else {
    pos = (long long)blockIdx.x * p.per;
    end = min(pos + (long long)p.per, p.total);
  }
  uint32_t cnt = 0;  // steps consumed so far by this CTA: stage = cnt & 1, phase = (cnt >> 1) & 1
  uint32_t issued = 0;  // warp 0: steps whose copies have been issued (sequence numbers [0, issued))
  const uint32_t wait_limit = p.wait_limit ? p.wait_limit : (1u << 22);
  bool ok = true, waited = false;
  auto wait_step = [&](uint32_t seq) -> bool {
    for (uint32_t it = 0; it < wait_limit; ++it) {
      if (mbar_try_wait(bar0 + 8 * (seq & 1), (seq >> 1) & 1)) return true;
      if (*s_abort) return false;
      if (it > 2048) __nanosleep(64);
    }
    *s_abort = 1;
    return false;
  };

  while (pos < end && ok) {
    const long long u = pos / p.steps;
    const int f0 = (int)(pos - u * p.steps);
    const int nst = (int)min((long long)(p.steps - f0), end - pos);   // steps of this segment
    const int nfs = max(0, min(p.fsteps - f0, nst));                   // ... the first nfs of them frames
    const UnitInfo ui = decode_unit(p, u);
    char* const* pages = p.tbl + ((long long)ui.l * p.qb.nQ + ui.qi) * p.ncf;
    const bool whole_unit = (nst == p.steps);
    const int ns = p.sb.nQ ? p.sb.cu[ui.qi + 1] - p.sb.cu[ui.qi] : 0;
    const int nq = p.qb.cu[ui.qi + 1] - p.qb.cu[ui.qi];
    // Step i of this segment into stage (cnt + i) & 1.  Frames: warp 0, a frame per lane.
    auto issue_frames = [&](int i) {
      const uint32_t seq = cnt + i, st = seq & 1;
      const int fr = (f0 + i) * p.F, n = min(p.F, p.ncf - fr);
      issued = seq + 1;
      if (p.skip_copy_entry >= 0 && blockIdx.x == 0 && (int)seq == p.skip_copy_entry) return;  // test-only
      const uint32_t bar = bar0 + 8 * st;
      if (lane == 0) mbar_expect_tx(bar, 4u * half_bytes * (uint32_t)n);
      __syncwarp();
      if (lane < n) {
        const char* kt = reinterpret_cast<const char*>(__ldcg(reinterpret_cast<const unsigned long long*>(pages) + fr + lane)) +
                         (long long)(ui.g * 2) * p.Nf * 256;
        const uint32_t dst = s_base + st * 2u * tile_bytes + (uint32_t)(lane * p.Npad) * 128u;
        if (DEC_GUARD(kt != nullptr && (reinterpret_cast<uintptr_t>(kt) & 15) == 0 && (half_bytes & 15) == 0, 1) &&
            DEC_GUARD(dst + tile_bytes + half_stride + half_bytes <= s_base + ring_bytes && (dst & 15) == 0, 2)) {
          bulk_g2s(dst, kt, half_bytes, bar);
          bulk_g2s(dst + half_stride, kt + half_bytes, half_bytes, bar);
          bulk_g2s(dst + tile_bytes, kt + 2 * half_bytes, half_bytes, bar);
          bulk_g2s(dst + tile_bytes + half_stride, kt + 3 * half_bytes, half_bytes, bar);
        }
      }
      __syncwarp();
    };
    // Tokens of X: all threads, rows in the pages' layout, zeros behind them up to a whole 16-token unit
    auto x_tokens = [&](int i) { return min(ns - (f0 + i - p.fsteps) * stage_rows, stage_rows); };
    auto issue_x = [&](int i) {
      const int x0 = (f0 + i - p.fsteps) * stage_rows, n = x_tokens(i), nu = (max(n, 0) + 15) >> 4;
      const uint32_t dst0 = s_base + ((cnt + i) & 1) * 2u * tile_bytes;
      for (int it = tid; it < nu * 16 * 32; it += DEC_THREADS) {
        const int c = it & 15, kv = (it >> 4) & 1, r = it >> 5;
        const __nv_bfloat16* src = (kv ? p.v_self : p.k_self) +
            (((long long)ui.l * p.sb.sumNq + p.sb.cu[ui.qi] + (r < n ? x0 + r : 0)) * p.Hkv + ui.g) * 128 + c * 8;
        cp_async16(dst0 + kv * tile_bytes + (c >> 3) * half_stride + r * 128 + (((c & 7) ^ (r & 7)) << 4), src, r < n ? 16u : 0u);
      }
    };
    auto units_of = [&](int i) {  // 16-row units of step i
      return i >= nfs ? (max(x_tokens(i), 0) + 15) >> 4 : min(p.F, p.ncf - (f0 + i) * p.F) * (p.Npad >> 4);
    };
    const int upf = p.Npad >> 4;                                       // units of a frame
    auto frame_pos = [&](int i, int un) {                              // position of the first token of unit un of frame step i
      const int f = p.F == 1 ? 0 : un / upf;
      return ((f0 + i) * p.F + f) * p.Nf + (un - f * upf) * 16;
    };
    if (warp == 0) {
      if (nfs > 0) issue_frames(0);
      if (nfs > 1) issue_frames(1);
    }
    // (cos, sin) of the query rows: token n of the question is token N_s - N_q + n of X
    float4 csq[4][2];
    auto ask_csq = [&](int nt) {
      const int r = 8 * nt + lg;
      const float2* t = p.tab + (long long)(p.pos_x + ns - nq + (r < ui.rows_q ? r / p.G : 0)) * 64 + 2 * lt;
#pragma unroll
      for (int kb = 0; kb < 4; ++kb)
#pragma unroll
        for (int e = 0; e < 2; ++e) csq[kb][e] = __ldg(reinterpret_cast<const float4*>(t + kb * 16 + e * 8));
    };
    int rotated = 0;   // steps whose keys are rotated already
    if (p.early && !waited) {
      if (ROPE && p.rot_ctx) {
        // Before the dependency wait, hidden behind the launch before: the keys of the first two steps are rotated in place,
        // each 16-token unit by the warp that will use it, eight rows at a time.  The next rows' (cos, sin) are asked for
        // before these are used, the first ones' before their frame has arrived.
        rotated = min(2, nfs);
        const int nu0 = rotated > 0 ? units_of(0) : 0, nu1 = rotated > 1 ? units_of(1) : 0;
        const int a0 = warp * nu0 / DEC_WARPS, n0 = (warp + 1) * nu0 / DEC_WARPS - a0;
        const int a1 = warp * nu1 / DEC_WARPS, n = n0 + (warp + 1) * nu1 / DEC_WARPS - a1;
        const int c = lane & 7;
        auto ask = [&](int h, float4 (&x)[2][4]) {
          const int k = h >> 1;
          const int at = (k < n0 ? frame_pos(0, a0 + k) : frame_pos(1, a1 + k - n0)) + (h & 1) * 8 + (lane >> 3);
#pragma unroll
          for (int j = 0; j < 2; ++j) {  // (pad rows: any position)
            const float4* t = reinterpret_cast<const float4*>(p.tab_c + (long long)min(at + 4 * j, p.n_pos - 1) * 64) + c;
#pragma unroll
            for (int w = 0; w < 4; ++w) x[j][w] = __ldg(t + 8 * w);
          }
        };
        auto turn = [&](int h, const float4 (&x)[2][4]) {
          const int k = h >> 1, i = k < n0 ? 0 : 1, un = i ? a1 + k - n0 : a0 + k;
          if (ok && (h == 0 || h == 2 * n0)) ok = wait_step(cnt + i);
          if (!ok) return;
          unsigned char* k0 = smem + ((cnt + i) & 1) * 2u * tile_bytes;
#pragma unroll
          for (int j = 0; j < 2; ++j) {
            const int r = un * 16 + (h & 1) * 8 + 4 * j + (lane >> 3);
            uint4* q = reinterpret_cast<uint4*>(k0 + r * 128 + ((c ^ (r & 7)) << 4));
            uint4* qh = reinterpret_cast<uint4*>(reinterpret_cast<unsigned char*>(q) + half_stride);
            uint4 lo = *q, hi = *qh;
            rotate_pair(lo.x, hi.x, x[j][0]);
            rotate_pair(lo.y, hi.y, x[j][1]);
            rotate_pair(lo.z, hi.z, x[j][2]);
            rotate_pair(lo.w, hi.w, x[j][3]);
            *q = lo;
            *qh = hi;
          }
        };
        float4 cs0[2][4], cs1[2][4];
        if (n > 0) ask(0, cs0);
#pragma unroll 1
        for (int h = 0; h < 2 * n; h += 2) {
          ask(h + 1, cs1);
          turn(h, cs0);
          if (h + 2 < 2 * n) ask(h + 2, cs0);
          turn(h + 1, cs1);
        }
        __syncwarp();
      }
      if (ROPE) ask_csq(0);
      grid_dep_wait();
      grid_dep_launch();
      waited = true;
    } else if (ROPE) {
      ask_csq(0);
    }
    if (nfs == 0) issue_x(0);
    if (nfs < 2 && nst > 1) issue_x(1);
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
      if (ROPE) {
        if (nt > 0) ask_csq(nt);
#pragma unroll
        for (int kb = 0; kb < 4; ++kb)
#pragma unroll
          for (int e = 0; e < 2; ++e) rotate_pair(qf[nt][kb][e], qf[nt][kb + 4][e], csq[kb][e]);
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
      const bool is_x = i >= nfs;
      const uint32_t st = (cnt + i) & 1;
      const int x0 = is_x ? (f0 + i - p.fsteps) * stage_rows : 0;      // a tile of X: its first token
      // this warp's tokens: whole 16-token units, spread as evenly as they go (none: X of a shorter question)
      const int nu = units_of(i);
      const int u0 = warp * nu / DEC_WARPS, u1 = (warp + 1) * nu / DEC_WARPS;
      const bool rot = ROPE && (is_x || (p.rot_ctx && i >= rotated));
      // (cos, sin) of a unit: tokens lg (+ 8), dims 16 kb + 2 lt (+ 8); asked for before the frame is waited for
      float4 cs[4][4];
      auto ask_cs = [&](int un) {
        const int at = (is_x ? p.pos_x + x0 + un * 16 : frame_pos(i, un)) + lg;
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
        cp_async_wait_all();
        __syncthreads();
        if (tid == 0) mbar_arrive(bar0 + 8 * st);   // (the stage's phases count all steps)
      } else if (ok) {
        ok = wait_step(cnt + i);
      }
      const uint32_t sK = s_base + st * 2u * tile_bytes, sV = sK + tile_bytes;
      // last row of its frame that a row of Q sees: all of a frame, X up to the row's own token
      int last[NT][2];
#pragma unroll
      for (int nt = 0; nt < NT; ++nt)
#pragma unroll
        for (int e = 0; e < 2; ++e) last[nt][e] = p.Nf - 1;
      if (is_x) {
#pragma unroll
        for (int nt = 0; nt < NT; ++nt)
#pragma unroll
          for (int e = 0; e < 2; ++e) last[nt][e] = ns - nq + (8 * nt + 2 * lt + e) / p.G - x0;
      }
#pragma unroll 1
      for (int un = u0; un < u1 && ok; ++un) {
        const int t0 = un * 16, tf = is_x || p.F == 1 ? t0 : (un % upf) * 16;   // first row of the unit in its stage, and in its frame
        if (!DEC_GUARD(t0 + 16 <= stage_rows, 3)) break;
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
          uint32_t a[4], b[4];
          const uint32_t addr = a0 ^ (uint32_t)(kb << 5);
          ldmatrix_x4(a[0], a[1], a[2], a[3], addr);
          ldmatrix_x4(b[0], b[1], b[2], b[3], addr + half_stride);
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
            const float s0 = tf + lg <= last[nt][e] ? sacc[nt][e] * p.scale_log2 : -INFINITY;
            const float s1 = tf + lg + 8 <= last[nt][e] ? sacc[nt][2 + e] * p.scale_log2 : -INFINITY;
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
          uint32_t v[4];
          ldmatrix_x4_trans(v[0], v[1], v[2], v[3], addr);
#pragma unroll
          for (int nt = 0; nt < NT; ++nt) mma_bf16_16816(oacc[nt][dm], v, pf[nt][0], pf[nt][1]);
        }
      }
      if (is_x || i < rotated) fence_proxy_async();  // (written by threads: a bulk copy may be the next to write it)
      __syncthreads();  // every warp is done with this stage
      if (*s_abort) ok = false;
      if (!ok) break;
      if (i + 2 < nfs) {
        if (warp == 0) issue_frames(i + 2);
      } else if (i + 2 < nst) {
        issue_x(i + 2);
      }
    }
    if (!ok) {
      // a copy never completed: record it and give the copies still in flight -- every thread's share of X, and the last two
      // steps of frames issued, one per stage (a bounded chance) -- time to land before the CTA's shared memory is given up
      cp_async_wait_all();
      if (tid == 0) {
        atomicExch(p.status, REKV_ERR_TIMEOUT);
        for (uint32_t e = issued > 2 ? issued - 2 : 0; e < issued; ++e)
          for (uint32_t it = 0; it < wait_limit && !mbar_try_wait(bar0 + 8 * (e & 1), (e >> 1) & 1); ++it)
            __nanosleep(64);
      }
      __syncthreads();
      break;
    }
    cnt += nst;

    // the unit's parts, and where they are kept (a CTA that works on two units has a part of each)
    const long long c_first = p.parts > 0 ? 0 : (u * p.steps) / p.per;
    const long long slot0 = p.parts > 0 ? u * p.parts : c_first + u;
    const int part = p.parts > 0 ? (int)(blockIdx.x / (unsigned)p.units) : (int)(blockIdx.x - c_first);
    const int n_parts = p.parts > 0 ? p.parts : (int)(((u + 1) * p.steps - 1) / p.per - c_first + 1);
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
      } else if (DEC_GUARD(slot0 + part < p.part_slots, 5)) {
        const long long slot = slot0 + part;  // a part: 16 rows
        __stcg(reinterpret_cast<float4*>(p.part_o + (slot * 16 + r) * 128) + lane, acc);
        if (lane == 0) __stcg(reinterpret_cast<float2*>(p.part_ml) + slot * 16 + r, make_float2(M, den));
      }
    }
    if (!whole_unit) {
      // The range covered a part of the unit.  The CTA that finishes a unit's last part merges all of them (no further
      // launch): parts are published with a fence, counted with an atomic, and the counter is left at zero for the next
      // launch.
      volatile int& s_last = *reinterpret_cast<volatile int*>(smem + ring_bytes + 24);  // beside the barriers
      __syncthreads();
      if (tid == 0) {
        __threadfence();   // (the CTA's parts, through the barrier)
        const int prev = atomicAdd(p.unit_cnt + u, 1);
        s_last = prev == n_parts - 1 ? 1 : 0;
        if (s_last) p.unit_cnt[u] = 0;
      }
      __syncthreads();
      if (s_last) {
        __threadfence();
        // A warp per row, a float4 of its 128 columns per lane; a lane's (max, sum) are those of parts k0 + lane and
        // k0 + 32 + lane.  The parts of a batch are all in flight at once, into shared memory, where a lane reads what it asked
        // for itself (28 layers, 37 parts each: twelve parts at a time in registers took 8 us of a layer's 20, this 4).
        const int cap = min((int)(ring_bytes / (DEC_WARPS * 512)), 64);   // parts of a batch
        unsigned char* mine = smem + (size_t)warp * cap * 512 + lane * 16;
        for (int r = warp; r < ui.rows_q; r += DEC_WARPS) {
          const float2* ml_r = reinterpret_cast<const float2*>(p.part_ml) + slot0 * 16 + r;
          const float4* o_r = reinterpret_cast<const float4*>(p.part_o + (slot0 * 16 + r) * 128) + lane;
          float M = -1e30f, den = 0.f;
          float4 acc = make_float4(0.f, 0.f, 0.f, 0.f);
          for (int k0 = 0; k0 < n_parts; k0 += cap) {
            const int kn = min(cap, n_parts - k0);
#pragma unroll 4
            for (int k = 0; k < kn; ++k) cp_async16(smem_u32(mine + k * 512), o_r + (long long)(k0 + k) * 16 * 32, 16u);
            const float2 ml0 = lane < kn ? __ldcg(ml_r + (k0 + lane) * 16) : make_float2(-INFINITY, 0.f);
            const float2 ml1 = 32 + lane < kn ? __ldcg(ml_r + (k0 + 32 + lane) * 16) : make_float2(-INFINITY, 0.f);
            float Mn = fmaxf(M, fmaxf(ml0.x, ml1.x));
            for (int o = 16; o; o >>= 1) Mn = fmaxf(Mn, __shfl_xor_sync(0xffffffffu, Mn, o));
            const float a = ex2(M - Mn), w0 = ex2(ml0.x - Mn), w1 = ex2(ml1.x - Mn);
            M = Mn;
            float d = fmaf(w0, ml0.y, w1 * ml1.y);
            for (int o = 16; o; o >>= 1) d += __shfl_xor_sync(0xffffffffu, d, o);
            den = fmaf(den, a, d);
            acc = make_float4(acc.x * a, acc.y * a, acc.z * a, acc.w * a);
            cp_async_wait_all();
#pragma unroll 8
            for (int k = 0; k < kn; ++k) {  // added in part order
              const float wk = __shfl_sync(0xffffffffu, k < 32 ? w0 : w1, k & 31);
              const float4 x = *reinterpret_cast<const float4*>(mine + k * 512);
              acc.x = fmaf(wk, x.x, acc.x);
              acc.y = fmaf(wk, x.y, acc.y);
              acc.z = fmaf(wk, x.z, acc.z);
              acc.w = fmaf(wk, x.w, acc.w);
            }
            __syncwarp();
          }
          const float inv = den > 0.f ? 1.f / den : 0.f;
          *reinterpret_cast<uint2*>(p.out + row_index(r) * 128 + lane * 4) =
              make_uint2(pack_bf16(acc.x * inv, acc.y * inv), pack_bf16(acc.z * inv, acc.w * inv));
        }
      }
    }
    if (pos + nst >= end) break;   // (nothing reads the stages any more)
    __syncthreads();  // the scratch is a K tile again from here on
    if (p.Npad > p.Nf) zero_pads();   // the merge scratch (or a tile of X) covered pad rows
    fence_proxy_async();  // the next range's bulk copies land where these generic-proxy accesses were
    __syncthreads();
    pos += nst;
  }
}


}  // namespace rekv_att

namespace {
// Frames of a step: of small frames so many that each of the eight warps has a 16-token unit (28 layers, one query token over 72 of
// 600 frames of 32 tokens, the whole question: 85 us with a frame per step, 50 with four).
int decode_frames(int Nf) { return std::max(1, rekv_att::DEC_WARPS / ((Nf + 15) >> 4)); }
size_t decode_smem(int Nf) {
  const int npad = (Nf + 15) & ~15;
  return std::max((size_t)4 * 2 * decode_frames(Nf) * npad * 128, (size_t)rekv_att::DEC_SCRATCH) + 64 + 1024;
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
  p.tab_c = full ? c->rope_tab_c : nullptr;
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
  p.F = decode_frames(s.Nf);
  p.fsteps = (ncf + p.F - 1) / p.F;
  p.steps = p.fsteps + (max_ns + p.F * p.Npad - 1) / (p.F * p.Npad);
  const long long units = (long long)(layer1 - layer0) * s.Hkv * p.MP;
  p.total = units * p.steps;
  const int n_sm = rekv_sm_count();
  long long grid;
  p.parts = 0;
  p.split = p.frame_parts = p.units = 0;
  // One layer: every unit gets CTAs of its own, since a CTA with parts of two units pays the end of a range twice.
  if (units * 4 <= n_sm && p.steps > 1) {
    // ... as few as the longest of them allows (24 steps on 18 CTAs are two steps each: twelve CTAs, twelve parts to join).
    // X, whose tokens are asked for only after the dependency wait, is a part of its own if there is room for one, else the last
    // part's besides its frames if it is one step.  The last blocks start last, on the SMs on which the launch before joined
    // its parts: X loses nothing there, having nothing to ask for early.
    const int room = (int)(n_sm / units);
    p.split = p.steps - p.fsteps <= 1 ? p.fsteps : p.steps;
    p.frame_parts = std::min(room, p.split);
    const int longest = (p.split + p.frame_parts - 1) / p.frame_parts;
    p.frame_parts = (p.split + longest - 1) / longest;
    p.parts = p.frame_parts + (p.split < p.steps && p.frame_parts < room ? 1 : 0);
    p.units = (int)units;
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
    for (auto k : {attend_decode_kernel<1, false>, attend_decode_kernel<1, true>, attend_decode_kernel<2, false>, attend_decode_kernel<2, true>})
      if (cudaError_t e1 = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, 227 * 1024)) return e1;
    return cudaSuccess;
  });
  if (e != cudaSuccess) return e;
  if (timed) cudaEventRecord(c->ev_t0, st);
  bool few = true;
  for (int i = 0; i < qb.nQ; ++i) few = few && (qb.cu[i + 1] - qb.cu[i]) * s.G <= 8;
  const auto kernel = few ? (p.tab ? attend_decode_kernel<1, true> : attend_decode_kernel<1, false>)
                          : (p.tab ? attend_decode_kernel<2, true> : attend_decode_kernel<2, false>);
  e = rekv_launch_pdl(kernel, dim3((unsigned)grid), dim3(DEC_THREADS), decode_smem(s.Nf), st, p);
  if (e != cudaSuccess) return e;
  if (timed) {
    cudaEventRecord(c->ev_t1, st);
    c->timing_valid = true;
    c->merge_timed = false;
  }
  c->launches += 1;
  return cudaGetLastError();
}
