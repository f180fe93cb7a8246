// Small kernels of the decode step: row planning + embedding gather, the
// draft's token selection from LM-head statistics, acceptance with KV
// commit / rollback, and helpers for tests.
#include <algorithm>
#include <climits>

#include "common.cuh"
#include "internal.h"

namespace pard {

#define PARD_LAUNCH(kernel, grid, block, smem, strm, pdl, ...)                       \
  do {                                                                                 \
    cudaLaunchConfig_t cfg_ = {};                                                      \
    cfg_.gridDim = dim3(grid);                                                         \
    cfg_.blockDim = dim3(block);                                                       \
    cfg_.dynamicSmemBytes = (smem);                                                    \
    cfg_.stream = (strm);                                                              \
    cudaLaunchAttribute at_[1];                                                        \
    at_[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;                    \
    at_[0].val.programmaticStreamSerializationAllowed = 1;                             \
    cfg_.attrs = at_;                                                                  \
    cfg_.numAttrs = (pdl) ? 1 : 0;                                                     \
    cudaError_t e_ = cudaLaunchKernelEx(&cfg_, kernel, __VA_ARGS__);                   \
    if (e_ != cudaSuccess) throw e_;                                                   \
  } while (0)

// ---------------------------------------------------------------------------
// Row plan + embedding.  One block per row of the pass (grid = row capacity).
//   draft  (Eq. 6): sequence b feeds its pend_cnt pending real tokens, then
//                   K-1 mask tokens (one shared id, or one id per offset),
//                   at positions n-p .. n+K-2; logits rows are the last real
//                   row and every mask row;
//   verify:         [last token, d_0..d_{K-1}] at positions n-1 .. n+K-1;
//   sequential draft (vanilla speculative decoding), pass i: i = 0 feeds
//                   the pending real tokens (logits row: the last), i > 0
//                   feeds candidate d_{i-1} at position n-1+i;
//   prefill:        a run of rows of the concatenated prompts.
// h = E[token]; x = h * g (hi/lo bf16 pairs); ssq[t][m] = sum of h^2 over
// the 128 columns of tile t.
// ---------------------------------------------------------------------------
__global__ void __launch_bounds__(128) embed_kernel(const __grid_constant__ EmbedArgs a) {
  pdl_wait();
  pdl_trigger();
  __shared__ int s_tok;
  const int m = blockIdx.x;
  if (threadIdx.x < 32) {
    // Rows of each sequence and their prefix: two sequences a lane, all
    // counts requested at once (one after the other they cost a memory
    // latency per sequence).
    const int lane = threadIdx.x;
    int b = 0, row0 = 0, total = 0;
    {
      const bool prompt = a.mode == EMB_PREFILL;
      int cnt[2];
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int sq = 2 * lane + e;
        cnt[e] = sq >= a.batch ? 0
                 : prompt                  ? a.plen[sq]
                 : a.mode == EMB_DRAFT     ? a.st.pend_cnt[sq] + a.K - 1
                 : a.mode == EMB_DRAFT_SEQ ? (a.seq_i == 0 ? a.st.pend_cnt[sq] : 1)
                                           : a.K + 1;
      }
      int inc = cnt[0] + cnt[1];
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int v = __shfl_up_sync(0xffffffffu, inc, o);
        if (lane >= o) inc += v;
      }
      total = prompt ? a.pf_rows : __shfl_sync(0xffffffffu, inc, 31);
      // first row of the lane's sequences in this pass (a prompt pass is a run
      // of rows of all prompts, one after the other; negative: it began earlier)
      const int start = inc - cnt[0] - cnt[1] - (prompt ? a.pf_row0 : 0);
      if (m == 0) {
        const int s0 = prompt ? a.pf_seq : 0, ns = prompt ? a.pf_nseq : a.batch;
#pragma unroll
        for (int e = 0; e < 2; ++e) {
          const int i = 2 * lane + e - s0;
          if (i >= 0 && i < ns) a.rp.seq_row0[i] = max(0, start + (e ? cnt[0] : 0));
        }
        if (lane == 0) a.rp.seq_row0[ns] = total;
      }
      // this row's sequence: the last one that starts at or before it (an
      // empty sequence starts where its successor does and is not the last)
      int mine = -1, mine0 = 0;
#pragma unroll
      for (int e = 0; e < 2; ++e) {
        const int at = start + (e ? cnt[0] : 0);
        if (2 * lane + e < a.batch && at <= m) { mine = 2 * lane + e; mine0 = at; }
      }
      const unsigned has = __ballot_sync(0xffffffffu, mine >= 0);
      const int src = 31 - __clz((int)has);
      b = __shfl_sync(0xffffffffu, mine, src);
      row0 = __shfl_sync(0xffffffffu, mine0, src);
    }
    if (m == 0 && lane == 0) {
      *a.rp.m_dev = total;
      if (a.call_out) *a.call_out = a.call;
      if (total > a.m_cap) set_status(a.status, ST_BAD_ROWS);
    }
    int tok = -1;
    if (m < total && m < a.m_cap) {
      int pos = 0, out = -1, gi = -1;
      if (a.mode == EMB_PREFILL) {
        tok = a.tokens[a.pf_row0 + m];
        pos = m - row0;
      } else {
        const int j = m - row0, kp = a.st.kmax + 1;
        // the sequence's facts, requested together
        const int n = a.st.n[b], p = a.st.pend_cnt[b];
        const int pend = lane < kp ? a.st.pend[b * kp + lane] : 0;
        if (a.mode == EMB_DRAFT) {
          const int mask = a.mask_ids ? a.mask_ids[max(0, min(j - p, a.K - 2))] : a.mask_id;
          const int real = __shfl_sync(0xffffffffu, pend, min(j, 31));
          tok = j < p ? real : mask;
          pos = n - p + j;
          if (j >= p - 1) { gi = j - (p - 1); out = b * a.K + gi; }
        } else if (a.mode == EMB_DRAFT_SEQ) {
          if (a.seq_i == 0) {
            tok = __shfl_sync(0xffffffffu, pend, min(j, 31));
            pos = n - p + j;
            if (j == p - 1) { gi = 0; out = b * a.K; }
          } else {
            tok = a.st.d[b * a.st.kmax + a.seq_i - 1];
            pos = n - 1 + a.seq_i;
            gi = a.seq_i;
            out = b * a.K + a.seq_i;
          }
        } else {
          const int cand = j > 0 ? a.d_in[b * a.K + j - 1] : 0;
          const int last = __shfl_sync(0xffffffffu, pend, min(max(p - 1, 0), 31));
          tok = j == 0 ? last : cand;
          if (j > 0 && lane == 0) a.st.d[b * a.st.kmax + j - 1] = tok;
          pos = n - 1 + j;
          out = b * (a.K + 1) + j;
        }
      }
      if (tok < 0 || tok >= a.vocab) {
        if (lane == 0) set_status(a.status, ST_BAD_TOKEN);
        tok = 0;
      }
      if (lane == 0) {
        a.rp.row_tok[m] = tok;
        a.rp.row_pos[m] = pos;
        a.rp.row_seq[m] = b;
        a.rp.row_out[m] = out;
        a.rp.row_gi[m] = gi;
      }
    }
    if (lane == 0) s_tok = tok;
  }
  __syncthreads();
  const int tok = s_tok;
  if (tok < 0) return;
  const uint4* e = reinterpret_cast<const uint4*>(a.embed + (size_t)tok * a.d);
  const uint4* g = reinterpret_cast<const uint4*>(a.gain0);
  // a thread takes eight columns at a time, half a warp one 128-column tile
  for (int c8 = threadIdx.x; c8 < a.d / 8; c8 += 128) {
    const uint4 ev = e[c8], gv = g[c8];
    const uint32_t ew[4] = {ev.x, ev.y, ev.z, ev.w}, gw[4] = {gv.x, gv.y, gv.z, gv.w};
    float h[8], x[8], ss = 0.f;
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      h[2 * k] = __uint_as_float(ew[k] << 16);
      h[2 * k + 1] = __uint_as_float(ew[k] & 0xffff0000u);
      x[2 * k] = h[2 * k] * __uint_as_float(gw[k] << 16);
      x[2 * k + 1] = h[2 * k + 1] * __uint_as_float(gw[k] & 0xffff0000u);
      ss += h[2 * k] * h[2 * k] + h[2 * k + 1] * h[2 * k + 1];
    }
    float4* hp = reinterpret_cast<float4*>(a.h + (size_t)m * a.d + c8 * 8);
    hp[0] = make_float4(h[0], h[1], h[2], h[3]);
    hp[1] = make_float4(h[4], h[5], h[6], h[7]);
    store_pair8(a.x, m, c8 * 8, 2 * a.m_cap, x);
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) ss += __shfl_xor_sync(0xffffu << (threadIdx.x & 16), ss, o, 16);
    if ((threadIdx.x & 15) == 0) a.ssq[(size_t)(c8 >> 4) * a.m_cap + m] = ss;
  }
}

// Failure-path self test: one thread waits, through the pipelines' bounded
// wait, on an mbarrier that nothing arrives on; the wait gives up after its
// limit (kWaitLimitNs) and flags ST_TIMEOUT_TMA, as a stalled pipeline would,
// and the kernel returns normally.
__global__ void stalled_wait_kernel(uint32_t* status) {
  __shared__ __align__(8) uint64_t bar;
  __shared__ int never_raised;
  if (threadIdx.x != 0) return;
  mbar_init(&bar, 1);
  never_raised = 0;
  fence_barrier_init();
  if (!mbar_wait(&bar, 0, &never_raised)) set_status(status, ST_TIMEOUT_TMA);
}

void launch_stalled_wait(uint32_t* status, cudaStream_t s) {
  PARD_LAUNCH(stalled_wait_kernel, 1, 32, 0, s, false, status);
}

void launch_embed(const EmbedArgs& a, int grid, cudaStream_t s, bool pdl) {
  PARD_LAUNCH(embed_kernel, grid, 128, 0, s, pdl, a);
}

// Copy activation rows (hi/lo pairs, packed layout) and their sum-of-squares partials.
__global__ void __launch_bounds__(256) gather_rows_kernel(const __grid_constant__ GatherArgs a) {
  pdl_wait();
  pdl_trigger();
  const int src = a.src[blockIdx.x], dst = a.dst0 + blockIdx.x;
  if (src < 0) return;
  for (int i = threadIdx.x; i < a.d / 4; i += blockDim.x) {  // 8 columns of the hi or the lo row
    const int c = i / 2 * 8, lo = i & 1;
    *reinterpret_cast<uint4*>(a.xg + xpk(dst, lo, c, a.xg_rows)) =
        *reinterpret_cast<const uint4*>(a.x + xpk(src, lo, c, a.x_rows));
  }
  for (int t = threadIdx.x; t < a.ssq_tiles; t += blockDim.x)
    a.ssqg[(size_t)t * a.m_cap_dst + dst] = a.ssq[(size_t)t * a.m_cap_src + src];
}

void launch_gather_rows(const GatherArgs& a, int n, cudaStream_t s, bool pdl) {
  PARD_LAUNCH(gather_rows_kernel, n, 256, 0, s, pdl, a);
}

// Weight packing: nblocks consecutive R-row blocks of a [N][K] matrix move
// between row-major order and the packed layout ([K/64][R][64] per block,
// 16-byte chunks of row r rotated by r mod 8).  tmp holds a copy of the
// blocks in the source order; w is overwritten in the destination order.
__global__ void pack_kernel(const __nv_bfloat16* tmp, __nv_bfloat16* w, int R, int K, int nblocks, int unpack) {
  const int kc = K / 64;
  const size_t chunks = (size_t)nblocks * R * kc * 8;
  for (size_t i = blockIdx.x * (size_t)blockDim.x + threadIdx.x; i < chunks; i += (size_t)gridDim.x * blockDim.x) {
    const int j = (int)(i % 8);
    size_t t = i / 8;
    const int kk = (int)(t % kc);
    t /= kc;
    const int r = (int)(t % R);
    const size_t b = t / R;
    const size_t rm = (b * R + r) * (size_t)K + (size_t)kk * 64 + (size_t)j * 8;
    const size_t pk = ((b * kc + kk) * R + r) * 64 + (size_t)((j ^ (r & 7)) << 3);
    if (!unpack)
      *reinterpret_cast<uint4*>(w + pk) = *reinterpret_cast<const uint4*>(tmp + rm);
    else
      *reinterpret_cast<uint4*>(w + rm) = *reinterpret_cast<const uint4*>(tmp + pk);
  }
}

void launch_pack(const __nv_bfloat16* tmp, __nv_bfloat16* w, int R, int K, int nblocks, bool unpack, cudaStream_t s) {
  const size_t chunks = (size_t)nblocks * R * (K / 64) * 8;
  const int grid = (int)std::min<size_t>((chunks + 255) / 256, 4096);
  PARD_LAUNCH(pack_kernel, grid, 256, 0, s, false, tmp, w, R, K, nblocks, unpack ? 1 : 0);
}

// ---------------------------------------------------------------------------
// Reductions of the LM-head tile statistics.
// (max, sum exp((x - max)/T)) pairs merge by rescaling to the larger max.
// ---------------------------------------------------------------------------
struct RowRed {
  float mx; int arg; float se; float gv; int gi;
};

__device__ __forceinline__ void merge_lse(float& m1, float& s1, float m2, float s2, float T) {
  if (m2 == -INFINITY) return;
  if (m1 == -INFINITY) { m1 = m2; s1 = s2; return; }
  const float M = fmaxf(m1, m2);
  s1 = s1 * expf(m1 / T - M / T) + s2 * expf(m2 / T - M / T);
  m1 = M;
}

__device__ __forceinline__ void merge_red(RowRed& r, const RowRed& o, float T) {
  float m1 = r.mx, s1 = r.se;
  merge_lse(m1, s1, o.mx, o.se, T);
  float v = r.mx;
  int i = r.arg;
  argmax_merge(v, i, o.mx, o.arg);
  r.arg = i;
  r.mx = m1;
  r.se = s1;
  argmax_merge(r.gv, r.gi, o.gv, o.gi);
}

// Block-wide reduction (256 threads) over the w_tiles tile statistics of one
// row; thread 0 returns the result.  Fixed order: strided per thread with all
// loads in flight, a shuffle tree per warp, then the warps in order.
__device__ RowRed reduce_row(const float4* stats, const int2* stats_i, int w_tiles, int m_cap, int m, float T,
                             RowRed* sred) {
  RowRed r{-INFINITY, INT_MAX, 0.f, -INFINITY, INT_MAX};
  for (int t0 = threadIdx.x; t0 < w_tiles; t0 += 4 * 256) {
    float4 s[4];
    int2 si[4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const size_t at = (size_t)min(t0 + k * 256, w_tiles - 1) * m_cap + m;
      s[k] = stats[at];
      si[k] = stats_i[at];
    }
#pragma unroll
    for (int k = 0; k < 4; ++k)
      if (t0 + k * 256 < w_tiles) merge_red(r, RowRed{s[k].x, si[k].x, s[k].y, s[k].z, si[k].y < 0 ? INT_MAX : si[k].y}, T);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    RowRed x;
    x.mx = __shfl_xor_sync(0xffffffffu, r.mx, o);
    x.arg = __shfl_xor_sync(0xffffffffu, r.arg, o);
    x.se = __shfl_xor_sync(0xffffffffu, r.se, o);
    x.gv = __shfl_xor_sync(0xffffffffu, r.gv, o);
    x.gi = __shfl_xor_sync(0xffffffffu, r.gi, o);
    merge_red(r, x, T);
  }
  if ((threadIdx.x & 31) == 0) sred[threadIdx.x >> 5] = r;
  __syncthreads();
  r = sred[0];
  if (threadIdx.x == 0)
    for (int w = 1; w < 8; ++w) merge_red(r, sred[w], T);
  return r;
}

// The same for rows m0 .. m0 + nrows - 1 at once (at most 32 rows), by a block of
// 32 warps: 32 / nrows warps share a row, each lane takes every 32nd of its
// warp's tiles and the warp merges by shuffles, then one thread a row merges
// the warps in order.  out[i] holds row i when the call returns.  (One row
// after the other through a block-wide tree cost about 2.5 us a row.)
// Rows nrows .. nrows + nrows2 - 1 are rows m2 .. of stats2 (row pitch m_cap2).
constexpr int kRowWarps = 32;
template <bool kLse>
__device__ void reduce_rows(const float4* stats, const int2* stats_i, int w_tiles, int m_cap, int m0, int nrows,
                            const float4* stats2, int m_cap2, int m2, int nrows2, float T, RowRed* part, RowRed* out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rows1 = nrows;
  nrows += nrows2;
  const int per = kRowWarps / nrows;  // warps a row
  if (warp < per * nrows) {
    const int row = warp / per;
    const bool second = row >= rows1;
    const int m = second ? m2 + row - rows1 : m0 + row;
    if (second) { stats = stats2; m_cap = m_cap2; }
    RowRed r{-INFINITY, INT_MAX, 0.f, -INFINITY, INT_MAX};
#pragma unroll 4
    for (int t = (warp % per) * 32 + lane; t < w_tiles; t += 32 * per) {
      const size_t at = (size_t)t * m_cap + m;
      if constexpr (kLse) {
        const float4 s = stats[at];
        merge_lse(r.mx, r.se, s.x, s.y, T);
      } else {
        argmax_merge(r.mx, r.arg, stats[at].x, stats_i[at].x);
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      const float m2 = __shfl_xor_sync(0xffffffffu, r.mx, o);
      if constexpr (kLse) {
        const float s2 = __shfl_xor_sync(0xffffffffu, r.se, o);
        merge_lse(r.mx, r.se, m2, s2, T);
      } else {
        const int a2 = __shfl_xor_sync(0xffffffffu, r.arg, o);
        argmax_merge(r.mx, r.arg, m2, a2);
      }
    }
    if (lane == 0) part[warp] = r;
  }
  __syncthreads();
  if ((int)threadIdx.x < nrows) {
    RowRed r = part[threadIdx.x * per];
    for (int i = 1; i < per; ++i) {
      const RowRed o = part[threadIdx.x * per + i];
      if constexpr (kLse) merge_lse(r.mx, r.se, o.mx, o.se, T);
      else argmax_merge(r.mx, r.arg, o.mx, o.arg);
    }
    out[threadIdx.x] = r;
  }
  __syncthreads();
}

// Draft tokens (argmax or Gumbel-max winner) and draft-row normalisers;
// or the prefill's first token and state initialisation.
__global__ void __launch_bounds__(256) select_kernel(const __grid_constant__ SelectArgs a) {
  pdl_wait();
  pdl_trigger();
  __shared__ RowRed sred[8];
  const float T = a.call->temp;
  const bool sample = a.call->sample != 0;
  int b, i = 0, m;
  if (a.mode == SEL_FIRST) {
    b = blockIdx.x;
    m = b;
  } else if (a.mode == SEL_DRAFT_SEQ) {
    b = blockIdx.x;
    i = a.seq_i;
    m = i == 0 ? a.seq_row0[b] + a.st.pend_cnt[b] - 1 : b;
  } else {
    b = blockIdx.x / a.K;
    i = blockIdx.x % a.K;
    m = a.mode == SEL_DRAFT ? a.seq_row0[b] + a.st.pend_cnt[b] - 1 + i : b * a.K + i;
  }
  const RowRed r = reduce_row(a.stats, a.stats_i, a.w_tiles, a.m_cap, m, T, sred);
  if (threadIdx.x != 0) return;
  const int tok = sample ? r.gi : r.arg;
  if (a.mode == SEL_FIRST) {
    a.out[b] = tok;
    const int kp = a.st.kmax + 1;
    a.st.n[b] = a.plen[b] + 1;
    a.st.pend_cnt[b] = 1;
    a.st.pend[b * kp] = tok;
    a.st.gen[b] = 1;
    a.st.max_new[b] = a.n_new;
    a.st.done[b] = a.n_new <= 1 ? 1 : 0;
    return;
  }
  a.st.dnorm[b * a.st.kmax + i] = make_float2(r.mx, r.se);
  if (a.mode == SEL_DRAFT || a.mode == SEL_DRAFT_SEQ || a.mode == SEL_DRAFT_GIVEN) {
    a.st.d[b * a.st.kmax + i] = tok;
    if (a.out) a.out[b * a.K + i] = tok;
  }
}

void launch_select(const SelectArgs& a, cudaStream_t s, bool pdl) {
  const int grid = (a.mode == SEL_FIRST || a.mode == SEL_DRAFT_SEQ) ? a.batch : a.batch * a.K;
  PARD_LAUNCH(select_kernel, grid, 256, 0, s, pdl, a);
}

// ---------------------------------------------------------------------------
// Commit / rollback of one sequence (a accepted candidates + one bonus).
// ---------------------------------------------------------------------------
__device__ void commit_seq(const AcceptArgs& a, int b, int acc, const int* emitted_tok) {
  const int K = a.K, kp = a.st.kmax + 1;
  if (a.st.done[b]) {
    if (a.accept_len) a.accept_len[b] = 0;
    if (a.n_emit) a.n_emit[b] = 0;
    for (int j = 0; j <= K; ++j) {
      if (a.emitted) a.emitted[b * (K + 1) + j] = -1;
      if (a.kv_slots) a.kv_slots[b * (K + 1) + j] = -1;
    }
    return;
  }
  const int n = a.st.n[b];
  const int room = a.st.max_new[b] - a.st.gen[b];
  const int take = acc + 1 < room ? acc + 1 : room;
  for (int j = 0; j <= K; ++j) {
    if (a.emitted) a.emitted[b * (K + 1) + j] = j < take ? emitted_tok[j] : -1;
    if (a.kv_slots) {
      int slot = -1;
      if (j <= acc) {
        const int pos = n - 1 + j;
        slot = a.page_table[(size_t)b * a.pt_ld + pos / a.page_size] * a.page_size + pos % a.page_size;
      }
      a.kv_slots[b * (K + 1) + j] = slot;
    }
  }
  for (int j = 0; j <= acc; ++j) a.st.pend[b * kp + j] = emitted_tok[j];
  a.st.pend_cnt[b] = acc + 1;
  a.st.n[b] = n + acc + 1;
  a.st.gen[b] += take;
  if (a.st.gen[b] >= a.st.max_new[b]) a.st.done[b] = 1;
  if (a.accept_len) a.accept_len[b] = acc;
  if (a.n_emit) a.n_emit[b] = take;
}

// Greedy: a = longest prefix with d_i == argmax y_i, bonus = argmax y_a.
__global__ void __launch_bounds__(32 * kRowWarps) accept_greedy_kernel(const __grid_constant__ AcceptArgs a) {
  pdl_wait();
  pdl_trigger();
  __shared__ RowRed s_part[kRowWarps], s_row[17];
  __shared__ int s_arg[17];
  const int b = blockIdx.x;
  reduce_rows<false>(a.stats, a.stats_i, a.w_tiles, a.m_cap, b * (a.K + 1), a.K + 1, nullptr, 0, 0, 0, 1.0f, s_part,
                     s_row);
  if ((int)threadIdx.x <= a.K) s_arg[threadIdx.x] = s_row[threadIdx.x].arg;
  __syncthreads();
  if (threadIdx.x != 0) return;
  int acc = 0;
  while (acc < a.K && a.st.d[b * a.st.kmax + acc] == s_arg[acc]) ++acc;
  // a candidate outside the vocabulary never equals an argmax (rejected); flag it
  for (int i = 0; i < a.K && a.status; ++i) {
    const int di = a.st.d[b * a.st.kmax + i];
    if (di < 0 || di >= a.vocab) set_status(a.status, ST_BAD_TOKEN);
  }
  int em[17];
  for (int j = 0; j < acc; ++j) em[j] = a.st.d[b * a.st.kmax + j];
  em[acc] = s_arg[acc];
  commit_seq(a, b, acc, em);
}

void launch_accept_greedy(const AcceptArgs& a, cudaStream_t s, bool pdl) {
  PARD_LAUNCH(accept_greedy_kernel, a.batch, 32 * kRowWarps, 0, s, pdl, a);
}

// Sampling, phase 1: row normalisers and the accept tests
// u_i * q_i(d_i) < p_i(d_i), p = softmax(y/T), q = softmax(z/T).
__global__ void __launch_bounds__(32 * kRowWarps) accept_test_kernel(const __grid_constant__ AcceptArgs a) {
  pdl_wait();
  pdl_trigger();
  __shared__ RowRed s_part[kRowWarps], s_row[kRowWarps];
  __shared__ float2 s_norm[17], s_dnorm[16];
  __shared__ int s_ok[16];  // candidate i's test: 1 accepted, 0 rejected, -1 outside the vocabulary
  const int b = blockIdx.x, tid = threadIdx.x;
  const float T = a.call.temp;
  // what the tests read besides the normalisers, requested before them
  int di = -1;
  float yv = 0.f, zv = 0.f;
  if (tid < a.K) {
    di = a.st.d[b * a.st.kmax + tid];
    if (di >= 0 && di < a.vocab) {
      yv = a.logits[((size_t)b * (a.K + 1) + tid) * a.vocab + di];
      zv = a.dlogits[((size_t)b * a.K + tid) * a.vocab + di];
    }
  }
  reduce_rows<true>(a.stats, a.stats_i, a.w_tiles, a.m_cap, b * (a.K + 1), a.K + 1, a.dstats, a.d_m_cap, b * a.K,
                    a.dstats ? a.K : 0, T, s_part, s_row);
  if (tid <= a.K) s_norm[tid] = make_float2(s_row[tid].mx, s_row[tid].se);
  if (tid < a.K) {
    const float2 yn = make_float2(s_row[tid].mx, s_row[tid].se);
    const float2 zn = a.dstats ? make_float2(s_row[a.K + 1 + tid].mx, s_row[a.K + 1 + tid].se)
                               : a.st.dnorm[b * a.st.kmax + tid];
    s_dnorm[tid] = zn;
    // a candidate outside the vocabulary has no probability: rejected
    int ok = -1;
    if (di >= 0 && di < a.vocab) {
      const float p = expf(yv / T - yn.x / T) / yn.y;
      const float q = expf(zv / T - zn.x / T) / zn.y;
      const float u = uniform01(philox_word(a.call.seed, STREAM_ACCEPT, a.call.step, (uint32_t)b, (uint32_t)tid, 0u));
      ok = u * q < p ? 1 : 0;
    }
    s_ok[tid] = ok;
  }
  __syncthreads();
  if (tid != 0) return;
  int j = 0;
  while (j < a.K && s_ok[j] == 1) ++j;
  if (j < a.K && s_ok[j] < 0 && a.status) set_status(a.status, ST_BAD_TOKEN);
  a.st.samp_a[b] = j;
  const float2 zn = j < a.K ? s_dnorm[j] : make_float2(0.f, 1.f);
  a.st.samp_norm[b] = make_float4(s_norm[j].x, s_norm[j].y, zn.x, zn.y);
}

// Sampling, phase 2: the bonus token by Gumbel-max over the vocabulary,
// from max(0, p_j - q_j) at the first rejection j, or from p_K; split over
// kResampleSplit blocks per sequence, the last one merges in block order
// and commits.
constexpr int kResampleThreads = 512;
// (value, index) maximum over the block, in s_v[0] and s_i[0]
__device__ __forceinline__ void block_argmax(float v, int i, float* s_v, int* s_i) {
  warp_argmax(v, i);
  __syncthreads();  // s_v and s_i may still be read
  if ((threadIdx.x & 31) == 0) { s_v[threadIdx.x >> 5] = v; s_i[threadIdx.x >> 5] = i; }
  __syncthreads();
  if (threadIdx.x < 32) {
    v = threadIdx.x < kResampleThreads / 32 ? s_v[threadIdx.x] : -INFINITY;
    i = threadIdx.x < kResampleThreads / 32 ? s_i[threadIdx.x] : INT_MAX;
    warp_argmax(v, i);
    if (threadIdx.x == 0) { s_v[0] = v; s_i[0] = i; }
  }
  __syncthreads();
}
__global__ void __launch_bounds__(kResampleThreads) resample_kernel(const __grid_constant__ AcceptArgs a) {
  pdl_wait();
  pdl_trigger();
  __shared__ float s_v[kResampleThreads / 32];
  __shared__ int s_i[kResampleThreads / 32];
  __shared__ int s_last;
  const int b = blockIdx.x / kResampleSplit, part = blockIdx.x % kResampleSplit;
  const float T = a.call.temp;
  const int j = a.st.samp_a[b];
  const float4 nm = a.st.samp_norm[b];
  const float* y = a.logits + ((size_t)b * (a.K + 1) + j) * a.vocab;
  const float* z = j < a.K ? a.dlogits + ((size_t)b * a.K + j) * a.vocab : nullptr;
  const int v0 = (int)((long)part * a.vocab / kResampleSplit), v1 = (int)((long)(part + 1) * a.vocab / kResampleSplit);
  float best = -INFINITY;
  int bi = INT_MAX;
  // A thread takes the four entries of one Philox block at a time.  An entry
  // whose noise cannot lift it over the warp's best so far is passed over
  // before the logarithms: its score beats `best` only if -log u < w exp(-best)
  // (w exp(-best) = exp(y/T - best) without a draft row), and -log u >= 1 - u.
  // The factor 1.0001 is far above the errors of the exponentials and of the
  // noise (1e-5 together), so the exact sum of an entry passed over is below
  // `best`; rounded, at whatever size y/T gives it, it is at most `best`, and
  // an equal score of a later entry does not win: the warp's best is of an
  // earlier round of the loop, whose indices are all lower.
  const uint64_t seed = a.call.seed;
  const uint32_t k0 = (uint32_t)seed, k1 = (uint32_t)(seed >> 32), step = (uint32_t)a.call.step;
  const float cy = nm.x / T, cz = nm.z / T;
  const bool unit = T == 1.f;  // no divisions
  for (int blk0 = v0 / 4; 4 * blk0 < v1; blk0 += blockDim.x) {
    const int blk = blk0 + threadIdx.x;
    float yv[4], zv[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int v = 4 * blk + e;
      const bool in = v >= v0 && v < v1;
      yv[e] = in ? y[v] : 0.f;
      zv[e] = in && z ? z[v] : 0.f;
    }
    const U4 pw = philox4x32_10(U4{(uint32_t)blk, (uint32_t)STREAM_BONUS << 16, (uint32_t)b, step}, k0, k1);
    const uint32_t wd[4] = {pw.x, pw.y, pw.z, pw.w};
    const float wbest = warp_max(best);
    const float inv_best = expf(-wbest);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int v = 4 * blk + e;
      if (v < v0 || v >= v1) continue;
      const float t = 1.0f - uniform_open01(wd[e]);  // exact
      if (z) {
        const float p = expf((unit ? yv[e] : yv[e] / T) - cy) / nm.y;
        const float q = expf((unit ? zv[e] : zv[e] / T) - cz) / nm.w;
        const float w = fmaxf(p - q, 0.f);
        if (w > 0.f && t > w * inv_best * 1.0001f) continue;
        argmax_merge(best, bi, w > 0.f ? logf(w) + gumbel(wd[e]) : -INFINITY, v);
      } else {
        const float x = unit ? yv[e] : yv[e] / T;
        if (t > expf(x - wbest) * 1.0001f) continue;
        argmax_merge(best, bi, x + gumbel(wd[e]), v);
      }
    }
  }
  block_argmax(best, bi, s_v, s_i);
  if (threadIdx.x == 0) {
    a.st.samp_part[b * kResampleSplit + part] = make_float2(s_v[0], __int_as_float(s_i[0]));
    __threadfence();
    const int old = atomicAdd(&a.st.samp_cnt[b], 1);
    s_last = old == kResampleSplit - 1;
  }
  __syncthreads();
  if (!s_last) return;
  __threadfence();
  if (threadIdx.x < 32) {
    // kResampleSplit partial draws, a lane each
    const float2 pv = __ldcg(&a.st.samp_part[b * kResampleSplit + threadIdx.x]);
    float gbest = pv.x;
    int gi = __float_as_int(pv.y);
    warp_argmax(gbest, gi);
    if (threadIdx.x == 0) {
      a.st.samp_cnt[b] = 0;
      s_i[0] = gi;
      s_v[0] = gbest;
    }
  }
  __syncthreads();
  if (s_v[0] == -INFINITY) {
    // max(0, p - q) vanished everywhere (p == q up to rounding): draw from p_j
    float bb = -INFINITY;
    int bj = INT_MAX;
    for (int v = threadIdx.x; v < a.vocab; v += blockDim.x) {
      const float g = gumbel(philox_word(a.call.seed, STREAM_BONUS, a.call.step, (uint32_t)b, 0u, (uint32_t)v));
      const float p = expf(y[v] / T - nm.x / T) / nm.y;
      argmax_merge(bb, bj, logf(p) + g, v);
    }
    block_argmax(bb, bj, s_v, s_i);
  }
  if (threadIdx.x != 0) return;
  int em[17];
  for (int k = 0; k < j; ++k) em[k] = a.st.d[b * a.st.kmax + k];
  em[j] = s_i[0];
  commit_seq(a, b, j, em);
}

void launch_accept_sample(const AcceptArgs& a, cudaStream_t s, bool pdl) {
  PARD_LAUNCH(accept_test_kernel, a.batch, 32 * kRowWarps, 0, s, pdl, a);
  static_assert(kResampleSplit == 32, "a lane per partial draw");
  PARD_LAUNCH(resample_kernel, a.batch * kResampleSplit, kResampleThreads, 0, s, true, a);
}

// Tile statistics of given logits rows (same layout as the LM-head
// epilogue): per 128-entry tile the max and argmax, the sum of exp((x - max)/T)
// and, when gumbel_stream >= 0 and the call samples, the Gumbel-max winner of
// the tile for row m = b * rows_per_seq + i (Philox row i of sequence b): the
// draw that the LM-head epilogue makes for a draft row, by scoring every entry
// exactly (the epilogue ranks roughly first).
__global__ void __launch_bounds__(128) row_stats_kernel(const float* logits, int vocab, int m_cap, const CallArgs* call,
                                                        int gumbel_stream, int rows_per_seq, float4* stats,
                                                        int2* stats_i) {
  pdl_wait();
  const int t = blockIdx.x, m = blockIdx.y;
  const int v = t * 128 + threadIdx.x;
  const float T = call->temp;
  const bool valid = v < vocab;
  const bool gumb = gumbel_stream >= 0 && call->sample != 0;
  const float x = valid ? logits[(size_t)m * vocab + v] : -INFINITY;
  __shared__ float s_v[4], s_g[4];
  __shared__ int s_i[4], s_gi[4];
  __shared__ float s_m;
  float mv = x;
  int mi = valid ? v : INT_MAX;
  warp_argmax(mv, mi);
  float gv = -INFINITY;
  int gi = INT_MAX;
  if (gumb && valid) {
    gv = gumbel_score(x, T, call->seed, (uint32_t)gumbel_stream, call->step, (uint32_t)(m / rows_per_seq),
                      (uint32_t)(m % rows_per_seq), (uint32_t)v);
    gi = v;
  }
  if (gumb) warp_argmax(gv, gi);
  const int w = threadIdx.x >> 5;
  if ((threadIdx.x & 31) == 0) { s_v[w] = mv; s_i[w] = mi; s_g[w] = gv; s_gi[w] = gi; }
  __syncthreads();
  if (threadIdx.x == 0) {
    float bv = s_v[0];
    int bi = s_i[0];
    for (int k = 1; k < 4; ++k) argmax_merge(bv, bi, s_v[k], s_i[k]);
    float bg = s_g[0];
    int bgi = s_gi[0];
    for (int k = 1; k < 4; ++k) argmax_merge(bg, bgi, s_g[k], s_gi[k]);
    s_m = bv;
    s_i[0] = bi;
    s_g[0] = bg;
    s_gi[0] = bgi;
  }
  __syncthreads();
  const float mxv = s_m;
  const int arg = s_i[0];
  float e = valid ? expf(x / T - mxv / T) : 0.f;
  e = warp_sum(e);
  __syncthreads();
  if ((threadIdx.x & 31) == 0) s_v[w] = e;
  __syncthreads();
  if (threadIdx.x == 0) {
    stats[(size_t)t * m_cap + m] =
        make_float4(mxv, ((s_v[0] + s_v[1]) + s_v[2]) + s_v[3], gumb ? s_g[0] : -INFINITY, 0.f);
    stats_i[(size_t)t * m_cap + m] = make_int2(arg, gumb ? s_gi[0] : -1);
  }
}

void launch_row_stats(const float* logits, int rows, int vocab, int w_tiles, int m_cap, const CallArgs* call,
                      int gumbel_stream, int rows_per_seq, float4* stats, int2* stats_i, cudaStream_t s) {
  PARD_LAUNCH(row_stats_kernel, dim3(w_tiles, rows), 128, 0, s, false, logits, vocab, m_cap, call, gumbel_stream,
              rows_per_seq > 0 ? rows_per_seq : 1, stats, stats_i);
}

// Statistics of given logits rows in tiles of kGivenTile entries (the max, and
// the argmax or, when sampling, the sum of exp((x - max)/T)): a warp takes a
// tile, four tiles a block, the target's rows first; block (0, 0) also resets
// the acceptance state.  Every logit is read once, 16 loads of 16 bytes in
// flight a lane, and no block reduction follows (batch 16, K = 6: 107 MB).
// The whole sampled acceptance takes 45 us, 231 us with one 512-byte
// tile a block, three block reductions each and one row after the other after
// it; the greedy one at batch 1, K = 8: 9.5 us, 51.7 before.
template <bool kSample>  // greedy acceptance reads the argmax only, sampled the maximum and the sum
__global__ void __launch_bounds__(128) given_stats_kernel(const __grid_constant__ GivenArgs a) {
  pdl_trigger();
  const int tid = threadIdx.x, lane = tid & 31, t = blockIdx.x * 4 + (tid >> 5);
  const bool target = (int)blockIdx.y < a.rows_t;
  const int m = target ? blockIdx.y : blockIdx.y - a.rows_t;
  const float* row = (target ? a.y : a.z) + (size_t)m * a.vocab;
  if (blockIdx.x == 0 && blockIdx.y == 0) {
    if (tid < a.batch) {
      a.st.n[tid] = 1;
      a.st.pend_cnt[tid] = 1;
      a.st.gen[tid] = 0;
      a.st.max_new[tid] = 1 << 30;
      a.st.done[tid] = 0;
      a.st.samp_cnt[tid] = 0;
    }
    for (int i = tid; i < a.batch * a.K; i += 128) a.st.d[i] = a.d[i];
  }
  if (t >= a.tiles) return;
  // lane's entries: 16 float4s, 512 contiguous bytes a warp and load
  float x[64];
  const int v0 = t * kGivenTile + lane * 4;
#pragma unroll
  for (int q = 0; q < 16; ++q) {
    const int v = v0 + q * 128;
    float4 f = make_float4(-INFINITY, -INFINITY, -INFINITY, -INFINITY);
    if (v < a.vocab) {  // vocab is a multiple of 8: all four entries or none
      if (a.vec) f = __ldcs(reinterpret_cast<const float4*>(row + v));
      else f = make_float4(row[v], row[v + 1], row[v + 2], row[v + 3]);
    }
    x[4 * q] = f.x; x[4 * q + 1] = f.y; x[4 * q + 2] = f.z; x[4 * q + 3] = f.w;
  }
  float mv = -INFINITY, se = 0.f;
  int mi = INT_MAX;
#pragma unroll
  for (int i = 0; i < 64; ++i) {
    const int v = v0 + (i >> 2) * 128 + (i & 3);
    if (kSample) mv = fmaxf(mv, x[i]);  // past the vocabulary: -infinity
    else if (v < a.vocab) argmax_merge(mv, mi, x[i], v);
  }
  const float T = a.call.temp;
  if (kSample) {
    mv = warp_max(mv);
    if (mv != -INFINITY) {  // past the vocabulary: exp(-infinity) = 0
      if (T == 1.f) {       // no divisions
#pragma unroll
        for (int i = 0; i < 64; ++i) se += expf(x[i] - mv);
      } else {
        const float c = mv / T;
#pragma unroll
        for (int i = 0; i < 64; ++i) se += expf(x[i] / T - c);
      }
    }
    se = warp_sum(se);
  } else {
    warp_argmax(mv, mi);
  }
  if (lane == 0) {
    const size_t at = (size_t)t * (target ? a.m_cap_t : a.m_cap_d) + m;
    (target ? a.stats_t : a.stats_d)[at] = make_float4(mv, se, -INFINITY, 0.f);
    if (!kSample) a.stats_it[at] = make_int2(mi, -1);
  }
}

void launch_given_stats(const GivenArgs& a, cudaStream_t s) {
  const dim3 grid((a.tiles + 3) / 4, a.rows_t + a.rows_d);
  if (a.sample) PARD_LAUNCH(given_stats_kernel<true>, grid, 128, 0, s, false, a);
  else PARD_LAUNCH(given_stats_kernel<false>, grid, 128, 0, s, false, a);
}

__global__ void set_call_kernel(CallArgs* dst, CallArgs v) {
  pdl_wait();
  pdl_trigger();
  *dst = v;
}
void launch_set_call(CallArgs* dst, CallArgs v, cudaStream_t s, bool pdl) {
  PARD_LAUNCH(set_call_kernel, 1, 1, 0, s, pdl, dst, v);
}

__global__ void read_kv_kernel(const __nv_bfloat16* kc, const __nv_bfloat16* vc, const int* pt, const int* pos, int n,
                               int hkv, int hd, int ps, __nv_bfloat16* ok, __nv_bfloat16* ov) {
  const int i = blockIdx.x;
  if (i >= n) return;
  const int p = pos[i];
  const int page = pt[p / ps];
  for (int e = threadIdx.x; e < hkv * hd; e += blockDim.x) {
    const int h = e / hd, c = e % hd;
    const size_t off = (((size_t)page * hkv + h) * ps + p % ps) * hd + c;
    ok[(size_t)i * hkv * hd + e] = kc[off];
    ov[(size_t)i * hkv * hd + e] = vc[off];
  }
}
void launch_read_kv(const __nv_bfloat16* kc, const __nv_bfloat16* vc, const int* page_table_row, const int* pos, int n,
                    int hkv, int hd, int page_size, __nv_bfloat16* ok, __nv_bfloat16* ov, cudaStream_t s) {
  PARD_LAUNCH(read_kv_kernel, n, 128, 0, s, false, kc, vc, page_table_row, pos, n, hkv, hd, page_size, ok, ov);
}

}  // namespace pard
