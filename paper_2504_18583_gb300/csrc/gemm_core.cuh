// Device code of the weight-streaming GEMMs (gemm.cu, gemm_wide.cu): the fused
// epilogues, and the narrow one's tile configuration and split-K finish.
#pragma once

#include <climits>

#include "common.cuh"
#include "internal.h"

namespace pard {

template <int TT>
struct GemmCfg {
  static constexpr int kABytes = kTileN * 128;       // 128 rows x 64 bf16
  static constexpr int kBBytes = 2 * TT * 128;       // 2*TT rows x 64 bf16
  static constexpr int kStageBytes = kABytes + kBBytes;
  // Ring capacity (a launch may use fewer).  At the 16-token tile the CTA
  // (about 106 KB of shared memory, at most 168 registers a thread) leaves
  // room on its SM for one CTA of the next launch, which then starts, fills
  // its ring and reaches its PDL wait while this one finishes.  The 64-token
  // tile runs one CTA per SM and takes a deeper ring (~200 KB) instead: with 4
  // stages it kept too few weight bytes in flight per SM.  (More than 64 rows:
  // gemm_wide.cu.)
  static constexpr int kStages = TT <= 16 ? 5 : 6;
  static constexpr int kAccCols = 2 * TT;
  static constexpr int kNumAcc = (2 * kAccCols <= 512) ? 2 : 1;
  static constexpr int kTmemCols = kNumAcc * kAccCols <= 32 ? 32 : kNumAcc * kAccCols <= 64 ? 64
                                   : kNumAcc * kAccCols <= 128 ? 128 : kNumAcc * kAccCols <= 256 ? 256 : 512;
  static constexpr int kChunks = TT / kEpiTok;
  // scratch after the stage ring
  // full, empty, accf x2, acce x2, drain, fix-up; rounded to 16 bytes
  static constexpr int kBarBytes = (8 * (2 * kStages + 6) + 15) / 16 * 16;
  static constexpr int kMiscBytes = 64;
  static constexpr int kScratchFloats = TT + kEpiTok * kTileN + 3 * kEpiTok;
  static constexpr int kSmem = 1024 + kStages * kStageBytes + kBarBytes + kMiscBytes + 4 * kScratchFloats;
};

// barrier of one epilogue group of 128 threads
__device__ __forceinline__ void epi_bar(int id = 1) { asm volatile("bar.sync %0, 128;" ::"r"(id) : "memory"); }
// epi_bar that also returns whether any of the 128 threads passed v != 0, so
// that all of them take the same branch after it
__device__ __forceinline__ bool epi_bar_any(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.or.pred q, 1, 128, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v)
      : "memory");
  return r != 0;
}

// The split of U units over G CTAs: 32-bit (the host checks that U G fits; a
// 64-bit division costs some hundred clocks, and each CTA has several on its
// way to the first copy and again to its last store).
__device__ __forceinline__ int owner_of(int u, int U, int G) { return ((u + 1) * G + U - 1) / U - 1; }
__device__ __forceinline__ int range_start(int c, int U, int G) { return c * U / G; }

__device__ __forceinline__ int seg_of(const GemmArgs& a, int w_tile) {
  int s = 0;
#pragma unroll
  for (int i = 1; i < kMaxSeg; ++i)
    if (i < a.nseg && w_tile >= a.seg_tile0[i]) s = i;
  return s;
}

struct EpiSmem {
  float* rs;     // [TT]   RMS row scale
  float* xch;    // [16][128] the chunk's accumulator, exchanged to row-major (16-byte aligned)
  int* ri;       // [3][16] per-row facts of the chunk, loaded once by 16 threads
  int bar;       // named barrier of the 128 threads
};

// Token j's value in the 32 accumulator columns of a 16-token chunk whose hi
// and lo parts have columns of their own (8 tokens: 8 hi, then 8 lo columns)
__device__ __forceinline__ float hilo(const uint32_t (&r)[32], int j) {
  return __uint_as_float(r[(j >> 3) * 16 + (j & 7)]) + __uint_as_float(r[(j >> 3) * 16 + 8 + (j & 7)]);
}

// Carves the epilogue scratch (GemmCfg<TT>::kScratchFloats floats) at p.
template <int TT>
__device__ __forceinline__ EpiSmem carve_epi(float* p) {
  EpiSmem S;
  S.rs = p;
  S.xch = S.rs + TT;
  S.ri = reinterpret_cast<int*>(S.xch + kEpiTok * kTileN);
  S.bar = 1;
  return S;
}

// Row-major phase of the epilogues.  After the accumulator columns of a
// 16-token chunk are exchanged through S.xch, thread et handles token
// jl = et / 8 and the tile columns 32 i + 4 l8 .. + 3 (l8 = et % 8, i = 0..3):
// the eight threads of a token read and write 128 contiguous bytes at a time
// (with 16 consecutive columns a thread every access was a 16-byte piece of
// another 64 bytes: 2.1k clocks a chunk for the residual epilogue, most of
// them in the stores), the exchange reads are free of bank conflicts, and
// RoPE's partner columns and a gate's up column are the thread's own.
__device__ __forceinline__ int epi_col(int i, int l8) { return 32 * i + 4 * l8; }

// Loads of one 16-token chunk's epilogue that do not depend on the tile's
// result: the residual and norm gains (O / down), the row's position, KV page
// and RoPE factors (QKV), the rows' output facts (LM head).  Taken before the
// split-K arrival, so that the CTA that finishes a tile has them in hand.
struct EpiPre {
  float4 f[4];    // O / down: h; QKV: (cos, sin) pairs of columns epi_col(i) mod (hd / 2), i = 0, 1, two float4 each
  uint2 g[4];     // O / down: norm gains
  int pos, page;  // QKV: position (-1 invalid) and KV page (-1 none) of the thread's token
  int ri[3];      // LM head, threads et < 16: logits row, Gumbel index, sequence of token et
};

template <int MODE>
__device__ __forceinline__ EpiPre epi_pre(const GemmArgs& a, int w_tile, int tok0, int et, int M) {
  EpiPre p;
  p.pos = -1;
  p.page = -1;
  const int jl = et >> 3, l8 = et & 7;
  const int mr = tok0 + jl;
  if constexpr (MODE == MODE_RESID) {
    if (mr < M) {
      const int n0 = w_tile * kTileN;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        // L2 loads: h was written by the previous kernel's CTAs
        p.f[i] = __ldcg(reinterpret_cast<const float4*>(a.h + (size_t)mr * a.h_ld + n0 + epi_col(i, l8)));
        p.g[i] = *reinterpret_cast<const uint2*>(a.g_next + n0 + epi_col(i, l8));
      }
    }
  } else if constexpr (MODE == MODE_QKV) {
    const int seg = seg_of(a, w_tile);
    if (mr < M) {
      const int pos = a.row_pos[mr];
      const bool pv = pos >= 0 && pos / a.page_size < a.pt_ld;
      if (!pv && l8 == 0) set_status(a.status, ST_BAD_POS);
      if (pv) {
        p.pos = pos;
        if (seg > 0) {
          const int page = a.page_table[(size_t)a.row_seq[mr] * a.pt_ld + pos / a.page_size];
          if (page >= 0 && page < a.n_pages) p.page = page;
          else if (l8 == 0) set_status(a.status, ST_BAD_PAGE);
        }
        if (seg < 2) {
          const int half = a.hd >> 1;  // 64: columns i and i + 2 are partners; 32: i and i ^ 1, the same factors twice
          const float4* cs = reinterpret_cast<const float4*>(a.rope + (size_t)pos * half);
#pragma unroll
          for (int i = 0; i < 2; ++i)
#pragma unroll
            for (int k = 0; k < 2; ++k) p.f[2 * i + k] = cs[(epi_col(i, l8) % half) / 2 + k];
        }
      }
    }
  } else if constexpr (MODE == MODE_LOGITS) {
    if (et < kEpiTok) {
      const int m = tok0 + et;
      const bool in = m < M;
      const bool sample = a.call->sample != 0 && a.row_gi != nullptr;
      p.ri[0] = in ? (a.row_out ? a.row_out[m] : m) : -1;
      p.ri[1] = (in && sample) ? a.row_gi[m] : -1;
      p.ri[2] = (in && sample) ? a.row_seq[m] : 0;
    }
  }
  return p;
}

// -log(u) for u = 1 - t to within 1e-3 of its value (t exact: 1 - u has no
// rounding for 24-bit u), to rank Gumbel scores before the exact ones.
__device__ __forceinline__ float neg_log_rough(float t) {
  const float series = t * (1.f + t * (0.5f + t * (0.33333334f + t * (0.25f + t * 0.2f))));
  return t < 0.25f ? series : -__logf(1.f - t);
}

// One 16-token chunk of the epilogue for the thread holding weight row fr;
// pre holds the chunk's result-independent loads (epi_pre).
template <int MODE>
__device__ __forceinline__ void epi_chunk(const GemmArgs& a, float (&v)[kEpiTok], int w_tile, int tok0, int rs_off, int fr,
                          int et, int M, const EpiSmem& S, const EpiPre& pre) {
  if constexpr (MODE != MODE_RESID) {  // the RMS-normalised inputs
#pragma unroll
    for (int j = 0; j < kEpiTok; ++j) v[j] *= S.rs[rs_off + j];
  }
  if constexpr (MODE == MODE_LOGITS) {
    // row facts of the chunk: logits row (-1: none), Gumbel index (-1: none), sequence
    if (et < kEpiTok) {
      S.ri[et] = pre.ri[0];
      S.ri[kEpiTok + et] = pre.ri[1];
      S.ri[2 * kEpiTok + et] = pre.ri[2];
    }
  }
#pragma unroll
  for (int j = 0; j < kEpiTok; ++j) S.xch[j * kTileN + fr] = v[j];
  epi_bar(S.bar);
  const int jl = et >> 3, l8 = et & 7;
  const int mr = tok0 + jl;
  float4 x[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) x[i] = *reinterpret_cast<const float4*>(S.xch + jl * kTileN + epi_col(i, l8));
  if constexpr (MODE == MODE_RESID) {
    const int n0 = w_tile * kTileN;
    float sq = 0.f;
    if (mr < M) {
      float* hp = a.h + (size_t)mr * a.h_ld + n0;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        const float4 h = make_float4(pre.f[i].x + x[i].x, pre.f[i].y + x[i].y, pre.f[i].z + x[i].z, pre.f[i].w + x[i].w);
        *reinterpret_cast<float4*>(hp + epi_col(i, l8)) = h;
        const float2 g0 = make_float2(__uint_as_float(pre.g[i].x << 16), __uint_as_float(pre.g[i].x & 0xffff0000u));
        const float2 g1 = make_float2(__uint_as_float(pre.g[i].y << 16), __uint_as_float(pre.g[i].y & 0xffff0000u));
        store_pair4(a.x_next, mr, n0 + epi_col(i, l8), a.x_rows,
                    make_float4(h.x * g0.x, h.y * g0.y, h.z * g1.x, h.w * g1.y));
        sq += h.x * h.x + h.y * h.y + h.z * h.z + h.w * h.w;
      }
    }
    // the tile's sum of squares of this token: its 8 threads are 8 adjacent lanes
    sq += __shfl_xor_sync(0xffffffffu, sq, 1);
    sq += __shfl_xor_sync(0xffffffffu, sq, 2);
    sq += __shfl_xor_sync(0xffffffffu, sq, 4);
    if (l8 == 0 && mr < M) a.ssq_out[(size_t)w_tile * a.m_cap + mr] = sq;
  } else if constexpr (MODE == MODE_QKV) {
    const int seg = seg_of(a, w_tile);
    const int n0 = (w_tile - a.seg_tile0[seg]) * kTileN;  // first column within the segment
    if (mr < M && pre.pos >= 0) {
      if (seg < 2) {
        // rotate-half RoPE: the partner half of a head is in the same 128-row tile
        auto rot = [](float4& lo, float4& hi, const float4& c0, const float4& c1) {
          const float4 l = lo, h = hi;
          lo = make_float4(l.x * c0.x - h.x * c0.y, l.y * c0.z - h.y * c0.w, l.z * c1.x - h.z * c1.y,
                           l.w * c1.z - h.w * c1.w);
          hi = make_float4(l.x * c0.y + h.x * c0.x, l.y * c0.w + h.y * c0.z, l.z * c1.y + h.z * c1.x,
                           l.w * c1.w + h.w * c1.z);
        };
        if (a.hd == 128) {
          rot(x[0], x[2], pre.f[0], pre.f[1]);
          rot(x[1], x[3], pre.f[2], pre.f[3]);
        } else {
          rot(x[0], x[1], pre.f[0], pre.f[1]);
          rot(x[2], x[3], pre.f[0], pre.f[1]);
        }
      }
      if (seg == 0) {
        float* qp = a.q_out + (size_t)mr * a.q_ld + n0;
#pragma unroll
        for (int i = 0; i < 4; ++i) *reinterpret_cast<float4*>(qp + epi_col(i, l8)) = x[i];
      } else if (pre.page >= 0) {
        __nv_bfloat16* base = seg == 1 ? a.kcache : a.vcache;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const int n = n0 + epi_col(i, l8);
          __nv_bfloat16* dst =
              base + (((size_t)pre.page * a.hkv + n / a.hd) * a.page_size + pre.pos % a.page_size) * a.hd + n % a.hd;
          uint2 w;
          w.x = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x[i].x)) |
                ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x[i].y)) << 16);
          w.y = (uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x[i].z)) |
                ((uint32_t)__bfloat16_as_ushort(__float2bfloat16_rn(x[i].w)) << 16);
          *reinterpret_cast<uint2*>(dst) = w;
        }
      }
    }
  } else if constexpr (MODE == MODE_SWIGLU) {
    // the tile's gate rows are columns 0..63 of the exchange, its up rows 64..127
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const int n = w_tile * 64 + epi_col(i, l8);
      if (mr < M && n < a.seg_rows[0])  // a multiple of 8: the four columns or none
        store_pair4(a.x_next, mr, n, a.x_rows,
                    make_float4(silu(x[i].x) * x[i + 2].x, silu(x[i].y) * x[i + 2].y, silu(x[i].z) * x[i + 2].z,
                                silu(x[i].w) * x[i + 2].w));
    }
  } else {  // MODE_LOGITS
    const float T = a.call->temp;
    const bool sample = a.call->sample != 0 && a.row_gi != nullptr;
    const int n0 = w_tile * kTileN;
    const int orow = S.ri[jl];
    float z[16];
    bool in[4];  // the vocabulary is a multiple of 8: four entries or none
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      z[4 * i] = x[i].x; z[4 * i + 1] = x[i].y; z[4 * i + 2] = x[i].z; z[4 * i + 3] = x[i].w;
      in[i] = n0 + epi_col(i, l8) < a.vocab;
    }
    if (a.logits && orow >= 0 && mr < M) {
      float* lp = a.logits + (size_t)orow * a.vocab + n0;
#pragma unroll
      for (int i = 0; i < 4; ++i)
        if (in[i]) *reinterpret_cast<float4*>(lp + epi_col(i, l8)) = x[i];
      if (a.logits_out) {  // the caller's copy (a copy afterwards reads and writes the rows once more)
        lp = a.logits_out + (size_t)orow * a.vocab + n0;
        const bool vec = (reinterpret_cast<uintptr_t>(a.logits_out) & 15) == 0;
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          float* q = lp + epi_col(i, l8);
          if (in[i] && vec) *reinterpret_cast<float4*>(q) = x[i];
          else if (in[i]) { q[0] = x[i].x; q[1] = x[i].y; q[2] = x[i].z; q[3] = x[i].w; }
        }
      }
    }
    // tile max and argmax (lowest index on ties) of token jl
    float mv = -INFINITY;
    int mi = INT_MAX;
#pragma unroll
    for (int k = 0; k < 16; ++k)
      if (in[k >> 2]) argmax_merge(mv, mi, z[k], n0 + epi_col(k >> 2, l8) + (k & 3));
#pragma unroll
    for (int o = 4; o > 0; o >>= 1) {
      const float v2 = __shfl_xor_sync(0xffffffffu, mv, o);
      const int i2 = __shfl_xor_sync(0xffffffffu, mi, o);
      argmax_merge(mv, mi, v2, i2);
    }
    // sum of exp((x - max) / T) over the tile; e: the single terms
    float e[16], se = 0.f;
    if (T == 1.f) {
#pragma unroll
      for (int k = 0; k < 16; ++k) e[k] = in[k >> 2] ? expf(z[k] - mv) : 0.f;
    } else {
      const float c = mv / T;
#pragma unroll
      for (int k = 0; k < 16; ++k) e[k] = in[k >> 2] ? expf(z[k] / T - c) : 0.f;
    }
#pragma unroll
    for (int k = 0; k < 16; ++k) se += e[k];
    se += __shfl_xor_sync(0xffffffffu, se, 4);
    se += __shfl_xor_sync(0xffffffffu, se, 2);
    se += __shfl_xor_sync(0xffffffffu, se, 1);
    // Gumbel-max draw of the tile (sampling draft rows only): the score
    // x / T - log(-log u) orders entries as exp(x / T) / -log u does, so a
    // rough quotient finds the few entries within its error of the tile's
    // best, and only those get the exact score.  (A full Philox block and two
    // logarithms for every entry: 374 us for the 96 rows of a batch-16 draft.)
    float gv = -INFINITY;
    int gi = INT_MAX;
    if (sample) {
      const int ri = mr < M ? S.ri[kEpiTok + jl] : -1;
      const uint32_t sq = (uint32_t)S.ri[2 * kEpiTok + jl];
      float rmax = 0.f;
      if (ri >= 0) {
#pragma unroll
        for (int i = 0; i < 4; ++i) {
          const uint32_t v0 = (uint32_t)(n0 + epi_col(i, l8));
          const U4 w = philox4x32_10(
              U4{v0 >> 2, ((uint32_t)(a.gumbel_stream & 0xFFFF) << 16) | ((uint32_t)ri & 0xFFFFu), sq, (uint32_t)a.call->step},
              (uint32_t)a.call->seed, (uint32_t)(a.call->seed >> 32));
          const uint32_t wd[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            e[4 * i + k] = __fdividef(e[4 * i + k], neg_log_rough(1.0f - uniform_open01(wd[k])));
            rmax = fmaxf(rmax, e[4 * i + k]);
          }
        }
      }
      rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, 4));
      rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, 2));
      rmax = fmaxf(rmax, __shfl_xor_sync(0xffffffffu, rmax, 1));
      if (ri >= 0) {
        // Left out: entries whose score is below the best by more than the
        // rough quotients' errors (1e-3 each) and an ulp of the score, which
        // is rounded at the size of x / T (2^-23 of it): two scores that round
        // to the same value are both in, so that the lower index wins.
        const float least = rmax * (0.99f - 2.4e-7f * fabsf(T == 1.f ? mv : mv / T));
#pragma unroll
        for (int k = 0; k < 16; ++k)
          if (in[k >> 2] && !(e[k] < least)) {  // NaN too
            const int n = n0 + epi_col(k >> 2, l8) + (k & 3);
            argmax_merge(gv, gi, gumbel_score(z[k], T, a.call->seed, (uint32_t)a.gumbel_stream, a.call->step, sq,
                                              (uint32_t)ri, (uint32_t)n), n);
          }
      }
#pragma unroll
      for (int o = 4; o > 0; o >>= 1) {
        const float v2 = __shfl_xor_sync(0xffffffffu, gv, o);
        const int i2 = __shfl_xor_sync(0xffffffffu, gi, o);
        argmax_merge(gv, gi, v2, i2);
      }
    }
    if (l8 == 0 && mr < M) {
      const size_t o = (size_t)w_tile * a.m_cap + mr;
      a.stats[o] = make_float4(mv, se, sample ? gv : -INFINITY, 0.f);
      a.stats_i[o] = make_int2(mi, sample ? gi : -1);
    }
  }
  epi_bar(S.bar);  // S.xch and the row facts are rewritten by the next chunk
}

// Bounded wait until every bit of `all` is set in *p, with acquire semantics
// on success.
__device__ __forceinline__ bool wait_mask(const unsigned long long* p, unsigned long long all, volatile int* abort) {
  if ((ld_acquire_u64(p) & all) == all) return true;
  const unsigned long long t0 = globaltimer();
  while (true) {
    if ((ld_acquire_u64(p) & all) == all) return true;
    if (*abort) return false;
    if (globaltimer() - t0 > kWaitLimitNs) return false;
  }
}
// bits of contributors 1..n of a tile (bit k - 1: the k-th after the finisher)
__device__ __forceinline__ unsigned long long contrib_bits(int n) { return n >= 64 ? ~0ull : ((1ull << n) - 1); }
// 4-token groups of a 16-token chunk that hold some of the pass's M rows: a
// partial tile stores and copies only those ([chunk][j4][row] layout)
__device__ __forceinline__ int chunk_groups(int M, int tok0) { return min(4, max(0, (M - tok0 + 3) / 4)); }

// Split-K with a designated finisher (per-phase kernel).  The first CTA of a
// tile in CTA order, cf, finishes it.  Its share of the tile is the last
// segment of its range (the tile starts inside the range and runs past its
// end), so when its epilogue gets there every MMA of the CTA has completed and
// the stage ring is idle.  The other contributors move on without a round
// trip: contributor k (the k-th CTA after cf) stores its partial and sets
// bit k - 1 of the tile's arrival mask with one release OR; cf copies each
// partial into the ring as soon as its bit is seen (so the copies of early
// contributors overlap the wait for late ones) and adds them to its own in
// CTA order (deterministic).  The contributors' ranges begin inside the tile,
// so their partials are in the first of their two slots.  With many chunks
// (wide tiles) the copies go in rounds of chunks once every bit is set.
// pre0: epi_pre of the segment's first chunk, taken by the caller before the
// accumulator was ready; only read for a whole tile or by cf.
// ring/ring_bytes: the stage ring; fx: an mbarrier whose phase r is round r
// of the one split tile a CTA finishes; fx_armed: 1 + the round whose copies
// may be in flight (0: none).  Partials hold only the 4-token groups with
// output rows (chunk_groups).  The arrival masks live in a.counters (64-bit
// words, tile t at word t; the host keeps every tile's contributors at 64 or
// fewer) and are cleared by the finisher.
template <int TT, int MODE>
__device__ bool epi_segment_owned(const GemmArgs& a, int t, int ub, int ue, int u0, int U, int G, int c,
                                  uint32_t tbase, int fr, int et, int M, const EpiSmem& S,
                                  const EpiPre& pre0, float* ring, uint32_t ring_bytes, uint64_t* fx,
                                  volatile int* fx_armed, volatile int* abort_flag, int* bcast) {
  using C = GemmCfg<TT>;
  constexpr int kTileF = kTileN * TT;  // floats of one partial tile
  // 16-token chunks holding at least one of the pass's M rows; the others are
  // neither finished nor exchanged (their rows are not outputs)
  const int nch = max(0, min(C::kChunks, (M + kEpiTok - 1) / kEpiTok));
  const int kChF = kTileN * kEpiTok;   // floats of one chunk of a partial tile
  if (ub == t * a.kc && ue == (t + 1) * a.kc) {
    EpiPre pre = pre0;  // one chunk's loads live at a time
#pragma unroll 1
    for (int ch = 0; ch < nch; ++ch) {
      if (ch > 0) pre = epi_pre<MODE>(a, t, ch * kEpiTok, et, M);
      uint32_t r[32];
      tmem_ld32(tbase + ch * 32, r);
      float v[kEpiTok];
#pragma unroll
      for (int j = 0; j < kEpiTok; ++j) v[j] = hilo(r, j);
      epi_chunk<MODE>(a, v, t, ch * kEpiTok, ch * kEpiTok, fr, et, M, S, pre);
    }
    return true;
  }
  const int cf = owner_of(t * a.kc, U, G), cl = owner_of((t + 1) * a.kc - 1, U, G);
  unsigned long long* mask = reinterpret_cast<unsigned long long*>(a.counters) + t;
  if (c != cf) {
    const int slot = (ub == u0) ? 0 : 1;
    float* mine = a.partials + ((size_t)c * 2 + slot) * kTileF;
#pragma unroll 1
    for (int ch = 0; ch < nch; ++ch) {
      uint32_t r[32];
      tmem_ld32(tbase + ch * 32, r);
      const int ng = chunk_groups(M, ch * kEpiTok);
      // [chunk][j4][row] float4s: a warp's accesses are 512 contiguous bytes
      float4* dst = reinterpret_cast<float4*>(mine + (size_t)ch * kTileN * kEpiTok) + fr;
#pragma unroll
      for (int j4 = 0; j4 < 4; ++j4)
        if (j4 < ng)
          dst[j4 * kTileN] =
              make_float4(hilo(r, 4 * j4), hilo(r, 4 * j4 + 1), hilo(r, 4 * j4 + 2), hilo(r, 4 * j4 + 3));
    }
    // the barrier orders every thread's partial before the one release OR
    // (cumulative)
    epi_bar();
    if (et == 0) red_release_or64(mask, 1ull << (c - cf - 1));
    return true;
  }
  if constexpr (C::kChunks == 1) {
    // 16-token tile: one chunk, so one staging round (the partials of up to
    // ring_bytes / 8 KB contributors) or direct loads
    const int n_other = cl - cf;
    // bytes copied of one contributor: the 4-token groups of its chunk with output rows
    const uint32_t part_bytes = nch > 0 ? (uint32_t)chunk_groups(M, 0) * kTileN * 16 : 0u;
    const bool staged = nch > 0 && (uint32_t)n_other * kChF * 4 <= ring_bytes;
    if (et == 0) {
      const unsigned long long all = contrib_bits(n_other);
      bool ok = true;
      if (staged) {
        *fx_armed = 1;
        mbar_arrive_expect_tx(fx, (uint32_t)n_other * part_bytes);
        // copy each contributor's partial as soon as its bit is seen
        unsigned long long seen = 0;
        const unsigned long long t0 = globaltimer();
        while (seen != all) {
          const unsigned long long m = ld_acquire_u64(mask) & all;
          unsigned long long nw = m & ~seen;
          if (nw) {
            // the partials were written through the generic proxy; the copies
            // read them through the async proxy
            fence_proxy_async();
            while (nw) {
              const int k = __ffsll((long long)nw) - 1;
              nw &= nw - 1;
              const int cc = cf + 1 + k;
              bulk_load(ring + (size_t)k * kChF, a.partials + ((size_t)cc * 2) * kTileF, part_bytes, fx);
            }
            seen = m;
          } else if (*abort_flag || globaltimer() - t0 > kWaitLimitNs) {
            ok = false;
            break;
          }
        }
      } else {
        ok = wait_mask(mask, all, abort_flag);
      }
      if (!ok) set_status(a.status, ST_TIMEOUT_EPI);
      bcast[0] = ok ? 1 : 0;
    }
    epi_bar();
    if (!bcast[0]) {
      *abort_flag = 1;
      return false;
    }
    const bool late = staged && nch > 0 && !mbar_wait(fx, 0, abort_flag);
    if (epi_bar_any(late)) {
      if (et == 0) set_status(a.status, ST_TIMEOUT_EPI);
      *abort_flag = 1;
      return false;
    }
    EpiPre pre = pre0;
  #pragma unroll 1
    for (int ch = 0; ch < nch; ++ch) {
      if (ch > 0) pre = epi_pre<MODE>(a, t, ch * kEpiTok, et, M);
      uint32_t r[32];
      tmem_ld32(tbase + ch * 32, r);
      float v[kEpiTok];
  #pragma unroll
      for (int j = 0; j < kEpiTok; ++j) v[j] = hilo(r, j);
      const size_t off = (size_t)ch * kTileN * kEpiTok;
      for (int k = 0; k < n_other; ++k) {
        float4 pv[4];
        if (staged) {
          const float4* p = reinterpret_cast<const float4*>(ring + (size_t)k * kChF + off) + fr;
  #pragma unroll
          for (int j4 = 0; j4 < 4; ++j4) pv[j4] = p[j4 * kTileN];
        } else {
          const int cc = cf + 1 + k;
          const float4* p = reinterpret_cast<const float4*>(a.partials + ((size_t)cc * 2) * kTileF + off) + fr;
  #pragma unroll
          for (int j4 = 0; j4 < 4; ++j4) pv[j4] = __ldcg(p + j4 * kTileN);
        }
  #pragma unroll
        for (int j4 = 0; j4 < 4; ++j4) {
          v[4 * j4 + 0] += pv[j4].x;
          v[4 * j4 + 1] += pv[j4].y;
          v[4 * j4 + 2] += pv[j4].z;
          v[4 * j4 + 3] += pv[j4].w;
        }
      }
      epi_chunk<MODE>(a, v, t, ch * kEpiTok, ch * kEpiTok, fr, et, M, S, pre);
    }
  } else {
    const int n_other = cl - cf;
    // Partials are staged in the idle ring in rounds of chunks: each round one
    // bulk copy per contributor brings the same run of chunks of every
    // partial ([chunk][j4][row] layout: a run of chunks is contiguous), so a
    // tile with many contributors or many chunks costs a few round trips
    // instead of one L2 load chain per chunk.
    const uint32_t ch_bytes = (uint32_t)kChF * 4;
    int per_round = n_other > 0 ? (int)(ring_bytes / ((uint32_t)n_other * ch_bytes)) : nch;
    if (per_round > nch) per_round = nch;
    const bool staged = per_round > 0 && nch > 0;
    if (et == 0) {
      const bool ok = wait_mask(mask, contrib_bits(n_other), abort_flag);
      if (!ok) set_status(a.status, ST_TIMEOUT_EPI);
      bcast[0] = ok ? 1 : 0;
    }
    epi_bar();
    if (!bcast[0]) {
      *abort_flag = 1;
      return false;
    }
    EpiPre pre = pre0;
    const int step = staged ? per_round : nch;
    for (int r0 = 0, round = 0; r0 < nch; r0 += step, ++round) {
      const int r1 = min(nch, r0 + step), nr = r1 - r0;
      if (staged) {
        if (et == 0) {
          // the partials were written through the generic proxy (and the ring
          // read through it by the previous round); the copies use the async proxy
          fence_proxy_async();
          *fx_armed = round + 1;
          mbar_arrive_expect_tx(fx, (uint32_t)n_other * nr * ch_bytes);
          for (int k = 0; k < n_other; ++k) {
            const int cc = cf + 1 + k;
            bulk_load(ring + (size_t)k * nr * kChF, a.partials + ((size_t)cc * 2) * kTileF + (size_t)r0 * kChF,
                      (uint32_t)nr * ch_bytes, fx);
          }
        }
        const bool late = !mbar_wait(fx, (uint32_t)(round & 1), abort_flag);
        if (epi_bar_any(late)) {
          if (et == 0) set_status(a.status, ST_TIMEOUT_EPI);
          *abort_flag = 1;
          return false;
        }
      }
  #pragma unroll 1
      for (int ch = r0; ch < r1; ++ch) {
        if (ch > 0) pre = epi_pre<MODE>(a, t, ch * kEpiTok, et, M);
        uint32_t r[32];
        tmem_ld32(tbase + ch * 32, r);
        float v[kEpiTok];
  #pragma unroll
        for (int j = 0; j < kEpiTok; ++j) v[j] = hilo(r, j);
        for (int k = 0; k < n_other; ++k) {
          float4 pv[4];
          if (staged) {
            const float4* p = reinterpret_cast<const float4*>(ring + ((size_t)k * nr + (ch - r0)) * kChF) + fr;
  #pragma unroll
            for (int j4 = 0; j4 < 4; ++j4) pv[j4] = p[j4 * kTileN];
          } else {
            const int cc = cf + 1 + k;
            const float4* p = reinterpret_cast<const float4*>(a.partials + ((size_t)cc * 2) * kTileF +
                                                              (size_t)ch * kChF) + fr;
  #pragma unroll
            for (int j4 = 0; j4 < 4; ++j4) pv[j4] = __ldcg(p + j4 * kTileN);
          }
  #pragma unroll
          for (int j4 = 0; j4 < 4; ++j4) {
            v[4 * j4 + 0] += pv[j4].x;
            v[4 * j4 + 1] += pv[j4].y;
            v[4 * j4 + 2] += pv[j4].z;
            v[4 * j4 + 3] += pv[j4].w;
          }
        }
        epi_chunk<MODE>(a, v, t, ch * kEpiTok, ch * kEpiTok, fr, et, M, S, pre);
      }
      if (staged && r1 < nch) epi_bar();  // the ring is read out before the next round's copies
    }
  }
  if (et == 0) *mask = 0ull;
  return true;
}

// RMS row scales of the pass's rows: all partial sums of squares in one round
// of loads, then a fixed-order sum per row.
template <int TT>
__device__ void epi_row_scale(const GemmArgs& a, int et, int M, const EpiSmem& S) {
  for (int c0 = 0; c0 < TT; c0 += kEpiTok) {
    const int nld = a.ssq_tiles * kEpiTok;
    for (int i = et; i < nld; i += 128) {
      const int tile = i / kEpiTok, j = i % kEpiTok;
      const int m = c0 + j;
      S.xch[i] = m < M ? __ldcg(a.ssq_in + (size_t)tile * a.m_cap + m) : 0.f;
    }
    epi_bar();
    if (et < kEpiTok) {
      float ss = 0.f;
      for (int t2 = 0; t2 < a.ssq_tiles; ++t2) ss += S.xch[t2 * kEpiTok + et];
      S.rs[c0 + et] = 1.0f / sqrtf(ss * a.inv_d + a.eps);
    }
    epi_bar();
  }
}

}  // namespace pard
