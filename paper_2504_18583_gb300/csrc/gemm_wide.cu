// GEMM of passes with more than 64 rows: batched decoding (112 verify rows at
// batch 16) and prompt passes (up to a whole prefill chunk).
//
// At these sizes a weight tile meets so many tokens that the traffic into the
// SMs bounds a kernel, not HBM: a CTA that multiplies 128 weight rows with 128
// tokens (hi and lo parts: 32 KB a 64-column step) takes 48 KB from L2 per
// 16 KB of weights.  Here a pair of CTAs (cta_group::2) shares a tile of 256
// weight rows and up to 256 tokens: each CTA loads its own 128 weight rows
// and half of the tokens, the tensor cores read the other half from the peer.
// Each 16 columns of K take two MMAs, one with the tokens' hi parts and one
// with their lo parts (selected by the descriptors' atom stride).  The tensor
// cores truncate at every accumulation, so hi and lo parts have accumulator
// columns of their own wherever tensor memory holds two buffers of them (tiles
// of at most 128 tokens), and in every tile of the QKV projection, whose keys
// and values are rounded to bf16 (one buffer, the whole of tensor memory,
// above 128 tokens).  The other projections' larger tiles sum both parts in
// one column: two 256-column buffers, so one tile's epilogue runs under the
// next tile's MMAs (sums a quarter as long changed the error of none of them).
//
// The tiles are shared out over the pairs whole, in equal parts or evenly by
// K-steps, whichever is expected to end first (wide_split).  A tile split
// between several pairs is finished by all of them: each stores its partial,
// then finishes its own share of the tile's 16-token chunks, summing the
// partials in pair order (deterministic).  (One finisher per tile gathers all
// partials of up to 128 KB each on one SM, which took longer than the
// multiplication.)  A pair waits for the others only after its last unit is
// multiplied and stored, and not for long: it gives its share up to one
// that arrives later, so that no CTA holds its SM for CTAs that have none yet.
//
// Roles per CTA: warp 0 streams, counting both CTAs' bytes on rank 0's
// barriers (TMA tensor copies can do that; the packed operands are tensors of
// 128-byte rows to them), warp 1 of rank 0 issues the MMAs, warps 2-5 and 6-9
// are two epilogue groups that take alternate chunks.
//
// Measured (one layer's launches, serialised, us; before: 64-token tiles, and a
// 128-token tile for gate/up and LM head, on single CTAs): 8B widths, 112 rows:
// QKV 36 -> 25, O 30 -> 24, gate/up 62 -> 54 (34 at the HBM rate), down 52 -> 38,
// LM head 236 -> 183; 512 rows: 82 -> 72, 57 -> 44, 197 -> 137, 138 -> 97.
// The main loop runs at 1.14k clocks per step of 256 x 256 x 64 (hi and lo: 2 x
// 8.4 MFLOP a pair) or at 7 TB/s of weights; what is left is each launch's start
// and its tail (partials, arrival, shares).
#include "gemm_core.cuh"

namespace pard {

namespace {

constexpr int kWideRing = 192 * 1024;  // stage ring; the stages' number follows from their size
constexpr int kWideMaxStages = 8;
constexpr int kWideThreads = 320;
constexpr int kWideBarBytes = (8 * (2 * kWideMaxStages + 6) + 15) / 16 * 16;
constexpr int kWideMiscBytes = 64;
constexpr int kWideGroupFloats = kEpiTok * kTileN + 3 * kEpiTok;  // exchange and row facts of one epilogue group
constexpr int kWideSmem =
    1024 + kWideRing + kWideBarBytes + kWideMiscBytes + 4 * (kWideMaxRows + 2 * kWideGroupFloats);
static_assert(kWideSmem <= 227 * 1024, "shared memory of one CTA");
static_assert(kWideGroupFloats % 4 == 0 && kWideMaxRows % 4 == 0 && kWideBarBytes % 16 == 0, "16-byte exchange reads");

__device__ __forceinline__ void all_epi_bar() { asm volatile("bar.sync 3, 256;" ::: "memory"); }

// all_epi_bar that also returns whether any of the 256 threads passed true
__device__ __forceinline__ bool all_epi_any(bool v) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\t"
      "setp.ne.u32 p, %1, 0;\n\t"
      "bar.red.or.pred q, 3, 256, p;\n\t"
      "selp.u32 %0, 1, 0, q;\n\t}"
      : "=r"(r)
      : "r"((uint32_t)v)
      : "memory");
  return r != 0;
}

// Epilogue values of one 16-token chunk straight from the accumulator; lo: how
// far behind the hi parts' columns the lo parts' are (0: in the same)
__device__ __forceinline__ void load_acc(uint32_t taddr, int lo, float (&v)[kEpiTok]) {
  uint32_t r[16];
  if (lo) {
    uint32_t l[16];
    tmem_ld16x2(taddr, taddr + lo, r, l);
#pragma unroll
    for (int j = 0; j < kEpiTok; ++j) v[j] = __uint_as_float(r[j]) + __uint_as_float(l[j]);
    return;
  }
  tmem_ld16(taddr, r);
#pragma unroll
  for (int j = 0; j < kEpiTok; ++j) v[j] = __uint_as_float(r[j]);
}

}  // namespace

// Shares of a complete tile that were given up go to whoever takes their bits
// out of its word.  The last contributor to arrive sees, after its own bit, all
// bits set before that; who gives up later sees the tile complete.  Both calls
// are rare and out of line: inlined, they lengthened every launch's tail (a
// batch-16 draft pass: 1640 us, 1599 so; 1545 before shares were given up).
static __device__ __noinline__ uint32_t claim_shares(unsigned long long* word, uint32_t given) {
  return (uint32_t)(atom_and64(word, ~((unsigned long long)given << kWideContrib)) >> kWideContrib) & given;
}
// gives up contributor i's share; which shares are the caller's all the same
static __device__ __noinline__ uint32_t give_share_up(unsigned long long* word, unsigned long long all, int i) {
  const unsigned long long own = 1ull << (kWideContrib + i), w = atom_or64(word, own) | own;
  return (w & all) == all ? claim_shares(word, (uint32_t)(w >> kWideContrib & all)) : 0u;
}

template <int MODE>
__global__ void __launch_bounds__(kWideThreads, 1) gemm_wide_kernel(const __grid_constant__ WideArgs w) {
  const GemmArgs& a = w.g;
  constexpr bool kPieces = MODE == MODE_QKV;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* ring = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint64_t* full = reinterpret_cast<uint64_t*>(ring + kWideRing);  // rank 0: both CTAs' stage has landed
  uint64_t* empty = full + kWideMaxStages;
  uint64_t* accf = empty + kWideMaxStages;
  uint64_t* acce = accf + 2;                 // rank 0: both CTAs' epilogue groups are done with the buffer
  uint64_t* drain = acce + 2;
  uint64_t* fx = drain + 1;                  // split tiles: partials copied into the idle ring
  uint32_t* misc = reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(full) + kWideBarBytes);
  uint32_t* tmem_slot = misc;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 1);
  int* bcast = reinterpret_cast<int*>(misc + 2);
  volatile int* fx_armed = reinterpret_cast<volatile int*>(misc + 3);  // rounds of copies issued
  int* live = reinterpret_cast<int*>(misc + 4);  // [0] token tiles, [1] tokens a tile
  uint32_t* extra = misc + 6;                    // [2] shares given up by others that fall to this CTA, per split tile
  float* rs = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(misc) + kWideMiscBytes);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const uint32_t rank = cluster_rank();
  const int c = blockIdx.x >> 1;  // this pair

  if (threadIdx.x == 0) {
    for (int s = 0; s < kWideMaxStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) { mbar_init(&accf[b], 1); mbar_init(&acce[b], 4); }
    mbar_init(drain, 1);
    mbar_init(fx, 1);
    *fx_armed = 0;
    *abort_flag = 0;
    // A row count written two or more launches back is read now, and the
    // tiles past it are neither loaded nor multiplied.
    int tiles = a.tok_tiles, n_tok = a.n_tok;
    if (a.m_early) wide_tiles(min(max(__ldcg(a.m_dev), 1), a.m_cap), tiles, n_tok);
    live[0] = tiles;
    live[1] = n_tok;
    fence_barrier_init();
  }
  __syncthreads();
  if (warp == 1) tmem_alloc2(tmem_slot, 512);
  tc_fence_before();
  __syncthreads();
  cluster_sync();  // the peer's barriers are initialised before anything arrives on them
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  const int tok_tiles = live[0], n_tok = live[1];
  // columns from the hi parts' accumulator to the lo parts' (0: one for both), and the buffers there are
  const int lo = n_tok <= kWideTok / 2 ? kWideTok / 2 : MODE == MODE_QKV ? kWideTok : 0;
  const int nacc = lo == kWideTok ? 1 : 2;
  const int kc = a.kc;
  // unit indices: 32 bits (the host checks that U times the pairs fits; 64-bit
  // divisions made up half of a short launch's tail)
  const int T = (a.w_tiles + 1) / 2 * tok_tiles, U = T * kc;
  const WideSplit split = wide_split(T, kc, a.max_pairs);
  const int G = split.pairs;  // pairs with work
  auto start_of = [&](int cc) { return split.tiles ? cc * T / G * kc : cc * U / G; };
  auto owner = [&](int u) { return ((u + 1) * G + U - 1) / U - 1; };
  const int u0 = c < G ? start_of(c) : 0, u1 = c < G ? start_of(c + 1) : 0;
  // QKV: this pair's share [tb, te) of the tile of unit u is summed in pieces
  // of equal length, at most `chain` units each: the end of u's piece.
  auto piece_end = [&](int u, int tb, int te) {
    if constexpr (!kPieces) return te;
    const int chain = kc > kWideChain ? kWideChain : kWideChainShort;
    const int pieces = (te - tb + chain - 1) / chain, len = (te - tb + pieces - 1) / pieces;
    return min(tb + ((u - tb) / len + 1) * len, te);
  };
  const uint32_t b_bytes = (uint32_t)n_tok * 128;  // half of the tile's tokens, hi and lo rows
  const uint32_t stage_bytes = (uint32_t)kTileN * 128 + b_bytes;
  const int R = min(kWideMaxStages, kWideRing / (int)stage_bytes);
  uint32_t armed = 0, armed_odd = 0;  // producer: slots armed at least once, and those armed an odd number of times

  if (warp == 0) {
    // ---------------- producer: this CTA's weight rows and half of the tokens ----------------
    // The whole warp runs the loop and one elected thread issues: in a loop
    // inside "if (lane == 0)" each copy took about 150 clocks to issue.
    if (u1 > u0) {
      // the weights are read again for every further token tile
      const uint64_t pol = tok_tiles == 1 ? policy_evict_first() : policy_evict_normal();
      if (elect_one()) {
        for (int i = 0; i < (a.pair ? 2 : a.nseg); ++i) tma_prefetch_desc(&a.wmap[i]);
        for (int i = 0; i < 3; ++i) tma_prefetch_desc(&w.x[i]);
      }
      const int n = u1 - u0;
      const int npre = min(n, R);
      int kk = u0 % kc;
      int wp = u0 / kc / tok_tiles, tok_tile = u0 / kc % tok_tiles;
      // coordinates of the current weight tile's step kk: (col0 + kk colstep, row0 + kk rowstep)
      const CUtensorMap *wmap0 = nullptr, *wmap1 = nullptr;
      int row0 = 0, rowstep = 0, colstep = 0;
      auto set_tile = [&]() {
        // an odd last tile is loaded by both CTAs and finished by rank 0 alone
        const int w_tile = min(2 * wp + (int)rank, a.w_tiles - 1);
        const int seg = a.pair ? 0 : seg_of(a, w_tile);
        const int blk = a.pair ? w_tile : w_tile - a.seg_tile0[seg];
        const int rows = a.pair ? 64 : kTileN;
        wmap0 = &a.wmap[seg];
        wmap1 = &a.wmap[1];
        const bool packed = a.wpk[seg] != nullptr;  // blocks of [rows][64] in steps of K
        row0 = packed ? blk * kc * rows : blk * rows;
        rowstep = packed ? rows : 0;
        colstep = packed ? 0 : kChunkK;
      };
      set_tile();
      const uint64_t polx = policy_evict_normal();
      const uint32_t full0 = mapa_shared(full, 0);  // rank 0's barriers
      auto issue_a = [&](int s) {
        uint8_t* dst = ring + (uint32_t)s * stage_bytes;
        const uint32_t bar = full0 + 8 * s;
        tma2_load_2d_hint(dst, wmap0, bar, kk * colstep, row0 + kk * rowstep, pol);
        if (a.pair) tma2_load_2d_hint(dst + kTileN * 64, wmap1, bar, kk * colstep, row0 + kk * rowstep, pol);
      };
      // this rank's half of a token tile: n_tok rows of 128 bytes
      auto issue_b = [&](int s, int kk_, int tok_) {
        uint8_t* dst = ring + (uint32_t)s * stage_bytes + kTileN * 128;
        const uint32_t bar = full0 + 8 * s;
        const int row = kk_ * a.x_rows + (2 * tok_ + (int)rank) * n_tok;
        if (n_tok == a.n_tok) {
          tma2_load_2d_hint(dst, &w.x[0], bar, 0, row, polx);
        } else {  // fewer rows than the launch was sized for
          int r = 0;
          for (; r + kWideBoxL <= n_tok; r += kWideBoxL) tma2_load_2d_hint(dst + r * 128, &w.x[1], bar, 0, row + r, polx);
          for (; r < n_tok; r += kWideBoxS) tma2_load_2d_hint(dst + r * 128, &w.x[2], bar, 0, row + r, polx);
        }
      };
      auto arm = [&](int s) {  // armed, armed_odd: by every thread of the warp
        armed |= rank == 0 ? 1u << s : 0u;
        armed_odd ^= rank == 0 ? 1u << s : 0u;
      };
      auto expect = [&](int s) {
        if (rank == 0) mbar_arrive_expect_tx(&full[s], 2 * stage_bytes);
      };
      auto advance = [&]() {
        if (++kk == kc) {
          kk = 0;
          if (++tok_tile == tok_tiles) { tok_tile = 0; ++wp; }
          set_tile();
        }
      };
      // weights first: they do not depend on the previous kernel
      const int kk0 = kk, tok0 = tok_tile;
      for (int i = 0; i < npre; ++i) {
        arm(i);
        if (elect_one()) {
          expect(i);
          issue_a(i);
        }
        __syncwarp();
        advance();
      }
      pdl_wait();
      for (int i = 0, k2 = kk0, t2 = tok0; i < npre; ++i) {
        if (elect_one()) issue_b(i, k2, t2);
        __syncwarp();
        if (++k2 == kc) { k2 = 0; if (++t2 == tok_tiles) t2 = 0; }
      }
      int s = npre % R;
      uint32_t ph = (uint32_t)((npre / R) & 1) ^ 1u;
      for (int i = npre; i < n; ++i) {
        if (!__all_sync(0xffffffffu, mbar_wait(&empty[s], ph, abort_flag))) {
          if (lane == 0) set_status(a.status, ST_TIMEOUT_TMA);
          *abort_flag = 1;
          break;
        }
        arm(s);
        if (elect_one()) {
          expect(s);
          issue_a(s);
          issue_b(s, kk, tok_tile);
        }
        __syncwarp();
        advance();
        if (++s == R) { s = 0; ph ^= 1u; }
      }
    }
    if (lane == 0) pdl_trigger();
  } else if (warp == 1) {
    if (rank == 0) {
      // ---------------- MMA issuer of the pair: the whole warp runs the loop, one thread issues ----------------
      // (a loop inside "if (lane == 0)" took about 100 clocks an MMA to issue)
      const uint32_t idesc = idesc_bf16(2 * kTileN, n_tok);
      int s = 0;
      uint32_t fph = 0;
      int seg_i = 0;
      bool ok = true;
      for (int u = u0; u < u1 && ok;) {
        const int tile0 = u / kc * kc;
        const int ub = u, ue = piece_end(u, max(tile0, u0), min(tile0 + kc, u1));
        const int ab = seg_i % nacc;
        ok = __all_sync(0xffffffffu, mbar_wait_cluster(&acce[ab], (uint32_t)((seg_i / nacc) & 1) ^ 1u, abort_flag));
        if (!ok) break;
        tc_fence_after();
        const uint32_t d = tmem + ab * kWideTok, dl = d + lo;
        for (; u < ue; ++u) {
          ok = __all_sync(0xffffffffu, mbar_wait(&full[s], fph, abort_flag));
          if (!ok) break;
          tc_fence_after();
          const uint32_t sa = smem_u32(ring) + (uint32_t)s * stage_bytes;
          const uint64_t ad = sw128_desc(sa);
          const uint64_t bh = sw128_desc(sa + kTileN * 128, 2048), bl = sw128_desc(sa + kTileN * 128 + 1024, 2048);
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < kChunkK / 16; ++k) {
              const uint32_t more = (u > ub || k > 0) ? 1u : 0u;
              umma2_bf16(d, ad + 2 * k, bh + 2 * k, idesc, more);
              umma2_bf16(dl, ad + 2 * k, bl + 2 * k, idesc, lo ? more : 1u);
            }
            umma2_commit(&empty[s], 3);
            if (u + 1 == ue) umma2_commit(&accf[ab], 3);
          }
          __syncwarp();
          if (++s == R) { s = 0; fph ^= 1u; }
        }
        ++seg_i;
      }
      if (!ok && lane == 0) {
        set_status(a.status, ST_TIMEOUT_MMA);
        *abort_flag = 1;
      }
    }
  } else {
    // ---------------- epilogue: two groups of 128 threads ----------------
    pdl_wait();
    const int et256 = threadIdx.x - 64, grp = et256 >> 7, et = et256 & 127;
    const int q = warp & 3, fr = q * 32 + lane;
    EpiSmem S;
    S.rs = rs;
    S.xch = rs + kWideMaxRows + grp * kWideGroupFloats;
    S.ri = reinterpret_cast<int*>(S.xch + kEpiTok * kTileN);
    S.bar = 1 + grp;
    int M = *a.m_dev;
    if (M > a.m_cap) {
      if (et256 == 0) set_status(a.status, ST_BAD_ROWS);
      M = a.m_cap;
    }
    constexpr int kTileF = kTileN * kWideTok;  // floats of one partial tile of one CTA
    constexpr int kChF = kTileN * kEpiTok;
    constexpr int kRingChunks = kWideRing / (kChF * 4);  // chunks the ring holds; more contributors are read from L2
    // RMS scales of all the pass's rows: a thread a token, its partial sums
    // requested sixteen at a time and added in tile order
    if constexpr (MODE != MODE_RESID) {
      for (int m = et256; m < M; m += 256) {
        float ss = 0.f;
        for (int t0 = 0; t0 < a.ssq_tiles; t0 += 16) {
          float p[16];
#pragma unroll
          for (int k = 0; k < 16; ++k)
            p[k] = t0 + k < a.ssq_tiles ? __ldcg(a.ssq_in + (size_t)(t0 + k) * a.m_cap + m) : 0.f;
#pragma unroll
          for (int k = 0; k < 16; ++k) ss += p[k];
        }
        rs[m] = 1.0f / sqrtf(ss * a.inv_d + a.eps);
      }
      for (int m = M + et256; m < min(M + kEpiTok, kWideMaxRows); m += 256) rs[m] = 0.f;  // the last chunk's other rows
      all_epi_bar();
    }
    auto chunks_of = [&](int w_tile, int tok_base) {
      return w_tile < a.w_tiles ? max(0, min(n_tok / kEpiTok, (M - tok_base + kEpiTok - 1) / kEpiTok)) : 0;
    };
    // A split tile this pair has stored its partial of, and its share of it:
    // contributor i of n finishes chunks [ceil(i nch / n), ceil((i + 1) nch / n))
    struct Share {
      int t, w_tile, tok_base, cf, n, nch, i, c0, c1;
    };
    Share sh0{0, 0, 0, 0, 1, 0, 0, 0, 0}, sh1{0, 0, 0, 0, 1, 0, 0, 0, 0};
    bool settled = false;  // it is known which shares are this CTA's
    uint32_t todo0 = 0, todo1 = 0;  // contributors whose shares it takes besides its own
    auto range_of = [](Share& h, int i) {
      h.c0 = (i * h.nch + h.n - 1) / h.n;
      h.c1 = ((i + 1) * h.nch + h.n - 1) / h.n;
    };
    auto mask_of = [&](int t) { return reinterpret_cast<unsigned long long*>(a.counters) + 2 * t + rank; };
    auto partial = [&](const Share& h, int k) {
      // only the tile's first contributor may begin before the tile
      const int sl = k > 0 || start_of(h.cf) >= h.t * kc ? 0 : 1;
      return a.partials + ((size_t)(2 * (h.cf + k) + rank) * 2 + sl) * kTileF;
    };
    auto claim = [&](const Share& h, unsigned long long w, int slot) {
      const uint32_t given = (uint32_t)(w >> kWideContrib & contrib_bits(h.n));
      if (given) extra[slot] |= claim_shares(mask_of(h.t), given);
    };
    auto look = [&](const Share& h, int slot) {
      if (h.nch <= 0 || h.c0 < h.c1) return;
      const unsigned long long all = contrib_bits(h.n), w = ld_acquire_u64(mask_of(h.t));
      if ((w & all) == all) claim(h, w, slot);
    };
    auto settle = [&](int mine) {
      settled = true;
      if (!(mine & 1)) sh0.c0 = sh0.c1;
      if (!(mine & 2)) sh1.c0 = sh1.c1;
      if (sh0.nch > 0) todo0 = extra[0];
      if (sh1.nch > 0) todo1 = extra[1];
    };
    int seg_i = 0, rounds = 0;
    bool ok = true;
    int u = u0;
    // Each turn of the loop takes one segment of this pair's range: a partial
    // is stored, a whole tile's chunks are finished from the accumulator; and
    // after the last segment one round of the shares, whose partials a bulk
    // copy per contributor brings into the ring (idle by then).
    while (true) {
      const bool from_acc = u < u1;
      int take0 = 0, take1 = 0, base1 = 0;  // chunks of this turn: of the tile / first share, of the second share
      bool staged = true;
      unsigned long long old0 = 0, old1 = 0;
      const float* sum = nullptr;  // from the accumulator: what earlier pieces of the tile added up to
      uint32_t tbase = 0;
      int wt0 = 0, wt1 = 0, tb0 = 0, tb1 = 0, n0 = 0, n1 = 0, ch0 = 0, ch1 = 0;  // tile, token, contributors, first chunk
      int ab = 0;
      if (from_acc) {
        const int t = u / kc;
        const int tb = max(t * kc, u0), te = min((t + 1) * kc, u1);
        const int ub = u, ue = piece_end(u, tb, te);
        u = ue;
        ab = seg_i % nacc;
        wt0 = 2 * (t / tok_tiles) + (int)rank;
        tb0 = t % tok_tiles * n_tok;
        const int nch = chunks_of(wt0, tb0);
        const bool whole = tb == t * kc && te == (t + 1) * kc;
        const bool last = ue == te;
        if (whole && last) take0 = nch;
        // this pair's sum so far, or its partial; a whole tile's is gone
        // before the range's last tile, which may be split, begins
        const int slot = !whole && tb == u0 ? 0 : 1;
        float* mine = a.partials + ((size_t)(2 * c + rank) * 2 + slot) * kTileF;
        sum = ub > tb ? mine : nullptr;
        ok = mbar_wait(&accf[ab], (uint32_t)((seg_i / nacc) & 1), abort_flag);
        if (all_epi_any(!ok)) {
          if (et256 == 0) set_status(a.status, ST_TIMEOUT_EPI);
          *abort_flag = 1;
          break;
        }
        ++seg_i;
        tc_fence_after();
        tbase = tmem + ab * kWideTok + ((uint32_t)(q * 32) << 16);
        if (!whole || !last) {
          // [chunk][j4][row] float4s: a warp's stores are 512 contiguous bytes
          auto put = [&](float4* dst, float4 f) {
            if (kPieces && sum) {
              const float4 o = __ldcg(dst);  // this thread's own
              f = make_float4(f.x + o.x, f.y + o.y, f.z + o.z, f.w + o.w);
            }
            *dst = f;
          };
          if (lo) {
#pragma unroll 1
            for (int ch = grp; ch < nch; ch += 2) {
              float v[kEpiTok];
              load_acc(tbase + ch * kEpiTok, lo, v);
              float4* dst = reinterpret_cast<float4*>(mine + (size_t)ch * kChF) + fr;
#pragma unroll
              for (int j4 = 0; j4 < 4; ++j4)
                put(dst + j4 * kTileN, make_float4(v[4 * j4], v[4 * j4 + 1], v[4 * j4 + 2], v[4 * j4 + 3]));
            }
          } else {
            // two chunks a turn: one accumulator read for both
#pragma unroll 1
            for (int ch = 2 * grp; ch < nch; ch += 4) {
              uint32_t r[32];
              tmem_ld32(tbase + ch * kEpiTok, r);
              float4* dst = reinterpret_cast<float4*>(mine + (size_t)ch * kChF) + fr;
#pragma unroll
              for (int j4 = 0; j4 < 8; ++j4)
                if (j4 < 4 || ch + 1 < nch)
                  put(dst + j4 * kTileN, make_float4(__uint_as_float(r[4 * j4]), __uint_as_float(r[4 * j4 + 1]),
                                                     __uint_as_float(r[4 * j4 + 2]), __uint_as_float(r[4 * j4 + 3])));
            }
          }
          tc_fence_before();
          // orders every thread's partial before the one release OR, and
          // before another thread's reads of a whole tile's sum
          all_epi_bar();
          if (et == 0) mbar_arrive_remote(&acce[ab], 0);
          if (!last) continue;
          const int cf = owner(t * kc), n = owner((t + 1) * kc - 1) - cf + 1, i = c - cf;
          if (et256 == 0) {
            if (nch > 0) red_release_or64(mask_of(t), 1ull << i);
            extra[slot] = 0;
          }
          Share h{t, wt0, tb0, cf, n, nch, i, 0, 0};
          range_of(h, i);
          if (slot == 0) sh0 = h;
          else sh1 = h;
          continue;
        }
      } else {
        // its own shares first; those that others gave up after them
        if (!settled && sh0.c0 >= sh0.c1 && sh1.c0 >= sh1.c1) {
          if (et256 == 0) {
            look(sh0, 0);
            look(sh1, 1);
          }
          all_epi_bar();
          settle(3);
        }
        while (sh0.c0 >= sh0.c1 && todo0) {
          range_of(sh0, __ffs((int)todo0) - 1);
          todo0 &= todo0 - 1;
        }
        while (sh1.c0 >= sh1.c1 && todo1) {
          range_of(sh1, __ffs((int)todo1) - 1);
          todo1 &= todo1 - 1;
        }
        const int rem0 = max(0, sh0.c1 - sh0.c0), rem1 = max(0, sh1.c1 - sh1.c0);
        if (rem0 + rem1 == 0) break;
        n0 = sh0.n; n1 = sh1.n;
        take0 = min(rem0, kRingChunks / n0);
        take1 = min(rem1, (kRingChunks - take0 * n0) / n1);
        staged = take0 + take1 > 0;
        if (!staged) {  // more contributors than the ring has places: summed from L2
          take0 = rem0;
          take1 = rem1;
        }
        base1 = take0 * n0;
        wt0 = sh0.w_tile; tb0 = sh0.tok_base; ch0 = sh0.c0;
        wt1 = sh1.w_tile; tb1 = sh1.tok_base; ch1 = sh1.c0;
      }
      // this group's chunks of the turn: every second of take0 + take1
      auto tile_of = [&](int i, int& w_tile, int& tok0) {
        w_tile = i < take0 ? wt0 : wt1;
        tok0 = i < take0 ? tb0 + (ch0 + i) * kEpiTok : tb1 + (ch1 + i - take0) * kEpiTok;
      };
      const int items = take0 + take1;
      EpiPre pre = {};
      if (grp < items) {
        int w_tile, tok0;
        tile_of(grp, w_tile, tok0);
        pre = epi_pre<MODE>(a, w_tile, tok0, et, M);
      }
      if (!from_acc) {
        if (et256 == 0) {
          uint32_t mine = 3;
          if (staged) fence_proxy_async_all();  // the ring was read by the previous round
          // copies of the contributors that have arrived since the last look;
          // the partials were written through the generic proxy, the copies
          // read them through the async proxy
          auto fetch = [&](const Share& h, unsigned long long all, unsigned long long& seen, int take, int at, int slot) {
            const unsigned long long w = settled ? all : ld_acquire_u64(mask_of(h.t)), m = w & all;
            if (m == all && !settled) claim(h, w, slot);
            unsigned long long nw = m & ~seen;
            if (!nw) return false;
            fence_proxy_async();
            for (; nw && staged && take; nw &= nw - 1) {
              const int k = __ffsll((long long)nw) - 1;
              const uint32_t bytes = (uint32_t)take * kChF * 4;
              mbar_expect_tx(fx, bytes);
              bulk_load(reinterpret_cast<float*>(ring) + (size_t)(at + k * take) * kChF, partial(h, k) + (size_t)h.c0 * kChF, bytes,
                        fx);
            }
            seen = m;
            return true;
          };
          // (a share without room in this round is settled all the same)
          const unsigned long long all0 = sh0.c0 < sh0.c1 ? contrib_bits(n0) : 0, all1 = sh1.c0 < sh1.c1 ? contrib_bits(n1) : 0;
          unsigned long long seen0 = 0, seen1 = 0;
          const unsigned long long t0 = globaltimer();
          while (seen0 != all0 || seen1 != all1) {
            bool any = false;
            if (seen0 != all0) any |= fetch(sh0, all0, seen0, take0, 0, 0);
            if (seen1 != all1) any |= fetch(sh1, all1, seen1, take1, base1, 1);
            if (!any && globaltimer() - t0 > (unsigned)w.share_wait_ns) {
              // not in time: the round is done anew, without what is no longer this CTA's
              mine = 7;
              if (seen0 != all0) {
                const uint32_t e = give_share_up(mask_of(sh0.t), all0, sh0.i);
                if (!(e >> sh0.i & 1)) mine &= ~1u;
                extra[0] |= e & ~(1u << sh0.i);
              }
              if (seen1 != all1) {
                const uint32_t e = give_share_up(mask_of(sh1.t), all1, sh1.i);
                if (!(e >> sh1.i & 1)) mine &= ~2u;
                extra[1] |= e & ~(1u << sh1.i);
              }
              break;
            }
          }
          if (staged) {
            *fx_armed = rounds + 1;
            mbar_arrive(fx);
          }
          if (!settled) {
            look(sh0, 0);
            look(sh1, 1);
            bcast[0] = (int)mine;
          }
          // last round of a share: count it in the mask's upper byte (read below)
          if (mine == 3 && take0 && sh0.c0 + take0 == sh0.c1) old0 = atomicAdd(mask_of(sh0.t), 1ull << kWideReadShift);
          if (mine == 3 && take1 && sh1.c0 + take1 == sh1.c1) old1 = atomicAdd(mask_of(sh1.t), 1ull << kWideReadShift);
        }
        ok = !staged || mbar_wait(fx, (uint32_t)(rounds & 1), abort_flag);
        if (all_epi_any(!ok)) {
          if (et256 == 0) set_status(a.status, ST_TIMEOUT_EPI);
          *abort_flag = 1;
          break;
        }
        if (!settled) {
          const int mine = bcast[0];
          settle(mine);
          if (mine != 3) {
            rounds += staged ? 1 : 0;
            continue;
          }
        }
      }
#pragma unroll 1
      for (int i = grp; i < items; i += 2) {
        const EpiPre now = pre;
        int w_tile, tok0;
        if (i + 2 < items) {
          tile_of(i + 2, w_tile, tok0);
          pre = epi_pre<MODE>(a, w_tile, tok0, et, M);
        }
        tile_of(i, w_tile, tok0);
        float v[kEpiTok];
        if (from_acc) {
          load_acc(tbase + i * kEpiTok, lo, v);
          if (kPieces && sum) {
            const float4* p = reinterpret_cast<const float4*>(sum + (size_t)i * kChF) + fr;
#pragma unroll
            for (int j4 = 0; j4 < 4; ++j4) {
              const float4 pv = __ldcg(p + j4 * kTileN);
              v[4 * j4 + 0] += pv.x;
              v[4 * j4 + 1] += pv.y;
              v[4 * j4 + 2] += pv.z;
              v[4 * j4 + 3] += pv.w;
            }
          }
        } else {
#pragma unroll
          for (int j = 0; j < kEpiTok; ++j) v[j] = 0.f;
          const int n = i < take0 ? n0 : n1, take = i < take0 ? take0 : take1;
          const int at = i < take0 ? i : base1 + i - take0;
#pragma unroll 2
          for (int k = 0; k < n; ++k) {
            const float4* p;
            if (staged)
              p = reinterpret_cast<const float4*>(reinterpret_cast<const float*>(ring) + (size_t)(at + k * take) * kChF) + fr;
            else
              p = reinterpret_cast<const float4*>((i < take0 ? partial(sh0, k) : partial(sh1, k)) +
                                                  (size_t)(i < take0 ? ch0 + i : ch1 + i - take0) * kChF) + fr;
#pragma unroll
            for (int j4 = 0; j4 < 4; ++j4) {
              const float4 pv = staged ? p[j4 * kTileN] : __ldcg(p + j4 * kTileN);
              v[4 * j4 + 0] += pv.x;
              v[4 * j4 + 1] += pv.y;
              v[4 * j4 + 2] += pv.z;
              v[4 * j4 + 3] += pv.w;
            }
          }
        }
        epi_chunk<MODE>(a, v, w_tile, tok0, tok0, fr, et, M, S, now);
      }
      if (from_acc) {
        tc_fence_before();
        epi_bar(S.bar);
        if (et == 0) mbar_arrive_remote(&acce[ab], 0);
      } else {
        all_epi_bar();  // the ring is read out before the next round
        if (et256 == 0) {
          // the last of the finishing CTAs clears the mask
          if (take0 && sh0.c0 + take0 == sh0.c1 && (int)(old0 >> kWideReadShift) == min(sh0.n, sh0.nch) - 1)
            *mask_of(sh0.t) = 0ull;
          if (take1 && sh1.c0 + take1 == sh1.c1 && (int)(old1 >> kWideReadShift) == min(sh1.n, sh1.nch) - 1)
            *mask_of(sh1.t) = 0ull;
        }
        sh0.c0 += take0;
        sh1.c0 += take1;
        rounds += staged ? 1 : 0;
      }
    }
  }

  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // let this CTA's copies and MMAs in flight land before its memory goes away
    if (warp == 0 && lane == 0)
      for (int s = 0; s < kWideMaxStages; ++s)
        if (armed >> s & 1u) mbar_drain(&full[s], (armed_odd >> s & 1u) ^ 1u);
    if (warp == 1 && rank == 0) {
      if (elect_one()) umma2_commit(drain, 1);
      __syncwarp();
      mbar_drain(drain, 0);
    }
    if (threadIdx.x == 64 && *fx_armed) mbar_drain(fx, (uint32_t)((*fx_armed - 1) & 1));
    __syncthreads();
  }
  __syncwarp();
  cluster_sync();  // the peer's MMAs read this CTA's memory, its threads arrive on this CTA's barriers
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc2(tmem, 512);
  }
}

using WideKernel = void (*)(WideArgs);
static WideKernel wide_kernel(int mode) {
  switch (mode) {
    case MODE_QKV: return gemm_wide_kernel<MODE_QKV>;
    case MODE_RESID: return gemm_wide_kernel<MODE_RESID>;
    case MODE_SWIGLU: return gemm_wide_kernel<MODE_SWIGLU>;
    default: return gemm_wide_kernel<MODE_LOGITS>;
  }
}

static void wide_launch_config(cudaLaunchConfig_t& cfg, cudaLaunchAttribute (&attr)[2], int pairs, cudaStream_t s,
                               bool pdl) {
  cfg.gridDim = dim3(2 * pairs);
  cfg.blockDim = dim3(kWideThreads);
  cfg.dynamicSmemBytes = kWideSmem;
  cfg.stream = s;
  attr[0].id = cudaLaunchAttributeClusterDimension;
  attr[0].val.clusterDim.x = 2;
  attr[0].val.clusterDim.y = 1;
  attr[0].val.clusterDim.z = 1;
  attr[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 2 : 1;
}

int gemm_wide_max_pairs(int sm) {
  int pairs = sm / 2;
  for (int mode = 0; mode < 4; ++mode) {
    cudaError_t e = cudaFuncSetAttribute(wide_kernel(mode), cudaFuncAttributeMaxDynamicSharedMemorySize, kWideSmem);
    if (e != cudaSuccess) throw e;
    cudaLaunchConfig_t cfg = {};
    cudaLaunchAttribute attr[2];
    wide_launch_config(cfg, attr, sm / 2, nullptr, false);
    int n = 0;
    e = cudaOccupancyMaxActiveClusters(&n, wide_kernel(mode), &cfg);
    if (e != cudaSuccess) throw e;
    if (n < pairs) pairs = n;
  }
  return pairs < 1 ? 1 : pairs;
}

void launch_gemm_wide(const WideArgs& a, int pairs, cudaStream_t s, bool pdl) {
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute attr[2];
  wide_launch_config(cfg, attr, pairs, s, pdl);
  const cudaError_t e = cudaLaunchKernelEx(&cfg, wide_kernel(a.g.mode), a);
  if (e != cudaSuccess) throw e;
}

}  // namespace pard
