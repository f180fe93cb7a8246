// Weight-streaming GEMM of passes of up to 64 rows: Y[m][n] = sum_k X[m][k] W[n][k]
// with W bf16 [N][K] streamed from HBM exactly once per launch and X a few
// activation rows (M = K+1 verify rows, up to 2K draft rows per sequence).
//
// GB300 design (one launch fills the GPU once; one CTA per SM, two where tiles
// of 16 tokens are shared out whole):
//  * operand swap: the weight tile is the UMMA A operand (M = 128 weight
//    rows), the activations the B operand (N = 2 x token tile), so a skinny
//    M=9 product still issues full 128-row tensor-core tiles;
//  * activations are carried as bf16 hi/lo pairs (x = hi + lo, each a row of
//    the B operand), which keeps fp32-level accuracy of the products
//    with bf16 tensor-core inputs; hi and lo columns are summed in the
//    epilogue;
//  * warp 0 streams 128x64 weight tiles and the matching activation tile
//    with TMA (128-byte swizzle) through a multi-stage mbarrier ring, warp 1
//    issues tcgen05.mma into a TMEM accumulator, warps 2-5 drain TMEM;
//  * the flattened (tile, K-chunk) index space is split evenly over the
//    CTAs, in whole tiles or with every tile in the same number of parts
//    (run_gemm chooses the number of CTAs so); a tile shared by several CTAs
//    is finished by the first of them, for which it is the last segment: the
//    others store their partials and set their bit of the tile's mask with one
//    release OR each, the finisher pulls all partials into its idle stage ring
//    with bulk copies and sums them in CTA order (deterministic);
//  * epilogues are fused: RMS row scaling, RoPE + paged KV write (QKV),
//    residual add + next norm's gain and sum of squares (O / down),
//    SiLU(gate) * up (gate/up pairs), logits + per-tile max / argmax /
//    sum-exp / Gumbel-max statistics (LM head);
//  * programmatic dependent launch: the weight tiles of the first stages
//    are requested before waiting on the previous kernel, since weights do
//    not depend on it.
#include "gemm_core.cuh"

namespace pard {

template <int TT, int MODE>
// two CTAs per SM at the 16-token tile: this launch's and the next one's
__global__ void __launch_bounds__(192, TT <= 16 ? 2 : 1) gemm_kernel(const __grid_constant__ GemmArgs a) {
  using C = GemmCfg<TT>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  uint8_t* sA = smem;
  uint8_t* sB = smem + C::kStages * C::kABytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(sB + C::kStages * C::kBBytes);
  uint64_t* empty = full + C::kStages;
  uint64_t* accf = empty + C::kStages;
  uint64_t* acce = accf + 2;
  uint64_t* drain = acce + 2;
  uint64_t* fx = drain + 1;  // split-K finish: partials pulled into the ring
  // the barrier block is rounded to 16 bytes: the epilogue scratch after
  // misc takes 16-byte vector accesses
  uint32_t* misc = reinterpret_cast<uint32_t*>(reinterpret_cast<uint8_t*>(full) + C::kBarBytes);
  static_assert(C::kStages * C::kStageBytes % 16 == 0 && C::kBarBytes % 16 == 0 && C::kMiscBytes % 16 == 0 &&
                    TT % 4 == 0,
                "epilogue scratch alignment");
  uint32_t* tmem_slot = misc;
  volatile int* abort_flag = reinterpret_cast<volatile int*>(misc + 1);
  int* bcast = reinterpret_cast<int*>(misc + 2);
  volatile int* fx_armed = reinterpret_cast<volatile int*>(misc + 3);
  float* scratch = reinterpret_cast<float*>(reinterpret_cast<uint8_t*>(misc) + C::kMiscBytes);
  const EpiSmem S = carve_epi<TT>(scratch);

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int G = gridDim.x;
  const int c = blockIdx.x;
  const int U = a.w_tiles * a.kc;  // one token tile
  const int u0 = range_start(c, U, G), u1 = range_start(c + 1, U, G);  // this CTA's units

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kStages; ++s) { mbar_init(&full[s], 1); mbar_init(&empty[s], 1); }
    for (int b = 0; b < 2; ++b) { mbar_init(&accf[b], 1); mbar_init(&acce[b], 128); }
    mbar_init(drain, 1);
    mbar_init(fx, 1);
    *abort_flag = 0;
    *fx_armed = 0;
    fence_barrier_init();
  }
  if (warp == 1) tmem_alloc(tmem_slot, C::kTmemCols);
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *tmem_slot;
  uint32_t armed = 0, armed_odd = 0;  // producer: slots armed at least once, and those armed an odd number of times
  constexpr int R = C::kStages;
  // token rows a tile's MMA covers: hi/lo pairs are the B rows, so N = 2 n_tok
  const int n_tok = min(a.n_tok, TT);
  const uint32_t b_bytes = (uint32_t)n_tok * 2 * 128;
  const uint32_t stage_bytes = (uint32_t)C::kABytes + b_bytes;

  if (warp == 0) {
    // ---------------- TMA producer ----------------
    // The whole warp runs the loop and one elected thread issues: inside "if
    // (lane == 0)" every copy (and every MMA below) takes about 100 clocks to issue.
    {
      const uint64_t pol = policy_evict_first();
      const int n = u1 - u0;
      const int npre = n < R ? n : R;
      // Unit cursor advanced incrementally: the producer issues one stage per
      // wake-up with no divisions on the path between the 'empty' signal and
      // the copies.
      int kk = u0 % a.kc;
      int w_tile = u0 / a.kc;
      const __nv_bfloat16* wsrc0 = nullptr;  // packed block base of the current weight tile (A)
      const __nv_bfloat16* wsrc1 = nullptr;  // second half (gate/up pairs)
      const CUtensorMap* wmap0 = nullptr;
      int wrow = 0;                          // row-major fallback: first row of the tile
      auto set_tile = [&]() {
        if (a.pair) {
          if (a.wpk[0]) {
            wsrc0 = a.wpk[0] + (size_t)w_tile * a.kc * 64 * 64;
            wsrc1 = a.wpk[1] + (size_t)w_tile * a.kc * 64 * 64;
          } else {
            wsrc0 = wsrc1 = nullptr;
            wrow = w_tile * 64;
          }
        } else {
          const int seg = seg_of(a, w_tile);
          const int blk = w_tile - a.seg_tile0[seg];
          wsrc0 = a.wpk[seg] ? a.wpk[seg] + (size_t)blk * a.kc * kTileN * 64 : nullptr;
          wmap0 = &a.wmap[seg];
          wrow = blk * kTileN;
        }
      };
      set_tile();
      const size_t x_blk = (size_t)a.x_rows * 64;         // elements between 64-column blocks
      auto issue_a = [&](int s) {
        uint8_t* dst = sA + s * C::kABytes;
        if (a.pair) {
          if (wsrc0) {
            bulk_load_hint(dst, wsrc0 + (size_t)kk * 64 * 64, C::kABytes / 2, &full[s], pol);
            bulk_load_hint(dst + C::kABytes / 2, wsrc1 + (size_t)kk * 64 * 64, C::kABytes / 2, &full[s], pol);
          } else {
            tma_load_2d_hint(dst, &a.wmap[0], &full[s], kk * kChunkK, wrow, pol);
            tma_load_2d_hint(dst + C::kABytes / 2, &a.wmap[1], &full[s], kk * kChunkK, wrow, pol);
          }
        } else if (wsrc0) {
          bulk_load_hint(dst, wsrc0 + (size_t)kk * kTileN * 64, C::kABytes, &full[s], pol);
        } else {
          tma_load_2d_hint(dst, wmap0, &full[s], kk * kChunkK, wrow, pol);
        }
      };
      auto issue_b = [&](int s, int kk_) {
        bulk_load(sB + s * C::kBBytes, a.x + (size_t)kk_ * x_blk, b_bytes, &full[s]);
      };
      auto advance = [&]() {
        if (++kk == a.kc) {
          kk = 0;
          ++w_tile;
          set_tile();
        }
      };
      // weights first: they do not depend on the previous kernel
      auto arm = [&](int s) {
        armed |= 1u << s;
        armed_odd ^= 1u << s;
      };
      const int kk0 = kk;
      for (int i = 0; i < npre; ++i) {
        arm(i);
        if (elect_one()) {
          mbar_arrive_expect_tx(&full[i], stage_bytes);
          issue_a(i);
        }
        __syncwarp();
        advance();
      }
      pdl_wait();
      for (int i = 0, k2 = kk0; i < npre; ++i) {
        if (elect_one()) issue_b(i, k2);
        __syncwarp();
        if (++k2 == a.kc) k2 = 0;
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
          mbar_arrive_expect_tx(&full[s], stage_bytes);
          issue_a(s);
          issue_b(s, kk);
        }
        __syncwarp();
        advance();
        if (++s == R) { s = 0; ph ^= 1u; }
      }
      if (lane == 0) pdl_trigger();
    }
  } else if (warp == 1) {
    // ---------------- MMA issuer ----------------
    {
      const uint32_t idesc = idesc_bf16(kTileN, 2 * n_tok);
      int s = 0;          // ring slot of the next unit
      uint32_t fph = 0;   // its 'full' phase parity
      int seg_i = 0;
      bool ok = true;
      for (int u = u0; u < u1 && ok;) {
        const int t = u / a.kc;
        const int ub = u, ue = (t + 1) * a.kc < u1 ? (t + 1) * a.kc : u1;
        const int ab = seg_i % C::kNumAcc;
        const uint32_t aph = (uint32_t)((seg_i / C::kNumAcc) & 1) ^ 1u;
        ok = __all_sync(0xffffffffu, mbar_wait(&acce[ab], aph, abort_flag));
        if (!ok) break;
        tc_fence_after();
        const uint32_t d = tmem + ab * C::kAccCols;
        for (; u < ue; ++u) {
          ok = __all_sync(0xffffffffu, mbar_wait(&full[s], fph, abort_flag));
          if (!ok) break;
          tc_fence_after();
          const uint64_t ad = sw128_desc(smem_u32(sA + s * C::kABytes));
          const uint64_t bd = sw128_desc(smem_u32(sB + s * C::kBBytes));
          if (elect_one()) {
#pragma unroll
            for (int k = 0; k < kChunkK / 16; ++k)
              umma_bf16(d, ad + 2 * k, bd + 2 * k, idesc, (u > ub || k > 0) ? 1u : 0u);
            umma_commit(&empty[s]);
            if (u + 1 == ue) umma_commit(&accf[ab]);
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
    // ---------------- epilogue (warps 2..5) ----------------
    pdl_wait();
    const int et = threadIdx.x - 64;
    const int q = warp & 3;
    const int fr = q * 32 + lane;
    int M = *a.m_dev;
    if (M > a.m_cap) {
      if (et == 0) set_status(a.status, ST_BAD_ROWS);
      M = a.m_cap;
    }
    int seg_i = 0;
    if (MODE != MODE_RESID && u0 < u1) epi_row_scale<TT>(a, et, M, S);
    for (int u = u0; u < u1;) {
      const int t = u / a.kc;
      const int ub = u, ue = (t + 1) * a.kc < u1 ? (t + 1) * a.kc : u1;
      u = ue;
      const int ab = seg_i % C::kNumAcc;
      // result-independent loads of a segment this CTA finishes (it starts
      // the tile), issued while the MMAs run
      EpiPre pre0 = {};
      if (ub == t * a.kc) pre0 = epi_pre<MODE>(a, t, 0, et, M);
      if (!mbar_wait(&accf[ab], (uint32_t)((seg_i / C::kNumAcc) & 1), abort_flag)) {
        if (et == 0) set_status(a.status, ST_TIMEOUT_EPI);
        *abort_flag = 1;
        break;
      }
      tc_fence_after();
      epi_bar();
      const uint32_t tbase = tmem + ab * C::kAccCols + ((uint32_t)(q * 32) << 16);
      if (!epi_segment_owned<TT, MODE>(a, t, ub, ue, u0, U, G, c, tbase, fr, et, M, S, pre0,
                                 reinterpret_cast<float*>(sA), (uint32_t)(C::kStages * C::kStageBytes), fx,
                                 fx_armed, abort_flag, bcast))
        break;
      tc_fence_before();
      mbar_arrive(&acce[ab]);
      epi_bar();
      ++seg_i;
    }
  }

  tc_fence_before();
  __syncthreads();
  if (*abort_flag) {
    // let this CTA's copies and MMAs in flight land before its memory goes away
    if (warp == 0 && lane == 0)
      for (int s = 0; s < C::kStages; ++s)
        if (armed >> s & 1u) mbar_drain(&full[s], (armed_odd >> s & 1u) ^ 1u);
    if (warp == 1) {
      if (elect_one()) umma_commit(drain);
      __syncwarp();
      mbar_drain(drain, 0);
    }
    // fx_armed: 1 + the staging round whose copies may be in flight
    if (threadIdx.x == 64 && *fx_armed) mbar_drain(fx, (uint32_t)((*fx_armed - 1) & 1));
    __syncthreads();
  }
  if (warp == 1) {
    __syncwarp();
    tc_fence_after();
    tmem_dealloc(tmem, C::kTmemCols);
  }
}

template <int TT, int MODE>
static cudaError_t launch_tt(const GemmArgs& a, int grid, cudaStream_t s, bool pdl) {
  static bool configured = false;
  const int smem = GemmCfg<TT>::kSmem;
  if (!configured) {
    cudaError_t e = cudaFuncSetAttribute(gemm_kernel<TT, MODE>, cudaFuncAttributeMaxDynamicSharedMemorySize, smem);
    if (e != cudaSuccess) return e;
    configured = true;
  }
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(192);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute attr[1];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = attr;
  cfg.numAttrs = pdl ? 1 : 0;
  return cudaLaunchKernelEx(&cfg, gemm_kernel<TT, MODE>, a);
}

template <int TT>
static cudaError_t launch_mode(const GemmArgs& a, int grid, cudaStream_t s, bool pdl) {
  switch (a.mode) {
    case MODE_QKV: return launch_tt<TT, MODE_QKV>(a, grid, s, pdl);
    case MODE_RESID: return launch_tt<TT, MODE_RESID>(a, grid, s, pdl);
    case MODE_SWIGLU: return launch_tt<TT, MODE_SWIGLU>(a, grid, s, pdl);
    default: return launch_tt<TT, MODE_LOGITS>(a, grid, s, pdl);
  }
}

void launch_gemm(const GemmArgs& a, int tt, int grid, cudaStream_t s, bool pdl) {
  const cudaError_t e = tt == 16 ? launch_mode<16>(a, grid, s, pdl) : launch_mode<64>(a, grid, s, pdl);
  if (e != cudaSuccess) throw e;
}

}  // namespace pard
