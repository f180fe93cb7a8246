// Host-side structures shared by the translation units of libpard.
#pragma once

#include <cuda.h>
#include <cuda_bf16.h>
#include <cuda_runtime.h>
#include <stdint.h>

#include <string>
#include <vector>

#include "../../include/pard.h"

namespace pard {

constexpr int kTileN = 128;     // weight rows per UMMA tile (MMA M)
constexpr int kChunkK = 64;     // K elements per pipeline stage (one 128-byte swizzle row)
constexpr int kEpiTok = 16;     // tokens per epilogue pass (32 TMEM columns: hi/lo pairs)
constexpr int kMaxSeg = 3;

enum GemmMode : int { MODE_QKV = 0, MODE_RESID = 1, MODE_SWIGLU = 2, MODE_LOGITS = 3 };

// Per-call scalars kept in device memory, so that captured launches read the
// current call's values.
struct CallArgs {
  uint64_t seed;
  uint64_t step;
  float temp;
  int32_t sample;
  int32_t K;
  int32_t pad;
};

struct GemmArgs {
  CUtensorMap wmap[kMaxSeg];  // weights (A operand), row-major or packed; pair mode: [0] gate, [1] up, 64-row boxes
  const __nv_bfloat16* wpk[kMaxSeg];  // packed weights (null: wmap is row-major)
  const __nv_bfloat16* x;     // packed activations (B operand), a hi and a lo row per token (xpk)
  int x_rows;                 // rows of the activation buffer (2 x row capacity)
  int nseg;
  int seg_tile0[kMaxSeg + 1]; // prefix sums of tiles per segment
  int seg_rows[kMaxSeg];      // rows of each segment
  int pair;
  int w_tiles, tok_tiles, kc; // tok_tiles: 1 in the narrow GEMM
  int n_tok;                  // token rows a tile's MMA covers (multiple of 8, <= the tile): a pass of fewer rows
                              // loads and multiplies only those
  int m_early;                // wide GEMM: m_dev was written two or more launches back, so it is read before the
                              // PDL wait, and the token tiles are laid out for the rows there are
  int mode;
  int m_cap;                  // row capacity of the activation/output buffers
  const int* m_dev;           // runtime row count
  float* partials;
  int* counters;              // split-K arrival masks: 64-bit word per output tile, zero between launches
  uint32_t* status;
  int max_pairs;              // wide GEMM: pairs the GPU holds at once
  // RMS row scale applied after the reduction (null: none)
  const float* ssq_in;
  int ssq_tiles;
  float inv_d, eps;
  // MODE_RESID
  float* h;
  int h_ld;
  float* ssq_out;
  __nv_bfloat16* x_next;      // packed, x_rows rows
  const __nv_bfloat16* g_next;
  // MODE_QKV
  float* q_out;
  int q_ld;
  __nv_bfloat16* kcache;
  __nv_bfloat16* vcache;
  const int* page_table;
  int pt_ld;
  const int* row_pos;
  const int* row_seq;
  const float2* rope;
  int hd, hkv, page_size, n_pages;
  // MODE_LOGITS
  float* logits;              // [rows_out][vocab] or null
  float* logits_out;          // the caller's copy of them (null: none; any 4-byte alignment)
  const int* row_out;         // row -> output row, -1: none (null: identity)
  const int* row_gi;          // row -> Philox row index for Gumbel draws, -1: none
  float4* stats;              // [w_tiles][m_cap] {max, sumexp(T), gumbel best, 0}
  int2* stats_i;              // [w_tiles][m_cap] {argmax, gumbel argmax}
  int vocab;
  int gumbel_stream;
  const CallArgs* call;
};

struct AttnArgs {
  const float* q;             // [rows][hq*hd] fp32, post-RoPE
  int q_ld;
  const __nv_bfloat16* kcache;
  const __nv_bfloat16* vcache;
  const int* page_table;
  int pt_ld;
  const int* row_pos;
  const int* seq_row0;        // [B+1] first row of each sequence in this pass
  int rows_per_seq;           // > 0: every sequence has this many rows (row0 = b x it), seq_row0 unread
  const int* m_dev;
  int batch;
  int hq, hkv, hd, n_pages;   // pages of kAttnPage tokens
  int row_blocks;             // row blocks per sequence (grid.y / ...)
  int n_split;                // key splits
  int prompt;                 // a prompt pass: units are launched longest first
  int nbuf;                   // K/V chunk buffers a CTA keeps (4, or 2 for ragged or crowded passes)
  float scale;                // log2(e) / sqrt(hd)
  __nv_bfloat16* x_out;       // packed [2*rows][hq*hd] hi/lo
  int x_rows;
  uint32_t* status;
  uint32_t* paths;            // combine paths taken (kAttnPath* bits, OR-ed; null: not recorded)
};

// Attention combine paths recorded in AttnArgs::paths: push or pull combine
// of the key splits, and bit kAttnPathSplit0 + n for clusters of n CTAs.
constexpr uint32_t kAttnPathPush = 1u << 0;
constexpr uint32_t kAttnPathPull = 1u << 1;
constexpr uint32_t kAttnPathRing2 = 1u << 2;  // the two-buffer K/V ring variant ran
constexpr int kAttnPathSplit0 = 3;


// Per-sequence decode state, in the workspace.
struct DevState {
  int* n;          // [B] tokens so far, the pending one included (target cache holds n-1)
  int* pend_cnt;   // [B] draft tokens waiting to be fed (a+1 after a commit)
  int* pend;       // [B][kmax+1]
  int* gen;        // [B] tokens generated (counted toward max_new)
  int* max_new;    // [B]
  int* done;       // [B]
  int* d;          // [B][kmax] current candidates
  float2* dnorm;   // [B][kmax] draft row (max logit, sum exp) at the draft temperature
  int* samp_a;     // [B] sampling: first rejected index (K: all accepted)
  float4* samp_norm;  // [B] (max_y, S_y, max_z, S_z) of the rejected row
  float2* samp_part;  // [B][kResampleSplit] (score, index) partial draws
  int* samp_cnt;      // [B]
  int kmax;        // row pitch of pend (kmax+1) and d (kmax)
};

constexpr int kResampleSplit = 32;

struct RowPlan {     // row layout of one forward pass
  int* row_tok;
  int* row_pos;
  int* row_seq;
  int* row_out;      // logits output row or -1
  int* row_gi;       // Philox row index for Gumbel draws or -1
  int* seq_row0;     // [B+1]
  int* m_dev;
};

struct EmbedArgs {
  int mode;          // EMB_PREFILL, EMB_DRAFT, EMB_VERIFY, EMB_DRAFT_SEQ
  int batch, K, mask_id, vocab, d;
  int seq_i;         // EMB_DRAFT_SEQ: pass index i (0: the pending tokens; i > 0: candidate i-1)
  const int* mask_ids;  // EMB_DRAFT: id of mask m_k per offset k (null: mask_id for all)
  const __nv_bfloat16* embed;
  const __nv_bfloat16* gain0;  // first layer's attention-norm gain
  const int* tokens;           // prefill: the prompts, concatenated
  const int* plen;             // prefill: their lengths
  int pf_row0, pf_rows;        // prefill: this pass's first row of the concatenation, its rows,
  int pf_seq, pf_nseq;         // its first sequence and the number of sequences it touches
  const int* d_in;             // verify: candidates to feed ([B][K])
  DevState st;
  RowPlan rp;
  float* h;
  __nv_bfloat16* x;            // packed, 2 * m_cap rows
  float* ssq;
  int m_cap;
  uint32_t* status;
  CallArgs call;               // the call's scalars, written to *call_out for the pass's other kernels (null: not)
  CallArgs* call_out;
};
enum { EMB_PREFILL = 0, EMB_DRAFT = 1, EMB_VERIFY = 2, EMB_DRAFT_SEQ = 3 };

struct SelectArgs {
  int mode;          // SEL_DRAFT, SEL_FIRST, SEL_NORM_ONLY, SEL_DRAFT_SEQ, SEL_DRAFT_GIVEN
  int batch, K, w_tiles, m_cap, vocab;
  int seq_i;         // SEL_DRAFT_SEQ: the candidate this pass picks
  const float4* stats;
  const int2* stats_i;
  const CallArgs* call;
  DevState st;
  const int* seq_row0;
  int* out;          // draft: [B][K]; first token: [B]
  const int* plen;   // first token: prompt lengths
  int n_new;
};
// SEL_DRAFT_GIVEN: candidates from given draft logits rows b * K + i
enum { SEL_DRAFT = 0, SEL_FIRST = 1, SEL_NORM_ONLY = 2, SEL_DRAFT_SEQ = 3, SEL_DRAFT_GIVEN = 4 };

struct AcceptArgs {
  int batch, K, w_tiles, m_cap, vocab;
  const float4* stats;
  const int2* stats_i;
  const float* logits;     // [B][K+1][V] (sampling)
  const float* dlogits;    // [B][K][V] (sampling)
  CallArgs call;
  DevState st;
  const int* page_table;
  int pt_ld, page_size;
  int* accept_len;
  int* emitted;
  int* kv_slots;
  int* n_emit;
  uint32_t* status;        // sticky device status word (null: none)
  const float4* dstats;    // sampling: tile statistics of the draft rows b K + i (null: their normalisers are in st.dnorm)
  int d_m_cap;
};

// Statistics of given logits in tiles of kGivenTile entries, for the
// acceptance that keeps its scratch in a fixed array (noalloc.cu).
constexpr int kGivenTile = 2048;
struct GivenArgs {
  const float* y;          // [rows_t][vocab]
  const float* z;          // [rows_d][vocab] (rows_d = 0: none)
  int rows_t, rows_d, m_cap_t, m_cap_d, vocab, tiles;
  int vec;                 // both arrays are 16-byte aligned
  int sample;
  float4 *stats_t, *stats_d;
  int2* stats_it;
  CallArgs call;
  DevState st;             // reset by block (0, 0)
  const int* d;            // [batch][K] candidates
  int batch, K;
};

constexpr int kMaxGemmTiles = 32768;  // output tiles (weight tile x token tile) of one GEMM launch
constexpr int kMaxQVRows = 64;          // query vectors of one attention work unit
constexpr int kMaxAttnSplit = 16;       // key splits (CTAs of one cluster) of one attention work unit

// Wide GEMM (gemm_wide.cu; passes of more than 64 rows): tiles of 256 weight
// rows and at most kWideTok tokens, multiplied by a pair of CTAs.
constexpr int kWideTok = 256;
// A split tile's mask word: a bit per contributor that has stored its partial,
// a bit per contributor whose given-up share nobody has claimed, and above them the number
// of finished shares.
constexpr int kWideContrib = 28, kWideReadShift = 2 * kWideContrib;
// A contributor waits this long for the others of its tile before it gives its
// share up to one that arrives later (usually all arrive within 10 us): every
// CTA of a launch ends in bounded time without the others, as it must where
// launches of two streams share the SMs and neither is wholly on them.
constexpr int kShareWaitNs = 100000;
// Units of the QKV projection that one accumulator sums before the epilogue
// adds it up in fp32 registers (kWideChainShort where K has kWideChain or
// fewer): the tensor cores truncate at every accumulation, and keys and values
// are rounded to bf16 afterwards, so that small differences become whole
// roundings.  Error against 64 bits: 6 layers of the 8B widths over a 512-row
// prompt 1.37e-3 on 64-token tiles; here 1.27e-3 without a limit, 1.22e-3 at 32
// units, 1.15e-3 at 16 (the pass 1.4% slower); 2 layers of the 70B widths
// 1.53e-3, then 1.40e-3, 1.22e-3 and 1.14e-3; the draft pass of 8 sequences on
// the 1B widths 1.007e-3, here 1.012e-3 in even shares of ten units, 0.994e-3
// at 8.  Cutting the other projections' sums to 16 units changed no error and
// made a 512-row pass 7% slower.
constexpr int kWideChain = 32, kWideChainShort = 8;
constexpr int kWideMaxRows = 2048;  // rows of one pass (64 sequences x 2 x 16)
constexpr int kWideBoxL = 32, kWideBoxS = 16;
struct WideArgs {
  GemmArgs g;              // packed matrices: wmap holds the packed array as a tensor of 128-byte rows
  CUtensorMap x[3];        // the activation buffer as one, boxes of g.n_tok, kWideBoxL and kWideBoxS rows
  int share_wait_ns;       // kShareWaitNs, or what a test asks for
};
// Token tiles of a pass of m rows, all of the same size (a multiple of 16).
__host__ __device__ inline void wide_tiles(int m, int& tiles, int& n_tok) {
  tiles = (m + kWideTok - 1) / kWideTok;
  n_tok = ((m + tiles - 1) / tiles + 15) / 16 * 16;
}
// How T tiles of kc units (64 columns of K) are shared out over at most
// max_pairs pairs: evenly by units (a pair may begin and end inside a tile),
// or with tiles whole, or each cut into the same number of parts.  Finishing
// a split tile costs a launch about kWideExchange units of time on top of its
// epilogue, and a pair with two split tiles kWideSecond more than with one, so
// the even split has to save more than that.  Measured (batch-16 draft and
// verify of 8 layers, 512-row prompt; us): always even 1673 / 1497 / 18007,
// with equal parts 1643 / 1426 / 17422, with whole tiles too 1549 / 1384 / 16785
// at (40, 8); 1566 / 1444 / 16999 at (12, 4), 1562 / 1387 / 16899 at (64, 8).
// Fewer tiles than pairs, and more than half as many, stay whole up to
// kWideWhole units, as the 1B draft's gate/up does; the even split makes its
// passes of more than 64 rows 5% to 8% slower.  With the limit above 64 units
// the QKV projection of the 8B widths would sum two pieces of kWideChain units
// a tile instead of even shares of 20: 1% to 2% off a 512-row prompt, but its
// error, and a batch-16 verify pass's, 3% to 4% larger.
constexpr int kWideExchange = 40, kWideSecond = 8, kWideWhole = 32;
struct WideSplit {
  int pairs;
  bool tiles;  // ranges are whole tiles
};
__host__ __device__ inline WideSplit wide_split(int T, int kc, int max_pairs) {
  // at least four units (64 KB of weights a CTA) a pair, and at most kWideContrib pairs to a tile
  const int least = kc > 4 * (kWideContrib - 2) ? (kc + kWideContrib - 3) / (kWideContrib - 2) : 4;
  const int most = T * kc / least < 1 ? 1 : (T * kc / least < max_pairs ? T * kc / least : max_pairs);
  const int even = (T * kc + most - 1) / most;
  if (T >= most) return {most, (T + most - 1) / most * kc <= even + kWideExchange};
  const int parts = most / T;
  if (parts == 1 && kc <= kWideWhole) return {T, true};
  if (parts > 1 && (kc + parts - 1) / parts <= even + kWideSecond) return {T * parts, false};
  return {most, false};
}

// launchers (gemm.cu, gemm_wide.cu, attention.cu, misc.cu)
void launch_embed(const EmbedArgs& a, int grid, cudaStream_t s, bool pdl);
constexpr int kMaxBatch = 64;
struct GatherArgs {            // row src[i] of x and of its sums of squares to row dst0 + i (src[i] < 0: none)
  const __nv_bfloat16* x;
  const float* ssq;
  __nv_bfloat16* xg;
  float* ssqg;
  int x_rows, xg_rows, ssq_tiles, m_cap_src, m_cap_dst, d, dst0;
  int src[kMaxBatch];
};
void launch_gather_rows(const GatherArgs& a, int n, cudaStream_t s, bool pdl);
void launch_pack(const __nv_bfloat16* tmp, __nv_bfloat16* w, int R, int K, int nblocks, bool unpack, cudaStream_t s);
void launch_select(const SelectArgs& a, cudaStream_t s, bool pdl);
void launch_given_stats(const GivenArgs& a, cudaStream_t s);
void launch_accept_greedy(const AcceptArgs& a, cudaStream_t s, bool pdl);
void launch_accept_sample(const AcceptArgs& a, cudaStream_t s, bool pdl);
void launch_row_stats(const float* logits, int rows, int vocab, int w_tiles, int m_cap, const CallArgs* call,
                      int gumbel_stream, int rows_per_seq, float4* stats, int2* stats_i, cudaStream_t s);
void launch_set_call(CallArgs* dst, CallArgs v, cudaStream_t s, bool pdl);
void launch_read_kv(const __nv_bfloat16* kc, const __nv_bfloat16* vc, const int* page_table_row, const int* pos, int n,
                    int hkv, int hd, int page_size, __nv_bfloat16* ok, __nv_bfloat16* ov, cudaStream_t s);

void launch_stalled_wait(uint32_t* status, cudaStream_t s);
constexpr int kCodMaxN = 4096;  // rows per subtask of one COD sample
void launch_cod(int N, int K, double r, double r_min, uint64_t seed, uint64_t sample_id, int32_t* keep,
                int32_t* counts, cudaStream_t s);
void launch_gemm(const GemmArgs& a, int tt, int grid, cudaStream_t s, bool pdl);
int gemm_wide_max_pairs(int sm);  // pairs an idle GPU holds at once: a launch has no more
void launch_gemm_wide(const WideArgs& a, int pairs, cudaStream_t s, bool pdl);
void launch_attention(const AttnArgs& a, int grid_x, cudaStream_t s, bool pdl);
int attention_rows_per_block(int group);

}  // namespace pard
