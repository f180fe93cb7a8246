// Conditional drop-token (COD) data construction (Section 3.2 and the
// appendix algorithm): which rows of the mask-token subtasks 2..K of one
// training sample are kept.
//
// Subtask k keeps n_k = round(N max(r^(k-1), r_min)) rows, chosen at random
// among its candidates: row j (position j, fed m_{k-2}, labelled x_{j+1}) is a
// candidate when its attention chain is complete -- subtask 2 rows always,
// subtask k >= 3 rows when row j-1 of subtask k-1 is kept (the integrity of
// prefix key-value states); rows j < k-2 have no chain.  The random choice
// keeps the candidates with the n_k smallest Philox words (stream 3, step =
// sample id, row k, v = j), ties to the lower j, so it is reproducible.
//
// One CTA per sample; subtasks run in order (each depends on the previous
// one's flags, kept in shared memory).  What bounds it is the chain of block
// synchronisations, K - 1 subtasks of five each.  Within a subtask the
// n_k-th smallest key is found by one histogram over the keys' top 12 bits
// (4096 bins for at most 4096 keys: the words are uniform, so the bin the
// threshold falls into holds a key or two) and a rank count among that bin's
// members alone, instead of every candidate counting over the whole subtask
// (2048 rows, K = 8: 18.8 us, 971 us with the O(n^2) count on one SM).  Thread t
// holds rows 4t .. 4t+3, the four words of one Philox block.
#include "common.cuh"
#include "internal.h"

namespace pard {

constexpr int kCodThreads = 1024;
constexpr int kCodBins = 4096;
constexpr uint32_t kStreamCod = 3;
static_assert(kCodThreads * 4 == kCodMaxN && kCodThreads * 4 == kCodBins, "four rows and four bins a thread");

__global__ void __launch_bounds__(kCodThreads) cod_kernel(int N, int K, double r, double r_min, uint64_t seed,
                                                          uint64_t sample_id, int32_t* keep, int32_t* counts) {
  __shared__ int4 s_hist[kCodBins / 4];          // keys per bin of the subtask at hand; zero between subtasks
  __shared__ uint32_t s_lkey[kCodMaxN];          // keys and rows of the threshold bin's members
  __shared__ uint16_t s_lrow[kCodMaxN];
  __shared__ uint32_t s_keep[kCodThreads];       // the previous subtask's flags, one byte a row
  __shared__ int s_warp[kCodThreads / 32];
  __shared__ int s_n[64];
  __shared__ int s_bin, s_need, s_total, s_members;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  int* hist = reinterpret_cast<int*>(s_hist);
  const int j0 = 4 * tid;
  const bool vec = N % 4 == 0 && (reinterpret_cast<uintptr_t>(keep) & 15) == 0;
  s_hist[tid] = make_int4(0, 0, 0, 0);
  if (tid == 0) counts[0] = N;
  // rows kept by each subtask, a thread a subtask: the double-precision unit is
  // too narrow for 32 warps to compute them in every subtask
  if (tid < K - 1) {
    double g = 1.0;
    for (int i = 0; i <= tid; ++i) g *= r;
    s_n[tid] = (int)floor((double)N * (g > r_min ? g : r_min) + 0.5);
  }
  __syncthreads();
  for (int k = 2; k <= K; ++k) {
    const int n = s_n[k - 2];
    // flags of rows j0 - 1 .. j0 + 2 of subtask k - 1, a byte each
    uint32_t prev = 0x01010101u;
    if (k > 2) prev = (s_keep[tid] << 8) | (tid > 0 ? s_keep[tid - 1] >> 24 : 0u);
    const U4 w = philox4x32_10(U4{(uint32_t)tid, (kStreamCod << 16) | ((uint32_t)k & 0xFFFFu), 0u, (uint32_t)sample_id},
                               (uint32_t)seed, (uint32_t)(seed >> 32));
    const uint32_t key[4] = {w.x, w.y, w.z, w.w};
    bool valid[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      valid[e] = j0 + e < N && j0 + e >= k - 2 && ((prev >> (8 * e)) & 1u) != 0;
      if (valid[e]) atomicAdd(&hist[key[e] >> 20], 1);
    }
    if (tid == 0) { s_bin = kCodBins; s_need = 0; s_members = 0; }  // bin 4096: every candidate is below the threshold
    __syncthreads();
    // exclusive prefix of the bins, four a thread
    const int4 h = s_hist[tid];
    s_hist[tid] = make_int4(0, 0, 0, 0);
    const int mine = h.x + h.y + h.z + h.w;
    int inc = mine;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += v;
    }
    if (lane == 31) s_warp[warp] = inc;
    __syncthreads();
    const int wv = s_warp[lane];
    int winc = wv;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int v = __shfl_up_sync(0xffffffffu, winc, o);
      if (lane >= o) winc += v;
    }
    int before = inc - mine + __shfl_sync(0xffffffffu, winc - wv, warp);  // candidates in bins below 4 tid
    if (tid == kCodThreads - 1) s_total = before + mine;
    const int hb[4] = {h.x, h.y, h.z, h.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      if (before <= n && n < before + hb[e]) { s_bin = 4 * tid + e; s_need = n - before; }
      before += hb[e];
    }
    __syncthreads();
    const int bin = s_bin, need = s_need;
#pragma unroll
    for (int e = 0; e < 4; ++e)
      if (valid[e] && (int)(key[e] >> 20) == bin) {
        const int at = atomicAdd(&s_members, 1);
        s_lkey[at] = key[e];
        s_lrow[at] = (uint16_t)(j0 + e);
      }
    __syncthreads();
    const int members = s_members;
    int kept[4];
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int kb = (int)(key[e] >> 20);
      kept[e] = valid[e] && kb < bin ? 1 : 0;
      if (valid[e] && kb == bin) {
        int rank = 0;
        for (int i = 0; i < members; ++i)
          rank += (s_lkey[i] < key[e] || (s_lkey[i] == key[e] && (int)s_lrow[i] < j0 + e)) ? 1 : 0;
        kept[e] = rank < need ? 1 : 0;
      }
    }
    s_keep[tid] = (uint32_t)kept[0] | ((uint32_t)kept[1] << 8) | ((uint32_t)kept[2] << 16) | ((uint32_t)kept[3] << 24);
    int32_t* out = keep + (size_t)(k - 2) * N + j0;
    if (vec && j0 < N) {
      *reinterpret_cast<int4*>(out) = make_int4(kept[0], kept[1], kept[2], kept[3]);
    } else {
#pragma unroll
      for (int e = 0; e < 4; ++e)
        if (j0 + e < N) out[e] = kept[e];
    }
    if (tid == 0) counts[k - 1] = n < s_total ? n : s_total;
    __syncthreads();  // the flags are read, and the bin, list and counters rewritten, by the next subtask
  }
}

void launch_cod(int N, int K, double r, double r_min, uint64_t seed, uint64_t sample_id, int32_t* keep,
                int32_t* counts, cudaStream_t s) {
  cod_kernel<<<1, kCodThreads, 0, s>>>(N, K, r, r_min, seed, sample_id, keep, counts);
  const cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) throw e;
}

}  // namespace pard
