// Adaptive number of selected blocks: an extension, NOT in the paper (which always keeps k blocks).  It applies the
// paper's dropped mass tau (the normalised block mass outside the kept set, Background, before Eq. prop-gqa) to the
// group score of Eq. prop-gqa:
//
//   k_adapt = the smallest k such that the k largest candidate scores hold at least (1 - tau) of the candidates'
//             total score, clamped to [k_min, topk] and to the number of candidates.
//
// The kernel trims an existing selection in place: the top-`topk` blocks of cobs_score_select (ascending index) and
// the scores the same call wrote.  One CTA per (sequence, KV head), four threads or more per selected block; topk <= 128.
// Sums are taken in double precision in a fixed order (no atomics), so the result does not depend on scheduling.
// It is all latency: two dependent reads, the ranks (each thread compares with a quarter of the others), the prefix
// sums of the ranked scores by one warp.  (Scoring, this and attention over 85 of 512 blocks, 32 units: 37.9 us; 43.8 with
// one thread adding up the ranked scores and 128 threads with a barrier per level of the total.)
#include "common.cuh"

namespace cobs {

namespace {

constexpr int kAThreads = 4 * COBS_MAX_TOPK;              // at most; a launch has four threads per block that may be selected

__global__ void __launch_bounds__(kAThreads) adaptive_trim_kernel(Params p, float tau, int k_min) {
  __shared__ double s_part[kAThreads / 32];
  __shared__ __align__(16) double s_sorted[COBS_MAX_TOPK];
  __shared__ float2 s_item[COBS_MAX_TOPK];               // score, id
  __shared__ int s_warp[kAThreads / 32];
  __shared__ int s_k;
  pdl_begin();
  const int u = blockIdx.x, tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, item = tid >> 2, quarter = tid & 3;
  const int nthr = blockDim.x, nw = nthr >> 5;
  const int b_idx = u / p.Hkv;
  const float *sc = p.scores + (size_t)u * p.NB;
  int32_t *out = p.sel_idx + (size_t)u * p.topk;
  const int T = tokens_of(p.seq_lens, b_idx), cnt = p.sel_cnt[u];
  int id = (item < p.topk) ? out[item] : -1;
  const int n_sum = min(T / p.L, p.NB);
  const int n_cand = min(window_start(T, p.window, p.L) / p.L, n_sum);
  const int k = min(min(cnt, p.topk), n_cand);
  // ---- the selected block of this thread and its three neighbours ------------------------------------------------
  float my = 0.f;
  if (item >= k) id = -1;
  else if (id < 0 || id >= n_cand) { if (quarter == 0) report(p.status, COBS_ERR_BOUNDS); id = -1; }
  else my = sc[id];
  // ---- total score of the candidates ------------------------------------------------------------------------------
  double part = 0.0;
  for (int b = tid; b < n_cand; b += nthr) part += (double)sc[b];
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) part += __shfl_xor_sync(0xffffffffu, part, o);
  if (lane == 0) s_part[warp] = part;
  if (quarter == 0) s_item[item] = make_float2(my, __int_as_float(id));
  const int valid = __syncthreads_count(quarter == 0 && id >= 0);
  // ---- rank among the selected: larger score first, lower index on ties ------------------------------------------
  int rank = 0;
#pragma unroll 4
  for (int j = quarter; j < k; j += 4) {
    const float2 o = s_item[j];
    const int oj = __float_as_int(o.y);
    rank += (oj >= 0 && (o.x > my || (o.x == my && oj < id))) ? 1 : 0;
  }
  rank += __shfl_xor_sync(0xffffffffu, rank, 1);
  rank += __shfl_xor_sync(0xffffffffu, rank, 2);
  if (quarter == 0 && id >= 0) s_sorted[rank] = (double)my;
  __syncthreads();
  if (warp == 0) {
    double total = (lane < nw) ? s_part[lane] : 0.0;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) total += __shfl_xor_sync(0xffffffffu, total, o);
    total = __shfl_sync(0xffffffffu, total, 0);
    const double need = (1.0 - (double)tau) * total;
    double c[4], sum = 0.0;                              // four ranks per lane
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      if (4 * lane + i < valid) sum += s_sorted[4 * lane + i];
      c[i] = sum;
    }
    double inc = sum;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const double t = __shfl_up_sync(0xffffffffu, inc, o);
      if (lane >= o) inc += t;
    }
    double before = __shfl_up_sync(0xffffffffu, inc, 1);
    if (lane == 0) before = 0.0;
    unsigned first = (unsigned)valid;
#pragma unroll
    for (int i = 3; i >= 0; --i)
      if (4 * lane + i < valid && before + c[i] >= need) first = 4 * lane + i + 1;
    const int ka = max((int)__reduce_min_sync(0xffffffffu, first), min(k_min, valid));
    if (lane == 0) s_k = min(ka, valid);
  }
  __syncthreads();
  const int ka = s_k;
  // ---- keep the ka best, in ascending index order (the order they came in) ------------------------------------------
  const bool keep = quarter == 0 && id >= 0 && rank < ka;
  const unsigned m = __ballot_sync(0xffffffffu, keep);
  if (lane == 0) s_warp[warp] = __popc(m);
  __syncthreads();
  int pos = __popc(m & ((1u << lane) - 1u));
#pragma unroll
  for (int w = 0; w < kAThreads / 32; ++w) pos += (w < warp) ? s_warp[w] : 0;      // (warp < nw)
  if (keep) out[pos] = id;                               // (every thread read its block before the first barrier)
  for (int i = ka + tid; i < p.topk; i += nthr) out[i] = -1;
  if (tid == 0) p.sel_cnt[u] = ka;
}

}  // namespace

cudaError_t launch_adaptive_trim(const Params &p, float tau, int k_min, cudaStream_t stream) {
  // four threads per block that may be selected, and no fewer than add up the candidates of a long sequence quickly (1 024 units of 16
  // blocks, 32 kept, L2 flushed: 21.2 us with 512 threads, 15.5 with 128)
  const int threads = min(kAThreads, max((4 * p.topk + 31) / 32 * 32, min(p.NB, kAThreads) / 32 * 32));
  return launch_chained(adaptive_trim_kernel, dim3(p.B * p.Hkv), dim3(threads), 0, stream, p, tau, k_min);
}

}  // namespace cobs
