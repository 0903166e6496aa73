// The decode step with one thread-block cluster per (sequence, KV head): block scoring, top-k selection, block-sparse
// attention and the split-KV merge (steps (b), (c), (d)).
//
// What bounds a step is, up to some tens of MB, not its bytes but the chain score -> log-sum-exp -> group score -> top-k ->
// page addresses -> attention -> merge.  A unit (one KV head of one sequence) is the scope of that whole chain, so here a
// unit belongs to one cluster of C CTAs with W warps each: the hand-offs are cluster barriers and distributed shared memory
// (about a microsecond each less than a counter in global memory with its fences), there is nothing to poll, no counter to
// clear, no order in which CTAs must run, and a grid of any size.
//
//   query    each CTA fetches its unit's 2 KB of query once, into shared memory (the caller's may lie in host memory)
//   score    the unit's 16-block chunks are dealt to the cluster's warps in contiguous ranges; a warp leaves e per block and
//            head in its CTA's buffer and keeps a running (max, sum) per head
//   lse      the CTAs exchange their (max, sum) pairs                                        (cluster barrier)
//   scores   every CTA turns its own e into group scores and writes them into all CTAs       (cluster barrier)
//   select   every CTA selects for itself, from its own copy of the scores: nothing to hand over
//   attend   the unit's 16-token groups are dealt to the cluster's warps; partials meet in shared memory, first within the
//            CTA, then across the cluster                                                    (cluster barrier)
//
// Measured against the persistent kernel with counters in global memory that this one replaced (a step among others, us):
// one sequence of 32k 31.9 -> 20.5, four of 32k with a subspace 37.0 -> 26.7, sixteen of 128k 115 -> 98 (80 % of the measured
// copy rate: 512 MB), 24 ragged ones of 12k (375 blocks, not a multiple of four: three launches before) 156 -> 45, fp32
// summaries at 2k (three launches before) 36.4 -> 18.5.  With programmatic dependent launch and the early end of the top-k
// search: 17.1, 23.4, 95-98, 43.5, 16.9; with the attention's accumulators apart and the query in shared memory: 16.1, 20.9,
// 93, 35.2, 16.4; with the merge by stores and the first loads together and the window fetched ahead: 14.6, 19.1, 91, 34.4, 13.3.  (One exchange of pairs and
// e, every CTA computing all scores, instead of pairs first and scores after: 15.4, 20.3, 93, 35.1, 13.6: not kept.)
//
// Data movement.  Every stream a warp consumes goes global -> shared into a ring that belongs to that warp alone.  Scoring: a
// chunk is three contiguous pieces of the summary arrays, fetched by three bulk copies (cp.async.bulk, completion on an
// mbarrier) issued by one lane, two stages.  Attention: K and V of a 16-token group share a stage of a three-stage cp.async ring
// (XOR-swizzled 16-byte chunks, read back with ldmatrix / ldmatrix.trans).
//
// Arithmetic.  mma.sync m16n8k16 with fp32 accumulation throughout:
//   scoring   rows = 16 block means, or factor i of 16 blocks; columns = the G query heads.  A thread owns two blocks (rows
//             gid, gid + 8), so all results of a block land in one thread.  bf16 rows multiply the raw bf16 query (exact
//             products); FP4 codes become f16 by the hardware conversion and multiply the query scaled by a per-head power
//             of two (exact in f16), or an f16 high + low split of the fp32 subspace query; fp32 rows are split into three
//             bf16 terms (24 bits), and so is the subspace query against them.
//   attention S^T = q K^T with the heads as rows (zero padded to 16) and 8 tokens as columns; the S accumulators are the A
//             fragments of P V as they sit in registers; P = bf16 high + low.
#include <atomic>
#include <type_traits>

#include "step_common.cuh"

namespace cobs {

// Phase times (the build with -DCOBS_TIMING, `python -m paper_2607_09052_b200.build --timing`, which makes
// libcobs_timing.so; read by `bench.py --phase-times`): thread 0 of every CTA records the global timer at the phase
// boundaries.  The production library carries none of this.
#ifdef COBS_TIMING
__device__ unsigned long long g_stamps[8][4096];
#define COBS_STAMP(k)                                                                   \
  do {                                                                                  \
    if (threadIdx.x == 0 && blockIdx.x < 4096) {                                        \
      unsigned long long t_;                                                            \
      asm volatile("mov.u64 %0, %%globaltimer;" : "=l"(t_));                            \
      g_stamps[k][blockIdx.x] = t_;                                                     \
    }                                                                                   \
  } while (0)
#else
#define COBS_STAMP(k) do { } while (0)
#endif

namespace {

constexpr int kMaxW = 8;                                     // warps per CTA: 8 (one CTA per SM) or 4 (two)
constexpr int kMaxC = 16;                                    // CTAs per cluster
constexpr int kStage = 13056;                                // scoring stage: means + factor rows + scales of a 16-block chunk
constexpr int kAttStages = 3;
constexpr int kAttStage = 2 * 16 * 128 * 2;                  // K + V of one 16-token group, D = 128
constexpr int kTable = 128;                                  // 16-token groups whose addresses a warp resolves at a time
constexpr int kRing = 2 * kStage;                            // 26112 bytes per warp
static_assert(kAttStages * kAttStage + kTable * 8 <= kRing, "the attention ring and its table must fit");
constexpr int kSmemOne = (227 - 9) * 1024;                   // dynamic shared memory of a CTA that has an SM to itself (static: 8960 bytes)
constexpr int kSmemTwo = 106752;                             // of two CTAs per SM (four warps each)
constexpr int kQRow = 128 + 8;                               // row stride of the query in shared memory (no bank conflicts)
constexpr int kMaxKeys = 24576;                              // score keys that fit over the rings of four warps

// how a launch lays out a CTA (chosen on the host, see launch_t)
struct Plan {
  int W, C;
  int u0;                                                    // the launch's first unit
  int key_off;                                               // byte offset of the score keys in dynamic shared memory
  int e_off;                                                 // of the e buffer, or -1: it is in the workspace
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }
__device__ __forceinline__ uint32_t mapa(uint32_t addr, int rank) {
  uint32_t r;
  asm("mapa.shared::cluster.u32 %0, %1, %2;\n" : "=r"(r) : "r"(addr), "r"(rank));
  return r;
}
__device__ __forceinline__ void st_cluster(uint32_t addr, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;\n" ::"r"(addr), "f"(v) : "memory");
}
__device__ __forceinline__ void st_cluster4(uint32_t addr, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};\n" ::"r"(addr), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void st_cluster2(uint32_t addr, float2 v) {
  asm volatile("st.shared::cluster.v2.f32 [%0], {%1, %2};\n" ::"r"(addr), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void cluster_arrive() { asm volatile("barrier.cluster.arrive.release;\n" ::: "memory"); }
__device__ __forceinline__ void cluster_wait() { asm volatile("barrier.cluster.wait.acquire;\n" ::: "memory"); }

__device__ __forceinline__ void bulk_prefetch_l2(const void *src, uint32_t bytes) {
  asm volatile("cp.async.bulk.prefetch.L2.global [%0], %1;\n" ::"l"(src), "r"(bytes) : "memory");
}

// running (max, sum of exponentials) of one head
struct Run { float m, s; };
__device__ __forceinline__ void run_add(Run &r, float a, float b) {
  const float m = fmaxf(r.m, fmaxf(a, b));
  r.s = r.s * __expf(r.m - m) + (__expf(a - m) + __expf(b - m));
  r.m = m;
}

// the warp's pair of every head, from the runs of threads that hold heads 2 tig and 2 tig + 1
__device__ __forceinline__ void reduce_runs(const Run (&rn)[2], float2 *pair, int lane) {
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    float m = rn[i].m;
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) m = fmaxf(m, __shfl_xor_sync(0xffffffffu, m, o));
    float s = rn[i].s * __expf(rn[i].m - m);
#pragma unroll
    for (int o = 4; o < 32; o <<= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane < 4) pair[2 * lane + i] = make_float2(m, s);
  }
}

// the first of n items that falls to worker i of w: floor(n i / w) without a 64-bit division (w <= 128)
__device__ __forceinline__ int share(int n, int i, int w) {
  const unsigned q = (unsigned)n / (unsigned)w, r = (unsigned)n - q * (unsigned)w;
  return (int)(q * (unsigned)i + r * (unsigned)i / (unsigned)w);
}

// what a warp needs to know about its unit
struct Unit {
  int u, b_idx, h, n_sum;
  float *eb;                                                 // [G][el]: e of the CTA's blocks, the first of which is b0
  int el, b0;
  const __nv_bfloat16 *q;                                    // [G][kQRow] the raw query in shared memory
  const float *qt;                                           // [G][Ds_pad] the subspace query in shared memory
};

// e of a thread's two blocks and two heads: into the buffer and into the running pairs.  eA0: block 16 ck + 2 gid, head 2 tig ...
__device__ __forceinline__ void put_e(const Unit &x, int G, int ck, int gid, int tig, float eA0, float eB0, float eA1, float eB1, Run (&run)[2]) {
  const int bA = ck * 16 + 2 * gid, g0 = 2 * tig, g1 = g0 + 1;
  if (bA >= x.n_sum) { eA0 = -INFINITY; eA1 = -INFINITY; }
  if (bA + 1 >= x.n_sum) { eB0 = -INFINITY; eB1 = -INFINITY; }
  float *d = x.eb + (bA - x.b0);
  if (g0 < G) *reinterpret_cast<float2 *>(d + (size_t)g0 * x.el) = make_float2(eA0, eB0);
  if (g1 < G) *reinterpret_cast<float2 *>(d + (size_t)g1 * x.el) = make_float2(eA1, eB1);
  run_add(run[0], eA0, eB0);
  run_add(run[1], eA1, eB1);
}

// Curvature term of a 16-block chunk whose packed E2M1 rows are full width (128 codes: one 16-byte read per thread and
// row) and whose rank R is a multiple of four: no clamps or row tests, four rows (four independent accumulator chains) at
// a time, the four scales of a block read in one go.  xa / xb: this thread's 16 bytes of row 0 of blocks 2 gid and
// 2 gid + 1 (rows 64 bytes apart); sp: the scales of block 2 gid (those of block 2 gid + 1 follow them).
// Adds sum_i (scale_i * (xi_i . q))^2 per block and head; the query's per-head factor is applied by the caller.
template <int R, bool SCALE_F32>
__device__ __forceinline__ void fp4_rows_full_width(uint32_t xa, uint32_t xb, uint32_t sp, const uint32_t (&bq)[8][2], float &sA0,
                                                    float &sA1, float &sB0, float &sB1) {
  static_assert(R % 4 == 0, "whole groups of four rows");
#pragma unroll 1                                 // rolled: half the code at rank 8 (instruction fetch is a visible stall of this kernel)
  for (int i0 = 0; i0 < R; i0 += 4) {
    uint4 wa[4], wb[4];
    float d[4][4];
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      wa[k] = lds128(xa + (i0 + k) * 64);
      wb[k] = lds128(xb + (i0 + k) * 64);
      d[k][0] = d[k][1] = d[k][2] = d[k][3] = 0.f;
    }
    float sa[4], sb[4];
    if (SCALE_F32) {
      const uint4 a = lds128(sp + i0 * 4), b = lds128(sp + R * 4 + i0 * 4);
      sa[0] = __uint_as_float(a.x); sa[1] = __uint_as_float(a.y); sa[2] = __uint_as_float(a.z); sa[3] = __uint_as_float(a.w);
      sb[0] = __uint_as_float(b.x); sb[1] = __uint_as_float(b.y); sb[2] = __uint_as_float(b.z); sb[3] = __uint_as_float(b.w);
    } else {
      const uint2 a = lds64(sp + i0 * 2), b = lds64(sp + R * 2 + i0 * 2);
      const float2 a0 = __half22float2(*reinterpret_cast<const __half2 *>(&a.x)), a1 = __half22float2(*reinterpret_cast<const __half2 *>(&a.y));
      const float2 b0 = __half22float2(*reinterpret_cast<const __half2 *>(&b.x)), b1 = __half22float2(*reinterpret_cast<const __half2 *>(&b.y));
      sa[0] = a0.x; sa[1] = a0.y; sa[2] = a1.x; sa[3] = a1.y;
      sb[0] = b0.x; sb[1] = b0.y; sb[2] = b1.x; sb[3] = b1.y;
    }
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        uint32_t ha[4], hb[4];
        e2m1x8_to_f16(j == 0 ? wa[k].x : j == 1 ? wa[k].y : j == 2 ? wa[k].z : wa[k].w, ha);
        e2m1x8_to_f16(j == 0 ? wb[k].x : j == 1 ? wb[k].y : j == 2 ? wb[k].z : wb[k].w, hb);
        mma16816_f16(d[k][0], d[k][1], d[k][2], d[k][3], ha[0], hb[0], ha[1], hb[1], bq[2 * j][0], bq[2 * j][1]);
        mma16816_f16(d[k][0], d[k][1], d[k][2], d[k][3], ha[2], hb[2], ha[3], hb[3], bq[2 * j + 1][0], bq[2 * j + 1][1]);
      }
    }
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float d0 = d[k][0] * sa[k], d1 = d[k][1] * sa[k], d2 = d[k][2] * sb[k], d3 = d[k][3] * sb[k];
      sA0 = fmaf(d0, d0, sA0); sA1 = fmaf(d1, d1, sA1); sB0 = fmaf(d2, d2, sB0); sB1 = fmaf(d3, d3, sB1);
    }
  }
}

// ---------------------------------------------------------------------------------------------------
// Scoring of chunks [cb, ce) of a unit by one warp.  DT: COBS_SUMM_BF16 | COBS_SUMM_FP4_E2M1.  WPT: 32-bit words of codes per
// thread per FP4 row (Ds_pad / 32).  NT: f16 terms of the query (1: full space, 2: fp32 subspace query).
// The first copies are issued by `start`, so that they fly while the CTA projects the query.
// `run` leaves the warp's (max, sum) pairs, and returns false when a wait for this warp's own copies ran out.
// ---------------------------------------------------------------------------------------------------
template <int DT, int D, int WPT, int NT>
struct Scorer {
  static constexpr int BLOCKS = 16;               // blocks of a chunk
  static constexpr bool FP4 = (DT == COBS_SUMM_FP4_E2M1);
  static constexpr int MCH = D / 32;              // 16-byte chunks of a bf16 row per thread
  static constexpr int KSM = D / 16;              // k-steps of a bf16 row
  static constexpr int KSQ = FP4 ? WPT * 2 : 1;   // k-steps of an FP4 row
  // stage layout: [16 block means, row stride MROW][16 blocks x rows of factors, block stride XS][scales]
  // The +32 bytes of padding per row / block put the rows of neighbouring quads in different bank halves.
  static constexpr int MROW = D * 2 + 32;
  static constexpr int MEAN_BYTES = 16 * MROW;
  static constexpr int ROWB = FP4 ? WPT * 16 : D * 2;                 // bytes of one factor row
  static constexpr int ROWS_CAP = (kStage - 16 * 32) / (16 * ROWB);
  static constexpr int ROWS_MAX = ROWS_CAP < COBS_MAX_RANK ? ROWS_CAP : COBS_MAX_RANK;   // rows a batch can hold at most
  static_assert((kStage - MEAN_BYTES - 16 * 32 - 16 * COBS_MAX_RANK * 4 - 16) / (16 * ROWB) >= 1, "stage too small");
  static constexpr int RG = 4;                    // FP4 factor rows decoded and multiplied together
  static size_t unit_bytes(const Params &p) {     // what a unit's scores are computed from
    return (size_t)p.NB * (D * 2 + p.r * (ROWB + (FP4 ? (p.scale_dtype == COBS_SCALE_FP16 ? 2 : 4) : 0)));
  }

  const Params &p;
  unsigned char *wsm;
  uint32_t ring, bar0;
  int lane, r, cap, scale_sz, scale_bytes, ROWS0, ROWSN, mrow, mean_bytes, XS0, XSN, n_batches;
  bool single;
  uint64_t pol;
  size_t rec_u;                                   // record of the unit's block 0
  size_t scale_total;                             // bytes of the whole scale array

  __device__ __forceinline__ Scorer(const Params &p_, const Unit &x, unsigned char *wsm_, uint64_t *bars, int lane_, bool one) : p(p_), wsm(wsm_), lane(lane_) {
    r = p.r;
    ring = smem_u32(wsm);
    bar0 = smem_u32(bars);
    scale_sz = (p.scale_dtype == COBS_SCALE_FP16) ? 2 : 4;
    // scales of a chunk, at the end of the stage; the copy starts on a 16-byte boundary below them
    scale_bytes = FP4 ? 16 * r * scale_sz + 16 : 0;
    // Common case: means, all r factor rows and scales of the 16 blocks fit one stage.  Then a chunk is three
    // contiguous pieces of the summary arrays and is fetched by three bulk copies in memory layout (`single`).
    // Otherwise the factor rows go in batches, each block copied on its own to a padded position.
    single = 16 * D * 2 + 16 * r * ROWB + scale_bytes <= kStage && r <= ROWS_MAX;
    // A warp with a single chunk gives it the whole ring if that saves batches (one sequence of 32k with bf16 summaries of rank 4:
    // 15.4 -> 14.6 us; not with a subspace, whose query is projected in the second stage).
    cap = (!single && one && !p.u_q && MEAN_BYTES + 16 * 32 + scale_bytes + 16 * r * ROWB <= kRing) ? kRing : kStage;
    ROWS0 = single ? r : min((int)COBS_MAX_RANK, (cap - MEAN_BYTES - 16 * 32 - scale_bytes) / (16 * ROWB));
    ROWSN = min(ROWS_MAX, (kStage - 16 * 32 - scale_bytes) / (16 * ROWB));
    mrow = single ? D * 2 : MROW;                                        // row stride of the mean area
    mean_bytes = 16 * mrow;
    XS0 = single ? r * ROWB : ROWS0 * ROWB + 32;                         // block stride of the factor area
    XSN = ROWSN * ROWB + 32;
    n_batches = (r <= ROWS0) ? 1 : 1 + (r - ROWS0 + ROWSN - 1) / ROWSN;
    pol = l2_evict_first_policy();
    rec_u = (size_t)x.u * p.NB;
    scale_total = (size_t)p.B * p.Hkv * p.NB * r * scale_sz;
  }
  __device__ __forceinline__ int scale_shift(int ck) const { return (int)(((rec_u + ck * 16) * r * scale_sz) & 15); }

  // bulk copies of (chunk ck, batch b) into stage st; completion is counted on the stage's mbarrier
  __device__ __forceinline__ void issue(int ck, int b, int st) {
    const int nblk = min(16, p.NB - ck * 16);
    const size_t rec0 = rec_u + ck * 16;
    const int row0 = (b == 0) ? 0 : ROWS0 + (b - 1) * ROWSN;
    const int rows = min(r - row0, (b == 0) ? ROWS0 : ROWSN);
    const uint32_t sbase = ring + st * kStage;
    const uint32_t xoff = (b == 0) ? mean_bytes : 0;
    const uint32_t xs = (b == 0) ? XS0 : XSN;
    const uint32_t soff = cap - scale_bytes;
    // the scales of a chunk start on any 2-byte boundary: the copy takes the 16-byte units that hold them, unless those
    // reach past the end of the array (then plain loads)
    const size_t sb0 = rec0 * r * scale_sz;
    const int shift = (int)(sb0 & 15), sbytes = (shift + nblk * r * scale_sz + 15) & ~15;
    const bool scales = FP4 && r > 0, scales_bulk = scales && sb0 - shift + sbytes <= scale_total;
    const uint32_t bar = bar0 + st * 8;
    if (lane == 0) {
      uint32_t tx = (uint32_t)nblk * (uint32_t)(rows > 0 ? rows * ROWB : 0);
      if (b == 0) tx += (uint32_t)nblk * (D * 2);
      if (scales_bulk) tx += (uint32_t)sbytes;
      mbar_expect_tx(bar, tx);
      if (single) {                               // the whole chunk: three contiguous pieces, one lane issues them
        bulk_g2s(sbase, (const char *)p.mean + rec0 * (size_t)(D * 2), nblk * D * 2, bar, pol);
        if (rows > 0) bulk_g2s(sbase + xoff, (const char *)p.xi + rec0 * r * (size_t)ROWB, nblk * r * ROWB, bar, pol);
      }
      if (scales_bulk) bulk_g2s(sbase + soff, (const char *)p.scale + (sb0 - shift), sbytes, bar, pol);
    }
    if (scales && !scales_bulk) {
      const uint16_t *ssrc = reinterpret_cast<const uint16_t *>((const char *)p.scale + sb0);
      uint16_t *dst = reinterpret_cast<uint16_t *>(wsm + st * kStage + soff + shift);
      for (int w = lane; w < nblk * r * scale_sz / 2; w += 32) dst[w] = ssrc[w];
    }
    if (single) return;
    __syncwarp();
    if (lane < 16) {
      if (lane < nblk && rows > 0)
        bulk_g2s(sbase + xoff + lane * xs, (const char *)p.xi + ((rec0 + lane) * r + row0) * (size_t)ROWB, rows * ROWB, bar, pol);
    } else if (b == 0 && lane - 16 < nblk) {
      bulk_g2s(sbase + (lane - 16) * mrow, (const char *)p.mean + (rec0 + lane - 16) * (size_t)(D * 2), D * 2, bar, pol);
    }
  }
  __device__ __forceinline__ void start(int cb, int ce) {
    if (cb < ce) issue(cb, 0, 0);
  }

  __device__ __forceinline__ bool run(const Unit &x, int cb, int ce, float2 *pair) {
    Run rn[2] = {{-1e30f, 0.f}, {-1e30f, 0.f}};
    const bool ok = cb >= ce || score(x, cb, ce, rn);
    reduce_runs(rn, pair, lane);
    return ok;
  }
  __device__ __forceinline__ bool score(const Unit &x, int cb, int ce, Run (&rn)[2]) {
    const int gid = lane >> 2, tig = lane & 3, G = p.G;
    const float inv_sqrt_d = 1.0f / sqrtf((float)D);
    const float ln_l = (float)(31 - __clz(p.L)) * 0.6931471805599453f;      // L is a power of two
    // ---- query fragments ------------------------------------------------------------------------------
    uint32_t bm[KSM][2];
    uint32_t bq[FP4 ? NT : 1][KSQ][2];
    float m0 = 0.f, m1 = 0.f;
    {
#pragma unroll
      for (int m = 0; m < KSM / 2; ++m) {
        uint4 v = make_uint4(0, 0, 0, 0);
        if (gid < G) v = *reinterpret_cast<const uint4 *>(x.q + gid * kQRow + (tig + 4 * m) * 8);
        bm[2 * m][0] = v.x; bm[2 * m][1] = v.y; bm[2 * m + 1][0] = v.z; bm[2 * m + 1][1] = v.w;
      }
      if (FP4) {
        // this thread's WPT * 8 query elements of head gid: the raw bf16 query (full space; the
        // 1/sqrt(D) factor is applied to the tile result) or the projected fp32 q~ (subspace)
        float e[WPT][8];
        float mx = 0.f;
#pragma unroll
        for (int j = 0; j < WPT; ++j) {
          if (NT == 2) {
            const float4 *src = reinterpret_cast<const float4 *>(x.qt + gid * p.Ds_pad + tig * (WPT * 8) + j * 8);
            float4 lo = make_float4(0.f, 0.f, 0.f, 0.f), hi = lo;
            if (gid < G) { lo = src[0]; hi = src[1]; }
            e[j][0] = lo.x; e[j][1] = lo.y; e[j][2] = lo.z; e[j][3] = lo.w;
            e[j][4] = hi.x; e[j][5] = hi.y; e[j][6] = hi.z; e[j][7] = hi.w;
          } else {
            uint4 v = make_uint4(0, 0, 0, 0);
            if (gid < G) v = *reinterpret_cast<const uint4 *>(x.q + gid * kQRow + tig * (WPT * 8) + j * 8);
            e[j][0] = bf16_lo(v.x); e[j][1] = bf16_hi(v.x); e[j][2] = bf16_lo(v.y); e[j][3] = bf16_hi(v.y);
            e[j][4] = bf16_lo(v.z); e[j][5] = bf16_hi(v.z); e[j][6] = bf16_lo(v.w); e[j][7] = bf16_hi(v.w);
          }
#pragma unroll
          for (int n = 0; n < 8; ++n) mx = fmaxf(mx, fabsf(e[j][n]));
        }
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        // mx in [2^(ex-1), 2^ex), from its exponent field (clamped: an all-zero or absurdly large query keeps
        // the powers of two below in range)
        const int ex = (int)(__float_as_uint(fminf(fmaxf(mx, 1e-30f), 1e30f)) >> 23) - 126;
        const float inv_s = __uint_as_float((uint32_t)(128 - ex) << 23);       // 2^(1-ex): brings max |q| into [1, 2)
        const float mult = __uint_as_float((uint32_t)(126 + ex) << 23) * (NT == 2 ? 1.0f : inv_sqrt_d);
#pragma unroll
        for (int j = 0; j < WPT; ++j) {
#pragma unroll
          for (int t = 0; t < NT; ++t) {
            float hi[8];
#pragma unroll
            for (int n = 0; n < 8; ++n) {
              const float v = (t == 0) ? e[j][n] * inv_s : e[j][n];
              hi[n] = __half2float(__float2half_rn(v));
              e[j][n] = v - hi[n];
            }
            bq[t][2 * j][0] = f16x2(hi[0], hi[1]); bq[t][2 * j][1] = f16x2(hi[2], hi[3]);
            bq[t][2 * j + 1][0] = f16x2(hi[4], hi[5]); bq[t][2 * j + 1][1] = f16x2(hi[6], hi[7]);
          }
        }
        // result columns 2 tig, 2 tig + 1 are heads whose factor sits in the lanes gid = 2 tig, 2 tig + 1
        m0 = __shfl_sync(0xffffffffu, mult, (2 * tig) * 4);
        m1 = __shfl_sync(0xffffffffu, mult, (2 * tig + 1) * 4);
      }
    }
    float fA0 = 0.f, fA1 = 0.f, fB0 = 0.f, fB1 = 0.f, sA0 = 0.f, sA1 = 0.f, sB0 = 0.f, sB1 = 0.f;
    int ck = cb, cur_b = 0, st = 0;
    uint32_t phase_bits = 0;                  // bit st = parity to wait for on stage st
    while (ck < ce) {
      int nck = ck, nxt_b = cur_b + 1;
      if (nxt_b >= n_batches) { nxt_b = 0; ++nck; }
      if (nck < ce) issue(nck, nxt_b, st ^ 1);
      const uint32_t sbase = ring + st * kStage;
      if (!mbar_wait(bar0 + st * 8, (phase_bits >> st) & 1u)) {     // bounded: the copies never landed
        if (lane == 0) report(p.status, COBS_ERR_TIMEOUT);
        return false;
      }
      phase_bits ^= 1u << st;
      __syncwarp();
      if (cur_b == 0) {
        // ---- first-order term: block means against the raw bf16 query ------------------------------------
        float c0 = 0.f, c1 = 0.f, c2 = 0.f, c3 = 0.f, e0 = 0.f, e1 = 0.f, e2 = 0.f, e3 = 0.f;   // two chains
        const uint32_t ma = sbase + (2 * gid) * mrow + tig * 16, mb = ma + mrow;
#pragma unroll
        for (int m = 0; m < MCH; ++m) {
          const uint4 va = lds128(ma + m * 64), vb = lds128(mb + m * 64);
          mma16816_bf16(c0, c1, c2, c3, va.x, vb.x, va.y, vb.y, bm[2 * m][0], bm[2 * m][1]);
          mma16816_bf16(e0, e1, e2, e3, va.z, vb.z, va.w, vb.w, bm[2 * m + 1][0], bm[2 * m + 1][1]);
        }
        fA0 = (c0 + e0) * inv_sqrt_d; fA1 = (c1 + e1) * inv_sqrt_d;
        fB0 = (c2 + e2) * inv_sqrt_d; fB1 = (c3 + e3) * inv_sqrt_d;
        sA0 = sA1 = sB0 = sB1 = 0.f;
      }
      // ---- curvature term: rows of this batch ----------------------------------------------------------
      const int row0 = (cur_b == 0) ? 0 : ROWS0 + (cur_b - 1) * ROWSN;
      const int rows = min(r - row0, (cur_b == 0) ? ROWS0 : ROWSN);
      const uint32_t xs = (cur_b == 0) ? XS0 : XSN;
      const uint32_t xa = sbase + ((cur_b == 0) ? mean_bytes : 0) + (2 * gid) * xs + tig * (FP4 ? WPT * 4 : 16), xb = xa + xs;
      bool rows_done = false;
      if constexpr (FP4 && WPT == 4 && NT == 1) {
        // full key space, rank 4 or 8, the whole chunk in one stage: straight-line code (the scales of a block then start
        // on a boundary of their vector reads: r * scale_sz divides 16 or is a multiple of it)
        if (single && (r == 8 || r == 4)) {
          const uint32_t spa = sbase + (kStage - scale_bytes) + scale_shift(ck) + (2 * gid) * r * scale_sz;
          if (r == 8) {
            if (scale_sz == 4) fp4_rows_full_width<8, true>(xa, xb, spa, bq[0], sA0, sA1, sB0, sB1);
            else fp4_rows_full_width<8, false>(xa, xb, spa, bq[0], sA0, sA1, sB0, sB1);
          } else {
            if (scale_sz == 4) fp4_rows_full_width<4, true>(xa, xb, spa, bq[0], sA0, sA1, sB0, sB1);
            else fp4_rows_full_width<4, false>(xa, xb, spa, bq[0], sA0, sA1, sB0, sB1);
          }
          rows_done = true;
        }
      }
      if (rows_done) {
      } else if (FP4) {
        // RG factor rows at a time: RG independent accumulator chains keep the tensor pipe busy
        const unsigned char *sp = wsm + st * kStage + (cap - scale_bytes) + scale_shift(ck) + (2 * gid) * r * scale_sz;
#pragma unroll 1
        for (int i0 = 0; i0 < rows; i0 += RG) {
          float d[RG][4];
          uint32_t wa[RG][4], wb[RG][4];
#pragma unroll
          for (int k = 0; k < RG; ++k) {
            // neighbouring quads walk the group's rows in a rotated order (their rows then sit in different
            // bank halves); a row past the end of the batch is read from the last row and weighted by zero
            const int i = min(i0 + ((k + gid) & (RG - 1)), rows - 1);
            if (WPT == 4) {
              const uint4 a = lds128(xa + i * ROWB), bb = lds128(xb + i * ROWB);
              wa[k][0] = a.x; wa[k][1] = a.y; wa[k][2] = a.z; wa[k][3] = a.w;
              wb[k][0] = bb.x; wb[k][1] = bb.y; wb[k][2] = bb.z; wb[k][3] = bb.w;
            } else {
#pragma unroll
              for (int j = 0; j < 4; ++j) {
                wa[k][j] = (j < WPT) ? lds_u32(xa + i * ROWB + j * 4) : 0u;
                wb[k][j] = (j < WPT) ? lds_u32(xb + i * ROWB + j * 4) : 0u;
              }
            }
            d[k][0] = d[k][1] = d[k][2] = d[k][3] = 0.f;
          }
#pragma unroll
          for (int j = 0; j < WPT; ++j) {
#pragma unroll
            for (int k = 0; k < RG; ++k) {
              uint32_t ha[4], hb[4];
              e2m1x8_to_f16(wa[k][j], ha);
              e2m1x8_to_f16(wb[k][j], hb);
#pragma unroll
              for (int t = 0; t < NT; ++t) {
                mma16816_f16(d[k][0], d[k][1], d[k][2], d[k][3], ha[0], hb[0], ha[1], hb[1], bq[t][2 * j][0], bq[t][2 * j][1]);
                mma16816_f16(d[k][0], d[k][1], d[k][2], d[k][3], ha[2], hb[2], ha[3], hb[3], bq[t][2 * j + 1][0],
                             bq[t][2 * j + 1][1]);
              }
            }
          }
          // scales of this lane's rows of the group (clamped like the rows themselves; a row past the end weighs
          // zero).  The per-head query factors m0, m1 are applied once per chunk, to the sums of squares.
          auto accumulate = [&](auto f32) {
#pragma unroll
            for (int k = 0; k < RG; ++k) {
              const int io = i0 + ((k + gid) & (RG - 1));
              const int ri = row0 + min(io, rows - 1);
              float sa, sb;
              if (decltype(f32)::value) {
                sa = reinterpret_cast<const float *>(sp)[ri];
                sb = reinterpret_cast<const float *>(sp)[r + ri];
              } else {
                sa = __half2float(reinterpret_cast<const __half *>(sp)[ri]);
                sb = __half2float(reinterpret_cast<const __half *>(sp)[r + ri]);
              }
              if (io >= rows) { sa = 0.f; sb = 0.f; }
              const float d0 = d[k][0] * sa, d1 = d[k][1] * sa, d2 = d[k][2] * sb, d3 = d[k][3] * sb;
              sA0 = fmaf(d0, d0, sA0); sA1 = fmaf(d1, d1, sA1); sB0 = fmaf(d2, d2, sB0); sB1 = fmaf(d3, d3, sB1);
            }
          };
          if (scale_sz == 4) accumulate(std::true_type{}); else accumulate(std::false_type{});
        }
      } else {
#pragma unroll 1
        for (int i0 = 0; i0 < rows; i0 += ROWS_MAX) {
#pragma unroll
          for (int k = 0; k < ROWS_MAX; ++k) {
            const int i = i0 + k;
            if (i < rows) {
              float d0 = 0.f, d1 = 0.f, d2 = 0.f, d3 = 0.f;
#pragma unroll
              for (int m = 0; m < MCH; ++m) {
                const uint4 va = lds128(xa + i * ROWB + m * 64), vb = lds128(xb + i * ROWB + m * 64);
                mma16816_bf16(d0, d1, d2, d3, va.x, vb.x, va.y, vb.y, bm[2 * m][0], bm[2 * m][1]);
                mma16816_bf16(d0, d1, d2, d3, va.z, vb.z, va.w, vb.w, bm[2 * m + 1][0], bm[2 * m + 1][1]);
              }
              d0 *= inv_sqrt_d; d1 *= inv_sqrt_d; d2 *= inv_sqrt_d; d3 *= inv_sqrt_d;
              sA0 = fmaf(d0, d0, sA0); sA1 = fmaf(d1, d1, sA1); sB0 = fmaf(d2, d2, sB0); sB1 = fmaf(d3, d3, sB1);
            }
          }
        }
      }
      if (cur_b == n_batches - 1) {
        // 1/2 of the sums of squared projections; for FP4 the squares still lack the query's per-head factor
        const float h0 = FP4 ? 0.5f * m0 * m0 : 0.5f, h1 = FP4 ? 0.5f * m1 * m1 : 0.5f;
        put_e(x, G, ck, gid, tig, ln_l + fA0 + h0 * sA0, ln_l + fB0 + h0 * sB0, ln_l + fA1 + h1 * sA1, ln_l + fB1 + h1 * sB1, rn);
      }
      __syncwarp();                           // all lanes are done with stage st before it is refilled
      ck = nck; cur_b = nxt_b; st ^= 1;
    }
    return true;
  }
};

// ---------------------------------------------------------------------------------------------------
// Scoring from rows of floats: fp32 summaries, bf16 factors in a subspace, the diagonal-skew variant.  Rows of Ds elements start
// on any element; a block's rows are fetched by one bulk copy of the 16-byte units that hold them, in batches of as many rows
// as fit a stage, and read back 16 bytes or (rows that are no multiple of 16 bytes) one element at a time.
// (Reading them straight from global memory, one row of 16 blocks in flight per warp, took 1366 us for 2.4 GB of fp32 summaries,
// 288 units; this way 688.)
// ---------------------------------------------------------------------------------------------------
__device__ __forceinline__ void split3(float x, float y, uint32_t &a, uint32_t &b, uint32_t &c) {
  a = bf16x2(x, y);
  const float x1 = x - bf16_lo(a), y1 = y - bf16_hi(a);
  b = bf16x2(x1, y1);
  c = bf16x2(x1 - bf16_lo(b), y1 - bf16_hi(b));
}
template <int DT, int D>
struct RowScorer {
  static constexpr int BLOCKS = 16;
  static constexpr bool F32 = (DT == COBS_SUMM_FP32);
  static constexpr int ES = F32 ? 4 : 2;
  static constexpr int KS = D / 32;               // groups of 32 elements (8 per lane of a quad)
  static constexpr int XT = F32 ? 3 : 1;          // bf16 terms of a stored value
  static constexpr int PAD = 32;                  // rows of neighbouring blocks start in different banks
  static constexpr int MROW = D * ES + PAD;
  static constexpr int ROOM = kStage / 16 - PAD - 32;       // bytes of a block's rows in a batch (the copy takes up to 15 more at either end)
  static_assert(ROOM >= D * ES, "a stage must hold a row of every block");
  static size_t unit_bytes(const Params &p) { return (size_t)p.NB * (D + p.r * p.Ds) * ES; }
  const Params &p;
  unsigned char *wsm;
  uint32_t ring, bar0;
  int lane, rowb, rows0, rows_n, n_batches;
  uint64_t pol;
  size_t rec_u, xi_total;

  __device__ __forceinline__ RowScorer(const Params &p_, const Unit &x, unsigned char *wsm_, uint64_t *bars, int lane_, bool one) : p(p_), wsm(wsm_), lane(lane_) {
    ring = smem_u32(wsm);
    bar0 = smem_u32(bars);
    rowb = p.Ds * ES;
    rows0 = min(p.r, max(0, ROOM - MROW) / rowb);            // rows beside the means
    rows_n = ROOM / rowb;
    n_batches = 1 + (p.r - rows0 + rows_n - 1) / rows_n;
    // a warp with a single chunk gives it the whole ring: one wait instead of one per batch (one sequence of 2k: 15.5 -> 13.9 us;
    // not with a subspace, whose query is projected in the second stage)
    if (one && n_batches > 1 && !p.u_q && p.r * rowb <= kRing / 16 - PAD - 32 - MROW) { rows0 = p.r; n_batches = 1; }
    pol = l2_evict_first_policy();
    rec_u = (size_t)x.u * p.NB;
    xi_total = (size_t)p.B * p.Hkv * p.NB * p.r * rowb;
  }
  __device__ __forceinline__ int first_row(int b) const { return (b == 0) ? 0 : rows0 + (b - 1) * rows_n; }
  __device__ __forceinline__ int n_rows(int b) const { return (b == 0) ? rows0 : min(p.r - first_row(b), rows_n); }
  __device__ __forceinline__ int stride(int b) const { return (((b == 0) ? rows0 : rows_n) * rowb + 16 + 15) / 16 * 16 + PAD; }
  __device__ __forceinline__ int shift(size_t rec, int b) const { return (int)(((rec * p.r + first_row(b)) * rowb) & 15); }

  __device__ __forceinline__ void issue(int ck, int b, int st) {
    const int nblk = min(16, p.NB - ck * 16), i = lane & 15;
    const size_t rec = rec_u + ck * 16 + i;
    const bool on = i < nblk, mean = lane >= 16;
    const int rows = n_rows(b);
    const uint32_t sbase = ring + st * kStage, bar = bar0 + st * 8;
    const char *src = nullptr;
    uint32_t dst = 0, bytes = 0;
    if (on && mean && b == 0) {
      src = (const char *)p.mean + rec * (size_t)(D * ES);
      dst = sbase + i * MROW;
      bytes = D * ES;
    } else if (on && !mean && rows > 0) {
      const size_t s0 = (rec * p.r + first_row(b)) * (size_t)rowb;
      const int sh = (int)(s0 & 15);
      src = (const char *)p.xi + (s0 - sh);
      dst = sbase + ((b == 0) ? 16 * MROW : 0) + i * stride(b);
      bytes = (sh + rows * rowb + 15) & ~15;
      if (s0 - sh + bytes > xi_total) {             // the end of the array: what is left of its last 16 bytes, element by element
        bytes = (uint32_t)(xi_total - (s0 - sh)) & ~15u;
        for (int k = (int)bytes / ES; k < (sh + rows * rowb) / ES; ++k) {
          if (F32) reinterpret_cast<float *>(wsm + (dst - ring))[k] = reinterpret_cast<const float *>(src)[k];
          else reinterpret_cast<uint16_t *>(wsm + (dst - ring))[k] = reinterpret_cast<const uint16_t *>(src)[k];
        }
      }
    }
    const uint32_t tx = __reduce_add_sync(0xffffffffu, bytes);
    if (lane == 0) mbar_expect_tx(bar, tx);
    __syncwarp();
    if (bytes) bulk_g2s(dst, src, bytes, bar, pol);
  }
  __device__ __forceinline__ void start(int cb, int ce) {
    if (cb < ce) issue(cb, 0, 0);
  }

  // eight elements from element j on of a row of n elements at address a, as bf16 pairs in XT terms (zeros beyond the row)
  __device__ __forceinline__ void load8(uint32_t a, int j, int n, bool vec, bool swap, uint32_t (&t)[XT][4]) const {
    if constexpr (F32) {
      float f[8];
      if (vec) {                                    // (n is a multiple of 4; odd gid reads the second half first: no bank conflicts)
        const uint4 z = make_uint4(0u, 0u, 0u, 0u);
        const int jx = j + (swap ? 4 : 0), jy = j + (swap ? 0 : 4);
        const uint4 v = (jx < n) ? lds128(a + jx * 4) : z, w = (jy < n) ? lds128(a + jy * 4) : z;
        const uint4 lo = swap ? w : v, hi = swap ? v : w;
        f[0] = __uint_as_float(lo.x); f[1] = __uint_as_float(lo.y); f[2] = __uint_as_float(lo.z); f[3] = __uint_as_float(lo.w);
        f[4] = __uint_as_float(hi.x); f[5] = __uint_as_float(hi.y); f[6] = __uint_as_float(hi.z); f[7] = __uint_as_float(hi.w);
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) f[i] = (j + i < n) ? lds_f32(a + (j + i) * 4) : 0.f;
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) split3(f[2 * i], f[2 * i + 1], t[0][i], t[XT > 1 ? 1 : 0][i], t[XT - 1][i]);
    } else {
      if (vec) {
        uint4 v = make_uint4(0u, 0u, 0u, 0u);
        if (j < n) v = lds128(a + j * 2);
        t[0][0] = v.x; t[0][1] = v.y; t[0][2] = v.z; t[0][3] = v.w;
      } else {
        const uint16_t *q = reinterpret_cast<const uint16_t *>(wsm + (a - ring)) + j;
#pragma unroll
        for (int i = 0; i < 4; ++i)
          t[0][i] = ((j + 2 * i < n) ? (uint32_t)q[2 * i] : 0u) | ((j + 2 * i + 1 < n) ? (uint32_t)q[2 * i + 1] << 16 : 0u);
      }
    }
  }

  __device__ __forceinline__ bool run(const Unit &x, int cb, int ce, float2 *pair) {
    Run rn[2] = {{-1e30f, 0.f}, {-1e30f, 0.f}};
    const bool ok = cb >= ce || score(x, cb, ce, rn);
    reduce_runs(rn, pair, lane);
    return ok;
  }
  __device__ __forceinline__ bool score(const Unit &x, int cb, int ce, Run (&rn)[2]) {
    const int gid = lane >> 2, tig = lane & 3, G = p.G, Ds = p.Ds;
    const bool sub = p.u_q != nullptr, vec = (rowb & 15) == 0, swap = gid & 1;
    const float inv_sqrt_d = 1.0f / sqrtf((float)D);
    const float ln_l = (float)(31 - __clz(p.L)) * 0.6931471805599453f;
    uint32_t bm[KS][4], bs[3][KS][4];               // the raw query; the subspace query in three bf16 terms
#pragma unroll
    for (int m = 0; m < KS; ++m) {
      uint4 v = make_uint4(0, 0, 0, 0);
      if (gid < G) v = *reinterpret_cast<const uint4 *>(x.q + gid * kQRow + (tig + 4 * m) * 8);
      bm[m][0] = v.x; bm[m][1] = v.y; bm[m][2] = v.z; bm[m][3] = v.w;
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float a = 0.f, b = 0.f;
        const int j = (tig + 4 * m) * 8 + 2 * i;
        if (sub && gid < G) {
          if (j < Ds) a = x.qt[gid * p.Ds_pad + j];
          if (j + 1 < Ds) b = x.qt[gid * p.Ds_pad + j + 1];
        }
        split3(a, b, bs[0][m][i], bs[1][m][i], bs[2][m][i]);
      }
    }
    // products of one row of the two blocks; `full` = against the raw query, else against the subspace query
    auto row_product = [&](uint32_t ra, uint32_t rb, int n, bool v, bool full, float (&d)[4]) {
      d[0] = d[1] = d[2] = d[3] = 0.f;
      float e[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int m = 0; m < KS; ++m) {
        uint32_t ta[XT][4], tb[XT][4];
        load8(ra, (tig + 4 * m) * 8, n, v, swap, ta);
        load8(rb, (tig + 4 * m) * 8, n, v, swap, tb);
        if (full) {
#pragma unroll
          for (int t = XT - 1; t >= 0; --t) {
            mma16816_bf16(d[0], d[1], d[2], d[3], ta[t][0], tb[t][0], ta[t][1], tb[t][1], bm[m][0], bm[m][1]);
            mma16816_bf16(e[0], e[1], e[2], e[3], ta[t][2], tb[t][2], ta[t][3], tb[t][3], bm[m][2], bm[m][3]);
          }
        } else {
#pragma unroll
          for (int t = XT - 1; t >= 0; --t)
#pragma unroll
            for (int s = 2 - t; s >= 0; --s) {        // terms below 2^-24 of the product are left out
              mma16816_bf16(d[0], d[1], d[2], d[3], ta[t][0], tb[t][0], ta[t][1], tb[t][1], bs[s][m][0], bs[s][m][1]);
              mma16816_bf16(e[0], e[1], e[2], e[3], ta[t][2], tb[t][2], ta[t][3], tb[t][3], bs[s][m][2], bs[s][m][3]);
            }
        }
      }
#pragma unroll
      for (int i = 0; i < 4; ++i) d[i] += e[i];
    };
    const float qs = sub ? 1.0f : inv_sqrt_d;
    float fA0 = 0.f, fA1 = 0.f, fB0 = 0.f, fB1 = 0.f, sA0 = 0.f, sA1 = 0.f, sB0 = 0.f, sB1 = 0.f;
    int ck = cb, b = 0, st = 0;
    uint32_t phase_bits = 0;
    while (ck < ce) {
      int nck = ck, nb = b + 1;
      if (nb >= n_batches) { nb = 0; ++nck; }
      if (nck < ce) issue(nck, nb, st ^ 1);
      if (!mbar_wait(bar0 + st * 8, (phase_bits >> st) & 1u)) {     // bounded: the copies never landed
        if (lane == 0) report(p.status, COBS_ERR_TIMEOUT);
        return false;
      }
      phase_bits ^= 1u << st;
      __syncwarp();
      const uint32_t sbase = ring + st * kStage;
      const size_t rec = rec_u + ck * 16 + 2 * gid;
      float d[4];
      if (b == 0) {
        const uint32_t ma = sbase + 2 * gid * MROW;
        row_product(ma, ma + MROW, D, true, true, d);
        fA0 = d[0] * inv_sqrt_d; fA1 = d[1] * inv_sqrt_d; fB0 = d[2] * inv_sqrt_d; fB1 = d[3] * inv_sqrt_d;
        sA0 = sA1 = sB0 = sB1 = 0.f;
      }
      const uint32_t xo = sbase + ((b == 0) ? 16 * MROW : 0) + 2 * gid * stride(b);
      const uint32_t xa = xo + shift(rec, b), xb = xo + stride(b) + shift(rec + 1, b);
      const int rows = n_rows(b), row0 = first_row(b);
#pragma unroll 1
      for (int i = 0; i < rows; ++i) {
        row_product(xa + i * rowb, xb + i * rowb, Ds, vec, !sub, d);
        float cA = 0.f, cB = 0.f;                    // (c / 6) / (1 / 2): folded into the sums that are halved below
        if (p.skew) {
          if (ck * 16 + 2 * gid < x.n_sum) cA = p.skew[rec * p.r + row0 + i] * (1.0f / 3.0f);
          if (ck * 16 + 2 * gid + 1 < x.n_sum) cB = p.skew[(rec + 1) * p.r + row0 + i] * (1.0f / 3.0f);
        }
        const float d0 = d[0] * qs, d1 = d[1] * qs, d2 = d[2] * qs, d3 = d[3] * qs;
        sA0 = fmaf(d0 * d0, fmaf(cA, d0, 1.0f), sA0); sA1 = fmaf(d1 * d1, fmaf(cA, d1, 1.0f), sA1);
        sB0 = fmaf(d2 * d2, fmaf(cB, d2, 1.0f), sB0); sB1 = fmaf(d3 * d3, fmaf(cB, d3, 1.0f), sB1);
      }
      if (b == n_batches - 1)
        put_e(x, G, ck, gid, tig, ln_l + fA0 + 0.5f * sA0, ln_l + fB0 + 0.5f * sB0, ln_l + fA1 + 0.5f * sA1, ln_l + fB1 + 0.5f * sB1, rn);
      __syncwarp();                           // all lanes are done with stage st before it is refilled
      ck = nck; b = nb; st ^= 1;
    }
    return true;
  }
};

// ---------------------------------------------------------------------------------------------------
// Exact block masses in place of estimates: e[g][b] = ln sum_{t in b} exp(q'_g . k_t) (Eq. bg-defs), for cobs_exact_select.  It reads
// every key, so what bounds it is HBM: a warp streams the 16-token groups of a contiguous range of blocks through a ring of its own
// without a stop at a block's end, five 4 KB stages in flight.  Logits by mma.sync with the heads as rows (zero padded to 16) and
// 8 tokens as columns; every lane keeps a running (max, sum) of its four tokens per group, merged once per block.
// (A kernel of its own with two stages per warp, drained at the end of every block, and a selection kernel behind it: 63 us
// for 268 MB; this way 50.)
// ---------------------------------------------------------------------------------------------------
template <int D>
struct ExactScorer {
  static constexpr int BLOCKS = 4;
  static constexpr int CH = D / 8, KS = D / 16, ROWB = D * 2, STAGE = 16 * ROWB, NCP = (16 * CH) / 32;
  static constexpr int NST = (D == 128) ? 6 : 12;   // 16-token groups in the ring: the two being used, 16 to 20 KB on their way
  static_assert(NST * STAGE <= kRing && NST % 2 == 0, "the ring must fit");
  static size_t unit_bytes(const Params &p) { return (size_t)p.NB * p.L * ROWB; }
  const Params &p;
  unsigned char *wsm;
  int lane;
  __device__ __forceinline__ ExactScorer(const Params &p_, const Unit &, unsigned char *wsm_, uint64_t *, int lane_, bool) : p(p_), wsm(wsm_), lane(lane_) {}
  __device__ __forceinline__ void start(int, int) {}
  __device__ __forceinline__ bool run(const Unit &x, int cb, int ce, float2 *pair) {
    const int gid = lane >> 2, tig = lane & 3, G = p.G, gpb = p.L >> 4;
    const int b0 = cb * BLOCKS, b1 = min(ce * BLOCKS, x.n_sum), n = max(0, b1 - b0) * gpb;
    Run rn = {-1e30f, 0.f};                         // of head gid
    const float sl = 1.0f / sqrtf((float)D);
    const uint32_t ring = smem_u32(wsm);
    const uint64_t pol = l2_evict_first_policy();
    const uint4 *kbase = reinterpret_cast<const uint4 *>(p.k_pages) + lane;
    uint32_t qa[KS][2];
    const uint32_t *qg = reinterpret_cast<const uint32_t *>(x.q + gid * kQRow);
#pragma unroll
    for (int s = 0; s < KS; ++s) {
      qa[s][0] = (gid < G) ? qg[8 * s + tig] : 0u;
      qa[s][1] = (gid < G) ? qg[8 * s + 4 + tig] : 0u;
    }
    uint32_t cdst[NCP];
#pragma unroll
    for (int j = 0; j < NCP; ++j) {
      const int i = lane + 32 * j, t = i / CH, c = i - t * CH;
      cdst[j] = t * ROWB + ((c ^ (t & 7)) << 4);
    }
    const int kt = ((lane >> 4) & 1) * 8 + (lane & 7), kc = (lane >> 3) & 1;
    // lane i holds the place of group 32 k + i (in groups from the pool's start; none: all ones), for two k at a time
    constexpr uint32_t kNone = 0xffffffffu;
    auto resolve = [&](int g) -> uint32_t {
      if (g >= n) return kNone;
      const int tok0 = b0 * p.L + g * 16, pg = page_of(p, x.b_idx, tok0);
      if (pg < 0 || pg >= p.n_pages) { report(p.status, COBS_ERR_BOUNDS); return kNone; }
      return group_place(p, pg, x.h, tok0);
    };
    uint32_t tab[2] = {resolve(lane), resolve(32 + lane)};
    auto issue = [&](int g, int st) {
      const uint32_t off = __shfl_sync(0xffffffffu, (g & 32) ? tab[1] : tab[0], g & 31);
      if (g < n && off != kNone) {
#pragma unroll
        for (int j = 0; j < NCP; ++j) cpa16(ring + st * STAGE + cdst[j], kbase + (size_t)off * (2 * D) + 32 * j, pol);
      }
      cpa_commit();
      return off;
    };
    uint32_t live = 0;                               // bit st: stage st holds a group
#pragma unroll
    for (int g = 0; g < NST - 2; ++g) live |= (issue(g, g) != kNone ? 1u : 0u) << g;
    int st = 0, in_blk = 0, blk = b0;
    float m_run = -1e30f, l_run = 0.f;
    // a lane's four logits of the group in stage s (natural-log units)
    auto logits = [&](int s_, float (&v)[4]) {
      const uint32_t sb = ring + s_ * STAGE;
      float sc[2][2][4] = {};                        // [tokens 0-7, 8-15][even, odd k steps]
#pragma unroll
      for (int s = 0; s < KS; ++s) {
        uint32_t r0, r1, r2, r3;
        ldsm_x4(r0, r1, r2, r3, sb + kt * ROWB + (((2 * s + kc) ^ (kt & 7)) << 4));
        float (&y0)[4] = sc[0][s & 1], (&y1)[4] = sc[1][s & 1];
        mma16816_bf16(y0[0], y0[1], y0[2], y0[3], qa[s][0], 0u, qa[s][1], 0u, r0, r1);
        mma16816_bf16(y1[0], y1[1], y1[2], y1[3], qa[s][0], 0u, qa[s][1], 0u, r2, r3);
      }
      v[0] = (sc[0][0][0] + sc[0][1][0]) * sl; v[1] = (sc[0][0][1] + sc[0][1][1]) * sl;
      v[2] = (sc[1][0][0] + sc[1][1][0]) * sl; v[3] = (sc[1][0][1] + sc[1][1][1]) * sl;
      if (!((live >> s_) & 1u)) v[0] = v[1] = v[2] = v[3] = -1e30f;
    };
    auto add = [&](const float (&v)[4], const float (&w)[4], bool both) {
      float m_new = fmaxf(m_run, fmaxf(fmaxf(v[0], v[1]), fmaxf(v[2], v[3])));
      if (both) m_new = fmaxf(m_new, fmaxf(fmaxf(w[0], w[1]), fmaxf(w[2], w[3])));
      float t = (__expf(v[0] - m_new) + __expf(v[1] - m_new)) + (__expf(v[2] - m_new) + __expf(v[3] - m_new));
      if (both) t += (__expf(w[0] - m_new) + __expf(w[1] - m_new)) + (__expf(w[2] - m_new) + __expf(w[3] - m_new));
      l_run = fmaf(l_run, __expf(m_run - m_new), t);
      m_run = m_new;
    };
    auto finish = [&]() {                            // the four lanes of a head hold different tokens: merge their pairs
#pragma unroll
      for (int o = 1; o <= 2; o <<= 1) {
        const float om = __shfl_xor_sync(0xffffffffu, m_run, o), ol = __shfl_xor_sync(0xffffffffu, l_run, o);
        const float nm = fmaxf(m_run, om);
        l_run = l_run * __expf(m_run - nm) + ol * __expf(om - nm);
        m_run = nm;
      }
      const float e = m_run + logf(l_run);
      if (gid < G && tig == 0) x.eb[(size_t)gid * x.el + (blk - x.b0)] = e;
      const float m = fmaxf(rn.m, e);
      rn.s = rn.s * __expf(rn.m - m) + __expf(e - m);
      rn.m = m;
      m_run = -1e30f; l_run = 0.f; in_blk = 0; ++blk;
    };
    // two groups at a time: their chains of products and exponentials run side by side
#pragma unroll 1
    for (int g = 0; g < n; g += 2) {
      if ((g & 31) == 0 && g > 0) {                  // the table's older half is used up to the last entry
        const uint32_t t = resolve(g + 32 + lane);
        if (g & 32) tab[0] = t; else tab[1] = t;
      }
#pragma unroll
      for (int i = 0; i < 2; ++i) {                  // into the two stages that were used last
        const int si = (st == 0) ? NST - 2 + i : st - 2 + i;
        const uint32_t off = issue(g + NST - 2 + i, si);
        live = (live & ~(1u << si)) | ((off != kNone ? 1u : 0u) << si);
      }
      cpa_wait<NST - 2>();
      __syncwarp();
      float v[4], w[4];
      logits(st, v);
      logits(st + 1, w);
      __syncwarp();
      st = (st == NST - 2) ? 0 : st + 2;
      if (gpb > 1) {
        add(v, w, true);
        in_blk += 2;
        if (in_blk == gpb) finish();
      } else {
        add(v, w, false);
        finish();
        if (g + 1 < n) { add(w, v, false); finish(); }
      }
    }
    cpa_wait<0>();
    __syncwarp();
    if (tig == 0) pair[gid] = (gid < G) ? make_float2(rn.m, rn.s) : make_float2(-1e30f, 0.f);
    return true;
  }
};

// ---------------------------------------------------------------------------------------------------
// Query projection q~ = U_Q^T (q / sqrt(D)) of a unit's heads, zero padded to Ds_pad, by the whole CTA (Method, "Per-step
// scoring": one O(s D) projection per step and head).  A warp takes (32 consecutive coordinates, a quarter of the head
// dimension): lane = coordinate, so the reads of U_Q [Hkv][D][Ds] are coalesced and serve all heads; the quarters are added in
// a fixed order.  qt: [G][Ds_pad] result; part: scratch of 4 KB per quarter, `stride` floats apart.
// ---------------------------------------------------------------------------------------------------
template <int D>
__device__ __forceinline__ void project_query(const Params &p, const Unit &x, float *qt, float *part, int stride, int warp, int lane, int W) {
  constexpr int DQ = D / 4;
  const int nsb = (p.Ds_pad + 31) / 32, G = p.G;
  const float inv_sqrt_d = 1.0f / sqrtf((float)D);
  for (int t = warp; t < 4 * nsb; t += W) {
    const int sb = t >> 2, quarter = t & 3, s = sb * 32 + lane;
    const bool live = s < p.Ds;
    const float *uq = p.u_q + ((size_t)x.h * D + quarter * DQ) * p.Ds + (live ? s : 0);
    float v[DQ];
#pragma unroll
    for (int j = 0; j < DQ; ++j) v[j] = live ? uq[(size_t)j * p.Ds] : 0.f;
#pragma unroll 1
    for (int g = 0; g < G; ++g) {
      const __nv_bfloat16 *q = x.q + g * kQRow + quarter * DQ;
      const float qv = (lane < DQ) ? __bfloat162float(q[lane]) * inv_sqrt_d : 0.f;
      float a = 0.f;
#pragma unroll
      for (int j = 0; j < DQ; ++j) a = fmaf(v[j], __shfl_sync(0xffffffffu, qv, j), a);
      part[quarter * stride + g * 128 + s] = a;
    }
  }
  __syncthreads();
  for (int i = threadIdx.x; i < G * p.Ds_pad; i += blockDim.x) {
    const int g = i / p.Ds_pad, s = i - g * p.Ds_pad;
    const float *q = part + g * 128 + s;
    qt[i] = ((q[0] + q[stride]) + q[2 * stride]) + q[3 * stride];
  }
  __syncthreads();
}

// ---------------------------------------------------------------------------------------------------
// Top-k of n keys in shared memory by the whole CTA: the k largest scores (>= 0, so that their bit patterns order like integers),
// lower index on ties, ascending output in sel.  1 <= k < n.  BPT: consecutive keys a thread holds in registers (0: any number,
// read from shared memory in every round: neighbouring threads take neighbouring keys, in the end every warp a contiguous part of
// them, 32 at a time.  With a contiguous part per thread all lanes of a warp met in one bank: one unit of 16 384 blocks, selected
// by each of its sixteen CTAs: step 120 -> 46 us; of 8 192: 67 -> 30).
// ---------------------------------------------------------------------------------------------------
template <int BPT>
__device__ __forceinline__ void select_topk(const float *keys_s, int n, int k, int *sel, uint32_t (*s_cnt)[2][kMaxW], int *s_scan, int tid, int W) {
  const int warp = tid >> 5, lane = tid & 31;
  const int b0 = tid * BPT;
  uint32_t key[BPT ? BPT : 1];
  if constexpr (BPT > 0) {
#pragma unroll
    for (int j = 0; j < BPT; j += 2) {               // (the array has a whole number of fours of keys)
      float2 v = make_float2(0.f, 0.f);
      if (b0 + j < n) v = *reinterpret_cast<const float2 *>(keys_s + b0 + j);
      key[j] = __float_as_uint(v.x);
      key[j + 1] = (b0 + j + 1 < n) ? __float_as_uint(v.y) : 0u;
    }
  }
  // one pass over this thread's keys
  auto each = [&](auto f) {
    if constexpr (BPT > 0) {
#pragma unroll
      for (int j = 0; j < BPT; ++j) f(key[j], b0 + j);
    } else {
      for (int b = tid; b < n; b += 32 * W) f(__float_as_uint(keys_s[b]), b);
    }
  };
  // theta = the largest T with #(key >= T) >= k (or any with exactly k), found two bits at a time: three trial counts packed, 10
  // bits each in one word while there are fewer than 1024 keys (BPT <= 2), else 16 bits each in two
  constexpr bool ONE = BPT == 1 || BPT == 2;
  uint32_t theta = 0u;
  int par = 0;
  for (int bit = 30; bit >= 0; bit -= 2) {          // bits 31 (zero), 30 | 29, 28 | ... | 1, 0
    const uint32_t ta = theta | (3u << bit), tb = theta | (2u << bit), tc = theta | (1u << bit);
    uint32_t c0 = 0, c1 = 0;
    each([&](uint32_t x, int) {
      if (ONE) c0 += (x >= ta ? 1u : 0u) + (x >= tb ? 1u << 10 : 0u) + (x >= tc ? 1u << 20 : 0u);
      else { c0 += (x >= ta ? 1u : 0u) + (x >= tb ? 1u << 16 : 0u); c1 += (x >= tc ? 1u : 0u); }
    });
    c0 = __reduce_add_sync(0xffffffffu, c0);
    if (!ONE) c1 = __reduce_add_sync(0xffffffffu, c1);
    if (lane == 0) { s_cnt[par][0][warp] = c0; if (!ONE) s_cnt[par][1][warp] = c1; }
    __syncthreads();
    uint32_t n0 = 0, n1 = 0;
#pragma unroll
    for (int w = 0; w < kMaxW; ++w) {                // (entries of absent warps are zero)
      n0 += s_cnt[par][0][w];
      if (!ONE) n1 += s_cnt[par][1][w];
    }
    par ^= 1;
    const uint32_t ku = (uint32_t)k;
    const uint32_t na = ONE ? n0 & 1023u : n0 & 0xffffu, nb = ONE ? (n0 >> 10) & 1023u : n0 >> 16, nc = ONE ? n0 >> 20 : n1;
    const uint32_t at = (na >= ku) ? na : (nb >= ku) ? nb : (nc >= ku) ? nc : 0u;
    if (na >= ku) theta = ta; else if (nb >= ku) theta = tb; else if (nc >= ku) theta = tc;
    if (at == ku) break;                             // (uniform) exactly k keys are >= theta: the bits below do not matter
  }
  // keep every key above theta and the lowest-index `need_eq` keys equal to it, in index order: one scan of the
  // packed (above, equal) counts gives both the totals and this thread's (BPT = 0: this warp's) position
  const int part = (n + 32 * W - 1) / (32 * W) * 32, p0 = warp * part, p1 = min(p0 + part, n);      // this warp's keys (BPT = 0)
  int v = 0;
  auto count = [&](uint32_t x) { v += (x > theta ? (1 << 16) : 0) + (x == theta ? 1 : 0); };
  if constexpr (BPT > 0) each([&](uint32_t x, int b) { if (b < n) count(x); });
  else for (int b = p0 + lane; b < p1; b += 32) count(__float_as_uint(keys_s[b]));
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  if (lane == 31) s_scan[warp] = inc;
  __syncthreads();
  int base = 0, total = 0;
#pragma unroll
  for (int q = 0; q < kMaxW; ++q) { const int t = s_scan[q]; total += t; base += (q < warp) ? t : 0; }
  const int need_eq = max(k - (total >> 16), 0);
  if constexpr (BPT > 0) {
    const int excl = base + inc - v;
    int eq_rank = excl & 0xffff, pos = (excl >> 16) + min(eq_rank, need_eq);
    each([&](uint32_t x, int b) {
      if (b < n) {
        bool keep = x > theta;
        if (x == theta) { keep = eq_rank < need_eq; ++eq_rank; }
        if (keep && pos < k) sel[pos++] = b;
      }
    });
  } else {
    const unsigned before = (1u << lane) - 1u;
    int above = base >> 16, equal = base & 0xffff;
    for (int b = p0 + lane; b - lane < p1; b += 32) {
      const uint32_t x = (b < p1) ? __float_as_uint(keys_s[b]) : 0u;
      const bool a = b < p1 && x > theta, e = b < p1 && x == theta;
      const unsigned ba = __ballot_sync(0xffffffffu, a), be = __ballot_sync(0xffffffffu, e);
      const int eq_rank = equal + __popc(be & before), pos = above + __popc(ba & before) + min(eq_rank, need_eq);
      if ((a || (e && eq_rank < need_eq)) && pos < k) sel[pos] = b;
      above += __popc(ba); equal += __popc(be);
    }
  }
  __syncthreads();
}

// The same for up to 32 KPL keys by one warp, which holds them all: a round costs no barrier, and a barrier is what a round of
// select_topk waits for.  Up to one key per thread of the CTA (16 steps of 16 sequences of 16k in blocks of 64: 731 -> 726 us; one sequence of 2k:
// 13.9 -> 13.4); sixteen keys per lane are too many instructions for one warp (one sequence of 32k: 14.6 us, 15.9 that way), and
// with four warps per CTA a barrier costs less (24 ragged sequences of 12k: 35.1 us, 35.3 with 256).
template <int KPL>
__device__ __forceinline__ void select_topk_warp(const float *keys_s, int n, int k, int *sel, int lane) {
  static_assert(KPL % 4 == 0 && 32 * KPL < 1024, "counts of ten bits");
  const int b0 = lane * KPL;
  uint32_t key[KPL];
#pragma unroll
  for (int j = 0; j < KPL; j += 4) {                 // (the array has a whole number of fours of keys)
    float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
    if (b0 + j < n) v = *reinterpret_cast<const float4 *>(keys_s + b0 + j);
    key[j] = __float_as_uint(v.x);
    key[j + 1] = (b0 + j + 1 < n) ? __float_as_uint(v.y) : 0u;
    key[j + 2] = (b0 + j + 2 < n) ? __float_as_uint(v.z) : 0u;
    key[j + 3] = (b0 + j + 3 < n) ? __float_as_uint(v.w) : 0u;
  }
  const uint32_t ku = (uint32_t)k;
  uint32_t theta = 0u;
#pragma unroll 1
  for (int bit = 30; bit >= 0; bit -= 2) {
    const uint32_t ta = theta | (3u << bit), tb = theta | (2u << bit), tc = theta | (1u << bit);
    uint32_t c = 0, d = 0;                           // (two chains)
#pragma unroll
    for (int j = 0; j < KPL; j += 2) {
      c += (key[j] >= ta ? 1u : 0u) + (key[j] >= tb ? 1u << 10 : 0u) + (key[j] >= tc ? 1u << 20 : 0u);
      d += (key[j + 1] >= ta ? 1u : 0u) + (key[j + 1] >= tb ? 1u << 10 : 0u) + (key[j + 1] >= tc ? 1u << 20 : 0u);
    }
    c = __reduce_add_sync(0xffffffffu, c + d);
    const uint32_t na = c & 1023u, nb = (c >> 10) & 1023u, nc = c >> 20;
    const uint32_t at = (na >= ku) ? na : (nb >= ku) ? nb : (nc >= ku) ? nc : 0u;
    if (na >= ku) theta = ta; else if (nb >= ku) theta = tb; else if (nc >= ku) theta = tc;
    if (at == ku) break;
  }
  int v = 0;
#pragma unroll
  for (int j = 0; j < KPL; ++j)
    if (b0 + j < n) v += (key[j] > theta ? (1 << 16) : 0) + (key[j] == theta ? 1 : 0);
  int inc = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int t = __shfl_up_sync(0xffffffffu, inc, o);
    if (lane >= o) inc += t;
  }
  const int total = __shfl_sync(0xffffffffu, inc, 31);
  const int need_eq = max(k - (total >> 16), 0), excl = inc - v;
  int eq_rank = excl & 0xffff, pos = (excl >> 16) + min(eq_rank, need_eq);
#pragma unroll
  for (int j = 0; j < KPL; ++j)
    if (b0 + j < n) {
      bool keep = key[j] > theta;
      if (key[j] == theta) { keep = eq_rank < need_eq; ++eq_rank; }
      if (keep && pos < k) sel[pos++] = b0 + j;
    }
}

// ---------------------------------------------------------------------------------------------------
// Attention over groups [g0, g1) of the unit by one warp: slots below n_sel are selected blocks, then the window's.
// Leaves acc [G][D] in the warp's ring and (max in natural log units, sum) per head in pair.
// ---------------------------------------------------------------------------------------------------
template <int D>
__device__ __forceinline__ void attend_groups(const Params &p, const Unit &x, int T, int n_cand, int win_blk, int n_sel, const int *sel, unsigned char *wsm,
                                              int g0, int g1, float2 *pair, int lane) {
  constexpr int CH = D / 8;                   // 16-byte chunks per row
  constexpr int KS = D / 16;
  constexpr int NTL = D / 8;                  // 8-wide output tiles
  constexpr int ROWB = D * 2;
  constexpr int VOFF = 16 * ROWB;             // V half of a stage
  constexpr int STAGE = 2 * VOFF;
  constexpr int NCP = (16 * CH) / 32;         // cp.async per lane per operand per stage
  const int gid = lane >> 2, tig = lane & 3;
  const int G = p.G, L = p.L;
  const int lgL = 31 - __clz(L), lgg = lgL - 4;      // L is a power of two: shifts, not divisions
  const uint32_t ring = smem_u32(wsm);
  uint32_t *goff = reinterpret_cast<uint32_t *>(wsm + kAttStages * kAttStage);
  int *gtok = reinterpret_cast<int *>(goff + kTable);
  const float sl2 = (1.0f / sqrtf((float)D)) * 1.4426950408889634f;
  const uint4 *kbase = reinterpret_cast<const uint4 *>(p.k_pages) + lane;
  const uint4 *vbase = reinterpret_cast<const uint4 *>(p.v_pages) + lane;
  const uint64_t pol = l2_evict_first_policy();
  uint32_t cdst[NCP];                          // destination of this lane's j-th 16-byte copy (swizzled)
#pragma unroll
  for (int j = 0; j < NCP; ++j) {
    const int i = lane + 32 * j, t = i / CH, c = i - t * CH;
    cdst[j] = t * ROWB + ((c ^ (t & 7)) << 4);
  }
  // ldmatrix row addresses.  K (not transposed): matrices (tokens 0-7, chunk 2s), (0-7, 2s+1), (8-15, 2s), (8-15, 2s+1)
  const int kt = ((lane >> 4) & 1) * 8 + (lane & 7), kc = (lane >> 3) & 1;
  // V (transposed): matrices (tokens 0-7, chunk 2np), (8-15, 2np), (0-7, 2np+1), (8-15, 2np+1)
  const int vt = ((lane >> 3) & 1) * 8 + (lane & 7), vc = lane >> 4;
  // query fragments: rows = heads (zero padded to 16), natural k order
  uint32_t qa[KS][2];
  {
    const uint32_t *qg = reinterpret_cast<const uint32_t *>(x.q + gid * kQRow);
#pragma unroll
    for (int s = 0; s < KS; ++s) {
      qa[s][0] = (gid < G) ? qg[8 * s + tig] : 0u;
      qa[s][1] = (gid < G) ? qg[8 * s + 4 + tig] : 0u;
    }
  }
  // P = bf16 high + low: the high parts are rows 0-7 of the A operand, the low parts rows 8-15, so that one mma takes both and
  // the two products meet at the end.  Every accumulator tile has its own four registers: with the unused rows of all tiles in
  // one pair, every mma waited for the one before it (192 ragged units of 64 groups: 21 us, now 12.5, which is 8 TB/s from L2 and
  // HBM; running the products with K a group ahead of those with V on top of it gains nothing)
  float o[NTL][4];
#pragma unroll
  for (int n = 0; n < NTL; ++n) o[n][0] = o[n][1] = o[n][2] = o[n][3] = 0.f;
  float m_run = -1e30f, l_run = 0.f;
#pragma unroll 1
  for (int gb = g0; gb < g1; gb += kTable) {
    const int n_groups = min(g1 - gb, kTable);
    __syncwarp();
    for (int g = lane; g < n_groups; g += 32) {
      const int gg = gb + g, it = gg >> lgg, sub = gg - (it << lgg);
      const int blk = (it < n_sel) ? sel[it] : win_blk + (it - n_sel);
      bool good = true;
      if (it < n_sel && (blk < 0 || blk >= n_cand)) { good = false; report(p.status, COBS_ERR_BOUNDS); }
      const int tok0 = blk * L + sub * 16;
      int first = -1;
      uint32_t off = 0;
      if (good && tok0 < T) {
        const int pg = page_of(p, x.b_idx, tok0);
        if (pg < 0 || pg >= p.n_pages) report(p.status, COBS_ERR_BOUNDS);
        else { first = tok0; off = group_place(p, pg, x.h, tok0); }
      }
      goff[g] = off;
      gtok[g] = first;
    }
    __syncwarp();
    auto issue = [&](int g, int st) {
      if (g < n_groups) {
        const int first = gtok[g];
        if (first >= 0) {
          const size_t off = (size_t)goff[g] * (2 * D);
          const uint4 *ks = kbase + off, *vs = vbase + off;
          const uint32_t dst = ring + st * STAGE;
          const int nv = T - first;
          if (nv >= 16) {
#pragma unroll
            for (int j = 0; j < NCP; ++j) { cpa16(dst + cdst[j], ks + 32 * j, pol); cpa16(dst + VOFF + cdst[j], vs + 32 * j, pol); }
          } else {                             // ragged tail: rows past the end of the sequence are zero filled
#pragma unroll
            for (int j = 0; j < NCP; ++j) {
              const int bytes = ((lane + 32 * j) / CH < nv) ? 16 : 0;
              cpa16z(dst + cdst[j], ks + 32 * j, bytes, pol);
              cpa16z(dst + VOFF + cdst[j], vs + 32 * j, bytes, pol);
            }
          }
        }
      }
      cpa_commit();
    };
    issue(0, 0);
    issue(1, 1);
    int st = 0, st2 = 2;
#pragma unroll 1
    for (int g = 0; g < n_groups; ++g) {
      issue(g + 2, st2);
      cpa_wait<2>();
      __syncwarp();
      const int first = gtok[g];
      if (first >= 0) {
        const uint32_t sb = ring + st * STAGE;
        // ---- S^T = q K^T: s0 tokens 0-7, s1 tokens 8-15 --------------------------------------------------
        float sc[2][2][4] = {};                // [tokens 0-7, 8-15][even, odd k steps]
#pragma unroll
        for (int s = 0; s < KS; ++s) {
          uint32_t b0, b1, b2, b3;
          ldsm_x4(b0, b1, b2, b3, sb + kt * ROWB + (((2 * s + kc) ^ (kt & 7)) << 4));
          float (&x0)[4] = sc[0][s & 1], (&x1)[4] = sc[1][s & 1];
          mma16816_bf16(x0[0], x0[1], x0[2], x0[3], qa[s][0], 0u, qa[s][1], 0u, b0, b1);
          mma16816_bf16(x1[0], x1[1], x1[2], x1[3], qa[s][0], 0u, qa[s][1], 0u, b2, b3);
        }
        float s00 = sc[0][0][0] + sc[0][1][0], s01 = sc[0][0][1] + sc[0][1][1];
        float s10 = sc[1][0][0] + sc[1][1][0], s11 = sc[1][0][1] + sc[1][1][1];
        const int nv = T - first;
        if (nv < 16) {                         // tokens past the end take no weight
          if (2 * tig >= nv) s00 = -1e30f;
          if (2 * tig + 1 >= nv) s01 = -1e30f;
          if (2 * tig + 8 >= nv) s10 = -1e30f;
          if (2 * tig + 9 >= nv) s11 = -1e30f;
        }
        float mx = fmaxf(fmaxf(s00, s01), fmaxf(s10, s11));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 1));
        mx = fmaxf(mx, __shfl_xor_sync(0xffffffffu, mx, 2));
        if (__any_sync(0xffffffffu, mx > m_run)) {       // rescale only when some head's running max moved
          const float m_new = fmaxf(m_run, mx);
          const float corr = ex2((m_run - m_new) * sl2);
          m_run = m_new;
          l_run *= corr;
          #pragma unroll
          for (int n = 0; n < NTL; ++n) { o[n][0] *= corr; o[n][1] *= corr; o[n][2] *= corr; o[n][3] *= corr; }
        }
        const float mb = m_run * sl2;
        const float p0 = ex2(fmaf(s00, sl2, -mb)), p1 = ex2(fmaf(s01, sl2, -mb));
        const float p2 = ex2(fmaf(s10, sl2, -mb)), p3 = ex2(fmaf(s11, sl2, -mb));
        l_run += (p0 + p1) + (p2 + p3);
        const uint32_t a0h = bf16x2(p0, p1), a2h = bf16x2(p2, p3);
        const uint32_t a0l = bf16x2(p0 - bf16_lo(a0h), p1 - bf16_hi(a0h));
        const uint32_t a2l = bf16x2(p2 - bf16_lo(a2h), p3 - bf16_hi(a2h));
        // ---- O += P V ---------------------------------------------------------------------------------------
#pragma unroll
        for (int np = 0; np < NTL / 2; ++np) {
          uint32_t b0, b1, b2, b3;
          ldsm_x4_t(b0, b1, b2, b3, sb + VOFF + vt * ROWB + (((2 * np + vc) ^ (vt & 7)) << 4));
          float (&o0)[4] = o[2 * np], (&o1)[4] = o[2 * np + 1];
          mma16816_bf16(o0[0], o0[1], o0[2], o0[3], a0h, a0l, a2h, a2l, b0, b1);
          mma16816_bf16(o1[0], o1[1], o1[2], o1[3], a0h, a0l, a2h, a2l, b2, b3);
        }
      }
      __syncwarp();                            // all lanes are done with the stage before it is refilled
      st = (st == kAttStages - 1) ? 0 : st + 1;
      st2 = (st2 == kAttStages - 1) ? 0 : st2 + 1;
    }
    cpa_wait<0>();
  }
  __syncwarp();
  // ---- this warp's partial -----------------------------------------------------------------------------
  l_run += __shfl_xor_sync(0xffffffffu, l_run, 1);
  l_run += __shfl_xor_sync(0xffffffffu, l_run, 2);
  if (gid < G) {
    float *dst = reinterpret_cast<float *>(wsm) + gid * D;
#pragma unroll
    for (int n = 0; n < NTL; ++n) *reinterpret_cast<float2 *>(dst + 8 * n + 2 * tig) = make_float2(o[n][0] + o[n][2], o[n][1] + o[n][3]);
    if (tig == 0) pair[gid] = make_float2((l_run > 0.f) ? m_run * (sl2 * 0.6931471805599453f) : -INFINITY, l_run);
  }
}

// ---------------------------------------------------------------------------------------------------
// the kernel: cluster = unit
// ---------------------------------------------------------------------------------------------------
template <class SCORER, int D>
__global__ void __launch_bounds__(kMaxW * 32, 1) unit_step_kernel(Params p, int phases, Plan pl) {
  extern __shared__ __align__(256) unsigned char fsm[];
  __shared__ __align__(8) uint64_t s_bars[kMaxW][2];       // one mbarrier per scoring stage per warp
  __shared__ __align__(16) float2 s_pair[kMaxW][8];        // per warp and head: (max, sum) of e, later of the attention logits
  __shared__ __align__(16) float2 s_cpair[kMaxC][8];       // per CTA of the cluster and head: (max, sum) of e, later of the attention logits
  __shared__ float s_max[8], s_inv[8];                     // per head: largest e, reciprocal of the sum of e^{e - largest}
  __shared__ __align__(16) __nv_bfloat16 s_q[8 * kQRow];
  __shared__ __align__(16) float s_qt[8 * 128 + 2 * kMaxC];
  __shared__ uint32_t s_cnt[2][2][kMaxW];
  __shared__ int s_scan[kMaxW];
  __shared__ int s_sel[COBS_MAX_TOPK];
  __shared__ int s_lost;                                   // a wait for copies ran out: the outputs are undefined, the rings not ours
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31, W = pl.W, C = pl.C, nthr = W * 32;
  const int u = pl.u0 + blockIdx.x / C, rank = blockIdx.x % C;
  const int G = p.G, L = p.L, NB = p.NB;
  if (C > 1) cluster_arrive();                             // (waited for before the first access to another CTA's memory)
  if (tid < 2 * 2 * kMaxW) (&s_cnt[0][0][0])[tid] = 0u;
  if (tid < kMaxW) s_scan[tid] = 0;
  if (tid == 0) s_lost = 0;
  if (lane == 0) {
    mbar_init(smem_u32(&s_bars[warp][0]), 1);
    mbar_init(smem_u32(&s_bars[warp][1]), 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
  }
  __syncthreads();
  pdl_begin();
  COBS_STAMP(0);
  Unit x;
  x.u = u; x.b_idx = u / p.Hkv; x.h = u - x.b_idx * p.Hkv;
  x.q = s_q;
  // the unit's query, once per CTA (it may lie in host memory): needed behind the next barrier, stored only when the first copies
  // of the summaries, which wait for the length, are on their way
  const int T = tokens_of(p.seq_lens, x.b_idx);
  const bool has_q = tid < G * (D / 8);
  uint4 qv = make_uint4(0u, 0u, 0u, 0u);
  if (has_q) qv = reinterpret_cast<const uint4 *>(p.q + ((size_t)x.b_idx * p.Hq + x.h * G) * D)[tid];
  auto store_q = [&]() {
    const int g = tid / (D / 8), c = tid - g * (D / 8);
    if (has_q) *reinterpret_cast<uint4 *>(s_q + g * kQRow + 8 * c) = qv;
  };
  x.n_sum = min(T / L, NB);
  const int ws = window_start(T, p.window, L);
  const int n_cand = (phases & PH_SCORE) ? min(ws / L, x.n_sum) : ws / L;
  const int n_win = (T - ws + L - 1) / L;
  unsigned char *wsm = fsm + warp * kRing;
  const int nw = C * W, wi = rank * W + warp;
  int n_sel = min(p.topk, n_cand);

  if (phases & PH_SCORE) {
    const int n_chunks = (x.n_sum + SCORER::BLOCKS - 1) / SCORER::BLOCKS;
    const int cb = share(n_chunks, wi, nw), ce = share(n_chunks, wi + 1, nw);
    const int c0 = share(n_chunks, rank * W, nw), c1 = share(n_chunks, rank * W + W, nw);
    x.b0 = c0 * SCORER::BLOCKS;
    x.el = (c1 - c0) * SCORER::BLOCKS;
    x.eb = (pl.e_off >= 0) ? reinterpret_cast<float *>(fsm + pl.e_off) : p.e + ((size_t)u * ((NB + 15) / 16 * 16) + x.b0) * G;
    x.qt = s_qt;
    SCORER sc(p, x, wsm, &s_bars[warp][0], lane, ce - cb == 1);
    sc.start(cb, ce);
    // Between the last scores and the first selected block HBM would be idle: the window's groups, known already, are fetched into
    // L2 meanwhile (sixteen sequences of 128k 93.4 -> 91.1 us; 16 steps of sixteen of 16k 727 -> 687).  Lane i < 4 looks up the page
    // of group nw i + wi: four groups of 8 KB per warp are the window of 512 tokens with eight warps per unit, and 38 MB in all.
    uint32_t ahead = 0xffffffffu;
    {
      const int tok = ws + 16 * (nw * lane + wi);
      if ((phases & PH_ATTEND) && lane < 4 && tok < T) {
        const int pg = page_of(p, x.b_idx, tok);
        if (pg >= 0 && pg < p.n_pages) ahead = group_place(p, pg, x.h, tok);
      }
    }
    store_q();
    __syncthreads();
    if (p.u_q) {                                            // (scratch: the second stages of four rings, not in use yet)
      project_query<D>(p, x, s_qt, reinterpret_cast<float *>(fsm + kStage), kRing / 4, warp, lane, W);
      fence_proxy_async();                                  // bulk copies follow where the scratch was written
    }
    // (max, sum) of e per head: over the warp, the CTA, the cluster
    if (!sc.run(x, cb, ce, s_pair[warp])) s_lost = 1;
    if (ahead != 0xffffffffu) {
      bulk_prefetch_l2(p.k_pages + (size_t)ahead * (16 * D), 16 * D * 2);
      bulk_prefetch_l2(p.v_pages + (size_t)ahead * (16 * D), 16 * D * 2);
    }
    __syncthreads();
    COBS_STAMP(1);
    if (C > 1) cluster_wait();
    if (tid < 8 * C) {                                      // thread = (destination CTA, head): the CTA's pair
      const int g = tid & 7, dst = tid >> 3;
      float m = -1e30f, s = 0.f;
      for (int w = 0; w < W; ++w) m = fmaxf(m, s_pair[w][g].x);
      for (int w = 0; w < W; ++w) s += s_pair[w][g].y * __expf(s_pair[w][g].x - m);
      const uint32_t a = mapa(smem_u32(&s_cpair[rank][g]), dst);
      st_cluster(a, m);
      st_cluster(a + 4, s);
    }
    if (C > 1) { cluster_arrive(); cluster_wait(); } else __syncthreads();
    if (tid < 8) {
      float m = -1e30f, s = 0.f;
      for (int c = 0; c < C; ++c) m = fmaxf(m, s_cpair[c][tid].x);
      for (int c = 0; c < C; ++c) s += s_cpair[c][tid].y * __expf(s_cpair[c][tid].x - m);
      s_max[tid] = m;
      s_inv[tid] = reciprocal(s);
    }
    __syncthreads();
    COBS_STAMP(2);
    // ---- group scores of the CTA's blocks, into every CTA that will select ---------------------------------------
    // (e - max is exact to its last bit where it counts, e - lse is not: every score of a head carried the rounding of its lse.
    // Error of the scores against 64 bits, root mean square: 2.8e-7 -> 1.2e-7)
    float *keys = reinterpret_cast<float *>(fsm + pl.key_off);
    {
      const uint32_t ka = smem_u32(keys);
      const int n_dst = (phases & PH_ATTEND) ? C : 1;       // without an attention phase CTA 0 alone selects
      const int n_loc = min(x.el, x.n_sum - x.b0);
      if (n_loc <= nthr) {                                  // few blocks: one per thread (0.6 us less than four on a quarter of them)
        if (tid < n_loc) {
          float s = 0.f;
#pragma unroll 4
          for (int g = 0; g < G; ++g) s = fmaf(__expf(x.eb[(size_t)g * x.el + tid] - s_max[g]), s_inv[g], s);
          const int b = x.b0 + tid;
          if (p.scores) p.scores[(size_t)u * NB + b] = s;
          if (C == 1) keys[b] = s;
          else for (int c = 0; c < n_dst; ++c) st_cluster(mapa(ka + 4 * b, c), s);
        }
      } else
      for (int i = 4 * tid; i < n_loc; i += 4 * nthr) {     // four blocks at a time (what lies beyond n_loc is not used)
        float4 v[8], s = make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
        for (int g = 0; g < 8; ++g)
          if (g < G) v[g] = *reinterpret_cast<const float4 *>(x.eb + (size_t)g * x.el + i);
#pragma unroll
        for (int g = 0; g < 8; ++g)
          if (g < G) {
            const float m = s_max[g], inv = s_inv[g];
            s.x = fmaf(__expf(v[g].x - m), inv, s.x); s.y = fmaf(__expf(v[g].y - m), inv, s.y);
            s.z = fmaf(__expf(v[g].z - m), inv, s.z); s.w = fmaf(__expf(v[g].w - m), inv, s.w);
          }
        const int b = x.b0 + i;
        if (p.scores) {
          float *d = p.scores + (size_t)u * NB + b;
          d[0] = s.x;
          if (i + 1 < n_loc) d[1] = s.y;
          if (i + 2 < n_loc) d[2] = s.z;
          if (i + 3 < n_loc) d[3] = s.w;
        }
        if (C == 1) *reinterpret_cast<float4 *>(keys + b) = s;
        else for (int c = 0; c < n_dst; ++c) st_cluster4(mapa(ka + 4 * b, c), s);
      }
    }
    if (C > 1) { cluster_arrive(); cluster_wait(); } else __syncthreads();
    COBS_STAMP(3);
    if (!(phases & PH_ATTEND) && rank != 0) return;         // (nothing of this CTA is read any more)
    // ---- top-k ------------------------------------------------------------------------------------------------------
    if (n_sel == n_cand) {
      for (int i = tid; i < n_sel; i += nthr) s_sel[i] = i;
      __syncthreads();
    } else if (n_cand <= nthr) {
      if (warp == 0) {
        if (n_cand <= 128) select_topk_warp<4>(keys, n_cand, n_sel, s_sel, lane);
        else select_topk_warp<8>(keys, n_cand, n_sel, s_sel, lane);
      }
      __syncthreads();
    } else if (n_cand <= 2 * nthr) {
      select_topk<2>(keys, n_cand, n_sel, s_sel, s_cnt, s_scan, tid, W);
    } else if (n_cand <= 8 * nthr) {
      select_topk<8>(keys, n_cand, n_sel, s_sel, s_cnt, s_scan, tid, W);
    } else {
      select_topk<0>(keys, n_cand, n_sel, s_sel, s_cnt, s_scan, tid, W);
    }
    if (rank == 0 && p.sel_idx) {
      if (tid == 0) p.sel_cnt[u] = n_sel;
      for (int i = tid; i < p.topk; i += nthr) p.sel_idx[(size_t)u * p.topk + i] = (i < n_sel) ? s_sel[i] : -1;
    }
    COBS_STAMP(4);
    if (!(phases & PH_ATTEND)) return;
  } else {
    n_sel = max(0, min(n_sel, p.sel_cnt[u]));
    for (int i = tid; i < n_sel; i += nthr) s_sel[i] = p.sel_idx[(size_t)u * p.topk + i];
    store_q();
    if (C > 1) cluster_wait();
    __syncthreads();
  }

  // ---- attention: the unit's groups dealt to the cluster's warps ---------------------------------------------------
  {
    const int n_groups = s_lost ? 0 : (n_sel + n_win) * (L >> 4);
    attend_groups<D>(p, x, T, n_cand, ws / L, n_sel, s_sel, wsm, share(n_groups, wi, nw), share(n_groups, wi + 1, nw),
                     s_pair[warp], lane);
  }
  __syncthreads();
  COBS_STAMP(5);
  // ---- merge: o = sum_s e^{m_s - M} acc_s / sum_s e^{m_s - M} l_s, over the CTA's warps, then over the cluster: CTA r finishes the
  // r-th part of the elements, and every CTA puts its sums where they are finished (stores that nothing waits for, one
  // barrier, local reads; fetching them from the other CTAs after the barrier: 0.5 us more per step) ------------------------------
  const int n2 = G * D / 2, per = (n2 + C - 1) / C;
  float *s_fin = s_qt;                                     // [C][per] float2: the subspace query is not needed any more
  for (int i = tid; i < n2; i += nthr) {
    const int g = i / (D / 2);
    float M = -INFINITY;
#pragma unroll
    for (int w = 0; w < kMaxW; ++w) if (w < W) M = fmaxf(M, s_pair[w][g].x);
    float2 acc = make_float2(0.f, 0.f);
    float l = 0.f;
#pragma unroll
    for (int w = 0; w < kMaxW; ++w) {
      if (w >= W) break;
      const float2 ml = s_pair[w][g];
      const float wt = (ml.x == -INFINITY) ? 0.f : __expf(ml.x - M);
      const float2 v = reinterpret_cast<const float2 *>(fsm + w * kRing)[i];
      acc.x = fmaf(wt, v.x, acc.x); acc.y = fmaf(wt, v.y, acc.y);
      l = fmaf(wt, ml.y, l);
    }
    if (C == 1) {
      const float inv = 1.0f / l;
      reinterpret_cast<float2 *>(p.out + ((size_t)x.b_idx * p.Hq + x.h * G) * D)[i] = make_float2(acc.x * inv, acc.y * inv);
      if (p.lse && i - g * (D / 2) == 0) p.lse[(size_t)x.b_idx * p.Hq + x.h * G + g] = M + __logf(l);
    } else {
      const int dst = i / per;
      st_cluster2(mapa(smem_u32(s_fin) + 8 * (rank * per + i - dst * per), dst), acc);
      if (i - g * (D / 2) < C) st_cluster2(mapa(smem_u32(&s_cpair[rank][g]), i - g * (D / 2)), make_float2(M, l));      // (C <= D / 2)
    }
  }
  COBS_STAMP(6);
  if (C == 1) return;
  cluster_arrive();
  cluster_wait();
  for (int j = tid; j < per; j += nthr) {
    const int i = rank * per + j;
    if (i >= n2) break;
    const int g = i / (D / 2);
    float M = -INFINITY;
    for (int c = 0; c < C; ++c) M = fmaxf(M, s_cpair[c][g].x);
    float2 acc = make_float2(0.f, 0.f);
    float l = 0.f;
    for (int c = 0; c < C; ++c) {
      const float2 ml = s_cpair[c][g], v = reinterpret_cast<const float2 *>(s_fin)[c * per + j];
      const float wt = (ml.x == -INFINITY) ? 0.f : __expf(ml.x - M);
      acc.x = fmaf(wt, v.x, acc.x); acc.y = fmaf(wt, v.y, acc.y);
      l = fmaf(wt, ml.y, l);
    }
    const float inv = 1.0f / l;
    reinterpret_cast<float2 *>(p.out + ((size_t)x.b_idx * p.Hq + x.h * G) * D)[i] = make_float2(acc.x * inv, acc.y * inv);
    if (p.lse && i - g * (D / 2) == 0) p.lse[(size_t)x.b_idx * p.Hq + x.h * G + g] = M + __logf(l);
  }
  COBS_STAMP(7);
}

// ---------------------------------------------------------------------------------------------------
// host side
// ---------------------------------------------------------------------------------------------------
template <class SCORER, int D>
cudaError_t launch_t(const Params &p, int phases, cudaStream_t stream) {
  constexpr int NBLK = SCORER::BLOCKS;
  auto kern = unit_step_kernel<SCORER, D>;
  static std::atomic<int> ready[64];                       // per device: attributes set, table filled
  static std::atomic<int> fit[64][kMaxC + 1];              // clusters of C CTAs, eight warps each, that are resident at a time
  int dev = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e != cudaSuccess) return e;
  if (dev < 0 || dev >= 64) return cudaErrorInvalidDevice;
  cudaLaunchConfig_t cfg = {};
  cudaLaunchAttribute at[2];
  at[0].id = cudaLaunchAttributeClusterDimension;
  at[0].val.clusterDim.y = 1; at[0].val.clusterDim.z = 1;
  at[1].id = cudaLaunchAttributeProgrammaticStreamSerialization;      // see pdl_begin
  at[1].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at; cfg.numAttrs = 1;
  if (!ready[dev].load(std::memory_order_acquire)) {       // (two threads may fill it with the same values)
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemOne)) != cudaSuccess) return e;
    if ((e = cudaFuncSetAttribute(kern, cudaFuncAttributeNonPortableClusterSizeAllowed, 1)) != cudaSuccess) return e;
    for (int c = 1; c <= kMaxC; ++c) {
      at[0].val.clusterDim.x = (unsigned)c;
      cfg.gridDim = dim3((unsigned)c); cfg.blockDim = dim3(kMaxW * 32); cfg.dynamicSmemBytes = kSmemOne;
      int n = 0;
      if (cudaOccupancyMaxActiveClusters(&n, kern, &cfg) != cudaSuccess) { n = 0; (void)cudaGetLastError(); }
      fit[dev][c].store(n, std::memory_order_relaxed);
    }
    ready[dev].store(1, std::memory_order_release);
  }
  // Eight warps per CTA and the largest cluster with which all units are resident at once; no larger than gives every warp a
  // chunk or a group.  (8 units of 32k: 20.5 us with clusters of 4 to 10, 36.7 with 16, of which only seven fit; 32 units:
  // 29.9 / 27.9 / 26.7 us with 2 / 3 / 4; 128 units of 128k: 98 us with one CTA of eight warps, 118 with two of four.)
  // More units than SMs: four warps per CTA, two CTAs per SM (192 ragged units of 12k: 45 us, 55 with eight warps in two waves); but
  // three waves of eight warps rather than two of four whose second is half empty, where there is work for eight (320 units of 32k
  // 85 -> 77 us, 440 88 -> 85, 448 would be 89 -> 101; ragged ones of 12k 50 -> 53 at 304, equal from 352 on; 320 with fp32 summaries
  // of 128 blocks 92 -> 84, of 64 it would be 71 -> 82).
  const int units = p.B * p.Hkv, n_chunks = (p.NB + NBLK - 1) / NBLK;
  const int groups = (p.topk + (p.window + p.L - 1) / p.L + 1) * (p.L / 16);
  // (the same for a scoring call and a whole step: the order of the sums, and so the selection's last bits, follow the split; a single
  // chunk has no order)
  const int work = (phases == PH_SCORE && n_chunks == 1) ? 1 : (phases & PH_SCORE) ? max(n_chunks, groups) : groups;
  const int full = max(1, fit[dev][1].load(std::memory_order_relaxed));      // CTAs of eight warps that are resident at a time: SMs
  auto launch = [&](int u0, int n) -> cudaError_t {
    Plan pl;
    pl.u0 = u0;
    pl.W = (n <= full || ((n + full - 1) / full == 3 && n_chunks >= kMaxW)) ? kMaxW : kMaxW / 2;
    pl.C = 1;
    for (int c = 2; c <= kMaxC && n <= full && (c - 1) * pl.W < work; ++c)
      if (fit[dev][c].load(std::memory_order_relaxed) >= n) pl.C = c;
    const int W = pl.W, C = pl.C, cap = (W == kMaxW) ? kSmemOne : kSmemTwo;
    const int key_bytes = (phases & PH_SCORE) ? (p.NB * 4 + 15) / 16 * 16 : 0;
    const int e_bytes = (phases & PH_SCORE) ? p.G * NBLK * ((n_chunks + C - 1) / C) * 4 : 0;
    int off = W * kRing;
    if (off + key_bytes <= cap) { pl.key_off = off; off += key_bytes; } else pl.key_off = 0;      // over the rings: scoring is over by then
    if (off + e_bytes <= cap) { pl.e_off = off; off += e_bytes; } else pl.e_off = -1;
    at[0].val.clusterDim.x = (unsigned)C;
    cfg.gridDim = dim3((unsigned)(n * C));
    cfg.blockDim = dim3((unsigned)(W * 32));
    cfg.dynamicSmemBytes = (size_t)off;
    cfg.stream = stream;
    cfg.numAttrs = 2;
    const cudaError_t err = cudaLaunchKernelEx(&cfg, kern, p, phases, pl);
    count_launch();
    return err;
  };
  // Up to a quarter more units than SMs, with 1.2 MB or more to score each: one unit per SM, then the others in clusters.  (With four
  // warps per CTA nearly every SM would have one such CTA.  160 / 184 units of 128k, 4 MB each: 147 -> 119 / 152 -> 135 us in a loop,
  // 149 -> 144 / 156 -> 157 with L2 flushed before each; fp32 at 32k, 152 / 176 units: 115 -> 93 / 122 -> 96, flushed 128 -> 119 / 132 -> 121;
  // exact masses of 32k, 152: 233 -> 209, 234 -> 225.  192 units of 128k: 152 -> 144, 160 -> 161, of 64k with
  // bf16 summaries 108 -> 114, 116 -> 146.  With 0.8 MB to score, 64k, 152: 114 -> 97,
  // 116 -> 124; with 0.3, 32k: 41 -> 44, 64 -> 72.)
  if ((phases & PH_SCORE) && units > full && units <= full + full / 4 && SCORER::unit_bytes(p) >= 1200000) {
    if ((e = launch(0, full)) != cudaSuccess) return e;
    return launch(full, units - full);
  }
  return launch(0, units);
}

}  // namespace

// Whether this kernel does a configuration's scoring: everything but the diagonal-skew variant of FP4 summaries, units whose scores
// do not fit a CTA's shared memory, and two kinds of call in which warps that score row by row (fp32 summaries, bf16 ones in a
// subspace or with the skew) are too few for long: one or two units with so much to score that sixteen SMs each take longer than the
// generic kernels' whole grid, and very many units of a single chunk, which one warp of each CTA scores.  Elements of a unit's
// means and factors, step with generic scoring / with this kernel (in a loop, and with L2 flushed before each pass):
//   1 unit   fp32  4.7M .93 / 1.07   8.9M .80 / 1.08   9.4M .74 / .84   18M .83 / .74   36M .57 / .55      drawn at 8M
//            bf16  12M 1.16 / 1.05   18M 1.25 / 1.00   24M .80 / .80   36M .72 / .83                       at 24M
//   2 units  fp32  9M 1.16 / 1.12   14M .98 / .94   18M .99 / 1.06   27M .91 / .98   36M .80 / .87         at 24M
//   fp32, rank 4 / 8, 4 blocks: 512 units .91 / .76, 1 024 .76 / .66; 16 blocks: 512 1.08 / 1.03, 1 024 .97 / .90, 2 048 1.00 / .90;
//   32 blocks: 1 024 1.18 / 1.11; bf16 in a subspace, 4 blocks: 1 024 1.04                                 at 64 units per block
//            bf16  24M 1.18 / 1.25   36M 1.11 / 1.14                       3 units  fp32  36M 1.07 / 1.21
bool unit_score_supported(const Params &p) {
  if (p.NB > kMaxKeys || (p.skew && p.summ_dtype == COBS_SUMM_FP4_E2M1)) return false;
  const long long units = (long long)p.B * p.Hkv, elements = (long long)p.NB * (p.D + p.r * p.Ds);
  const bool fp32 = p.summ_dtype == COBS_SUMM_FP32, rows = fp32 || (p.summ_dtype == COBS_SUMM_BF16 && (p.u_q || p.skew));
  if (fp32 && p.NB <= 16 && units > 296 && units >= 64LL * p.NB) return false;
  if (!rows || units > 2) return true;
  return (units == 1) ? elements < (fp32 ? 8LL << 20 : 24LL << 20) : !fp32 || elements < 24LL << 20;
}
// The same for the exact masses: all but few units with many keys, whose clusters are a few dozen SMs against the whole grid of
// exact_mass_kernel.  (One unit of 131 072 tokens, D 128, L 64, four heads: 24.6 us there, 36.6 here; of 65 536: 20.5 / 22.4; of 32 768:
// 18.5 / 14.0.  Two of 131 072: 28.7 / 36.8; three: 32.8 / 37.3; four: 43.7 / 37.7.  Eight heads, whose selection costs that route more:
// one unit of 98 304: 32.8 / 30.1, of 131 072: 32.8 / 36.9, two 37.3 / 37.2, three 43.0 / 37.2.  Blocks of 16, whose number does: one of
// 131 072 with D 64 47.1 / 43.4.  Blocks of 128, 512 of them, a group of blocks per warp: 20.5 / 15.3; 1 024 of them: 20.5 / 25.1.)
bool unit_exact_supported(const Params &p) {
  const bool many = p.L >= 64 && p.NB >= 1024 && (long long)p.NB * p.L * p.D * 2 >= (16LL << 20) * (p.G > 4 ? 2 : 1);
  return p.NB <= kMaxKeys && !(many && p.B * p.Hkv <= (p.G > 4 ? 2 : 3));
}

// Exact block masses, group scores and selection.
cudaError_t launch_unit_exact(const Params &p, cudaStream_t stream) {
  return p.D == 128 ? launch_t<ExactScorer<128>, 128>(p, PH_SCORE, stream) : launch_t<ExactScorer<64>, 64>(p, PH_SCORE, stream);
}

cudaError_t launch_unit_step(const Params &p, int phases, cudaStream_t stream) {
  const bool bf16_full = p.summ_dtype == COBS_SUMM_BF16 && !p.u_q && !p.skew;
  if (!(phases & PH_SCORE) || bf16_full)
    return p.D == 128 ? launch_t<Scorer<COBS_SUMM_BF16, 128, 1, 1>, 128>(p, phases, stream) : launch_t<Scorer<COBS_SUMM_BF16, 64, 1, 1>, 64>(p, phases, stream);
  if (p.summ_dtype == COBS_SUMM_FP32)
    return p.D == 128 ? launch_t<RowScorer<COBS_SUMM_FP32, 128>, 128>(p, phases, stream) : launch_t<RowScorer<COBS_SUMM_FP32, 64>, 64>(p, phases, stream);
  if (p.summ_dtype == COBS_SUMM_BF16)
    return p.D == 128 ? launch_t<RowScorer<COBS_SUMM_BF16, 128>, 128>(p, phases, stream) : launch_t<RowScorer<COBS_SUMM_BF16, 64>, 64>(p, phases, stream);
  const int wpt = p.Ds_pad / 32;
  if (!p.u_q)
    return p.D == 128 ? launch_t<Scorer<COBS_SUMM_FP4_E2M1, 128, 4, 1>, 128>(p, phases, stream) : launch_t<Scorer<COBS_SUMM_FP4_E2M1, 64, 2, 1>, 64>(p, phases, stream);
#define COBS_CASE(DD, WW) \
  if (p.D == DD && wpt == WW) return launch_t<Scorer<COBS_SUMM_FP4_E2M1, DD, WW, 2>, DD>(p, phases, stream);
  COBS_CASE(128, 4) COBS_CASE(128, 3) COBS_CASE(128, 2) COBS_CASE(128, 1) COBS_CASE(64, 2) COBS_CASE(64, 1)
#undef COBS_CASE
  return cudaErrorInvalidValue;
}

}  // namespace cobs

#ifdef COBS_TIMING
extern "C" int cobs_debug_stamps(unsigned long long *host_out) {
  return (int)cudaMemcpyFromSymbol(host_out, cobs::g_stamps, sizeof(unsigned long long) * 8 * 4096);
}
#endif
