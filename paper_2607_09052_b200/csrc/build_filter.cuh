// The r <= 8 leading eigenvectors of a block's Gram matrix by Chebyshev-filtered subspace iteration.
//
//   V (16 vectors)  ->  T_m(G) V, m products with G  ->  orthonormal again  ->  ...  ->  H = V G V^T (16 x 16)
//   ->  its eigenvectors U by one-sided Jacobi rotations  ->  w = U V, each checked: |G w - theta w|
//
// A tridiagonal form takes L - 2 dependent reflections whatever is asked for; here the chain is as long as the r leading
// directions need to stand out from the seventeenth on (7 to 40 products with G in all), and every product is a
// contraction for the tensor pipe.  (Y. Zhou, Y. Saad, "A Chebyshev-Davidson algorithm for large symmetric eigenproblems",
// 2007, for the filter; H. Rutishauser, "Simultaneous iteration method for symmetric matrices", 1970, for the scheme.)
//
// Layout.  Vectors are rows: V is 16 x L, and thread (gid, tig) holds rows gid and gid + 8, columns 8 g + 2 tig + {0, 1} of
// every 8-token tile g, which is the accumulator of mma.sync m16n8k16 and, packed, its A operand: the result of one product
// is the operand of the next without a shuffle.  G is symmetric, so its accumulators are the B operand in the same way.
// Operands are split into f16 high and low parts (23 bits with the low part's sign, one less than fp32) and products are summed in fp32 (mma_split); the first round, which
// only has to find the neighbourhood, takes the high parts alone.
// Four warps hold every fourth tile each; V goes through shared memory for each product, one barrier.
//
// Products with G and orthonormalisations of a block of 128 (medians; 1 % to 99 %), and time of 8 192 blocks, three per SM, by the
// tridiagonal form and by this:
//                                              rank 4                             rank 8
//   flat spectrum                              21 (18-24); 4    3 130 -> 1 470 us    25 (22-30); 4     3 450 -> 1 700 us
//   sixteen directions over noise               9 (8-11); 4     3 130 -> 1 160       11 (8-14); 4      3 460 -> 1 310
//   one channel ten times the others           30 (26-34); 16   3 130 -> 2 490       33 (33-42); 17    3 460 -> 2 840
//   thirty times                               32 (19-33); 17   3 130 -> 2 820       33 (22-35); 17    3 460 -> 3 610
//   a hundred times (left to the other)         -               3 130 -> 3 730        -                3 450 -> 4 030
//   24 eigenvalues within 5 % (the same)        -               3 130 -> 3 980        -                3 450 -> 4 370
// A product is 2 200 cycles, an orthonormalisation 4 200, the small eigenproblem 33 000, of which the rotations of one warp 22 000:
// latency, not the tensor pipe (20 products are 15 400 cycles of it).  168 registers for three blocks per SM, 350 bytes of them spilled
// (in a subspace 255 for two, 116 bytes).
#pragma once

#include <type_traits>

#include "build_mma.cuh"

namespace cobs {
namespace {

template <int L>
struct Filter {
  static constexpr int W = 4;                         // warps per block
  static constexpr int NT = L / 8 / W;                // 8-token tiles of a warp: tile a is tile W a + warp of the block
  static constexpr int KT = L / 16;                   // 16-token steps of a product
  // shared memory, in floats: the low halves of G as B fragments (the high ones stay in registers)
  static constexpr int G_FLOATS = L * L / 2;
  static constexpr int V_FLOATS = 2 * KT * 2 * 128;   // two buffers of V as A fragments
  static constexpr int X_FLOATS = 2 * W * 32 * 8;     // two buffers of the warps' partial sums
  static constexpr int U_FLOATS = 256;
};

__device__ __forceinline__ uint32_t movm(uint32_t x) {          // 8 x 8 transpose of f16 pairs over the warp
  uint32_t r;
  asm volatile("movmatrix.sync.aligned.m8n8.trans.b16 %0, %1;\n" : "=r"(r) : "r"(x));
  return r;
}
__device__ __forceinline__ float rsqrt_ftz(float x) {
  float r;
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}
__device__ __forceinline__ float quad_sum(float v) {
  v += __shfl_xor_sync(0xffffffffu, v, 1);
  return v + __shfl_xor_sync(0xffffffffu, v, 2);
}
__device__ __forceinline__ float rows_max(float v) {            // over the lanes of all rows
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 4));
  v = fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 8));
  return fmaxf(v, __shfl_xor_sync(0xffffffffu, v, 16));
}
__device__ __forceinline__ float pow2(int e) { return __uint_as_float((uint32_t)(127 + e) << 23); }
__device__ __forceinline__ int ilog2(float x) { return (int)(__float_as_uint(x) >> 23) - 127; }
// exp(-acosh(x)), 1 below 1: the reciprocal of what a step of the filter lets grow
__device__ __forceinline__ float cheb_damp(float x) {
  x = fmaxf(x, 1.0f);
  return rcp(x + sqrtf(fmaf(x, x, -1.0f)));
}

// A 16 x 16 matrix over a warp: rows gid and gid + 8, columns 2 tig + {0, 1} and 8 + 2 tig + {0, 1} (an accumulator's two tiles).
__device__ __forceinline__ void split16(const float (&u)[8], float f, uint32_t (&h)[4], uint32_t (&l)[4]) {      // as A fragments
  split_f16(u[0] * f, u[1] * f, h[0], l[0]);
  split_f16(u[4] * f, u[5] * f, h[1], l[1]);
  split_f16(u[2] * f, u[3] * f, h[2], l[2]);
  split_f16(u[6] * f, u[7] * f, h[3], l[3]);
}
__device__ __forceinline__ void from_tiles(const float (&c)[2][4], float (&o)[8]) {
  o[0] = c[0][0]; o[1] = c[0][1]; o[2] = c[1][0]; o[3] = c[1][1];
  o[4] = c[0][2]; o[5] = c[0][3]; o[6] = c[1][2]; o[7] = c[1][3];
}
// A B^T; SYM: to the bit the transpose of B A^T (the mixed products are added before the high ones)
template <bool SYM>
__device__ __forceinline__ void mul16_bt(const uint32_t (&ah)[4], const uint32_t (&al)[4], const uint32_t (&bh)[4], const uint32_t (&bl)[4], float (&o)[8]) {
  float c[2][4];
#pragma unroll
  for (int n = 0; n < 2; ++n) {
    if constexpr (!SYM) {
      mma_split<true>(c[n], ah, al, bh[n], bh[2 + n], bl[n], bl[2 + n]);
      continue;
    }
    float t[4];
    mma_f16_zero(c[n], ah[0], ah[1], ah[2], ah[3], bl[n], bl[2 + n]);
    mma_f16_zero(t, al[0], al[1], al[2], al[3], bh[n], bh[2 + n]);
    add4(c[n], t);
    mma_f16_zero(t, ah[0], ah[1], ah[2], ah[3], bh[n], bh[2 + n]);
    add4(c[n], t);
  }
  from_tiles(c, o);
}
__device__ __forceinline__ void diag16(const float (&s)[8], int lane, float &d0, float &d1) {      // elements gid and gid + 8
  const int gid = lane >> 2, src = (lane & 28) | (gid >> 1);
  d0 = __shfl_sync(0xffffffffu, (gid & 1) ? s[1] : s[0], src);
  d1 = __shfl_sync(0xffffffffu, (gid & 1) ? s[7] : s[6], src);
}

// All 120 pairs of sixteen rows (x: gid, y: gid + 8; four elements per lane, four lanes per row) made orthogonal by a rotation
// each, eight at a time: first each row x with all rows y, in Gray code, then, regrouped, halves, quarters and eighths of each.
// True if a pair whose larger squared norm exceeds `thr` and whose smaller one `noise` had a cosine above 2^-7.5.
__device__ __forceinline__ bool jacobi_sweep(u64 (&x)[2], u64 (&y)[2], float thr, float noise, int lane) {
  float nx, ny;                                         // squared norms, carried along
  {
    const u64 a = fma2(x[1], x[1], mul2(x[0], x[0])), b = fma2(y[1], y[1], mul2(y[0], y[0]));
    nx = quad_sum(lo(a) + hi(a)); ny = quad_sum(lo(b) + hi(b));
  }
  bool big = false;
#pragma unroll 1
  for (int step = 0;; ++step) {
    const u64 p = fma2(x[1], y[1], mul2(x[0], y[0]));
    const float g = quad_sum(lo(p) + hi(p));
    const float d = nx - ny, gg = g * g;
    big |= gg > 3e-5f * nx * ny && fmaxf(nx, ny) > thr && fminf(nx, ny) > noise;
    const bool turn = gg > 1e-36f;
    const float u = rsqrt_ftz(fmaf(d, d, 4.0f * gg)), c2 = turn ? fmaf(0.5f * fabsf(d), u, 0.5f) : 1.f, r = rsqrt_ftz(c2);      // cos^2 of the angle
    const float c = c2 * r, s = turn ? copysignf(1.0f, d) * (g * u) * r : 0.f;
    const u64 cc = pk(c, c), ss = pk(s, s), ms = pk(-s, -s);
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const u64 a = fma2(ss, y[i], mul2(cc, x[i])), b = fma2(ms, x[i], mul2(cc, y[i]));
      x[i] = a; y[i] = b;
    }
    const float t = fmaf(c * c, nx, fmaf(s * s, ny, 2.0f * (c * s) * g));
    ny = fmaxf(nx + ny - t, 0.f);
    nx = t;
    if (step == 14) break;
    // lanes 1, 2, 1, 4, 1, 2, 1 apart, then regroup over 4; 1, 2, 1, over 2; 1, over 1
    constexpr uint32_t kApart = (1u << 2) | (2u << 6) | (1u << 10) | (2u << 14) | (1u << 18) | (1u << 22);
    const int m = 4 << ((kApart >> (2 * step)) & 3u);
    const bool up = ((0x2880u >> step) & 1u) && (lane & m);      // lanes without the bit keep x and take the other's x for y
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const u64 v = __shfl_xor_sync(0xffffffffu, up ? x[i] : y[i], m);
      if (up) x[i] = v; else y[i] = v;
    }
    const float v = __shfl_xor_sync(0xffffffffu, up ? nx : ny, m);
    if (up) nx = v; else ny = v;
  }
  return __any_sync(0xffffffffu, big);
}

// Rows u, nearly the eigenvectors of the pair (h, g): h u = lambda g u, g nearly 1, to the rounding of the products (T. Ogita,
// K. Aishima, "Iterative refinement for symmetric eigenvalue decomposition", 2018): u_j += sum_i e_ij u_i with
// e_ij = (s_ij + lambda_j r_ij) / (lambda_j - lambda_i), r = 1 - u g u^T, s = u h u^T; for close pairs, and on the diagonal,
// r_ij / 2.  Both are made symmetric, to the bit, and so is what decides between the two: e_ij + e_ji has to be r_ij however close
// the pair (or the factors of four nearly equal eigenvalues come out 1e-4 off the right angle).  (The rotations alone leave the
// rounding of some fifty steps, 5e-7 of the largest eigenvalue.)  g: times 256.  Returns the largest |e_ij| of the first n rows:
// what is left after the pass is its square.
__device__ __forceinline__ float refine16(float (&u)[8], const float (&h)[8], const float (&g)[8], int n, int lane) {
  const int gid = lane >> 2, tig = lane & 3;
  uint32_t uh[4], ul[4], th[4], tl[4];
  float t[8], s[8], r[8];
  auto form = [&](const float (&x)[8], float (&o)[8]) {      // 256 u x u^T, twice
    split16(x, 1.f, th, tl);
    mul16_bt<false>(uh, ul, th, tl, t);                 // 256 u x
    split16(t, 1.f / 256.f, th, tl);
    mul16_bt<true>(th, tl, uh, ul, o);
    mul16_bt<true>(uh, ul, th, tl, t);
#pragma unroll
    for (int i = 0; i < 8; ++i) o[i] += t[i];
  };
  split16(u, 256.f, uh, ul);
  form(h, s);
  form(g, r);
  float l0, l1;
  diag16(s, lane, l0, l1);
  const float lmax = __shfl_sync(0xffffffffu, l0, 0);
  float most = 0.f;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int row = gid + 8 * (i >> 2), col = 8 * ((i >> 1) & 1) + 2 * tig + (i & 1);
    const float lc = __shfl_sync(0xffffffffu, ((i >> 1) & 1) ? l1 : l0, 4 * (2 * tig + (i & 1))), lr = (i >> 2) ? l1 : l0;
    const float ri = fmaf(r[i], -1.f / 131072.f, (row == col) ? 1.f : 0.f);
    // e_ij = r_ij / 2 + f_ij, f_ij = -f_ji; a numerator of rounding noise does not tell two close directions apart
    const float num = fmaf(0.5f * (lr + lc), ri, s[i]), gap = lr - lc, an = fabsf(num), ag = fabsf(gap);
    const bool turn = row != col && an < 0.25f * ag && (an > 2.5e-7f * lmax || an < 1e-4f * ag);
    t[i] = 0.5f * ri + (turn ? __fdividef(num, gap) : 0.f);
    // (rows of rounding noise may be nearly parallel: in full steps they grow without bound)
    if (row != col && row >= n && col >= n) t[i] = fminf(fmaxf(t[i], -0.12f), 0.12f);
    if (row != col && row < n) most = fmaxf(most, fabsf(t[i]));
  }
  split16(t, 4096.f, th, tl);
#pragma unroll
  for (int i = 0; i < 4; ++i) { uh[i] = movm(uh[i]); ul[i] = movm(ul[i]); }
  float c[2][4];
  mma_split<true>(c[0], th, tl, uh[0], uh[1], ul[0], ul[1]);
  mma_split<true>(c[1], th, tl, uh[2], uh[3], ul[2], ul[3]);
  from_tiles(c, t);
#pragma unroll
  for (int i = 0; i < 8; ++i) u[i] = fmaf(t[i], 1.f / (4096.f * 256.f), u[i]);
  return warp_max(most);
}

// w: unit vector gid at tokens 8 (W a + warp) + 2 tig + {0, 1}, zeros where a direction is null; top[0..RP): index or -1.  True if
// the block has to be left to the tridiagonal form.  A: the Gram matrix, rows 8 (W a + warp) + gid, columns 8 n + 2 tig + {0, 1}.
// sm: Filter's G_FLOATS, free; buf: V_FLOATS + X_FLOATS; ub: U_FLOATS.  null_at: eigenvalues up to it
// count as none.
template <int L, int RP>
__device__ __forceinline__ bool filter_solve(u64 (&A)[Filter<L>::NT][L / 8], float (&w)[Filter<L>::NT][2], float *sm, float *buf, float *ub,
                                             int *top, int r_eff, float null_at, int warp, int lane) {
  using F = Filter<L>;
  constexpr int W = F::W, NT = F::NT, KT = F::KT;
  const int gid = lane >> 2, tig = lane & 3;
  float *xbuf = buf + F::V_FLOATS;
  int xpar = 0, vpar = 0;
  // sums over the block's warps; two buffers, so that one barrier per call is enough
  auto xsum = [&](auto &v) {
    constexpr int N = sizeof(v) / sizeof(float);
    float *b = xbuf + xpar * W * 256;
    xpar ^= 1;
#pragma unroll
    for (int i = 0; i < N; ++i) b[warp * 256 + 32 * i + lane] = v[i];
    __syncthreads();
#pragma unroll
    for (int i = 0; i < N; ++i) v[i] = (b[32 * i + lane] + b[256 + 32 * i + lane]) + (b[512 + 32 * i + lane] + b[768 + 32 * i + lane]);
  };

  // ---- scale: the trace to [2^12, 2^13), so that elements and eigenvalues fit f16 with their low parts ---------------------------
  float gs, mu, fro2;
  {
    float t[1] = {0.f};
#pragma unroll
    for (int a = 0; a < NT; ++a)
#pragma unroll
      for (int w = 0; w < W; ++w)
        if (warp == w && tig == gid >> 1) t[0] += (gid & 1) ? hi(A[a][W * a + w]) : lo(A[a][W * a + w]);
    t[0] = warp_sum(t[0]);
    xsum(t);
    const float tr = t[0];
    if (!(tr < 1e30f) || !(tr > 0.f)) return true;      // (uniform) infinite or not a number
    gs = pow2(min(max(12 - ilog2(tr), -120), 120));
    mu = tr * gs * (1.0f / (float)L);
    const u64 g2 = pk(gs, gs);
    u64 f0 = 0ull, f1 = 0ull;
#pragma unroll
    for (int a = 0; a < NT; ++a)
#pragma unroll
      for (int n = 0; n < L / 8; n += 2) {
        A[a][n] = mul2(A[a][n], g2); A[a][n + 1] = mul2(A[a][n + 1], g2);
        f0 = fma2(A[a][n], A[a][n], f0); f1 = fma2(A[a][n + 1], A[a][n + 1], f1);
      }
    f0 = add2(f0, f1);
    float f[1] = {warp_sum(lo(f0) + hi(f0))};
    xsum(f);
    fro2 = f[0];
  }
  // (uniform) one direction holds nearly all of the trace: the others' eigenvalues are left to the tridiagonal form
  if (r_eff > 1 && fro2 > 0.93f * ((float)L * mu) * ((float)L * mu)) return true;
  // ---- G as B fragments -----------------------------------------------------------------------------------------------------------
  uint2 gh[NT][KT];                                     // the high halves
  uint2 *gl = reinterpret_cast<uint2 *>(sm) + warp * (NT * KT * 32) + lane;
#pragma unroll
  for (int kt = 0; kt < KT; ++kt)
#pragma unroll
    for (int a = 0; a < NT; ++a) {
      uint2 l;
      split_f16(lo(A[a][2 * kt]), hi(A[a][2 * kt]), gh[a][kt].x, l.x);
      split_f16(lo(A[a][2 * kt + 1]), hi(A[a][2 * kt + 1]), gh[a][kt].y, l.y);
      gl[(kt * NT + a) * 32] = l;
    }

  // ---- start: fixed vectors of no structure (odd multiples of 1/8 below 4) ---------------------------------------------------------------
  float V[NT][4], Vp[NT][4], P[NT][4];
#pragma unroll
  for (int a = 0; a < NT; ++a)
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const int vec = gid + 8 * (i >> 1), tok = 8 * (W * a + warp) + 2 * tig + (i & 1);
      uint32_t x = (uint32_t)(vec * 256 + tok + 1) * 0x9E3779B1u;
      x ^= x >> 15;
      x *= 0x85EBCA77u;
      x ^= x >> 13;
      V[a][i] = (float)(2 * (int)(x >> 27) - 31) * 0.125f;
      Vp[a][i] = 0.f;
    }

  // A fragments of tiles (a, a + 1) of rows scaled by s0 (gid) and s1 (gid + 8)
  auto split_pair = [&](const float (&X)[NT][4], int a, float s0, float s1, uint32_t (&h)[4], uint32_t (&l)[4]) {
    split_f16(X[a][0] * s0, X[a][1] * s0, h[0], l[0]);
    split_f16(X[a][2] * s1, X[a][3] * s1, h[1], l[1]);
    split_f16(X[a + 1][0] * s0, X[a + 1][1] * s0, h[2], l[2]);
    split_f16(X[a + 1][2] * s1, X[a + 1][3] * s1, h[3], l[3]);
  };
  // P = V G; 0: in f16 alone, 1: in split parts, 2: and their products added by rounding
  auto product = [&](auto mode_) {
    constexpr int MODE = decltype(mode_)::value;
    constexpr bool FULL = MODE > 0;
#pragma unroll
    for (int a = 0; a < NT; ++a) P[a][0] = P[a][1] = P[a][2] = P[a][3] = 0.f;
    auto step = [&](float (&c)[4], const uint32_t (&h)[4], const uint32_t (&l)[4], uint32_t bh0, uint32_t bh1, uint32_t bl0, uint32_t bl1) {
      if constexpr (MODE == 2) mma_split(c, h, l, bh0, bh1, bl0, bl1);
      else if constexpr (MODE == 1) mma_chain(c, h, l, bh0, bh1, bl0, bl1);
      else mma_f16(c, h[0], h[1], h[2], h[3], bh0, bh1);
    };
    // tile g of the block is half (g & 1) of step g / 2
    unsigned char *vb = reinterpret_cast<unsigned char *>(buf + vpar * KT * 256);
    vpar ^= 1;
#pragma unroll
    for (int a = 0; a < NT; ++a) {
      const int g = W * a + warp;
      uint2 h, l;
      split_f16(V[a][0], V[a][1], h.x, l.x);
      split_f16(V[a][2], V[a][3], h.y, l.y);
      unsigned char *d = vb + ((g >> 1) * 64 + lane) * 16 + (g & 1) * 8;
      *reinterpret_cast<uint2 *>(d) = h;
      if (FULL) *reinterpret_cast<uint2 *>(d + 512) = l;
    }
    __syncthreads();
#pragma unroll
    for (int kt = 0; kt < KT; ++kt) {
      const uint4 vh = *reinterpret_cast<const uint4 *>(vb + (kt * 64 + lane) * 16);
      uint4 vl = make_uint4(0u, 0u, 0u, 0u);
      if (FULL) vl = *reinterpret_cast<const uint4 *>(vb + (kt * 64 + 32 + lane) * 16);
      const uint32_t h[4] = {vh.x, vh.y, vh.z, vh.w}, l[4] = {vl.x, vl.y, vl.z, vl.w};
#pragma unroll
      for (int a = 0; a < NT; ++a) {
        uint2 bl = make_uint2(0u, 0u);
        if (FULL) bl = gl[(kt * NT + a) * 32];
        step(P[a], h, l, gh[a][kt].x, gh[a][kt].y, bl.x, bl.y);
      }
    }
  };
  // s = X Y^T (16 x 16) over all tokens, rows of X scaled by x0 and x1, those of Y by y0 and y1
  auto gram16 = [&](const float (&X)[NT][4], const float (&Y)[NT][4], float x0, float x1, float y0, float y1, float (&s)[8]) {
    float c[2][4];
#pragma unroll
    for (int a = 0; a < NT; a += 2) {
      uint32_t xh[4], xl[4], yh[4], yl[4];
      split_pair(X, a, x0, x1, xh, xl);
      split_pair(Y, a, y0, y1, yh, yl);
      if (a == 0) {
        mma_split<true>(c[0], xh, xl, yh[0], yh[2], yl[0], yl[2]);
        mma_split<true>(c[1], xh, xl, yh[1], yh[3], yl[1], yl[3]);
      } else {
        mma_split(c[0], xh, xl, yh[0], yh[2], yl[0], yl[2]);
        mma_split(c[1], xh, xl, yh[1], yh[3], yl[1], yl[3]);
      }
    }
    from_tiles(c, s);
    xsum(s);
  };
  // X = M X, M (16 x 16) as A fragments, rows of X scaled by s0 and s1
  auto rotate = [&](const uint32_t (&mh)[4], const uint32_t (&ml)[4], float (&X)[NT][4], float s0, float s1) {
#pragma unroll
    for (int a = 0; a < NT; ++a) {
      uint32_t h0, l0, h1, l1;
      split_f16(X[a][0] * s0, X[a][1] * s0, h0, l0);
      split_f16(X[a][2] * s1, X[a][3] * s1, h1, l1);
      h0 = movm(h0); h1 = movm(h1); l0 = movm(l0); l1 = movm(l1);
      mma_split<true>(X[a], mh, ml, h0, h1, l0, l1);
    }
  };
  auto row_dot = [&](const float (&X)[NT][4], const float (&Y)[NT][4], float &o0, float &o1) {      // (this warp's tokens)
    u64 t0 = 0ull, t1 = 0ull;
#pragma unroll
    for (int a = 0; a < NT; ++a) {
      t0 = fma2(pk(X[a][0], X[a][1]), pk(Y[a][0], Y[a][1]), t0);
      t1 = fma2(pk(X[a][2], X[a][3]), pk(Y[a][2], Y[a][3]), t1);
    }
    o0 = quad_sum(lo(t0) + hi(t0)); o1 = quad_sum(lo(t1) + hi(t1));
  };
  // V <- orthonormal rows (of length 16) of the same span: S = V V^T, rows of the inverse of its Cholesky factor by elimination.
  // What is left of a row's square, 256 to 1024 by the power of two that scales it, may be too near the rounding of S to be used:
  // below kPivot (2e-5 to 8e-5 of it) nothing is eliminated with the row.  Less the earlier rows it goes on to the next round, or
  // is left out of the solution (`final`), which then has to account for it.  n: squared norms of V's rows.
  auto orthonormalise = [&](const float (&n)[2], bool final) {
    constexpr float kPivot = 2e-2f;
    float s[8], m[8];
    // (a power of two: rows of length 16 to 32)
    const float s0 = pow2(4 - (min(max(ilog2(n[0]), -100), 120) >> 1)), s1 = pow2(4 - (min(max(ilog2(n[1]), -100), 120) >> 1));
    gram16(V, V, s0, s1, s0, s1, s);
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const int col = 8 * (e >> 1) + 2 * tig + (e & 1);
      m[e] = (col == gid) ? 1.f : 0.f;
      m[4 + e] = (col == gid + 8) ? 1.f : 0.f;
    }
    float p0 = 1.f, p1 = 1.f;
    auto eliminate = [&](auto E_, int j) {              // row j; E = 2 (j / 8) + (j & 1)
      constexpr int E = decltype(E_)::value, H = E >> 1, hj = 4 * H;
      const int src = (j & 7) * 4, ct = (j & 7) >> 1;
      float f0 = __shfl_sync(0xffffffffu, s[E], (lane & 28) | ct), f1 = __shfl_sync(0xffffffffu, s[4 + E], (lane & 28) | ct);
      const float raw = __shfl_sync(0xffffffffu, s[hj + E], src | ct), piv = fmaxf(raw, kPivot), inv = (raw < kPivot) ? 0.f : rcp(piv);
      f0 = (gid > j) ? -f0 * inv : 0.f;
      f1 = (gid + 8 > j) ? -f1 * inv : 0.f;
      if (gid == j) p0 = piv;
      if (gid + 8 == j) p1 = piv;
#pragma unroll
      for (int e = 2 * H; e < 4; ++e) {                 // (columns of earlier rows are not needed any more)
        const float pr = __shfl_sync(0xffffffffu, s[hj + e], src | tig);
        s[e] = fmaf(f0, pr, s[e]); s[4 + e] = fmaf(f1, pr, s[4 + e]);
      }
#pragma unroll
      for (int e = 0; e < 2 + 2 * H; ++e) {             // (nor are there columns of the inverse beyond j)
        const float pm = __shfl_sync(0xffffffffu, m[hj + e], src | tig);
        m[e] = fmaf(f0, pm, m[e]); m[4 + e] = fmaf(f1, pm, m[4 + e]);
      }
    };
#pragma unroll 1
    for (int j = 0; j < 8; j += 2) { eliminate(std::integral_constant<int, 0>{}, j); eliminate(std::integral_constant<int, 1>{}, j + 1); }
#pragma unroll 1
    for (int j = 8; j < 16; j += 2) { eliminate(std::integral_constant<int, 2>{}, j); eliminate(std::integral_constant<int, 3>{}, j + 1); }
    // rows of the inverse to [2^11, 2^12) at their largest: those of small pivots are long
    const float r0 = (final && p0 <= kPivot) ? 0.f : 16.f * rsqrtf(p0), r1 = (final && p1 <= kPivot) ? 0.f : 16.f * rsqrtf(p1);
    float q0 = 0.f, q1 = 0.f;
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      m[e] *= r0; m[4 + e] *= r1;
      q0 = fmaxf(q0, fabsf(m[e])); q1 = fmaxf(q1, fabsf(m[4 + e]));
    }
    q0 = fmaxf(q0, __shfl_xor_sync(0xffffffffu, q0, 1)); q1 = fmaxf(q1, __shfl_xor_sync(0xffffffffu, q1, 1));
    q0 = fmaxf(q0, __shfl_xor_sync(0xffffffffu, q0, 2)); q1 = fmaxf(q1, __shfl_xor_sync(0xffffffffu, q1, 2));
    const int x0 = 11 - min(max(ilog2(q0), -60), 60), x1 = 11 - min(max(ilog2(q1), -60), 60);
    const float w0 = pow2(x0), w1 = pow2(x1), o0 = pow2(-x0), o1 = pow2(-x1);
#pragma unroll
    for (int e = 0; e < 4; ++e) { m[e] *= w0; m[4 + e] *= w1; }
    uint32_t mh[4], ml[4];
    split16(m, 1.f, mh, ml);
    rotate(mh, ml, V, s0, s1);
#pragma unroll
    for (int a = 0; a < NT; ++a) { V[a][0] *= o0; V[a][1] *= o0; V[a][2] *= o1; V[a][3] *= o1; }
  };

  // ---- rounds of a filter and an orthonormalisation -----------------------------------------------------------------------------------
  // The filter of degree m damps eigenvalues in [0, b] and lets those above grow like T_m(2 x / b - 1).  First b from the
  // trace and the norm (the mean eigenvalue and 0.6 of their spread: about the upper quarter), then the smallest of the sixteen
  // vectors' Rayleigh quotients.  credit: the logarithm of the r-th direction's gain so far; when it would reach `need` with
  // this round, the small problem is solved.  What limits m: the leading direction's share of the other rows grows with it, and
  // takes their bits where it is left too large.
  constexpr float kCoarse = 4.f;                        // what vectors rounded to f16 can gain
  constexpr float kTol = 4e-7f, kTol1 = 2e-7f;      // |G w - theta w| over theta, and over theta_1
  float b = mu + 0.6f * sqrtf(fmaxf(fro2 * (1.0f / (float)L) - mu * mu, 0.f));
  float credit = 0.f, extra = 0.f, grown = 3.4f, parted = 1.f, s0 = 1.f, s1 = 1.f;      // (the first round lets vectors grow 30 times)
  bool last = false, failed = false;
  int m = 5, k = 0, round = 0, solves = 0;
#pragma unroll 1
  for (;;) {
    if (last && k == 0) product(std::integral_constant<int, 2>{});
    else if (round > 0) product(std::integral_constant<int, 1>{});
    else product(std::integral_constant<int, 0>{});
    float f1, f2, f3;                                   // V <- f1 P + f2 V + f3 Vp, rows scaled by s0, s1 per step
    if (k > 0) {
      f1 = __fdividef(4.0f, b); f2 = -2.0f; f3 = -1.0f;
    } else {
      f2 = -1.0f; f3 = 0.f;
      if (round > 0) {
        // Rayleigh quotients: the largest, the smallest, and the smallest of the first r rows but for rounding noise (the rows come
        // about in the order of their quotients)
        float d[4];
        row_dot(V, P, d[0], d[1]);
        row_dot(V, V, d[2], d[3]);
        xsum(d);
        d[0] = __fdividef(d[0], fmaxf(d[2], 1e-20f)); d[1] = __fdividef(d[1], fmaxf(d[3], 1e-20f));
        const float d_max = rows_max(fmaxf(d[0], d[1])), noise = 2e-6f * d_max;
        const int live = (__popc(__ballot_sync(0xffffffffu, d[2] > 0.f)) + __popc(__ballot_sync(0xffffffffu, d[3] > 0.f))) >> 2;
        const float least_live = -rows_max(-fminf((d[2] > 0.f) ? d[0] : d_max, (d[3] > 0.f) ? d[1] : d_max));
        const float d_min = (live > r_eff + 3) ? least_live : 0.f;      // (rows left out of a solution are zero)
        const float d_r = fminf(1.f / rows_max((gid < r_eff && d[0] > noise) ? 1.f / d[0] : 0.f), d_max);
        if (round == 1) credit = fminf(fmaxf(fmaf(-(float)m, __logf(cheb_damp(__fdividef(2.0f * d_r, b) - 1.0f)), -0.7f), 0.f), kCoarse);
        if (last) {
          // ---- H = V G V^T, its eigenvectors -----------------------------------------------------------------------------------
          float s[8], g[8];
          gram16(V, P, 1.f, 1.f, 1.f / 64.f, 1.f / 64.f, s);
          gram16(V, V, 1.f, 1.f, 1.f, 1.f, g);
          if (warp == 0) {
            u64 x[2] = {pk(s[0], s[1]), pk(s[2], s[3])}, y[2] = {pk(s[4], s[5]), pk(s[6], s[7])};
            const float thr = 8.f * d_r * d_r;          // (the squared norm of the r-th row is 16 d_r^2)
            const float null2 = 16.f * 5.8e-14f * d_max * d_max;      // 2^-22 of the largest is the error of any eigenvalue: none, then
#pragma unroll 1
            for (int sweep = 0; sweep < 8; ++sweep)
              if (!jacobi_sweep(x, y, thr, null2, lane)) break;
            float nx, ny;
            {
              const u64 a = fma2(x[1], x[1], mul2(x[0], x[0])), c = fma2(y[1], y[1], mul2(y[0], y[0]));
              nx = quad_sum(lo(a) + hi(a)); ny = quad_sum(lo(c) + hi(c));
            }
            // rows in descending order
            int q0 = 0, q1 = 0;
#pragma unroll 4
            for (int i = 0; i < 8; ++i) {
              const float o0 = __shfl_sync(0xffffffffu, nx, 4 * i), o1 = __shfl_sync(0xffffffffu, ny, 4 * i);
              q0 += (o0 > nx || (o0 == nx && i < gid)) + (o1 > nx);
              q1 += (o0 >= ny) + (o1 > ny || (o1 == ny && i < gid));
            }
            const float u0 = (nx > null2) ? rsqrtf(nx) : 0.f, u1 = (ny > null2) ? rsqrtf(ny) : 0.f;
            const u64 v0 = pk(u0, u0), v1 = pk(u1, u1);
            u64 *o = reinterpret_cast<u64 *>(ub) + tig;
            __syncwarp();
            o[q0 * 8] = mul2(x[0], v0); o[q0 * 8 + 4] = mul2(x[1], v0);
            o[q1 * 8] = mul2(y[0], v1); o[q1 * 8 + 4] = mul2(y[1], v1);
          }
          __syncthreads();
          uint32_t uh[4], ul[4];
          bool settled;                                 // (else the vectors need not be orthogonal to their rounding)
          {
            const u64 *o = reinterpret_cast<const u64 *>(ub) + gid * 8 + tig;
            const u64 t0 = o[0], t1 = o[4], t2 = o[64], t3 = o[68];
            float u[8] = {lo(t0), hi(t0), lo(t1), hi(t1), lo(t2), hi(t2), lo(t3), hi(t3)};
            float e = 1.f;
#pragma unroll 1
            for (int pass = 0; pass < 6 && e > 5e-5f; ++pass) e = refine16(u, s, g, r_eff, lane);
            settled = e < 3e-4f;
            split16(u, 256.f, uh, ul);
          }
          // the basis turned into the eigenvectors' (times 256)
          rotate(uh, ul, V, 1.f, 1.f);
          rotate(uh, ul, P, 1.f / 64.f, 1.f / 64.f);
          float q[2];                                   // x . x, x . G x / 64
          {
            u64 t0 = 0ull, t1 = 0ull;
#pragma unroll
            for (int a = 0; a < NT; ++a) {
              t0 = fma2(pk(V[a][0], V[a][1]), pk(V[a][0], V[a][1]), t0);
              t1 = fma2(pk(V[a][0], V[a][1]), pk(P[a][0], P[a][1]), t1);
            }
            q[0] = quad_sum(lo(t0) + hi(t0)); q[1] = quad_sum(lo(t1) + hi(t1));
            xsum(q);
          }
          const float th = (q[0] > 0.f) ? q[1] / q[0] : 0.f, xn = (q[0] > 0.f) ? rsqrtf(q[0]) : 0.f;      // eigenvalue gid over 64
          float e2[1] = {0.f};
#pragma unroll
          for (int a = 0; a < NT; ++a) {
            const float e0 = fmaf(-th, V[a][0], P[a][0]), e1 = fmaf(-th, V[a][1], P[a][1]);
            e2[0] = fmaf(e0, e0, fmaf(e1, e1, e2[0]));
          }
          e2[0] = quad_sum(e2[0]);
          xsum(e2);
          const float th1 = __shfl_sync(0xffffffffu, th, 0), thn = __shfl_down_sync(0xffffffffu, th, 4);
          const float err = sqrtf(e2[0]) * xn;
          // null rule: a direction below 1e-12 of the mean squared key norm is stored as zeros
          const bool keep = gid < r_eff && th * 64.f > null_at * gs;
          const bool sane = th1 > 0.f && th1 < 1e30f;
          // (a direction of rounding noise is one as well as another)
          const float allowed = (th > 1e-6f * th1) ? fmaf(kTol, th, kTol1 * th1) : 1e-6f * th1;
          const bool ok = sane && settled && __all_sync(0xffffffffu, !keep || err <= allowed);
          // A direction that is left out, or a faint one, stands for what the block has only if the others make up the trace, to its own
          // rounding or to what may follow after the r-th: rows end below the pivot, or come out as another pair's, because rounding
          // noise along the leading direction grows with it (one channel of deviation 100, rank 8: an eigenvalue 7e-6 of the largest missed).
          const float rest = mu * (float)L / 64.f - 0.25f * warp_sum((gid < r_eff) ? fmaxf(th, 0.f) : 0.f);
          const float least = -rows_max((gid < r_eff) ? -th : -th1), after = (least > 3e-4f * th1) ? 2.f * least : 0.f;
          const bool lost = !(least > 1.5e-3f * th1) && !(rest <= fmaf(2e-7f, th1, 1.5e-7f / 64.f * (mu * (float)L)) + after);
          // Two equal eigenvalues: any basis of their plane is right, and the careful kernel has the say.
          const bool equal = keep && gid + 1 < r_eff && thn > 2.4e-7f * th1 && th - thn <= 2.4e-7f * th;
          ++round;
          if (ok || lost || !sane || round > 20 || ++solves == 3) {
            failed = !ok || lost || __any_sync(0xffffffffu, equal);
            const float wn = keep ? xn : 0.f;
#pragma unroll
            for (int a = 0; a < NT; ++a) { w[a][0] = V[a][0] * wn; w[a][1] = V[a][1] * wn; }
            if (warp == 0 && tig == 0 && gid < RP) top[gid] = keep ? gid : -1;
            break;
          }
          const float far = warp_max(keep ? __fdividef(err, allowed) : 0.f);
          extra = fminf(extra + 1.5f * __logf(fminf(fmaxf(far, 1.f), 1e6f)) + 3.0f, 40.f);
          last = false;
#pragma unroll
          for (int a = 0; a < NT; ++a)
#pragma unroll
            for (int i = 0; i < 4; ++i) V[a][i] *= 1.f / 256.f;
          continue;
        }
        // Left to the tridiagonal form: wanted directions so far below the leading one that its rounding outgrows them, and sixteen
        // directions too close to one another to be parted soon.
        failed = d_max < 1.17f * d_min || (round > 4 && d_r < 2e-4f * d_max);
        if (failed) break;
        b = fmaxf(fmaxf(d_min, 0.02f * d_r), 1e-5f * d_max);      // (lower, and the leading rows drown the others)
        const float ib = __fdividef(2.0f, b);
        const float xr = -__logf(cheb_damp(fmaf(d_r, ib, -1.0f))), x1 = fmaxf(-__logf(cheb_damp(fmaf(d_max, ib, -1.0f))), 0.5f);
        const float need = __logf(1.0f / kTol) + 6.0f + 0.5f * __logf(__fdividef(d_max, d_r)) + extra;
        // The other rows' share of the leading direction is what the rounds so far have left: it may grow to some fifty times the
        // rows themselves, and in the rows that are wanted to no more than a few times.
        const float cap = fminf(__fdividef(fminf(grown + 4.f, 15.f), x1), __fdividef(parted + 1.5f, fmaxf(x1 - xr, 0.1f)));
        m = (int)fminf(ceilf(__fdividef(need - credit + 0.7f, fmaxf(xr, 0.05f))), cap);
        m = min(max(m, 1), 12);
        grown = fmaf((float)m, x1, grown); parted = fmaf((float)m, x1 - xr, parted);
        credit += fmaxf(fmaf((float)m, xr, -0.7f), 0.f);
        last = credit >= need || round >= 16;
        // a row is damped by its own growth, and by so much that what it may hold of the leading direction stays within f16
        const float least = __expf(__fdividef(6.5f, (float)m) - x1);
        s0 = fminf(cheb_damp(fmaf(d[0], ib, -1.0f)), least); s1 = fminf(cheb_damp(fmaf(d[1], ib, -1.0f)), least);
      }
      f1 = __fdividef(2.0f, b);
    }
    float n[2];
    {
      const u64 a0 = pk(f1 * s0, f1 * s0), b0 = pk(f2 * s0, f2 * s0), c0 = pk(f3 * s0 * s0, f3 * s0 * s0);
      const u64 a1 = pk(f1 * s1, f1 * s1), b1 = pk(f2 * s1, f2 * s1), c1 = pk(f3 * s1 * s1, f3 * s1 * s1);
#pragma unroll
      for (int a = 0; a < NT; ++a) {
        const u64 v = pk(V[a][0], V[a][1]), w = pk(V[a][2], V[a][3]);
        const u64 nv = fma2(a0, pk(P[a][0], P[a][1]), fma2(b0, v, mul2(c0, pk(Vp[a][0], Vp[a][1]))));
        const u64 nw = fma2(a1, pk(P[a][2], P[a][3]), fma2(b1, w, mul2(c1, pk(Vp[a][2], Vp[a][3]))));
        Vp[a][0] = lo(v); Vp[a][1] = hi(v); Vp[a][2] = lo(w); Vp[a][3] = hi(w);
        V[a][0] = lo(nv); V[a][1] = hi(nv); V[a][2] = lo(nw); V[a][3] = hi(nw);
      }
    }
    ++k;
    if (k == m || round == 0) {
      row_dot(V, V, n[0], n[1]);
      xsum(n);
      // (the first round, whose growth is not known, ends when the vectors have grown some 30 times)
      if (round == 0 && warp_max(fmaxf(n[0], n[1])) > 3e5f) m = k;
      if (k == m) {
        k = 0;
        ++round;
        orthonormalise(n, last);
      }
    }
  }
  __syncthreads();                                      // G and the sums have been read by all warps
  return failed;
}

}  // namespace
}  // namespace cobs
