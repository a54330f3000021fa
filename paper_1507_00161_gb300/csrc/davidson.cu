// Davidson's vector algebra and its projected (Ritz) problem.
//
// One Davidson iteration after its product A v_k is a chain of short dependent pieces on a
// few vectors of n elements (a few hundred in the sd shell, 10^5 at M = 4096):
//     h = V^T (A v_k),   lowest Ritz pair,   x = V y, r = A V y - theta x,  t = r / (theta - D),
//     t <- t - V (V^T t) twice,   v_{k+1} = t / |t|.
// The chain is bound by launches and by the latency of each piece, not by bytes: at n = 1000
// the vectors are 0.2 MB.  It runs as five launches with one readback (dav_chain).  The last
// block of a launch to finish adds the partial sums of all blocks (a counter, no waiting), so
// reductions need no launches of their own; the first launch's last block also solves the
// Ritz problem.  The correction and the next vector are computed before the host has seen the
// residual; a run that ends there ignores them.
//
// Every sum keeps one fixed shape whatever kernel forms it: 264 chunks of the vector, in a
// chunk 256 partial sums (elements t, t + 256, ...), each 32 of them added as a binary tree,
// the eight trees in order; the chunk sums are added the same way.  Far from convergence
// theta lies inside the range of the diagonal, and the correction amplifies a last-bit
// difference by orders of magnitude per iteration, so a run is only reproducible if the sums
// are the same to the bit in every kernel.  A warp forms the eight trees together: after the
// first level half of its lanes would idle, so two trees share each instruction from there on
// (9 FP64 additions instead of 40; FP64 runs at 1.7 lanes per clock and SM here).
//
// Short chunks (n up to 8448) are one tree, its empty levels left out; x and A x of an element are
// formed by different warps.
//
// Measured (GB300), chain and Ritz problem together, against 15 launches and two readbacks per
// iteration, the same results to the bit in every run compared: with the products' changes a Davidson run of pf 4p+4n
// (n = 700, ~55 products) 45.9 -> 19.2 ms, an sd-shell sweep at M = 64 200 -> 120 ms, five instances
// in batch mode 505 -> 316 ms; residual and first orthogonalisation at n = 300 13.7 + 11.5 -> 9.3 + 7.8 us.
#include <math.h>
#include <stdint.h>

#include <mutex>

#include "common.h"
#include "newton.cuh"

namespace dmrg {

namespace {

constexpr int kThr = 256;
constexpr int kWarps = kThr / 32;
constexpr int kChunks = 264;          // chunks of a vector = blocks of a launch

// sum of 256 values, p[t] held as p[w] = value 32 w + lane: the binary tree over each 32
// (lane l + lane l + 16, then 8, 4, 2, 1), the eight trees added in order; every lane
__device__ __forceinline__ double tree_sum(const double (&p)[kWarps]) {
  const unsigned all = 0xffffffffu;
  const int lane = threadIdx.x & 31;
  double a[4], b[2], c;
  const bool h16 = lane & 16, h8 = lane & 8, h4 = lane & 4;
#pragma unroll
  for (int i = 0; i < 4; ++i) {   // lanes 0-15: tree 2 i, lanes 16-31: tree 2 i + 1
    const double mine = h16 ? p[2 * i + 1] : p[2 * i];
    const double give = h16 ? p[2 * i] : p[2 * i + 1];
    a[i] = mine + __shfl_xor_sync(all, give, 16);
  }
#pragma unroll
  for (int i = 0; i < 2; ++i) {
    const double mine = h8 ? a[2 * i + 1] : a[2 * i];
    const double give = h8 ? a[2 * i] : a[2 * i + 1];
    b[i] = mine + __shfl_xor_sync(all, give, 8);
  }
  {
    const double mine = h4 ? b[1] : b[0];
    const double give = h4 ? b[0] : b[1];
    c = mine + __shfl_xor_sync(all, give, 4);
  }
  c += __shfl_xor_sync(all, c, 2);
  c += __shfl_xor_sync(all, c, 1);
  // tree 4 x + 2 y + z sits in the lanes with bit 2 = x, bit 3 = y, bit 4 = z
  double s = 0.0;
#pragma unroll
  for (int w = 0; w < kWarps; ++w)
    s += __shfl_sync(all, c, (w & 4) | ((w & 2) << 2) | ((w & 1) << 4));
  return s;
}

// the sum of v[i] w[i] over a chunk of len elements, one warp (valid in lane 0)
__device__ __forceinline__ double chunk_dot(const double* v, const double* w, int len) {
  const int lane = threadIdx.x & 31;
  if (len <= 32) {   // one tree, whose levels of at least len only add zeros
    double x = lane < len ? fma(v[lane], w[lane], 0.0) : 0.0;
    for (int o = 16; o > 0; o >>= 1)
      if (o < len) x += __shfl_xor_sync(0xffffffffu, x, o);
    return x;
  }
  double p[kWarps];
#pragma unroll
  for (int q = 0; q < kWarps; ++q) p[q] = 0.0;
  for (int base = 0; base < len; base += kThr)
#pragma unroll
    for (int q = 0; q < kWarps; ++q) {
      const int i = base + 32 * q + lane;
      if (i < len) p[q] = fma(v[i], w[i], p[q]);
    }
  return tree_sum(p);
}

// the sum of a launch's kChunks chunk sums, one warp
__device__ __forceinline__ double chunks_sum(const double* part) {
  const int lane = threadIdx.x & 31;
  double p[kWarps];
#pragma unroll
  for (int q = 0; q < kWarps; ++q) p[q] = 0.0 + __ldcg(part + 32 * q + lane);
  if (lane < kChunks - kThr) p[0] += __ldcg(part + kThr + lane);
  return tree_sum(p);
}

// the sum of one value per thread, in thread 0 (shared by all launches of the chain)
__device__ __forceinline__ double block_sum(double v, double* sh) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_down_sync(0xffffffffu, v, o);
  if ((threadIdx.x & 31) == 0) sh[threadIdx.x >> 5] = v;
  __syncthreads();
  double r = 0.0;
  if (threadIdx.x == 0)
    for (int w = 0; w < kWarps; ++w) r += sh[w];
  return r;
}

// true in every thread of the block that arrives last; *count is left at zero.  What the
// other blocks wrote before is visible to it.
__device__ __forceinline__ bool last_block(int* count) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(count, 1) == int(gridDim.x) - 1;
    if (s_last) *count = 0;
    __threadfence();
  }
  __syncthreads();
  return s_last != 0;
}

struct Chunk {
  int64_t i0;
  int len;
};
__device__ __forceinline__ Chunk my_chunk(int64_t n) {
  const int64_t c = (n + gridDim.x - 1) / gridDim.x;
  const int64_t i0 = int64_t(blockIdx.x) * c;
  return {i0, int(max(int64_t(0), min(n, i0 + c) - i0))};
}

// out[j] = vecs[j] . w, j < k
__global__ void __launch_bounds__(kThr)
k_dav_dots(const double* const* vecs, int k, const double* __restrict__ w, int64_t n,
           double* part, double* __restrict__ out, int* count) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Chunk c = my_chunk(n);
  for (int j = warp; j < k; j += kWarps) {
    const double s = chunk_dot(vecs[j] + c.i0, w + c.i0, c.len);
    if (lane == 0) part[j * kChunks + blockIdx.x] = s;
  }
  if (!last_block(count)) return;
  for (int j = warp; j < k; j += kWarps) {
    const double s = chunks_sum(part + j * kChunks);
    if (lane == 0) out[j] = s;
  }
}

// x, r, t; sums[0] = |r|^2, sums[1] = |t|^2, sums[2 ..] = V^T t
__global__ void __launch_bounds__(kThr)
k_dav_residual(const double* const* V, const double* const* AV, const double* __restrict__ y,
               const double* __restrict__ theta, const double* __restrict__ diag, int k,
               int64_t n, double* x, double* r, double* t,
               double* part, double* __restrict__ sums, int* count) {
  __shared__ double sy[64], s_ax[kThr / 2];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid < k) sy[tid] = y[tid];
  __syncthreads();
  const Chunk c = my_chunk(n);
  const double th = *theta;
  auto sum = [&](const double* const* W, int64_t i) {
    double v = 0.0;
#pragma unroll 4
    for (int j = 0; j < k; ++j) v = fma(sy[j], W[j][i], v);
    return v;
  };
  auto finish = [&](int64_t i, double xs, double as) {
    const double rv = fma(-th, xs, as);
    double den = th - diag[i];
    if (fabs(den) < 1e-8) den = den < 0.0 ? -1e-8 : 1e-8;
    x[i] = xs;
    r[i] = rv;
    t[i] = rv / den;
  };
  if (c.len <= kThr / 2) {   // a short chunk: x and A x of an element by different warps
    const int e = tid & (kThr / 2 - 1);
    double xs = 0.0;
    if (e < c.len) {
      if (tid < kThr / 2) xs = sum(V, c.i0 + e);
      else s_ax[e] = sum(AV, c.i0 + e);
    }
    __syncthreads();
    if (tid < c.len) finish(c.i0 + tid, xs, s_ax[tid]);
  } else {
    for (int64_t i = c.i0 + tid; i < c.i0 + c.len; i += kThr) finish(i, sum(V, i), sum(AV, i));
  }
  __syncthreads();   // the chunk is read by other warps below
  for (int j = warp; j < k + 2; j += kWarps) {
    const double* u = (j == 0 ? r : t) + c.i0;
    const double s = chunk_dot(j < 2 ? u : V[j - 2] + c.i0, u, c.len);
    if (lane == 0) part[j * kChunks + blockIdx.x] = s;
  }
  if (!last_block(count)) return;
  for (int j = warp; j < k + 2; j += kWarps) {
    const double s = chunks_sum(part + j * kChunks);
    if (lane == 0) sums[j] = s;
  }
}

// t <- t - V h; then h <- V^T t, or (LAST) *h = |t|^2
template <bool LAST>
__global__ void __launch_bounds__(kThr)
k_dav_orth(const double* const* V, int k, int64_t n, const double* __restrict__ h, double* t,
           double* part, double* __restrict__ out, int* count) {
  __shared__ double sh[64], red[kWarps];
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  if (tid < k) sh[tid] = h[tid];
  __syncthreads();
  const Chunk c = my_chunk(n);
  double tt = 0.0;
  for (int64_t i = c.i0 + tid; i < c.i0 + c.len; i += kThr) {
    double s = t[i];
#pragma unroll 4
    for (int j = 0; j < k; ++j) s = fma(-sh[j], V[j][i], s);
    t[i] = s;
    if (LAST) tt = fma(s, s, tt);
  }
  if (LAST) {
    const double s = block_sum(tt, red);
    if (tid == 0) part[blockIdx.x] = s;
  } else {
    __syncthreads();
    for (int j = warp; j < k; j += kWarps) {
      const double s = chunk_dot(V[j] + c.i0, t + c.i0, c.len);
      if (lane == 0) part[j * kChunks + blockIdx.x] = s;
    }
  }
  if (!last_block(count)) return;
  for (int j = warp; j < (LAST ? 1 : k); j += kWarps) {
    const double s = chunks_sum(part + j * kChunks);
    if (lane == 0) out[j] = s;
  }
}

// v = t / |t|; sc[0..3] = {theta, |r|^2, |t|^2 before and after}
__global__ void __launch_bounds__(kThr)
k_dav_next(const double* __restrict__ t, const double* __restrict__ tt,
           const double* __restrict__ sums, const double* __restrict__ theta, int64_t n,
           double* __restrict__ v, double* __restrict__ sc) {
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    sc[0] = *theta;
    sc[1] = sums[0];
    sc[2] = sums[1];
    sc[3] = *tt;
  }
  const double f = 1.0 / sqrt(*tt);
  for (int64_t i = int64_t(blockIdx.x) * kThr + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * kThr)
    v[i] = t[i] * f;
}

// ------------------------------------------------------------------------------------
// Ritz problem: H (k x k, row j holds <v_i, A v_j> for i <= j, leading dimension ld) -> the two
// lowest eigenvalues w[0..1] and their coefficients Y[0 ..], Y[64 ..], each with its largest
// |component| positive (lowest index on ties): cyclic Jacobi with the round-robin pairs and the
// rotations of jacobi.cuh, the same operations on every element in the same order, in one block.
//
// One FP64 instruction of a warp occupies its scheduler's FP64 unit for 64 clocks (19 per SM with
// four or more warps), whatever its active lanes and however independent the next one is, so
// the time is the count of FP64 instructions on the critical path.  A rotation takes 30 of them
// here against 47 with library divisions and roots, comparisons included; a round rotates the
// matrix in 4.
//   - Warp 0 forms the rotations of the next round while the other warps apply this round's to A
//     and V: it first rotates the three elements per pair that it needs itself (A is double-
//     buffered), so the chain of divisions and roots never waits for the matrix.  Signs, zeros
//     and powers of two are handled as integers.
//   - Rows and columns of A are rotated in one pass, four lanes per 2 x 2 block (the rows of one
//     pair, the columns of another): one element each, exchanged by shuffles.
// Measured (GB300) against rotations, rows, columns one after the other with library divisions:
// 3900 clocks per round against 5700; 8 vectors 65 us, 16 vectors 170 us, 24 vectors 340 us.
// ------------------------------------------------------------------------------------
constexpr int kMaxK = 64;

// rotation that annihilates a_pq: theta = (a_qq - a_pp) / (2 a_pq), t = sgn(theta) /
// (|theta| + sqrt(theta^2 + 1)), c = 1 / sqrt(t^2 + 1), s = t c; none for a_pq = 0.  All lanes
// of `lanes` call it.  A warp whose operands all stay in the middle of the exponent range
// (theta below 2^180) takes the straight line; otherwise the library's operations.
__device__ __forceinline__ void rotation(unsigned lanes, double app, double aqq, double apq,
                                         double& c, double& s) {
  const double diff = aqq - app;
  const bool none = is_zero(apq);
  const bool fine = none || (mid_range(apq) && mid_range(diff) && exponent(diff) - exponent(apq) < 180);
  if (__all_sync(lanes, fine)) {
    const double th = quick_div(diff, times_pow2(apq, 1));
    const double u = quick_rcp(fabs(th) + quick_sqrt(fma(th, th, 1.0)));
    const double t = flip_if(u, __double2hiint(th) < 0);
    c = quick_rcp(quick_sqrt(fma(t, t, 1.0)));
    s = t * c;
  } else {
    const double th = diff / (2.0 * apq);
    const double t = (th >= 0.0 ? 1.0 : -1.0) / (fabs(th) + sqrt(fma(th, th, 1.0)));
    c = 1.0 / sqrt(fma(t, t, 1.0));
    s = t * c;
  }
  if (none) {
    c = 1.0;
    s = 0.0;
  }
}

// round-robin pair number a of round r among m players
__device__ __forceinline__ void pair_of(int m, int r, int a, int& p, int& q) {
  int x = m - 1, y = r;
  if (a > 0) {
    x = r + a;
    if (x >= m - 1) x -= m - 1;
    y = r - a;
    if (y < 0) y += m - 1;
  }
  p = min(x, y);
  q = max(x, y);
}

struct RitzShared {
  double c[2][kMaxK / 2], s[2][kMaxK / 2];   // rotations, double-buffered by round
  int p[2][kMaxK / 2], q[2][kMaxK / 2];
  double norm[2 * kWarps], w[kMaxK];   // off-diagonal and whole norm by warp
  int low[2];
  // pair a of round r at [r * half + a]: p, q, and of each its partner and its pair's number in
  // the round before (6 bits each)
  uint32_t low_bits[(kMaxK - 1) * kMaxK / 2], high_bits[(kMaxK - 1) * kMaxK / 2];
};
struct PairOf {
  int p, q, p_mate, q_mate, p_pair, q_pair;
};
__device__ __forceinline__ PairOf pair_entry(const RitzShared& sh, int at) {
  const uint32_t l = sh.low_bits[at], h = sh.high_bits[at];
  return {int(l & 63), int(l >> 6 & 63), int(l >> 12 & 63), int(l >> 18 & 63), int(h & 63),
          int(h >> 6 & 63)};
}

// x_p, x_q -> c x_p - s x_q, s x_p + c x_q (first product fused, second rounded)
__device__ __forceinline__ double rotated(double xp, double xq, double c, double s, bool is_q) {
  return fma(is_q ? s : c, xp, flip_if((is_q ? c : s) * xq, !is_q));
}

// element (i, j) of A (k x k) after the rotations of buffer buf: i was paired with i_mate in pair
// i_pair, j likewise
__device__ __forceinline__ double element_after(const double* A, int k, const RitzShared& sh, int buf,
                                                int i, int i_mate, int i_pair, int j, int j_mate,
                                                int j_pair) {
  const double ca = sh.c[buf][i_pair], sa = sh.s[buf][i_pair];
  const double cb = sh.c[buf][j_pair], sb = sh.s[buf][j_pair];
  const int i2 = min(i_mate, k - 1), j2 = min(j_mate, k - 1);   // (a bye has no rotation)
  const double x_ij = A[i * k + j], x_2j = A[i2 * k + j], x_i2 = A[i * k + j2], x_22 = A[i2 * k + j2];
  const bool lo = i > i_mate, right = j > j_mate;
  double y = x_ij, y2 = x_i2;
  if (!is_zero(sa)) {
    y = rotated(lo ? x_2j : x_ij, lo ? x_ij : x_2j, ca, sa, lo);
    y2 = rotated(lo ? x_22 : x_i2, lo ? x_i2 : x_22, ca, sa, lo);
  }
  return is_zero(sb) ? y : rotated(right ? y2 : y, right ? y : y2, cb, sb, right);
}

// rotations of round r into buffer buf (one warp): the elements read from A, or (after) as they
// will be once the rotations of buffer buf ^ 1 (the round before) have been applied to A
__device__ __forceinline__ void round_rotations(const double* A, int k, int half, int r, bool after,
                                                RitzShared& sh, int buf) {
  const int lane = threadIdx.x & 31;
  // lane -> pair a, and which of its elements (p, p), (q, q), (p, q) the lane rotates first
  int g = 0, a = lane;
  if (3 * half <= 32) {
    g = lane >= 2 * half ? 2 : lane >= half ? 1 : 0;
    a = lane - g * half;
  } else if (half <= 16) {
    g = lane >> 4;
    a = lane & 15;
  }
  const PairOf e = pair_entry(sh, r * half + min(a, half - 1));
  const int p = e.p, q = e.q;
  const bool bye = q >= k;
  double app, aqq = 0.0, apq = 0.0;
  if (!after) {
    app = A[p * k + p];
    if (!bye) {
      aqq = A[q * k + q];
      apq = A[p * k + q];
    }
  } else if (3 * half <= 32) {   // the three elements of all pairs at once
    const bool iq = g == 1, jq = g > 0;   // (p, p), (q, q), (p, q)
    const double x =
        bye && g > 0 ? 0.0
                     : element_after(A, k, sh, buf ^ 1, iq ? q : p, iq ? e.q_mate : e.p_mate,
                                     iq ? e.q_pair : e.p_pair, jq ? q : p, jq ? e.q_mate : e.p_mate,
                                     jq ? e.q_pair : e.p_pair);
    app = x;
    aqq = __shfl_sync(0xffffffffu, x, (lane + half) & 31);
    apq = __shfl_sync(0xffffffffu, x, (lane + 2 * half) & 31);
  } else {
    const bool is_q = g == 1;
    app = is_q && bye ? 0.0
                      : element_after(A, k, sh, buf ^ 1, is_q ? q : p, is_q ? e.q_mate : e.p_mate,
                                      is_q ? e.q_pair : e.p_pair, is_q ? q : p,
                                      is_q ? e.q_mate : e.p_mate, is_q ? e.q_pair : e.p_pair);
    if (half <= 16)
      aqq = __shfl_sync(0xffffffffu, app, (lane + 16) & 31);
    else if (!bye)
      aqq = element_after(A, k, sh, buf ^ 1, q, e.q_mate, e.q_pair, q, e.q_mate, e.q_pair);
    if (!bye) apq = element_after(A, k, sh, buf ^ 1, p, e.p_mate, e.p_pair, q, e.q_mate, e.q_pair);
  }
  if (lane >= half || bye) apq = 0.0;   // (spare lanes and a bye: no rotation)
  double c, s;
  rotation(0xffffffffu, app, aqq, apq, c, s);
  if (lane < half) {
    sh.p[buf][lane] = p;
    sh.q[buf][lane] = q;
    sh.c[buf][lane] = c;
    sh.s[buf][lane] = s;
  }
}

__device__ void ritz_block(const double* H, int ld, int k, double* sm, double* w, double* Y) {
  __shared__ RitzShared sh;
  const int tid = threadIdx.x, warp = tid >> 5, lane = tid & 31;
  double* A = sm;              // before a round
  double* B = sm + k * k;      // after it
  double* V = sm + 2 * k * k;
  double off = 0.0, tot = 0.0;   // off-diagonal Frobenius norm against the full norm
  auto norms = [&](double x, bool diagonal) {
    tot = fma(x, x, tot);
    if (!diagonal) off = fma(x, x, off);
  };
  auto norms_out = [&] {   // lanes 0-15 add the one, 16-31 the other
    const bool up = lane & 16;
    double x = (up ? tot : off) + __shfl_xor_sync(0xffffffffu, up ? off : tot, 16);
    for (int o = 8; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    if ((lane & 15) == 0) sh.norm[(up ? kWarps : 0) + warp] = x;
    off = tot = 0.0;
  };
  auto converged = [&] {   // the same sums in every warp
    double x = sh.norm[lane & 15];
    for (int o = 4; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
    const double o = __shfl_sync(0xffffffffu, x, 0), t = __shfl_sync(0xffffffffu, x, 8);
    return o <= 1e-30 * t || t == 0.0;
  };
  for (int i = tid; i < k * k; i += kThr) {
    const int r = i / k, c = i - r * k;
    const double x = (r >= c) ? __ldcg(H + r * ld + c) : __ldcg(H + c * ld + r);
    A[i] = x;
    V[i] = r == c ? 1.0 : 0.0;
    norms(x, r == c);
  }
  norms_out();
  const int m = (k + 1) & ~1, half = m / 2;
  for (int i = tid; i < (m - 1) * half; i += kThr) {
    const int r = i / half;
    int p, q;
    pair_of(m, r, i - r * half, p, q);
    const int before = r ? r - 1 : m - 2;
    auto mate = [&](int x, int& pair) {   // partner and pair of player x in the round before
      int e = x == m - 1 ? 0 : x - before;
      if (e < 0) e += m - 1;
      pair = e < half ? e : m - 1 - e;
      int y, z;
      pair_of(m, before, pair, y, z);
      return x == y ? z : y;
    };
    int pp, qp;
    const int pm = mate(p, pp), qm = mate(q, qp);
    sh.low_bits[i] = uint32_t(p | q << 6 | pm << 12 | qm << 18);
    sh.high_bits[i] = uint32_t(pp | qp << 6);
  }
  __syncthreads();
  const int inv = 65536 / max(half, 1) + 1;   // x / half = (x inv) >> 16 for x < half^2 <= 1024
  int buf = 0;
  if (k > 1 && !converged()) {
    if (warp == 0) round_rotations(A, k, half, 0, false, sh, 0);
    __syncthreads();
    for (int sweep = 0; sweep < 40; ++sweep) {
      for (int r = 0; r < m - 1; ++r) {
        const bool last = r == m - 2;
        if (warp == 0) {
          round_rotations(A, k, half, last ? 0 : r + 1, true, sh, buf ^ 1);
        } else {
          // B <- P^T A P: rows of pair a, columns of pair b; lane bit 1 = row, bit 0 = column of
          // the block (whole groups of four lanes take part)
          const int nel = 4 * half * half;
          for (int e0 = (tid & ~31) - 32; e0 < nel; e0 += kThr - 32) {
            const int e = e0 + lane;
            const int blk = min(e, nel - 1) >> 2, a = (blk * inv) >> 16, b = blk - a * half;
            const bool lo = tid & 2, right = tid & 1;
            const int pa = sh.p[buf][a], qa = sh.q[buf][a], pb = sh.p[buf][b], qb = sh.q[buf][b];
            const bool ra = qa < k, rb = qb < k;   // (an odd k has one pair with a bye)
            const int row = lo ? qa : pa, col = right ? qb : pb;
            const bool mine = e < nel && row < k && col < k;
            double x = mine ? A[row * k + col] : 0.0;
            const double sa = sh.s[buf][a], ca = sh.c[buf][a];
            const double up = __shfl_xor_sync(0xffffffffu, x, 2);
            if (ra && !is_zero(sa)) x = rotated(lo ? up : x, lo ? x : up, ca, sa, lo);
            const double sb = sh.s[buf][b], cb = sh.c[buf][b];
            const double side = __shfl_xor_sync(0xffffffffu, x, 1);
            if (rb && !is_zero(sb)) x = rotated(right ? side : x, right ? x : side, cb, sb, right);
            if (mine) {
              B[row * k + col] = x;
              if (last) norms(x, row == col);
            }
          }
          for (int e = tid - 32; e < half * k; e += kThr - 32) {   // V <- V P
            const int a = e / k, row = e - a * k;
            const int p = sh.p[buf][a], q = sh.q[buf][a];
            const double c = sh.c[buf][a], s = sh.s[buf][a];
            if (q >= k || is_zero(s)) continue;
            const double vp = V[row * k + p], vq = V[row * k + q];
            V[row * k + p] = fma(c, vp, -(s * vq));
            V[row * k + q] = fma(s, vp, c * vq);
          }
        }
        if (last) norms_out();
        __syncthreads();
        double* t = A;
        A = B;
        B = t;
        buf ^= 1;
      }
      if (converged()) break;   // (the rotations formed ahead are dropped)
      __syncthreads();
    }
  }
  if (tid < k) sh.w[tid] = A[tid * k + tid];
  if (tid < 2) sh.low[tid] = min(tid, k - 1);   // (stays only if the weights are NaN)
  __syncthreads();
  // ranks 0 and 1, ties by index
  if (tid < k) {
    const double wi = sh.w[tid];
    int rank = 0;
    for (int j = 0; j < k; ++j) rank += sh.w[j] < wi || (sh.w[j] == wi && j < tid);
    if (rank < 2) sh.low[rank] = tid;
  }
  __syncthreads();
  if (warp < min(k, 2)) {
    const int col = sh.low[warp];
    double bv = -1.0, sg = 1.0;
    int bi = 0x7fffffff;
    for (int i = lane; i < k; i += 32) {
      const double v = V[i * k + col], a = fabs(v);
      if (a > bv) {
        bv = a;
        bi = i;
        sg = v < 0.0 ? -1.0 : 1.0;
      }
    }
    for (int o = 16; o > 0; o >>= 1) {
      const double ov = __shfl_xor_sync(0xffffffffu, bv, o), os = __shfl_xor_sync(0xffffffffu, sg, o);
      const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
      if (ov > bv || (ov == bv && oi < bi)) {
        bv = ov;
        bi = oi;
        sg = os;
      }
    }
    for (int i = lane; i < k; i += 32) Y[64 * warp + i] = sg * V[i * k + col];
    if (lane == 0) w[warp] = sh.w[col];
  }
}

__global__ void __launch_bounds__(kThr)
k_ritz(const double* H, int ld, int k, double* __restrict__ w, double* __restrict__ Y) {
  extern __shared__ double sm[];
  ritz_block(H, ld, k, sm, w, Y);
}

// H[k - 1][j] = V[j] . Av, j < k, then the Ritz problem, by the last block
__global__ void __launch_bounds__(kThr)
k_dav_ritz(const double* const* V, int k, const double* __restrict__ Av, int64_t n, double* part,
           double* H, int ld, double* __restrict__ w, double* __restrict__ Y, int* count) {
  extern __shared__ double sm[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const Chunk c = my_chunk(n);
  for (int j = warp; j < k; j += kWarps) {
    const double s = chunk_dot(V[j] + c.i0, Av + c.i0, c.len);
    if (lane == 0) part[j * kChunks + blockIdx.x] = s;
  }
  if (!last_block(count)) return;
  for (int j = warp; j < k; j += kWarps) {
    const double s = chunks_sum(part + j * kChunks);
    if (lane == 0) __stcg(H + (k - 1) * ld + j, s);
  }
  __threadfence_block();
  __syncthreads();
  ritz_block(H, ld, k, sm, w, Y);
}

}  // namespace

static size_t ritz_smem(int k) {
  DMRG_REQUIRE(k >= 1 && k <= kMaxK, DMRG_EINVAL, "internal: Ritz problem too large");
  static std::once_flag once;
  std::call_once(once, [] {
    const int most = int(sizeof(double) * 3 * kMaxK * kMaxK);
    DMRG_CUDA(cudaFuncSetAttribute(k_ritz, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
    DMRG_CUDA(cudaFuncSetAttribute(k_dav_ritz, cudaFuncAttributeMaxDynamicSharedMemorySize, most));
  });
  return sizeof(double) * 3 * size_t(k) * k;
}

void multidot(const double* const* d_vecs, int k, const double* w, int64_t n, double* d_out,
              double* d_partials, int* d_count, cudaStream_t s) {
  if (k <= 0) return;
  k_dav_dots<<<kChunks, kThr, 0, s>>>(d_vecs, k, w, n, d_partials, d_out, d_count);
  DMRG_LAUNCHED();
}

void ritz_solve(const double* d_H, int ld, int k, double* d_w, double* d_Y, cudaStream_t s) {
  k_ritz<<<1, kThr, ritz_smem(k), s>>>(d_H, ld, k, d_w, d_Y);
  DMRG_LAUNCHED();
}

void dav_chain(const DavChain& c, cudaStream_t s) {
  double* sums = c.sc + 8;      // |r|^2, |t|^2, V^T t
  double* h2 = sums + 66;       // V^T t of the second pass
  double* tt = h2 + 64;         // |t|^2
  k_dav_ritz<<<kChunks, kThr, ritz_smem(c.k), s>>>(c.V, c.k, c.Av, c.n, c.part, c.H, c.ldh, c.w,
                                                   c.Y, c.count);
  DMRG_LAUNCHED();
  k_dav_residual<<<kChunks, kThr, 0, s>>>(c.V, c.AV, c.Y, c.w, c.diag, c.k, c.n, c.x, c.r, c.t,
                                          c.part, sums, c.count);
  DMRG_LAUNCHED();
  k_dav_orth<false><<<kChunks, kThr, 0, s>>>(c.V, c.k, c.n, sums + 2, c.t, c.part, h2, c.count);
  DMRG_LAUNCHED();
  k_dav_orth<true><<<kChunks, kThr, 0, s>>>(c.V, c.k, c.n, h2, c.t, c.part, tt, c.count);
  DMRG_LAUNCHED();
  const int blocks = int(std::max<int64_t>(1, std::min<int64_t>((c.n + kThr - 1) / kThr, 152 * 8)));
  k_dav_next<<<blocks, kThr, 0, s>>>(c.t, tt, sums, c.w, c.n, c.next, c.sc);
  DMRG_LAUNCHED();
}

}  // namespace dmrg
