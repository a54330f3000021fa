// Mixed superblock product on the tensor cores (FP32 storage, FP32 accumulate)
//     psi'(b') = sum_k s_k L_k[Q_L' <- Q_L] psi(b) R_k[Q_R' <- Q_R]^T
// for the output blocks between the small-block kernel and the grouped passes (up to the
// big-block edge, dmrg_set_tuning): a few to ~100 states wide, below what a CTA-level MMA of 64
// or 128 rows fills, so the warp-level instruction is the one that fits them.
//     X (dLi x n)  = psi (dLi x dRi) R^T        (M = dLi, N = n, K = dRi)
//     Y (m x n)   += s L (m x dLi) X             (M = m,   N = n, K = dLi)
// Both products run as MMAs m16n8k8 on TF32 operands split into high and low parts,
//     a b  ~  a_hi b_hi + a_hi b_lo + a_lo b_hi   (three MMAs, FP32 accumulation),
// which keeps FP32-level accuracy (the dropped a_lo b_lo term is ~2^-22 relative).
//
// Work unit (one thread block, four warps), as in heff.cu: one output tile (at most 32 x 32), one
// group of at most 64 terms, one of four slots (every fourth term of the group, in order).  The
// warps share a term: each takes up to two of the m16n8 tiles of X, then of Y.  A term runs in
// pieces of 32 rows and 32 inner columns of psi; the blocks of the next piece travel to the other
// shared-memory buffer while this one is multiplied (terms up to 32 wide whole, 16 bytes a copy;
// of wider ones a 32 x 32 part, rows of 36 words).  32 KB per unit, so seven units (28 warps) on
// an SM, against twelve warps with a ring of terms per warp; terms wider than 32 are pipelined
// like the others instead of staged and waited for.  On starting-state blocks the first version, with
// 4-byte copies, was bound by instruction issue (74 % of the slots), so the copies and the bounds are
// what is kept short; on small terms the kernel now waits for their loads (37 % of the slots).
//   The high part is rounded with integer operations (add half a unit, cut): the conversion
// instruction runs at a quarter of their rate and was half of the inner loop's time with two per
// operand element.  The low part keeps it, so that a NaN stays one.
// The slots of a group are added in order and the groups in order (heff.cu): deterministic, and
// the same bit for bit as one warp per slot.
// Measured (GB300): pf 8p+8n at position 12, M0 = 4096 (2.9 GFLOP) 999 -> 650 us; pf 4p+5n at
// position 9, M0 = 777 (296 tiles) 58 -> 37 us; pf 8p+8n, M0 = 512 (115,000 terms of 5 to 20
// states) 163 -> 159 us.
#include <stdint.h>

#include "common.h"

namespace dmrg {
namespace tc {

constexpr int kT = 32;              // edge of tiles and pieces
constexpr int kLd = 36;             // row stride in words
constexpr int kTile = kT * kLd;
constexpr int kNarrow = 16;         // tiles up to this many columns: two warps per unit
constexpr int kSlots = 4;

__device__ __forceinline__ void copy4(float* dst, const float* src) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4;\n" ::"r"(s), "l"(src) : "memory");
}
__device__ __forceinline__ void copy16(float* dst, const float* src) {
  const unsigned s = static_cast<unsigned>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16;\n" ::"r"(s), "l"(src) : "memory");
}

// row stride in shared memory of a whole block with d <= 32 columns: as in memory, unless that
// puts the rows of a fragment into the same banks
__device__ __forceinline__ int stride_of(int d) { return (d & 7) ? d : d + 4; }

// a whole block (rows x d, contiguous, starting on 16 bytes; up to 3 elements behind it are read)
template <int W>
__device__ __forceinline__ void stage_whole(float* dst, const float* src, int rows, int d) {
  if (d & 7) {
    for (int v = threadIdx.x; v < (rows * d + 3) >> 2; v += 32 * W) copy16(dst + 4 * v, src + 4 * v);
  } else {
    const int q = d >> 2, inv = 65536 / q + 1;   // v / q = (v inv) >> 16 for v < 256
    for (int v = threadIdx.x; v < rows * q; v += 32 * W) {
      const int r = (v * inv) >> 16;
      copy16(dst + 4 * (v + r), src + 4 * v);
    }
  }
}
// rows x cols (at most 32 x 32) of a wider block with leading dimension ld, row stride kLd
template <int W>
__device__ __forceinline__ void stage_part(float* dst, const float* src, int ld, int rows, int cols) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  if (ld & 3) {
    dst += warp * kLd + lane;
    src += int64_t(warp) * ld + lane;
    if (lane < cols)
      for (int r = warp; r < rows; r += W, dst += W * kLd, src += int64_t(W) * ld) copy4(dst, src);
  } else {   // rows of whole 16-byte pieces
    const int r0 = threadIdx.x >> 3, c = 4 * (threadIdx.x & 7);
    if (c < cols)
      for (int r = r0; r < rows; r += 4 * W) copy16(dst + r * kLd + c, src + int64_t(r) * ld + c);
  }
}

__device__ __forceinline__ void split(float x, uint32_t& hi, uint32_t& lo) {
  hi = (__float_as_uint(x) + 0x1000u) & 0xffffe000u;   // nearest, ties away from zero
  asm("cvt.rna.tf32.f32 %0, %1;\n" : "=r"(lo) : "f"(x - __uint_as_float(hi)));
}
__device__ __forceinline__ void mma(float (&d)[4], const uint32_t (&a)[4], const uint32_t (&b)[2]) {
  asm volatile(
      "mma.sync.aligned.m16n8k8.row.col.f32.tf32.tf32.f32 {%0,%1,%2,%3}, {%4,%5,%6,%7}, "
      "{%8,%9}, {%0,%1,%2,%3};\n"
      : "+f"(d[0]), "+f"(d[1]), "+f"(d[2]), "+f"(d[3])
      : "r"(a[0]), "r"(a[1]), "r"(a[2]), "r"(a[3]), "r"(b[0]), "r"(b[1]));
}

__device__ __forceinline__ float keep(float x, bool in) { return in ? x : 0.f; }

// d0 (and d1, if two) += A B over k < kdim: A rows r and r + 8 at A and A8; B element k of the
// lane's column at B0[k bk] (B1).  Small products first, the two chains interleaved.  Only the
// last step looks at kdim: what lies behind the blocks in shared memory never enters a sum.
__device__ __forceinline__ void tile_mma(float (&d0)[4], float (&d1)[4], bool two, const float* A,
                                         const float* A8, const float* B0, const float* B1, int bk,
                                         int kdim, int tig) {
  for (int k0 = tig; k0 < kdim + tig; k0 += 8) {
    const int k1 = k0 + 4;
    float a[4] = {A[k0], A8[k0], A[k1], A8[k1]};
    float b[2] = {B0[k0 * bk], B0[k1 * bk]};
    float c[2] = {0.f, 0.f};
    if (two) {
      c[0] = B1[k0 * bk];
      c[1] = B1[k1 * bk];
    }
    if (k0 - tig + 8 > kdim) {
      const bool in0 = k0 < kdim, in1 = k1 < kdim;
      a[0] = keep(a[0], in0), a[1] = keep(a[1], in0), a[2] = keep(a[2], in1), a[3] = keep(a[3], in1);
      b[0] = keep(b[0], in0), b[1] = keep(b[1], in1);
      c[0] = keep(c[0], in0), c[1] = keep(c[1], in1);
    }
    uint32_t ah[4], al[4], bh[2], bl[2];
#pragma unroll
    for (int i = 0; i < 4; ++i) split(a[i], ah[i], al[i]);
#pragma unroll
    for (int i = 0; i < 2; ++i) split(b[i], bh[i], bl[i]);
    if (two) {
      uint32_t ch[2], cl[2];
#pragma unroll
      for (int i = 0; i < 2; ++i) split(c[i], ch[i], cl[i]);
      mma(d0, al, bh);
      mma(d1, al, ch);
      mma(d0, ah, bl);
      mma(d1, ah, cl);
      mma(d0, ah, bh);
      mma(d1, ah, ch);
    } else {
      mma(d0, al, bh);
      mma(d0, ah, bl);
      mma(d0, ah, bh);
    }
  }
}

// the m16n8 tiles of a warp in an MT x NT grid of them: row tile mt, column tiles n0 and n1
struct Mine {
  int mt, n0, n1;
  bool any, two;
};
template <int W>
__device__ __forceinline__ Mine my_tiles(int MT, int NT, int warp) {
  Mine w;
  constexpr int half = W / 2;   // warps per row tile when there are two
  w.mt = MT == 2 ? warp / half : 0;
  w.n0 = MT == 2 ? warp % half : warp;
  w.n1 = MT == 2 ? w.n0 + half : 4;
  w.any = w.n0 < NT;
  w.two = w.n1 < NT;
  return w;
}

// W = 4 warps for tiles of up to 32 columns, 2 for narrow ones when they have a launch of their own
// (half of the warps would have no MMA tile there)
template <int W>
__global__ void __launch_bounds__(32 * W, W == 4 ? 7 : 8)
k_heff_tc(const HeffTile* __restrict__ tiles, const int32_t* __restrict__ order,
          const HeffItem* __restrict__ items, const HeffPtrs<float> ptrs) {
  __shared__ __align__(16) float Ps[2][kTile], Rs[2][kTile * W / 4], Ls[2][kTile], Xs[kTile];
  const HeffTile t = tiles[order[blockIdx.x / kSlots]];
  const int slot = blockIdx.x % kSlots;
  if (ptrs.active && !ptrs.active[t.inst]) return;   // whole block: uniform
  const float* __restrict__ L = ptrs.L[t.inst];
  const float* __restrict__ R = ptrs.R[t.inst];
  const float* __restrict__ X = ptrs.X[t.inst];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int gid = lane >> 2, tig = lane & 3;
  const int m = t.m, n = t.n, mn = m * n;
  const int NT = (n + 7) >> 3, MT2 = (m + 15) >> 4;
  const Mine out = my_tiles<W>(MT2, NT, warp);
  float y0[4] = {0.f, 0.f, 0.f, 0.f}, y1[4] = {0.f, 0.f, 0.f, 0.f};

  // copies of one piece: psi and R chunks, with the last inner chunk also the L chunk
  auto fetch = [&](const HeffItem& it, int k0, int r0, int buf) {
    const float* Lt = L + it.loff + int64_t(t.r0) * it.dLi;
    const float* Rt = R + it.roff + int64_t(t.c0) * it.dRi;
    if (it.dLi <= kT && it.dRi <= kT) {
      stage_whole<W>(Ps[buf], X + it.xoff, it.dLi, it.dRi);
      stage_whole<W>(Rs[buf], Rt, n, it.dRi);
      stage_whole<W>(Ls[buf], Lt, m, it.dLi);
      return;
    }
    const int kc = min(kT, it.dLi - k0), rc = min(kT, it.dRi - r0);
    stage_part<W>(Ps[buf], X + it.xoff + int64_t(k0) * it.dRi + r0, it.dRi, kc, rc);
    stage_part<W>(Rs[buf], Rt + r0, it.dRi, n, rc);
    if (r0 + kT >= it.dRi) stage_part<W>(Ls[buf], Lt + k0, it.dLi, m, kc);
  };

  int j = t.i0 + slot, buf = 0;
  HeffItem it{}, next{};
  if (j < t.i1) {
    it = items[j];
    fetch(it, 0, 0, 0);
  }
  asm volatile("cp.async.commit_group;\n" ::: "memory");
  int k0 = 0, r0 = 0;
  float x0[4], x1[4];
  while (j < t.i1) {
    // the following piece
    int nj = j, nk = k0, nr = r0 + kT;
    if (nr >= it.dRi) {
      nr = 0;
      nk += kT;
      if (nk >= it.dLi) {
        nk = 0;
        nj += kSlots;
      }
    }
    next = it;
    if (nj != j && nj < t.i1) next = items[nj];
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    __syncthreads();   // this piece has arrived, the other buffer is free
    if (nj < t.i1) fetch(next, nk, nr, buf ^ 1);
    asm volatile("cp.async.commit_group;\n" ::: "memory");

    const int kc = min(kT, it.dLi - k0), rc = min(kT, it.dRi - r0);
    const bool whole = it.dLi <= kT && it.dRi <= kT;
    const int sr = whole ? stride_of(rc) : kLd, sl = whole ? stride_of(kc) : kLd;
    const Mine w = my_tiles<W>((kc + 15) >> 4, NT, warp);
    if (r0 == 0)
#pragma unroll
      for (int e = 0; e < 4; ++e) x0[e] = x1[e] = 0.f;
    if (w.any) {
      const float* A = Ps[buf] + (16 * w.mt + gid) * sr;
      tile_mma(x0, x1, w.two, A, A + 8 * sr, Rs[buf] + (8 * w.n0 + gid) * sr,
               Rs[buf] + (8 * w.n1 + gid) * sr, 1, rc, tig);
    }
    if (r0 + kT >= it.dRi) {
      if (w.any) {
        float* x = Xs + (16 * w.mt + gid) * kLd + 2 * tig;
        const float sg = it.sign;
        x[8 * w.n0] = sg * x0[0];
        x[8 * w.n0 + 1] = sg * x0[1];
        x[8 * kLd + 8 * w.n0] = sg * x0[2];
        x[8 * kLd + 8 * w.n0 + 1] = sg * x0[3];
        if (w.two) {
          x[8 * w.n1] = sg * x1[0];
          x[8 * w.n1 + 1] = sg * x1[1];
          x[8 * kLd + 8 * w.n1] = sg * x1[2];
          x[8 * kLd + 8 * w.n1 + 1] = sg * x1[3];
        }
      }
      __syncthreads();
      if (out.any) {
        const float* A = Ls[buf] + (16 * out.mt + gid) * sl;
        tile_mma(y0, y1, out.two, A, A + 8 * sl, Xs + 8 * out.n0 + gid, Xs + 8 * out.n1 + gid, kLd, kc,
                 tig);
      }
    }
    j = nj;
    k0 = nk;
    r0 = nr;
    it = next;
    buf ^= 1;
  }
  float* __restrict__ P = ptrs.P[t.inst] + t.qoff + int64_t(slot) * mn;
  if (out.any) {
    const int r = 16 * out.mt + gid;
    auto put = [&](const float (&y)[4], int c) {
      if (r < m && c < n) P[r * n + c] = y[0];
      if (r < m && c + 1 < n) P[r * n + c + 1] = y[1];
      if (r + 8 < m && c < n) P[(r + 8) * n + c] = y[2];
      if (r + 8 < m && c + 1 < n) P[(r + 8) * n + c + 1] = y[3];
    };
    put(y0, 8 * out.n0 + 2 * tig);
    if (out.two) put(y1, 8 * out.n1 + 2 * tig);
  }
}

}  // namespace tc

void heff_tc(const HeffTile* d_tiles, const int32_t* d_order, int64_t n_wide, int64_t n_tiles,
             const HeffItem* d_items, const HeffPtrs<float>& ptrs, cudaStream_t s,
             cudaStream_t s_narrow) {
  if (n_wide > 0) {
    tc::k_heff_tc<4><<<int(n_wide * tc::kSlots), 128, 0, s>>>(d_tiles, d_order, d_items, ptrs);
    DMRG_LAUNCHED();
  }
  if (n_tiles > n_wide) {
    tc::k_heff_tc<2><<<int((n_tiles - n_wide) * tc::kSlots), 64, 0, s_narrow>>>(
        d_tiles, d_order + n_wide, d_items, ptrs);
    DMRG_LAUNCHED();
  }
}

int64_t heff_tc_order(const std::vector<HeffTile>& tiles, bool apart, std::vector<int32_t>& order) {
  order.clear();
  order.reserve(tiles.size());
  for (size_t i = 0; i < tiles.size(); ++i)
    if (!apart || tiles[i].n > tc::kNarrow) order.push_back(int32_t(i));
  const int64_t n_wide = int64_t(order.size());
  if (!apart) return n_wide;
  for (size_t i = 0; i < tiles.size(); ++i)
    if (tiles[i].n <= tc::kNarrow) order.push_back(int32_t(i));
  return n_wide;
}

}  // namespace dmrg
