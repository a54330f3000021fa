// Superblock product for small blocks:  psi'(b') += s_k L_k psi(b) R_k^T  (the two-site
// H_eff of the superblock "Xi_l (x) Lambda (x) Lambda (x) Xi_r") for output blocks whose
// dimensions and whose terms' inner dimensions are all at most 16.
//
// At large M the sector count grows with M, so most wave-function blocks are a few states
// on a side: a term is a handful of multiply-adds, and a warp that takes the terms one after the
// other waits for its loads (descriptor, psi and R, L) at every one of them.  The terms of a
// group only meet in the sum  acc <- acc + s_k (L_k X_k),  so one thread block takes an (output
// block, group of at most 16 terms): its warps form the products  D_k = L_k (psi R_k^T)  of
// different terms side by side and leave them in shared memory, then the block adds them in term
// order.  Lane map for an m x n output block: elements are numbered through and dealt to the
// lanes 32 at a time (an FP64 instruction takes as long with half of its lanes); per term
//     X[a][c] = sum_b psi[a][b] R[c][b]     (X in shared memory, per warp)
//     D[i][c] = sum_a L[i][a] X[a][c]
// Terms are added in list order; groups of one block are added in group order by the
// reduction kernels: the result is deterministic.
// Measured (GB300) against one warp per group, FP32: pf 4p+5n, M0 = 777 (615 groups) 16.8 -> 4.7 us,
// pf 8p+8n at M = 4096, position 15 (1135 groups) 20.6 -> 7.9 us.
#include <stdint.h>

#include "common.h"

namespace dmrg {

namespace {

constexpr int kSmWarps = 8;
constexpr int kSmTerms = 16;   // most terms of a group

template <class T>
__global__ void __launch_bounds__(kSmWarps * 32)
k_heff_small(const HeffTile* __restrict__ tiles, const HeffItem* __restrict__ items,
             const HeffPtrs<T> ptrs) {
  constexpr int kE = kSmallEdge * kSmallEdge;
  __shared__ T Xs[kSmWarps][kE];
  extern __shared__ __align__(16) unsigned char small_sm[];
  T* const D = reinterpret_cast<T*>(small_sm);   // products of the terms, m n elements each
  const HeffTile t = tiles[blockIdx.x];
  if (ptrs.active && !ptrs.active[t.inst]) return;
  const T* __restrict__ L = ptrs.L[t.inst];
  const T* __restrict__ R = ptrs.R[t.inst];
  const T* __restrict__ X = ptrs.X[t.inst];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int m = t.m, n = t.n, mn = m * n;
  const int inv_n = 65536 / n + 1;   // e / n = (e inv_n) >> 16 for e < 256
  T* Xw = Xs[warp];
  const int cnt = t.i1 - t.i0;
  for (int j = warp; j < cnt; j += kSmWarps) {
    const HeffItem it = items[t.i0 + j];
    const int dLi = it.dLi, dRi = it.dRi;
    const T* __restrict__ Lb = L + it.loff + int64_t(t.r0) * dLi;
    const T* __restrict__ Rb = R + it.roff + int64_t(t.c0) * dRi;
    const T* __restrict__ Xb = X + it.xoff;
    for (int e = lane; e < dLi * n; e += 32) {
      const int a = (e * inv_n) >> 16, c = e - a * n;
      const T* xr = Xb + a * dRi;
      const T* rr = Rb + c * dRi;
      T s = T(0);
#pragma unroll 4
      for (int b = 0; b < dRi; ++b) s = fma(xr[b], rr[b], s);
      Xw[e] = s;
    }
    __syncwarp();
    for (int e = lane; e < mn; e += 32) {
      const int i = (e * inv_n) >> 16, c = e - i * n;
      const T* lr = Lb + i * dLi;
      T s = T(0);
#pragma unroll 4
      for (int a = 0; a < dLi; ++a) s = fma(lr[a], Xw[a * n + c], s);
      D[j * mn + e] = it.sign < 0.f ? -s : s;
    }
    __syncwarp();
  }
  __syncthreads();
  T* __restrict__ Y = t.poff < 0 ? ptrs.Y[t.inst] + t.yoff + int64_t(t.r0) * t.ld + t.c0
                                 : ptrs.P[t.inst] + t.poff;
  const int ld = t.poff < 0 ? t.ld : n;
  for (int e = threadIdx.x; e < mn; e += kSmWarps * 32) {
    T acc = T(0);
    for (int j = 0; j < cnt; ++j) acc += D[j * mn + e];
    const int i = (e * inv_n) >> 16, c = e - i * n;
    Y[int64_t(i) * ld + c] = acc;
  }
}

}  // namespace

template <class T>
void heff_small(const HeffTile* d_tiles, int64_t n_tiles, const HeffItem* d_items,
                const HeffPtrs<T>& ptrs, cudaStream_t s) {
  if (n_tiles <= 0) return;
  const size_t smem = sizeof(T) * kSmTerms * kSmallEdge * kSmallEdge;
  k_heff_small<T><<<int(n_tiles), kSmWarps * 32, smem, s>>>(d_tiles, d_items, ptrs);
  DMRG_LAUNCHED();
}
template void heff_small<float>(const HeffTile*, int64_t, const HeffItem*, const HeffPtrs<float>&,
                                cudaStream_t);
template void heff_small<double>(const HeffTile*, int64_t, const HeffItem*,
                                 const HeffPtrs<double>&, cudaStream_t);

}  // namespace dmrg
