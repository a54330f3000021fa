// FP64 superblock product  psi'(b') = sum_k s_k L_k[Q_L' <- Q_L] psi(b) R_k[Q_R' <- Q_R]^T
// (the two-site H_eff of the superblock "Xi_l (x) Lambda (x) Lambda (x) Xi_r") for the output
// blocks between the small-block kernel and the grouped passes.
//
// FP64 on this chip is one warp instruction per 19 clocks and SM (64 per scheduler), whatever the
// instruction's active lanes and however independent the next one is.  So the kernel is bound by
// the count of FP64 warp instructions, i.e. by lanes left idle, and by having four warps ready;
// operand traffic is cheap beside it (two operands per 19 clocks).  Hence
//   - the elements of a term's intermediate, and of the output tile, are numbered through and
//     dealt to the warps 32 at a time (a 25 x 25 tile fills 20 instructions instead of 25 rows
//     of 25 lanes), with one element per thread in flight and the sums in shared memory;
//   - psi and L are read where they are (a warp reads one to three rows, broadcast from the L1);
//     only the R tile is staged, because its rows run across the lanes;
//   - a work unit is one output tile (at most 32 x 32), one group of at most 64 terms and one of
//     four slots: every fourth term of the group, in order.  25 KB of shared memory and four
//     warps per unit put eight units on an SM, so one unit's loads and barriers are covered by
//     the others, and a superblock with few tiles still fills the chip.
// Per term: X = psi R^T (chunks of 32 rows of psi), then acc += L (s X); terms small enough use
// the cheaper association of the tile ((L psi) first).  The four slots of a group are added in
// order and the groups in order by k_heff_reduce: the result is deterministic, and the same bit
// for bit as one thread block running the group with one warp per slot.
// Measured (GB300) against one thread block per group (a row of lanes per tile row, wide terms
// staged in synchronous chunks): pf 8p+8n at position 12, M0 = 3000 (2.0 GFLOP) 9.48 -> 2.55 ms,
// 0.78 of the 1.07 TFLOP/s that FP64 reaches here; pf 4p+4n at M = 1024, position 20 (0.25 GFLOP)
// 1.99 -> 0.39 ms; pf 4p+4n, position 9, M0 = 256 (152 tiles) 170 -> 33 us.
#include <stdint.h>

#include "common.h"

namespace dmrg {

namespace {

constexpr int kT = 32;         // output tile edge, chunk of the inner dimensions
constexpr int kLd = kT + 1;    // row stride in shared memory: no bank conflicts down a column
constexpr int kThr = 128;
constexpr int kSlots = 4;
// L-first association: terms with inner dimensions up to kT whose three blocks together have at
// most this many elements (each rounded up to 16 bytes)
constexpr int kTermMost = 1536;

__device__ __forceinline__ int even(int e) { return (e + 1) & ~1; }
__device__ __forceinline__ double negate_if(double x, int sign_bit) {
  return __hiloint2double(__double2hiint(x) ^ sign_bit, __double2loint(x));
}

__global__ void __launch_bounds__(kThr, 8)
k_heff_fused(const HeffTile* __restrict__ tiles, const HeffItem* __restrict__ items,
             const HeffPtrs<double> ptrs) {
  __shared__ double Xs[kT * kLd], Rs[kT * kLd], acc[kT * kT];
  const HeffTile t = tiles[blockIdx.x / kSlots];
  const int slot = blockIdx.x % kSlots;
  if (ptrs.active && !ptrs.active[t.inst]) return;   // whole block: uniform
  const double* __restrict__ L = ptrs.L[t.inst];
  const double* __restrict__ R = ptrs.R[t.inst];
  const double* __restrict__ X = ptrs.X[t.inst];
  const int tid = threadIdx.x;
  const int m = t.m, n = t.n, mn = m * n;
  const int inv_n = 65536 / n + 1;   // e / n = (e inv_n) >> 16 for e < 1024, n <= 32
  for (int e = tid; e < mn; e += kThr) acc[e] = 0.0;   // (read by the same thread only)
  for (int j = t.i0 + slot; j < t.i1; j += kSlots) {
    const HeffItem it = items[j];
    const int dLi = it.dLi, dRi = it.dRi;
    const int neg = it.sign < 0.f ? int(0x80000000) : 0;
    const double* __restrict__ Lb = L + it.loff + int64_t(t.r0) * dLi;
    const double* __restrict__ Rb = R + it.roff + int64_t(t.c0) * dRi;
    const double* __restrict__ Pb = X + it.xoff;
    if (dLi <= kT && dRi <= kT && even(m * dLi) + even(n * dRi) + even(dLi * dRi) <= kTermMost &&
        int64_t(m) * dRi * (dLi + n) < int64_t(n) * dLi * (dRi + m)) {
      // Z = L psi (m x dRi), then acc += Z (s R)^T
      const int inv_r = 65536 / dRi + 1;
      for (int e = tid; e < n * dRi; e += kThr) {
        const int c = (e * inv_r) >> 16, b = e - c * dRi;
        Rs[c * kLd + b] = negate_if(Rb[e], neg);
      }
      for (int e = tid; e < m * dRi; e += kThr) {
        const int i = (e * inv_r) >> 16, b = e - i * dRi;
        const double* lr = Lb + i * dLi;
        const double* pr = Pb + b;
        double s = 0.0;
#pragma unroll 4
        for (int a = 0; a < dLi; ++a) s = fma(lr[a], pr[a * dRi], s);
        Xs[i * kLd + b] = s;
      }
      __syncthreads();
      for (int e = tid; e < mn; e += kThr) {
        const int i = (e * inv_n) >> 16, c = e - i * n;
        const double* zr = Xs + i * kLd;
        const double* rr = Rs + c * kLd;
        double a = acc[e];
#pragma unroll 4
        for (int b = 0; b < dRi; ++b) a = fma(zr[b], rr[b], a);
        acc[e] = a;
      }
      __syncthreads();
      continue;
    }
    for (int k0 = 0; k0 < dLi; k0 += kT) {
      const int kc = min(kT, dLi - k0);
      for (int r0 = 0; r0 < dRi; r0 += kT) {
        const int rc = min(kT, dRi - r0);
        // columns of the R tile: a warp reads rows of rc consecutive elements
        if (k0 == 0 || dRi > kT) {
          if (rc == dRi) {
            const int inv_r = 65536 / rc + 1;
            for (int e = tid; e < n * rc; e += kThr) {
              const int c = (e * inv_r) >> 16, b = e - c * rc;
              Rs[c * kLd + b] = Rb[e];
            }
          } else {
            for (int e = tid; e < n * kT; e += kThr) {
              const int c = e >> 5, b = e & 31;
              if (b < rc) Rs[c * kLd + b] = Rb[int64_t(c) * dRi + r0 + b];
            }
          }
          __syncthreads();
        }
        const bool last = r0 + kT >= dRi;
        for (int e = tid; e < kc * n; e += kThr) {
          const int i = (e * inv_n) >> 16, c = e - i * n;
          const double* pr = Pb + int64_t(k0 + i) * dRi + r0;
          const double* rr = Rs + c * kLd;
          double s = r0 ? Xs[i * kLd + c] : 0.0;
#pragma unroll 4
          for (int r = 0; r < rc; ++r) s = fma(pr[r], rr[r], s);
          Xs[i * kLd + c] = last ? negate_if(s, neg) : s;
        }
        __syncthreads();
      }
      for (int e = tid; e < mn; e += kThr) {
        const int i = (e * inv_n) >> 16, c = e - i * n;
        const double* lr = Lb + int64_t(i) * dLi + k0;
        const double* xr = Xs + c;
        double a = acc[e];
#pragma unroll 4
        for (int k = 0; k < kc; ++k) a = fma(lr[k], xr[k * kLd], a);
        acc[e] = a;
      }
      __syncthreads();
    }
  }
  double* __restrict__ P = ptrs.P[t.inst] + t.qoff + int64_t(slot) * mn;
  for (int e = tid; e < mn; e += kThr) P[e] = acc[e];
}

// psi' tile = sum over groups (in group order) of the partial tiles, each the sum of its slots
// in order: red[0 .. n_plain) have one partial tile per group (poff; the small-block kernel),
// the others four (qoff)
template <class T>
__global__ void __launch_bounds__(128)
k_heff_reduce_slots(const HeffRed* __restrict__ red, int64_t n_plain, const HeffPtrs<T> ptrs) {
  const HeffRed r = red[blockIdx.x];
  if (ptrs.active && !ptrs.active[r.inst]) return;
  const bool plain = blockIdx.x < n_plain;
  const T* __restrict__ P = ptrs.P[r.inst] + (plain ? r.poff : r.qoff);
  T* __restrict__ Y = ptrs.Y[r.inst];
  const int mn = r.m * r.n;
  // the outputs of a tile are spread over blockIdx.y: a tile has few of them and many addends
  // (one block per tile took 28 us for 900 tiles, four take 10)
  for (int e = blockIdx.y * blockDim.x + threadIdx.x; e < mn; e += gridDim.y * blockDim.x) {
    T s = T(0);
    if (plain) {
#pragma unroll 4
      for (int g = 0; g < r.groups; ++g) s += P[int64_t(g) * mn + e];
    } else {
#pragma unroll 4
      for (int g = 0; g < r.groups; ++g) {
        const T* q = P + int64_t(g) * kSlots * mn + e;
        T u = q[0];
#pragma unroll
        for (int w = 1; w < kSlots; ++w) u += q[int64_t(w) * mn];
        s = r.groups > 1 ? s + u : u;
      }
    }
    const int i = e / r.n, c = e - i * r.n;
    Y[r.yoff + int64_t(r.r0 + i) * r.ld + r.c0 + c] = s;
  }
}

}  // namespace

// psi' tile = sum over groups (in group order) of the partial tiles
template <class T>
__global__ void k_heff_reduce(const HeffRed* __restrict__ red, const HeffPtrs<T> ptrs) {
  const HeffRed r = red[blockIdx.x];
  if (ptrs.active && !ptrs.active[r.inst]) return;
  const T* __restrict__ P = ptrs.P[r.inst];
  T* __restrict__ Y = ptrs.Y[r.inst];
  const int mn = r.m * r.n;
  for (int e = threadIdx.x; e < mn; e += blockDim.x) {
    T s = T(0);
    for (int g = 0; g < r.groups; ++g) s += P[r.poff + (int64_t)g * mn + e];
    const int i = e / r.n, c = e - i * r.n;
    Y[r.yoff + (int64_t)(r.r0 + i) * r.ld + r.c0 + c] = s;
  }
}

// psi blocks into a 16-byte aligned copy (optionally converted): one block per thread block
template <class TI, class TO>
__global__ void k_pad_psi(const TI* __restrict__ x, TO* __restrict__ xp,
                          const int64_t* __restrict__ src_off, const int64_t* __restrict__ dst_off,
                          const int32_t* __restrict__ len) {
  const int b = blockIdx.x;
  const TI* s = x + src_off[b];
  TO* d = xp + dst_off[b];
  for (int i = threadIdx.x; i < len[b]; i += blockDim.x) d[i] = TO(s[i]);
}

template <class T>
void heff_reduce(const HeffRed* d_red, int64_t n_red, const HeffPtrs<T>& ptrs, cudaStream_t s) {
  if (n_red <= 0) return;
  k_heff_reduce<T><<<int(n_red), 128, 0, s>>>(d_red, ptrs);
  DMRG_LAUNCHED();
}
template void heff_reduce<float>(const HeffRed*, int64_t, const HeffPtrs<float>&, cudaStream_t);
template void heff_reduce<double>(const HeffRed*, int64_t, const HeffPtrs<double>&, cudaStream_t);

template <class T>
void heff_reduce_slots(const HeffRed* d_red, int64_t n_plain, int64_t n_red, const HeffPtrs<T>& ptrs,
                       cudaStream_t s) {
  if (n_red <= 0) return;
  k_heff_reduce_slots<T><<<dim3(unsigned(n_red), 4), 128, 0, s>>>(d_red, n_plain, ptrs);
  DMRG_LAUNCHED();
}
template void heff_reduce_slots<float>(const HeffRed*, int64_t, int64_t, const HeffPtrs<float>&,
                                       cudaStream_t);
template void heff_reduce_slots<double>(const HeffRed*, int64_t, int64_t, const HeffPtrs<double>&,
                                        cudaStream_t);

void heff_fused64(const HeffTile* d_tiles, int64_t n_tiles, const HeffItem* d_items,
                  const HeffPtrs<double>& ptrs, cudaStream_t s) {
  if (n_tiles <= 0) return;
  k_heff_fused<<<int(n_tiles * kSlots), kThr, 0, s>>>(d_tiles, d_items, ptrs);
  DMRG_LAUNCHED();
}

// staging with the vector pointer read from device memory (graph replay on new vectors)
template <class TO>
__global__ void k_pad_psi_ind(const double* const* __restrict__ xptr, TO* __restrict__ xp,
                              const int64_t* __restrict__ src_off,
                              const int64_t* __restrict__ dst_off,
                              const int32_t* __restrict__ len, const int32_t* __restrict__ active) {
  if (active && !active[0]) return;
  const int b = blockIdx.x;
  const double* s = xptr[0] + src_off[b];
  TO* d = xp + dst_off[b];
  for (int i = threadIdx.x; i < len[b]; i += blockDim.x) d[i] = TO(s[i]);
}

template <class TI>
__global__ void k_out_to_f64_ind(const TI* __restrict__ y, double* const* __restrict__ optr,
                                 int64_t n, const int32_t* __restrict__ active) {
  if (active && !active[0]) return;
  double* o = optr[0];
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x)
    o[i] = double(y[i]);
}

template <class TO>
void pad_psi_ind(const double* const* x_ptr, TO* xp, const int64_t* src_off,
                 const int64_t* dst_off, const int32_t* len, int nblocks, const int32_t* active,
                 cudaStream_t s) {
  if (nblocks <= 0) return;
  k_pad_psi_ind<TO><<<nblocks, 128, 0, s>>>(x_ptr, xp, src_off, dst_off, len, active);
  DMRG_LAUNCHED();
}
template void pad_psi_ind<float>(const double* const*, float*, const int64_t*, const int64_t*,
                                 const int32_t*, int, const int32_t*, cudaStream_t);
template void pad_psi_ind<double>(const double* const*, double*, const int64_t*, const int64_t*,
                                  const int32_t*, int, const int32_t*, cudaStream_t);

template <class TI>
void out_to_f64_ind(const TI* y, double* const* out_ptr, int64_t n, const int32_t* active,
                    cudaStream_t s) {
  if (n <= 0) return;
  const int blocks = int(std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 16)));
  k_out_to_f64_ind<TI><<<blocks, 256, 0, s>>>(y, out_ptr, n, active);
  DMRG_LAUNCHED();
}
template void out_to_f64_ind<float>(const float*, double* const*, int64_t, const int32_t*,
                                    cudaStream_t);
template void out_to_f64_ind<double>(const double*, double* const*, int64_t, const int32_t*,
                                     cudaStream_t);

template <class TO>
void pad_psi(const double* x, TO* xp, const int64_t* src_off, const int64_t* dst_off,
             const int32_t* len, int nblocks, cudaStream_t s) {
  if (nblocks <= 0) return;
  k_pad_psi<double, TO><<<nblocks, 128, 0, s>>>(x, xp, src_off, dst_off, len);
  DMRG_LAUNCHED();
}
template void pad_psi<double>(const double*, double*, const int64_t*, const int64_t*,
                              const int32_t*, int, cudaStream_t);
template void pad_psi<float>(const double*, float*, const int64_t*, const int64_t*,
                             const int32_t*, int, cudaStream_t);

}  // namespace dmrg
