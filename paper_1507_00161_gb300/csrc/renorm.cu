// Renormalization of block operators onto the kept states (the block basis update after
// the density-matrix truncation):  O'[n_o, n_i] = U_o^T  O[Q_o, Q_i]  U_i  for every block
// of every normal and complementary operator, U_Q = kept eigenvectors of the reduced
// density matrix in enlarged sector Q (D_Q x m_Q, row-major).
//
// FP64 is one warp instruction per 19 clocks and SM on this chip, whatever its active lanes, so
// the elements of T = O U_i and of U_o^T T are numbered through and dealt to the lanes 32 at a
// time, and nothing is computed for padding; the operands are read where they are (rows of O and
// columns of U_o broadcast, rows of U_i consecutive).  Driven by the block table itself:
//  - blocks with D_o, D_i <= 16: one warp each, T in shared memory;
//  - larger blocks: units of a block and some columns of U_i, one thread block each, T in shared
//    memory: 32 columns of blocks of up to 32 rows, 8 columns of taller ones, 128 rows at a time
//    (with more rows the result grows chunk by chunk in its place).  The tallest block's units are
//    the tail of the launch, and narrow ones keep that short.
// FP64 throughout, every sum in index order (deterministic).
// Measured (GB300) against 32 x 32 tiles in two passes through a scratch and one warp per block up to
// 32, kernels of all right blocks: pf 8p+8n, M0 = 4096, 361 -> 249 ms (270 with 32 columns), pf 4p+4n,
// M0 = 2000, 235 -> 187 ms (270), sd 2p+2n, M0 = 512, 5.3 -> 5.1 ms (11.5), M0 = 128 1.18 -> 0.97 ms
// (1.35); at M = 4096, position 15, the two steps of a pair 1.5 -> 0.5 ms each.
#include <stdint.h>

#include "common.h"

namespace dmrg {

namespace {

constexpr int kThr = 128;
constexpr int kTiny = kProjTiny, kTinyLd = kTiny + 1;
constexpr int kTinyWarps = 4;

// c[r * 1] ... sum_k a[k sa] b[k sb], k < n, in order
__device__ __forceinline__ double dot_strided(const double* __restrict__ a, int64_t sa,
                                              const double* b, int64_t sb, int n, double s) {
#pragma unroll 4
  for (int k = 0; k < n; ++k) s = fma(a[k * sa], b[k * sb], s);
  return s;
}

template <int ROWS, int COLS>
__global__ void __launch_bounds__(kThr, ROWS == 32 ? 12 : 6)
k_project(const ProjTask* __restrict__ units, const int32_t* __restrict__ D,
          const int32_t* __restrict__ m, const int64_t* __restrict__ uoff,
          const double* __restrict__ X, const double* __restrict__ U, double* __restrict__ Y) {
  constexpr int kLd = COLS + 1;
  __shared__ double T[ROWS * kLd];
  const ProjTask pt = units[blockIdx.x];
  const int Do = D[pt.so], Di = D[pt.si], mo = m[pt.so], mi = m[pt.si];
  const int n = min(COLS, mi - pt.c0);
  const double* __restrict__ Xb = X + pt.xoff;
  const double* __restrict__ Ui = U + uoff[pt.si] + pt.c0;
  const double* __restrict__ Uo = U + uoff[pt.so];
  double* __restrict__ Yb = Y + pt.yoff + pt.c0;
  // e / n = (e inv) >> 16 for e < 1024: elements are dealt in runs of kRun rows of n
  const int inv = 65536 / n + 1;
  constexpr int kRun = 32;
  for (int i0 = 0; i0 < Do; i0 += ROWS) {
    const int rows = min(ROWS, Do - i0);
    for (int r0 = 0; r0 < rows; r0 += kRun) {
      const int cnt = min(kRun, rows - r0) * n;
      for (int e = threadIdx.x; e < cnt; e += kThr) {
        const int i = (e * inv) >> 16, c = e - i * n;
        T[(r0 + i) * kLd + c] =
            dot_strided(Xb + int64_t(i0 + r0 + i) * Di, 1, Ui + c, mi, Di, 0.0);
      }
    }
    __syncthreads();
    for (int a0 = 0; a0 < mo; a0 += kRun) {
      const int cnt = min(kRun, mo - a0) * n;
      for (int e = threadIdx.x; e < cnt; e += kThr) {
        const int a = (e * inv) >> 16, c = e - a * n;
        double* y = Yb + int64_t(a0 + a) * mi + c;
        *y = dot_strided(Uo + int64_t(i0) * mo + a0 + a, mo, T + c, kLd, rows, i0 ? *y : 0.0);
      }
    }
    __syncthreads();
  }
}

__global__ void __launch_bounds__(kTinyWarps * 32)
k_project_tiny(const ProjTask* __restrict__ tasks, int64_t n, const int32_t* __restrict__ D,
               const int32_t* __restrict__ m, const int64_t* __restrict__ uoff,
               const double* __restrict__ X, const double* __restrict__ U,
               double* __restrict__ Y) {
  __shared__ double Ts[kTinyWarps][kTiny * kTinyLd];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  double* T = Ts[warp];
  const int64_t b = int64_t(blockIdx.x) * kTinyWarps + warp;
  if (b >= n) return;
  const ProjTask pt = tasks[b];
  const int Do = D[pt.so], Di = D[pt.si], mo = m[pt.so], mi = m[pt.si];
  const double* __restrict__ Xb = X + pt.xoff;
  const double* __restrict__ Ui = U + uoff[pt.si];
  const double* __restrict__ Uo = U + uoff[pt.so];
  const int inv = 65536 / mi + 1;
  for (int e = lane; e < Do * mi; e += 32) {
    const int i = (e * inv) >> 16, c = e - i * mi;
    T[i * kTinyLd + c] = dot_strided(Xb + i * Di, 1, Ui + c, mi, Di, 0.0);
  }
  __syncwarp();
  for (int e = lane; e < mo * mi; e += 32) {
    const int a = (e * inv) >> 16, c = e - a * mi;
    Y[pt.yoff + e] = dot_strided(Uo + a, mo, T + c, kTinyLd, Do, 0.0);
  }
}

}  // namespace

void project_blocks(const ProjTask* units, const int64_t (&begin)[4], const int32_t* D,
                    const int32_t* m, const int64_t* uoff, const double* X, const double* U,
                    double* Y, cudaStream_t s) {
  const int64_t n0 = begin[1] - begin[0], n1 = begin[2] - begin[1], n2 = begin[3] - begin[2];
  if (n2 > 0) {   // the widest first
    k_project<128, project_cols(2)><<<int(n2), kThr, 0, s>>>(units + begin[2], D, m, uoff, X, U, Y);
    DMRG_LAUNCHED();
  }
  if (n1 > 0) {
    k_project<32, project_cols(1)><<<int(n1), kThr, 0, s>>>(units + begin[1], D, m, uoff, X, U, Y);
    DMRG_LAUNCHED();
  }
  if (n0 > 0) {
    k_project_tiny<<<int((n0 + kTinyWarps - 1) / kTinyWarps), kTinyWarps * 32, 0, s>>>(
        units + begin[0], n0, D, m, uoff, X, U, Y);
    DMRG_LAUNCHED();
  }
}

}  // namespace dmrg
