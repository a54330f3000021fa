// Device functions of the FP64 symmetric eigensolver of the density-matrix kernels (kernels.cu).  The
// Ritz problem of Davidson has its own, with the same pairing and rotations (davidson.cu).
#pragma once
#include <cuda_runtime.h>
#include <math.h>

namespace dmrg {

// ------------------------------------------------------------------------------------
// symmetric eigensolver: parallel cyclic Jacobi (round-robin pairing), one block per matrix
// A (n x n, row-major, overwritten: diagonal -> eigenvalues), V (n x n) eigenvectors in
// columns.  Rotation of (Numerical Recipes): theta = (a_qq - a_pp) / (2 a_pq),
// t = sgn(theta)/(|theta| + sqrt(theta^2+1)), c = 1/sqrt(t^2+1), s = t c, A' = P^T A P.
// ------------------------------------------------------------------------------------
static __device__ void jacobi_block(double* A, double* V, int n, double* cs, int* pp, int* qq,
                             double* red) {
  const int tid = threadIdx.x, nt = blockDim.x;
  for (int i = tid; i < n * n; i += nt) V[i] = (i / n == i % n) ? 1.0 : 0.0;
  __syncthreads();
  if (n <= 1) return;
  const int m = (n + 1) & ~1;   // even number of players (a dummy when n is odd)
  for (int sweep = 0; sweep < 40; ++sweep) {
    // convergence: off-diagonal Frobenius norm against the full norm
    double off = 0.0, tot = 0.0;
    for (int i = tid; i < n * n; i += nt) {
      double a = A[i];
      tot += a * a;
      if (i / n != i % n) off += a * a;
    }
    for (int o = 16; o > 0; o >>= 1) {
      off += __shfl_down_sync(0xffffffffu, off, o);
      tot += __shfl_down_sync(0xffffffffu, tot, o);
    }
    __syncthreads();
    if ((tid & 31) == 0) {
      red[2 * (tid >> 5)] = off;
      red[2 * (tid >> 5) + 1] = tot;
    }
    __syncthreads();
    if (tid == 0) {
      double o2 = 0.0, t2 = 0.0;
      for (int w = 0; w < (nt + 31) / 32; ++w) { o2 += red[2 * w]; t2 += red[2 * w + 1]; }
      red[64] = (o2 <= 1e-30 * t2 || t2 == 0.0) ? 1.0 : 0.0;
    }
    __syncthreads();
    if (red[64] != 0.0) break;
    for (int r = 0; r < m - 1; ++r) {
      // round-robin tournament: player m-1 fixed, the others rotate
      for (int k = tid; k < m / 2; k += nt) {
        int a, b;
        if (k == 0) {
          a = m - 1;
          b = r;
        } else {
          a = (r + k) % (m - 1);
          b = (r - k + (m - 1)) % (m - 1);
        }
        int p = min(a, b), q = max(a, b);
        double c = 1.0, s = 0.0;
        if (q < n) {
          double apq = A[p * n + q];
          if (apq != 0.0) {
            double th = (A[q * n + q] - A[p * n + p]) / (2.0 * apq);
            double t = (th >= 0.0 ? 1.0 : -1.0) / (fabs(th) + sqrt(th * th + 1.0));
            c = 1.0 / sqrt(t * t + 1.0);
            s = t * c;
          }
        }
        pp[k] = p;
        qq[k] = q;
        cs[2 * k] = c;
        cs[2 * k + 1] = s;
      }
      __syncthreads();
      // rows: A <- P^T A
      for (int e = tid; e < (m / 2) * n; e += nt) {
        int k = e / n, col = e - k * n;
        int p = pp[k], q = qq[k];
        if (q >= n) continue;
        double c = cs[2 * k], s = cs[2 * k + 1];
        if (s == 0.0) continue;
        double ap = A[p * n + col], aq = A[q * n + col];
        A[p * n + col] = c * ap - s * aq;
        A[q * n + col] = s * ap + c * aq;
      }
      __syncthreads();
      // columns: A <- A P ; V <- V P
      for (int e = tid; e < (m / 2) * n; e += nt) {
        int k = e / n, row = e - k * n;
        int p = pp[k], q = qq[k];
        if (q >= n) continue;
        double c = cs[2 * k], s = cs[2 * k + 1];
        if (s == 0.0) continue;
        double ap = A[row * n + p], aq = A[row * n + q];
        A[row * n + p] = c * ap - s * aq;
        A[row * n + q] = s * ap + c * aq;
        double vp = V[row * n + p], vq = V[row * n + q];
        V[row * n + p] = c * vp - s * vq;
        V[row * n + q] = s * vp + c * vq;
      }
      __syncthreads();
    }
  }
}

// rank-sort of eigenpairs (descending or ascending), ties by original index; clip <0 to 0
// when requested; eigenvector sign: largest |component| positive (lowest row on ties)
static __device__ void sort_and_fix(const double* A, const double* V, int n, double* w_out,
                             double* V_out, int descending, int clip, int rs, int cs_) {
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    double wi = A[i * n + i];
    int rank = 0;
    for (int j = 0; j < n; ++j) {
      double wj = A[j * n + j];
      bool before = descending ? (wj > wi) : (wj < wi);
      if (before || (wj == wi && j < i)) ++rank;
    }
    w_out[rank] = (clip && wi < 0.0) ? 0.0 : wi;
    // sign of column i
    int best = 0;
    double bv = -1.0;
    for (int rr = 0; rr < n; ++rr) {
      double a = fabs(V[rr * n + i]);
      if (a > bv) { bv = a; best = rr; }
    }
    double sg = V[best * n + i] < 0.0 ? -1.0 : 1.0;
    for (int rr = 0; rr < n; ++rr) V_out[rr * rs + rank * cs_] = sg * V[rr * n + i];
  }
}

}  // namespace dmrg
