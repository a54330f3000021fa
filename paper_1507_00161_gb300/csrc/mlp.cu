// Learned Davidson preconditioner: a per-element network 4 -> 256 -> 256 -> 256 -> 1
// (ReLU), trained on the GPU by the kernels of this file (not in the paper; the method's
// own Davidson steps provide the training pairs, diagonal Davidson is the fallback).
//
// Parameters (packed, row-major): W1 (256 x 4), b1, W2 (256 x 256), b2, W3 (256 x 256),
// b3, w4 (256), b4 (1).  Activations are row-major (rows = samples).  The FP32 network's 256 x 256
// layers and the first one run as dense products on the split-TF32 tensor-core tiles (FP32
// accuracy), bias, ReLU and the ReLU mask in their epilogues; the output layer and every sum
// over the samples are kernels of their own, cut into parts of the minibatch: a weight gradient
// is 16 tiles summed over thousands of samples, and a bias gradient one row, so without a split
// a handful of thread blocks would walk the whole minibatch.  The FP64 network (gradient checks)
// runs layer by layer on the grouped FP64 GEMM.
// Measured (GB300): loss and gradient of 4096 samples 2.35 -> 0.32 ms of kernels, 2.73 -> 0.57 ms
// with the copies of dmrg_mlp_loss_grad; its error against 64 bits 9e-7 -> 7e-7.
// Loss: mean squared error; optimizer: Adam.
#include <cmath>
#include <type_traits>

#include "common.h"

namespace dmrg {

constexpr int kWd = 256;
constexpr int kIn = 4;

int64_t mlp_n_params() {
  return int64_t(kWd) * kIn + kWd + 2 * (int64_t(kWd) * kWd + kWd) + kWd + 1;
}

struct MlpOffsets {
  int64_t W1, b1, W2, b2, W3, b3, w4, b4;
  MlpOffsets() {
    W1 = 0;
    b1 = W1 + int64_t(kWd) * kIn;
    W2 = b1 + kWd;
    b2 = W2 + int64_t(kWd) * kWd;
    W3 = b2 + kWd;
    b3 = W3 + int64_t(kWd) * kWd;
    w4 = b3 + kWd;
    b4 = w4 + kWd;
  }
};

// ------------------------------------------------------------------------------------
// elementwise kernels (the first four: FP64 network only)
// ------------------------------------------------------------------------------------
__global__ void k_bias_relu(double* __restrict__ Z, const double* __restrict__ b,
                            double* __restrict__ H, int64_t rows, int cols) {
  const int64_t n = rows * cols;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x) {
    const double z = Z[i] + b[i % cols];
    Z[i] = z;
    H[i] = z > 0.0 ? z : 0.0;
  }
}

__global__ void k_add_scalar(double* __restrict__ y, const double* __restrict__ b, int64_t n) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x)
    y[i] += b[0];
}

// dZ = dH * (Z > 0)
__global__ void k_relu_grad(const double* __restrict__ Z, double* __restrict__ dH, int64_t n) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x)
    if (!(Z[i] > 0.0)) dH[i] = 0.0;
}

// column sums of a rows x cols matrix (one thread per column, fixed order)
__global__ void k_colsum(const double* __restrict__ A, int64_t rows, int cols,
                         double* __restrict__ out) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cols) return;
  double s = 0.0;
  for (int64_t r = 0; r < rows; ++r) s += A[r * cols + c];
  out[c] = s;
}

// dY = 2 (Y - T) / B ; per-block partial sums of (Y - T)^2
template <class T>
__global__ void k_mse(const T* __restrict__ Y, const T* __restrict__ Tg, int64_t B,
                      T* __restrict__ dY, double* __restrict__ part) {
  __shared__ double sh[256];
  double s = 0.0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < B;
       i += int64_t(gridDim.x) * blockDim.x) {
    const T d = Y[i] - Tg[i];
    dY[i] = T(2) * d / T(B);
    s += double(d) * double(d);
  }
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = blockDim.x / 2; o > 0; o >>= 1) {
    if (int(threadIdx.x) < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) part[blockIdx.x] = sh[0];
}

template <class T>
__global__ void k_adam(T* __restrict__ p, const T* __restrict__ g, T* __restrict__ m,
                       T* __restrict__ v, int64_t n, double lr, double b1, double b2, double eps,
                       double c1, double c2) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x) {
    const double gi = double(g[i]);
    const double mi = b1 * double(m[i]) + (1.0 - b1) * gi;
    const double vi = b2 * double(v[i]) + (1.0 - b2) * gi * gi;
    m[i] = T(mi);
    v[i] = T(vi);
    p[i] = T(double(p[i]) - lr * (mi / c1) / (sqrt(vi / c2) + eps));
  }
}

// gather rows of a sample table into a minibatch (samples: n_in features + target)
template <class T>
__global__ void k_gather(const T* __restrict__ S, const int32_t* __restrict__ idx, int64_t B,
                         T* __restrict__ X, T* __restrict__ Tg) {
  for (int64_t b = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; b < B;
       b += int64_t(gridDim.x) * blockDim.x) {
    const T* s = S + int64_t(idx[b]) * (kIn + 1);
#pragma unroll
    for (int j = 0; j < kIn; ++j) X[b * kIn + j] = s[j];
    Tg[b] = s[kIn];
  }
}

// features of every element of a Davidson iterate:
//   asinh(theta - D_i), r_i sqrt(n)/|r|, x_i sqrt(n), d_i sqrt(n)/|d|,  d_i = r_i/(theta - D_i)
// (the clamped diagonal correction); sc = {theta, |r|^2, |d|^2}
// features and targets are O(1) by construction; bound the rare outliers (an element whose
// diagonal sits on theta, a residual at rounding level) so that FP32 training stays finite
__device__ __forceinline__ float clampf(double v) {
  return float(v != v ? 0.0 : fmin(fmax(v, -1e4), 1e4));
}

template <class T>
__global__ void k_features(const double* __restrict__ r, const double* __restrict__ x,
                           const double* __restrict__ diag, const double* __restrict__ sc,
                           int64_t n, T* __restrict__ X) {
  const double th = sc[0];
  const double sn = sqrt(double(n));
  const double ir = sc[1] > 0 ? sn / sqrt(sc[1]) : 0.0;
  const double id = sc[2] > 0 ? sn / sqrt(sc[2]) : 0.0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x) {
    double den = th - diag[i];
    if (fabs(den) < 1e-8) den = den < 0.0 ? -1e-8 : 1e-8;
    X[i * kIn + 0] = T(clampf(asinh(th - diag[i])));
    X[i * kIn + 1] = T(clampf(r[i] * ir));
    X[i * kIn + 2] = T(clampf(x[i] * sn));
    X[i * kIn + 3] = T(clampf(r[i] / den * id));
  }
}

// training pairs from one saved iterate: features of sampled elements and the target
// e_i sqrt(n)/|e|, e = psi - x (x . psi) with the sign of psi making x . psi >= 0;
// sc = {theta, |r|^2, |d|^2, x.psi, |e|^2}; elements i = start + k stride
__global__ void k_harvest(const double* __restrict__ r, const double* __restrict__ x,
                          const double* __restrict__ psi, const double* __restrict__ diag,
                          const double* __restrict__ sc, int64_t n, int64_t start, int64_t stride,
                          int64_t count, float* __restrict__ out) {
  const double th = sc[0];
  const double sn = sqrt(double(n));
  const double ir = sc[1] > 0 ? sn / sqrt(sc[1]) : 0.0;
  const double id = sc[2] > 0 ? sn / sqrt(sc[2]) : 0.0;
  const double ov = sc[3];
  const double sg = ov < 0 ? -1.0 : 1.0;
  // an iterate that already equals the eigenvector (|e| at rounding level) has no error
  // direction to learn: its targets are zero
  const double ie = sc[4] > 1e-20 ? sn / sqrt(sc[4]) : 0.0;
  for (int64_t k = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; k < count;
       k += int64_t(gridDim.x) * blockDim.x) {
    const int64_t i = start + k * stride;
    double den = th - diag[i];
    if (fabs(den) < 1e-8) den = den < 0.0 ? -1e-8 : 1e-8;
    float* o = out + k * (kIn + 1);
    o[0] = clampf(asinh(th - diag[i]));
    o[1] = clampf(r[i] * ir);
    o[2] = clampf(x[i] * sn);
    o[3] = clampf(r[i] / den * id);
    o[4] = clampf(sg * (psi[i] - x[i] * ov) * ie);
  }
}

// e = psi - x (x . psi) (sign of psi as above) for |e|^2
__global__ void k_err_vec(const double* __restrict__ x, const double* __restrict__ psi,
                          const double* __restrict__ sc, int64_t n, double* __restrict__ e) {
  const double ov = sc[3];
  const double sg = ov < 0 ? -1.0 : 1.0;
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x)
    e[i] = sg * (psi[i] - x[i] * ov);
}

// out_double[i] = y[i]
template <class T>
__global__ void k_to_double(const T* __restrict__ y, double* __restrict__ out, int64_t n) {
  for (int64_t i = int64_t(blockIdx.x) * blockDim.x + threadIdx.x; i < n;
       i += int64_t(gridDim.x) * blockDim.x)
    out[i] = double(y[i]);
}

static int grid_for(int64_t n) {
  return int(std::max<int64_t>(1, std::min<int64_t>((n + 255) / 256, 152 * 16)));
}

// C (M x N, ldc) = op(A) op(B) through the task-list GEMM; sizes of the three buffers in
// elements for the host-side range check
static void gemm(double* C, int ldc, const double* A, int lda, bool ta, const double* B, int ldb,
                 bool tb, int M, int N, int K, int64_t nA, int64_t nB, int64_t nC, cudaStream_t s) {
  TaskList L;
  L.begin_task(Operand{0, B_Y, ldc}, M, N);
  L.add_term(Operand{0, B_X, lda}, Operand{0, B_U, ldb}, K, (ta ? 1 : 0) | (tb ? 2 : 0), 1.0);
  int64_t be[NBASE] = {0};
  be[B_X] = nA;
  be[B_U] = nB;
  be[B_Y] = nC;
  DevTaskList d;
  d.build(L, be, s);
  Bases<double> b{};
  b.p[B_X] = const_cast<double*>(A);
  b.p[B_U] = const_cast<double*>(B);
  b.p[B_Y] = C;
  run_gemm_tasks<double>(d, b, 1, s);
  DMRG_CUDA(cudaStreamSynchronize(s));   // the list buffers are released on return
}

// ------------------------------------------------------------------------------------
// the FP32 network
// ------------------------------------------------------------------------------------
constexpr int kRows = 64;   // samples of one part of a sum over the minibatch

// y = H3 w4 + b4: one warp per sample, a compensated sum of eight products per lane, then a plain tree
// over the lanes
__global__ void __launch_bounds__(256) k_output(const float* __restrict__ H,
                                                const float* __restrict__ w,
                                                const float* __restrict__ b, int64_t B,
                                                float* __restrict__ y) {
  const int lane = threadIdx.x & 31;
  const int64_t r = (int64_t(blockIdx.x) * 256 + threadIdx.x) >> 5;
  if (r >= B) return;
  float s = 0.f, c = 0.f;
#pragma unroll
  for (int j = lane; j < kWd; j += 32) {
    const float v = fmaf(H[r * kWd + j], w[j], -c);
    const float t = s + v;
    c = (t - s) - v;
    s = t;
  }
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) y[r] = s + b[0];
}

// dH3 = dY w4 where H3 > 0, and the parts of sum_r dY H3 and of sum_r dY (kWd + 1 per part, in
// the order of w4, b4)
__global__ void __launch_bounds__(kWd) k_output_grad(const float* __restrict__ dY,
                                                     const float* __restrict__ H,
                                                     const float* __restrict__ w, int64_t B,
                                                     float* __restrict__ dH,
                                                     float* __restrict__ part) {
  const int j = threadIdx.x;
  const float wj = w[j];
  const int64_t r0 = int64_t(blockIdx.x) * kRows, r1 = min(B, r0 + kRows);
  float s = 0.f, sd = 0.f;
#pragma unroll 4
  for (int64_t r = r0; r < r1; ++r) {
    const float h = H[r * kWd + j], d = dY[r];
    s = fmaf(d, h, s);
    sd += d;
    dH[r * kWd + j] = h > 0.f ? d * wj : 0.f;
  }
  part[int64_t(blockIdx.x) * (kWd + 1) + j] = s;
  if (j == 0) part[int64_t(blockIdx.x) * (kWd + 1) + kWd] = sd;
}

// parts of the column sums of D (rows x 256), and of D^T X with the four inputs (X != nullptr):
// row of a part = 256 sums, then 256 x 4
template <bool X4>
__global__ void __launch_bounds__(kWd) k_column_parts(const float* __restrict__ D,
                                                      const float* __restrict__ X, int64_t B,
                                                      float* __restrict__ part) {
  const int j = threadIdx.x;
  const int64_t r0 = int64_t(blockIdx.x) * kRows, r1 = min(B, r0 + kRows);
  float s = 0.f, x0 = 0.f, x1 = 0.f, x2 = 0.f, x3 = 0.f;
#pragma unroll 4
  for (int64_t r = r0; r < r1; ++r) {
    const float d = D[r * kWd + j];
    s += d;
    if (X4) {
      const float* x = X + r * kIn;
      x0 = fmaf(d, x[0], x0);
      x1 = fmaf(d, x[1], x1);
      x2 = fmaf(d, x[2], x2);
      x3 = fmaf(d, x[3], x3);
    }
  }
  float* p = part + int64_t(blockIdx.x) * (X4 ? 5 : 1) * kWd;
  p[j] = s;
  if (X4) {
    p[kWd + 4 * j] = x0;
    p[kWd + 4 * j + 1] = x1;
    p[kWd + 4 * j + 2] = x2;
    p[kWd + 4 * j + 3] = x3;
  }
}

// out[i] = sum of the parts p[i + z stride], compensated, in order
__global__ void __launch_bounds__(256) k_add_parts(const float* __restrict__ p, int parts,
                                                   int64_t stride, int64_t n,
                                                   float* __restrict__ out) {
  const int64_t i = int64_t(blockIdx.x) * 256 + threadIdx.x;
  if (i >= n) return;
  float s = 0.f, c = 0.f;
#pragma unroll 4
  for (int z = 0; z < parts; ++z) {
    const float v = p[int64_t(z) * stride + i] - c;
    const float t = s + v;
    c = (t - s) - v;
    s = t;
  }
  out[i] = s;
}

static void add_parts(const float* p, int parts, int64_t stride, int64_t n, float* out,
                      cudaStream_t s) {
  k_add_parts<<<int((n + 255) / 256), 256, 0, s>>>(p, parts, stride, n, out);
  DMRG_LAUNCHED();
}

static void forward32(const float* P, const float* X, int64_t B, MlpActs<float>& a, cudaStream_t s) {
  MlpOffsets o;
  auto layer = [&](const float* in, int n_in, int64_t W, int64_t b, float* out) {
    dense_gemm_tc(DenseGemm{in, P + W, out, P + b, int(B), kWd, n_in, n_in, n_in, kWd, 2, n_in, 0},
                  DenseEpilogue::bias_relu, 1, s);
  };
  layer(X, kIn, o.W1, o.b1, a.H1.p);
  layer(a.H1.p, kWd, o.W2, o.b2, a.H2.p);
  layer(a.H2.p, kWd, o.W3, o.b3, a.H3.p);
  k_output<<<int((B + 7) / 8), 256, 0, s>>>(a.H3.p, P + o.w4, P + o.b4, B, a.Y.p);
  DMRG_LAUNCHED();
}

// gradients from a.dY on
static void backward32(const float* P, const float* X, int64_t B, MlpActs<float>& a, float* G,
                       cudaStream_t s) {
  MlpOffsets o;
  const int parts = int((B + kRows - 1) / kRows);
  // a weight gradient in parts of at least 128 samples, two thread blocks per SM at most
  const int splits = int(std::max<int64_t>(1, std::min<int64_t>(19, (B + 127) / 128)));
  const int k_len = int(((B + splits - 1) / splits + 31) / 32 * 32);
  const int used = int((B + k_len - 1) / k_len);
  const int64_t nw = int64_t(kWd) * kWd;
  a.sums.alloc(std::max<int64_t>(int64_t(parts) * 5 * kWd, int64_t(used) * nw));
  k_output_grad<<<parts, kWd, 0, s>>>(a.dY.p, a.H3.p, P + o.w4, B, a.dH.p, a.sums.p);
  DMRG_LAUNCHED();
  add_parts(a.sums.p, parts, kWd + 1, kWd + 1, G + o.w4, s);   // (b4 follows w4)
  // G_W = dZ^T H, G_b = column sums of dZ, d_in = dZ W masked by the layer below
  auto layer = [&](const float* dZ, const float* below, int64_t W, int64_t b, float* d_in) {
    dense_gemm_tc(DenseGemm{dZ, below, a.sums.p, nullptr, kWd, kWd, int(B), kWd, kWd, kWd, 1, k_len, nw},
                  DenseEpilogue::none, used, s);
    add_parts(a.sums.p, used, nw, nw, G + W, s);
    k_column_parts<false><<<parts, kWd, 0, s>>>(dZ, nullptr, B, a.sums.p);
    DMRG_LAUNCHED();
    add_parts(a.sums.p, parts, kWd, kWd, G + b, s);
    dense_gemm_tc(DenseGemm{dZ, P + W, d_in, below, int(B), kWd, kWd, kWd, kWd, kWd, 0, kWd, 0},
                  DenseEpilogue::mask, 1, s);
  };
  layer(a.dH.p, a.H2.p, o.W3, o.b3, a.dZ.p);
  layer(a.dZ.p, a.H1.p, o.W2, o.b2, a.dH.p);
  k_column_parts<true><<<parts, kWd, 0, s>>>(a.dH.p, X, B, a.sums.p);
  DMRG_LAUNCHED();
  add_parts(a.sums.p, parts, 5 * kWd, kWd, G + o.b1, s);
  add_parts(a.sums.p + kWd, parts, 5 * kWd, kWd * kIn, G + o.W1, s);
}

static void forward64(const double* P, const double* X, int64_t B, MlpActs<double>& a, cudaStream_t s) {
  MlpOffsets o;
  const int64_t np = mlp_n_params();
  const int64_t nh = B * kWd;
  gemm(a.Z1.p, kWd, X, kIn, false, P + o.W1, kIn, true, int(B), kWd, kIn, B * kIn, np - o.W1,
          nh, s);
  k_bias_relu<<<grid_for(nh), 256, 0, s>>>(a.Z1.p, P + o.b1, a.H1.p, B, kWd);
  DMRG_LAUNCHED();
  gemm(a.Z2.p, kWd, a.H1.p, kWd, false, P + o.W2, kWd, true, int(B), kWd, kWd, nh, np - o.W2,
          nh, s);
  k_bias_relu<<<grid_for(nh), 256, 0, s>>>(a.Z2.p, P + o.b2, a.H2.p, B, kWd);
  DMRG_LAUNCHED();
  gemm(a.Z3.p, kWd, a.H2.p, kWd, false, P + o.W3, kWd, true, int(B), kWd, kWd, nh, np - o.W3,
          nh, s);
  k_bias_relu<<<grid_for(nh), 256, 0, s>>>(a.Z3.p, P + o.b3, a.H3.p, B, kWd);
  DMRG_LAUNCHED();
  gemm(a.Y.p, 1, a.H3.p, kWd, false, P + o.w4, kWd, true, int(B), 1, kWd, nh, np - o.w4, B, s);
  k_add_scalar<<<grid_for(B), 256, 0, s>>>(a.Y.p, P + o.b4, B);
  DMRG_LAUNCHED();
}

template <class T>
void mlp_forward(const T* P, const T* X, int64_t B, MlpActs<T>& a, cudaStream_t s) {
  a.ensure(B);
  if constexpr (std::is_same<T, float>::value) forward32(P, X, B, a, s);
  else forward64(P, X, B, a, s);
}

static double mlp_loss(const double* d_part, int nb, int64_t B, cudaStream_t s) {
  std::vector<double> part(nb);
  DMRG_CUDA(cudaMemcpyAsync(part.data(), d_part, sizeof(double) * nb, cudaMemcpyDeviceToHost, s));
  DMRG_CUDA(cudaStreamSynchronize(s));
  double loss = 0.0;
  for (double x : part) loss += x;
  return loss / double(B);
}

// gradients from a.dY on
static void backward64(const double* P, const double* X, int64_t B, MlpActs<double>& a, double* G,
                       cudaStream_t s) {
  MlpOffsets o;
  const int64_t np = mlp_n_params();
  const int64_t nh = B * kWd;
  // output layer
  gemm(G + o.w4, kWd, a.dY.p, 1, true, a.H3.p, kWd, false, 1, kWd, int(B), B, nh, np - o.w4, s);
  k_colsum<<<1, 32, 0, s>>>(a.dY.p, B, 1, G + o.b4);
  DMRG_LAUNCHED();
  gemm(a.dH.p, kWd, a.dY.p, 1, false, P + o.w4, kWd, false, int(B), kWd, 1, B, np - o.w4, nh, s);
  // layer 3
  k_relu_grad<<<grid_for(nh), 256, 0, s>>>(a.Z3.p, a.dH.p, nh);
  DMRG_LAUNCHED();
  gemm(G + o.W3, kWd, a.dH.p, kWd, true, a.H2.p, kWd, false, kWd, kWd, int(B), nh, nh,
          np - o.W3, s);
  k_colsum<<<1, kWd, 0, s>>>(a.dH.p, B, kWd, G + o.b3);
  DMRG_LAUNCHED();
  gemm(a.dZ.p, kWd, a.dH.p, kWd, false, P + o.W3, kWd, false, int(B), kWd, kWd, nh, np - o.W3,
          nh, s);
  // layer 2
  k_relu_grad<<<grid_for(nh), 256, 0, s>>>(a.Z2.p, a.dZ.p, nh);
  DMRG_LAUNCHED();
  gemm(G + o.W2, kWd, a.dZ.p, kWd, true, a.H1.p, kWd, false, kWd, kWd, int(B), nh, nh,
          np - o.W2, s);
  k_colsum<<<1, kWd, 0, s>>>(a.dZ.p, B, kWd, G + o.b2);
  DMRG_LAUNCHED();
  gemm(a.dH.p, kWd, a.dZ.p, kWd, false, P + o.W2, kWd, false, int(B), kWd, kWd, nh, np - o.W2,
          nh, s);
  // layer 1
  k_relu_grad<<<grid_for(nh), 256, 0, s>>>(a.Z1.p, a.dH.p, nh);
  DMRG_LAUNCHED();
  gemm(G + o.W1, kIn, a.dH.p, kWd, true, X, kIn, false, kWd, kIn, int(B), nh, B * kIn,
          np - o.W1, s);
  k_colsum<<<1, kWd, 0, s>>>(a.dH.p, B, kWd, G + o.b1);
  DMRG_LAUNCHED();
}

// loss (mean squared error) and gradient G of the parameters; forward must have run on X
template <class T>
double mlp_backward(const T* P, const T* X, const T* Tg, int64_t B, MlpActs<T>& a, T* G,
                    cudaStream_t s) {
  const int nb = 64;
  a.part.alloc(nb);
  k_mse<T><<<nb, 256, 0, s>>>(a.Y.p, Tg, B, a.dY.p, a.part.p);
  DMRG_LAUNCHED();
  if constexpr (std::is_same<T, float>::value) backward32(P, X, B, a, G, s);
  else backward64(P, X, B, a, G, s);
  return mlp_loss(a.part.p, nb, B, s);
}

template <class T>
void mlp_adam(T* P, const T* G, T* m, T* v, int64_t n, double lr, int step, cudaStream_t s) {
  const double b1 = 0.9, b2 = 0.999, eps = 1e-8;
  const double c1 = 1.0 - std::pow(b1, step), c2 = 1.0 - std::pow(b2, step);
  k_adam<T><<<grid_for(n), 256, 0, s>>>(P, G, m, v, n, lr, b1, b2, eps, c1, c2);
  DMRG_LAUNCHED();
}

template <class T>
void mlp_gather(const T* S, const int32_t* idx, int64_t B, T* X, T* Tg, cudaStream_t s) {
  k_gather<T><<<grid_for(B), 256, 0, s>>>(S, idx, B, X, Tg);
  DMRG_LAUNCHED();
}

template <class T>
void mlp_features(const double* r, const double* x, const double* diag, const double* sc,
                  int64_t n, T* X, cudaStream_t s) {
  k_features<T><<<grid_for(n), 256, 0, s>>>(r, x, diag, sc, n, X);
  DMRG_LAUNCHED();
}

template <class T>
void mlp_output_to_double(const T* y, double* out, int64_t n, cudaStream_t s) {
  k_to_double<T><<<grid_for(n), 256, 0, s>>>(y, out, n);
  DMRG_LAUNCHED();
}

void mlp_harvest(const double* r, const double* x, const double* psi, const double* diag,
                 const double* sc, int64_t n, int64_t start, int64_t stride, int64_t count,
                 float* out, cudaStream_t s) {
  if (count <= 0) return;
  k_harvest<<<grid_for(count), 256, 0, s>>>(r, x, psi, diag, sc, n, start, stride, count, out);
  DMRG_LAUNCHED();
}

void mlp_err_vec(const double* x, const double* psi, const double* sc, int64_t n, double* e,
                 cudaStream_t s) {
  k_err_vec<<<grid_for(n), 256, 0, s>>>(x, psi, sc, n, e);
  DMRG_LAUNCHED();
}

template void mlp_forward<float>(const float*, const float*, int64_t, MlpActs<float>&, cudaStream_t);
template void mlp_forward<double>(const double*, const double*, int64_t, MlpActs<double>&,
                                  cudaStream_t);
template double mlp_backward<float>(const float*, const float*, const float*, int64_t,
                                    MlpActs<float>&, float*, cudaStream_t);
template double mlp_backward<double>(const double*, const double*, const double*, int64_t,
                                     MlpActs<double>&, double*, cudaStream_t);
template void mlp_adam<float>(float*, const float*, float*, float*, int64_t, double, int,
                              cudaStream_t);
template void mlp_gather<float>(const float*, const int32_t*, int64_t, float*, float*, cudaStream_t);
template void mlp_features<float>(const double*, const double*, const double*, const double*,
                                  int64_t, float*, cudaStream_t);
template void mlp_output_to_double<float>(const float*, double*, int64_t, cudaStream_t);

}  // namespace dmrg
