// Newton initial-guess network: inference (warp mma.sync, BF16 weights, FP32
// accumulation), training forward/backward and Adam in FP32, all in own
// kernels.  Parameter vector layout (FP32, 4609 + 12): W1[64][5], b1[64],
// W2[64][64], b2[64], W3[64], b3, in_mean[5], in_std[5], out_mean, out_std.
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <numeric>
#include <random>
#include <string>
#include <vector>

#include "mlp.cuh"
#include "sbiem.h"

namespace sbiem {

// ----------------------------------------------------------- deployment
__global__ void k_mlp_pack(const float* __restrict__ p, MlpDev* out) {
  const float* W1 = p;
  const float* b1 = W1 + kMlpH * kMlpIn;
  const float* W2 = b1 + kMlpH;
  const float* b2 = W2 + kMlpH * kMlpH;
  const float* W3 = b2 + kMlpH;
  const float* b3 = W3 + kMlpH;
  const float* nrm = b3 + 1;
  for (int i = threadIdx.x; i < kMlpH * 8; i += blockDim.x) {
    const int n = i / 8, j = i % 8;
    const float lo = (2 * j < kMlpIn) ? W1[n * kMlpIn + 2 * j] : 0.f;
    const float hi = (2 * j + 1 < kMlpIn) ? W1[n * kMlpIn + 2 * j + 1] : 0.f;
    out->w1p[n][j] = pack_bf16(lo, hi);
  }
  for (int i = threadIdx.x; i < kMlpH * 32; i += blockDim.x) {
    const int n = i / 32, j = i % 32;
    out->w2p[n][j] = pack_bf16(W2[n * kMlpH + 2 * j], W2[n * kMlpH + 2 * j + 1]);
  }
  for (int i = threadIdx.x; i < kMlpH; i += blockDim.x) {
    out->b1[i] = b1[i];
    out->b2[i] = b2[i];
    out->w3[i] = W3[i];
  }
  if (threadIdx.x == 0) {
    out->b3 = b3[0];
    for (int k = 0; k < kMlpIn; ++k) {
      out->in_mean[k] = nrm[k];
      out->in_std[k] = nrm[kMlpIn + k];
    }
    out->out_mean = nrm[2 * kMlpIn];
    out->out_std = nrm[2 * kMlpIn + 1];
  }
}

// One warp per 32 feature rows (raw features, [n][5]); out[n] = predicted residual.
__global__ void k_mlp_predict(const MlpDev* __restrict__ net, const float* __restrict__ X, int64_t n,
                              float* __restrict__ out) {
  __shared__ MlpDev m;
  for (int i = threadIdx.x; i < static_cast<int>(sizeof(MlpDev) / 4); i += blockDim.x)
    reinterpret_cast<uint32_t*>(&m)[i] = reinterpret_cast<const uint32_t*>(net)[i];
  __syncthreads();
  const int64_t row = static_cast<int64_t>(blockIdx.x) * blockDim.x + threadIdx.x;
  float feat[kMlpIn];
#pragma unroll
  for (int k = 0; k < kMlpIn; ++k) feat[k] = row < n ? X[row * kMlpIn + k] : m.in_mean[k];
  const float y = mlp_residual_warp(m, feat);
  if (row < n) out[row] = y;
}

// ------------------------------------------------------------- training
// Loss and gradient of the mean-squared error on normalized rows, FP32: three
// 64 x 64 x 64 products a tile of 64 rows (Z2 = H1 W2^T, dH1 = dZ2 W2, dW2 =
// dZ2^T H1), the rest elementwise.  A CTA of 16 x 16 threads owns tiles t,
// t + grid, ...; each thread computes 4 x 4 blocks of the products from
// shared memory (16 FMA per two 128-bit reads) and keeps its 4 x 4 block of
// dW2 and its column sums (dW1, db1, db2, dW3) in registers over all its
// tiles, so a gradient leaves the CTA once.  H1 and dZ2 are kept in both
// orientations, so every product reads rows; the leading dimension of 68
// keeps the 128-bit accesses of a warp (8 x 4 threads) at four wavefronts.
// Bound by FP32 issue (erff and expf of 128 activations a row and 12,288 FMA):
// sbiem_mlp_grad of 100,003 rows 1730 us with a thread per row and 32-way bank
// conflicts (the kernel 1298 us of it), 340 us so (most of it the copies in).
constexpr int kTrainRows = 128;   // smallest batch sbiem_mlp_train takes
constexpr int kTileRows = 64;
constexpr int kTrainThreads = 256;
constexpr int kLd = 68;           // leading dimension of the 64 x 64 tiles

// GELU and its derivative.
__device__ __forceinline__ void gelu_pair(float z, float* g, float* d) {
  const float cdf = 0.5f * (1.f + erff(z * 0.70710678118654752f));
  *g = z * cdf;
  *d = fmaf(z * 0.3989422804014327f, expf(-0.5f * z * z), cdf);
}

// acc[i][j] += sum_k A[k][a0 + i] B[k][b0 + j], k < 64 in order.
__device__ __forceinline__ void tile_product(const float* __restrict__ A, const float* __restrict__ B, int a0, int b0,
                                             float (&acc)[4][4]) {
#pragma unroll 8
  for (int k = 0; k < kMlpH; ++k) {
    const float4 a = *reinterpret_cast<const float4*>(A + k * kLd + a0);
    const float4 b = *reinterpret_cast<const float4*>(B + k * kLd + b0);
    const float av[4] = {a.x, a.y, a.z, a.w}, bv[4] = {b.x, b.y, b.z, b.w};
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(av[i], bv[j], acc[i][j]);
  }
}

// A thread's 4 x 4 block, rows r0.., columns c0.., row-major and transposed.
__device__ __forceinline__ void put_block(float* R, float* T, int r0, int c0, const float (&v)[4][4]) {
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    *reinterpret_cast<float4*>(R + (r0 + i) * kLd + c0) = make_float4(v[i][0], v[i][1], v[i][2], v[i][3]);
    *reinterpret_cast<float4*>(T + (c0 + i) * kLd + r0) = make_float4(v[0][i], v[1][i], v[2][i], v[3][i]);
  }
}

struct TrainSmem {
  float W2[kMlpH * kLd], W2T[kMlpH * kLd];
  float H1R[kTileRows * kLd], H1T[kTileRows * kLd], D2R[kTileRows * kLd], D2T[kTileRows * kLd];
  float W1[kMlpH][kMlpIn], b1[kMlpH], b2[kMlpH], W3[kMlpH];
  float X[kTileRows][kMlpIn], t[kTileRows];
  float part[4][kTileRows];  // row sums of the output layer by column quarter
  float dy[kTileRows];
  float db3[kTileRows];
  double loss[kTileRows];
};

// Rows idx[b0 .. b0 + B) of X[n][5], t[n] (idx NULL: rows b0 ..).  Each CTA
// writes its partial gradient (scaled by 2/B) and partial loss.
__global__ void __launch_bounds__(kTrainThreads, 2)
    k_mlp_grad(const float* __restrict__ p, const float* __restrict__ X, const float* __restrict__ t,
               const int* __restrict__ idx, int64_t b0, int B, float* __restrict__ partial,
               double* __restrict__ loss_partial) {
  extern __shared__ __align__(16) unsigned char train_raw[];
  TrainSmem& s = *reinterpret_cast<TrainSmem*>(train_raw);
  const float* gW1 = p;
  const float* gb1 = gW1 + kMlpH * kMlpIn;
  const float* gW2 = gb1 + kMlpH;
  const float* gb2 = gW2 + kMlpH * kMlpH;
  const float* gW3 = gb2 + kMlpH;
  const float b3 = gW3[kMlpH];
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;
  for (int i = tid; i < kMlpH * kMlpH; i += kTrainThreads) {
    const int j = i / kMlpH, k = i % kMlpH;
    const float w = gW2[i];
    s.W2[j * kLd + k] = w;
    s.W2T[k * kLd + j] = w;
  }
  for (int i = tid; i < kMlpH * kMlpIn; i += kTrainThreads) s.W1[i / kMlpIn][i % kMlpIn] = gW1[i];
  if (tid < kMlpH) {
    s.b1[tid] = gb1[tid];
    s.b2[tid] = gb2[tid];
    s.W3[tid] = gW3[tid];
  }
  // a warp holds 8 row groups x 4 column groups of the 16 x 16 blocks
  const int rg = (wid >> 2) * 8 + (lane & 7), cg = (wid & 3) * 4 + (lane >> 3);
  const int r0 = 4 * rg, c0 = 4 * cg;
  float dW2[4][4] = {}, dW1[4][kMlpIn] = {}, db1[4] = {}, db2[4] = {}, dW3[4] = {};
  float db3 = 0.f;      // threads below kTileRows
  double loss = 0.0;
  const float scale = 2.f / static_cast<float>(B);
  const int tiles = (B + kTileRows - 1) / kTileRows;
  for (int tile = blockIdx.x; tile < tiles; tile += gridDim.x) {
    __syncthreads();  // the last tile's reads are over
    for (int i = tid; i < kTileRows * (kMlpIn + 1); i += kTrainThreads) {
      const int r = i / (kMlpIn + 1), k = i % (kMlpIn + 1);
      const int64_t q = static_cast<int64_t>(tile) * kTileRows + r;
      float v = 0.f;
      if (q < B) {
        const int64_t row = idx ? idx[b0 + q] : b0 + q;
        v = k < kMlpIn ? X[row * kMlpIn + k] : t[row];
      }
      if (k < kMlpIn) s.X[r][k] = v;
      else s.t[r] = v;
    }
    __syncthreads();
    float x[4][kMlpIn], h[4][4], gp1[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int k = 0; k < kMlpIn; ++k) x[i][k] = s.X[r0 + i][k];
    // H1 = GELU(X W1^T + b1)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
#pragma unroll
      for (int i = 0; i < 4; ++i) {
        float z = s.b1[c0 + j];
#pragma unroll
        for (int k = 0; k < kMlpIn; ++k) z = fmaf(s.W1[c0 + j][k], x[i][k], z);
        gelu_pair(z, &h[i][j], &gp1[i][j]);
      }
    }
    put_block(s.H1R, s.H1T, r0, c0, h);
    __syncthreads();
    // Z2 = H1 W2^T + b2, y = GELU(Z2) . W3 + b3
    float z[4][4], gp2[4][4];
#pragma unroll
    for (int j = 0; j < 4; ++j)
#pragma unroll
      for (int i = 0; i < 4; ++i) z[i][j] = s.b2[c0 + j];
    tile_product(s.H1T, s.W2T, r0, c0, z);
    float yp[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      yp[i] = 0.f;
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        gelu_pair(z[i][j], &h[i][j], &gp2[i][j]);  // h: GELU(Z2)
        yp[i] = fmaf(s.W3[c0 + j], h[i][j], yp[i]);
      }
      yp[i] += __shfl_xor_sync(0xffffffffu, yp[i], 8);
      yp[i] += __shfl_xor_sync(0xffffffffu, yp[i], 16);
    }
    if (lane < 8) *reinterpret_cast<float4*>(&s.part[wid & 3][r0]) = make_float4(yp[0], yp[1], yp[2], yp[3]);
    __syncthreads();
    if (tid < kTileRows) {
      const bool valid = static_cast<int64_t>(tile) * kTileRows + tid < B;
      const float y = b3 + ((s.part[0][tid] + s.part[1][tid]) + (s.part[2][tid] + s.part[3][tid]));
      const float res = valid ? y - s.t[tid] : 0.f;
      s.dy[tid] = scale * res;
      db3 += scale * res;
      loss += static_cast<double>(res) * static_cast<double>(res);
    }
    __syncthreads();
    // dZ2 = dy W3 GELU'(Z2)
    float d2[4][4];
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      const float dy = s.dy[r0 + i];
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        d2[i][j] = dy * s.W3[c0 + j] * gp2[i][j];
        dW3[j] = fmaf(dy, h[i][j], dW3[j]);
        db2[j] += d2[i][j];
      }
    }
    put_block(s.D2R, s.D2T, r0, c0, d2);
    __syncthreads();
    // dZ1 = (dZ2 W2) GELU'(Z1); dW1, db1 are its column sums
    float d1[4][4] = {};
    tile_product(s.D2T, s.W2, r0, c0, d1);
#pragma unroll
    for (int i = 0; i < 4; ++i)
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const float d = d1[i][j] * gp1[i][j];
        db1[j] += d;
#pragma unroll
        for (int k = 0; k < kMlpIn; ++k) dW1[j][k] = fmaf(d, x[i][k], dW1[j][k]);
      }
    // dW2 (rows: its output unit, columns: its input unit) over the tile's rows
    tile_product(s.D2R, s.H1R, r0, c0, dW2);
  }
  // column sums by row group, in the tiles' place
  float(*col)[kMlpH][kMlpIn + 3] = reinterpret_cast<float(*)[kMlpH][kMlpIn + 3]>(s.H1R);
  static_assert(sizeof(float) * 16 * kMlpH * (kMlpIn + 3) <= sizeof(s.H1R) + sizeof(s.H1T), "fits the two H1 tiles");
  __syncthreads();
  float* out = partial + static_cast<int64_t>(blockIdx.x) * kMlpParams;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) out[kMlpH * kMlpIn + kMlpH + (r0 + i) * kMlpH + c0 + j] = dW2[i][j];
#pragma unroll
  for (int j = 0; j < 4; ++j) {
    float* c = col[rg][c0 + j];
#pragma unroll
    for (int k = 0; k < kMlpIn; ++k) c[k] = dW1[j][k];
    c[kMlpIn] = db1[j];
    c[kMlpIn + 1] = db2[j];
    c[kMlpIn + 2] = dW3[j];
  }
  if (tid < kTileRows) {
    s.db3[tid] = db3;
    s.loss[tid] = loss;
  }
  __syncthreads();
  for (int i = tid; i < kMlpH * (kMlpIn + 3); i += kTrainThreads) {
    const int j = i / (kMlpIn + 3), k = i % (kMlpIn + 3);
    float v = 0.f;
    for (int g = 0; g < 16; ++g) v += col[g][j][k];
    const int tail = kMlpH * kMlpIn + kMlpH + kMlpH * kMlpH;
    out[k < kMlpIn ? j * kMlpIn + k : k == kMlpIn ? kMlpH * kMlpIn + j : k == kMlpIn + 1 ? tail + j : tail + kMlpH + j] =
        v;
  }
  if (tid == 0) {
    float v = 0.f;
    double l = 0.0;
    for (int r = 0; r < kTileRows; ++r) {
      v += s.db3[r];
      l += s.loss[r];
    }
    out[kMlpParams - 1] = v;
    loss_partial[blockIdx.x] = l;
  }
}

// grad[p] = sum over CTAs of partial[c][p], fixed order (eight interleaved
// subsums a parameter, so that the reads of one parameter overlap); optional
// Adam step.
__global__ void __launch_bounds__(256)
    k_mlp_reduce(const float* __restrict__ partial, int nblk, float* __restrict__ grad, float* p, float* m1, float* m2,
                 float lr, float beta1, float beta2, float epsa, int step) {
  __shared__ float sub[8][32];
  const int lane = threadIdx.x & 31, slice = threadIdx.x >> 5;
  const int pi = blockIdx.x * 32 + lane;
  float g = 0.f;
  if (pi < kMlpParams)
    for (int c = slice; c < nblk; c += 8) g += partial[static_cast<int64_t>(c) * kMlpParams + pi];
  sub[slice][lane] = g;
  __syncthreads();
  if (slice > 0 || pi >= kMlpParams) return;
  g = 0.f;
#pragma unroll
  for (int q = 0; q < 8; ++q) g += sub[q][lane];
  if (grad) grad[pi] = g;
  if (m1) {
    const float a = beta1 * m1[pi] + (1.f - beta1) * g;
    const float b = beta2 * m2[pi] + (1.f - beta2) * g * g;
    m1[pi] = a;
    m2[pi] = b;
    const float ah = a / (1.f - powf(beta1, static_cast<float>(step)));
    const float bh = b / (1.f - powf(beta2, static_cast<float>(step)));
    p[pi] -= lr * ah / (sqrtf(bh) + epsa);
  }
}
constexpr int kReduceCtas = (kMlpParams + 31) / 32;

// CTAs of k_mlp_grad for B rows: one a tile up to two on each of a GB300's 152
// SMs, all that are resident there.  Each leaves a partial gradient, so their
// number sets the order of the sums: it follows from the rows alone, not from
// the SMs that a device or a partition of it offers.
constexpr int kTrainCtas = 304;
int train_ctas(int64_t B) {
  return static_cast<int>(std::max<int64_t>(1, std::min<int64_t>((B + kTileRows - 1) / kTileRows, kTrainCtas)));
}
cudaError_t configure_train() {
  return cudaFuncSetAttribute(k_mlp_grad, cudaFuncAttributeMaxDynamicSharedMemorySize,
                              static_cast<int>(sizeof(TrainSmem)));
}

}  // namespace sbiem

using namespace sbiem;

namespace {
thread_local std::string g_mlp_err;
#define MCK(call)                                                   \
  do {                                                              \
    cudaError_t e_ = (call);                                        \
    if (e_ != cudaSuccess) {                                        \
      g_mlp_err = std::string(#call) + ": " + cudaGetErrorString(e_); \
      rc = SBIEM_ERR_CUDA;                                          \
      goto done;                                                    \
    }                                                               \
  } while (0)
}  // namespace

extern "C" {

int sbiem_mlp_predict(const float* params, const float* X, int64_t n, float* out) {
  if (!params || !X || !out || n < 0) return SBIEM_ERR_INVALID;
  int rc = SBIEM_OK;
  float *dp = nullptr, *dX = nullptr, *dout = nullptr;
  MlpDev* net = nullptr;
  MCK(cudaMalloc(&dp, sizeof(float) * (kMlpParams + kMlpNorm)));
  MCK(cudaMalloc(&net, sizeof(MlpDev)));
  MCK(cudaMalloc(&dX, sizeof(float) * kMlpIn * std::max<int64_t>(n, 1)));
  MCK(cudaMalloc(&dout, sizeof(float) * std::max<int64_t>(n, 1)));
  MCK(cudaMemcpy(dp, params, sizeof(float) * (kMlpParams + kMlpNorm), cudaMemcpyHostToDevice));
  MCK(cudaMemcpy(dX, X, sizeof(float) * kMlpIn * n, cudaMemcpyHostToDevice));
  k_mlp_pack<<<1, 256>>>(dp, net);
  if (n > 0) k_mlp_predict<<<static_cast<unsigned>((n + 31) / 32), 32>>>(net, dX, n, dout);
  MCK(cudaGetLastError());
  MCK(cudaMemcpy(out, dout, sizeof(float) * n, cudaMemcpyDeviceToHost));
done:
  cudaFree(dp);
  cudaFree(net);
  cudaFree(dX);
  cudaFree(dout);
  return rc;
}

int sbiem_mlp_grad(const float* params, const float* X, const float* t, int64_t n, float* grad, float* loss) {
  if (!params || !X || !t || !grad || n < 1 || n > (1 << 24)) return SBIEM_ERR_INVALID;
  int rc = SBIEM_OK;
  const int nblk = train_ctas(n);
  // one device allocation: loss partials, parameters, gradient, rows,
  // targets, gradient partials (each part a multiple of 16 bytes)
  auto up16 = [](size_t k) { return (k + 3) / 4 * 4; };
  const size_t np = up16(kMlpParams), nx = up16(static_cast<size_t>(kMlpIn) * n), nt = up16(static_cast<size_t>(n));
  double* lp = nullptr;
  float *dp = nullptr, *dg = nullptr, *dX = nullptr, *dt = nullptr, *part = nullptr;
  std::vector<double> lh(nblk);
  MCK(cudaMalloc(&lp, sizeof(double) * up16(nblk) + sizeof(float) * (2 * np + nx + nt + static_cast<size_t>(kMlpParams) * nblk)));
  dp = reinterpret_cast<float*>(lp + up16(nblk));
  dg = dp + np;
  dX = dg + np;
  dt = dX + nx;
  part = dt + nt;
  MCK(cudaMemcpy(dp, params, sizeof(float) * kMlpParams, cudaMemcpyHostToDevice));
  MCK(cudaMemcpy(dX, X, sizeof(float) * kMlpIn * n, cudaMemcpyHostToDevice));
  MCK(cudaMemcpy(dt, t, sizeof(float) * n, cudaMemcpyHostToDevice));
  MCK(configure_train());
  k_mlp_grad<<<nblk, kTrainThreads, sizeof(TrainSmem)>>>(dp, dX, dt, nullptr, 0, static_cast<int>(n), part, lp);
  k_mlp_reduce<<<kReduceCtas, 256>>>(part, nblk, dg, nullptr, nullptr, nullptr, 0.f, 0.f, 0.f, 0.f, 0);
  MCK(cudaGetLastError());
  MCK(cudaMemcpy(grad, dg, sizeof(float) * kMlpParams, cudaMemcpyDeviceToHost));
  MCK(cudaMemcpy(lh.data(), lp, sizeof(double) * nblk, cudaMemcpyDeviceToHost));
  if (loss) {
    double l = 0.0;
    for (double v : lh) l += v;
    *loss = static_cast<float>(l / static_cast<double>(n));
  }
done:
  cudaFree(lp);
  return rc;
}

int sbiem_mlp_train(const float* samples, int64_t n, int epochs, int batch, float lr, uint64_t seed,
                    float* params, float* final_loss) {
  // samples: n rows of (ln V_prev, ln theta, tau/sigma, a, b, ln V*)
  if (!samples || !params || n < 2 || epochs < 1 || batch < kTrainRows || !(lr > 0)) return SBIEM_ERR_INVALID;
  int rc = SBIEM_OK;
  // normalization: per-feature mean / std of the inputs and of the residual
  double mean[kMlpIn] = {0}, var[kMlpIn] = {0}, rm = 0.0, rv = 0.0;
  for (int64_t i = 0; i < n; ++i) {
    const float* r = samples + i * 6;
    for (int k = 0; k < kMlpIn; ++k) mean[k] += r[k];
    rm += r[5] - r[0];
  }
  for (int k = 0; k < kMlpIn; ++k) mean[k] /= n;
  rm /= n;
  for (int64_t i = 0; i < n; ++i) {
    const float* r = samples + i * 6;
    for (int k = 0; k < kMlpIn; ++k) var[k] += (r[k] - mean[k]) * (r[k] - mean[k]);
    const double d = r[5] - r[0] - rm;
    rv += d * d;
  }
  float in_mean[kMlpIn], in_std[kMlpIn];
  for (int k = 0; k < kMlpIn; ++k) {
    in_mean[k] = static_cast<float>(mean[k]);
    in_std[k] = static_cast<float>(std::max(std::sqrt(var[k] / n), 1e-6));
  }
  const float out_mean = static_cast<float>(rm), out_std = static_cast<float>(std::max(std::sqrt(rv / n), 1e-6));
  std::vector<float> Xn(static_cast<size_t>(n) * kMlpIn), tn(n);
  for (int64_t i = 0; i < n; ++i) {
    const float* r = samples + i * 6;
    for (int k = 0; k < kMlpIn; ++k) Xn[i * kMlpIn + k] = (r[k] - in_mean[k]) / in_std[k];
    tn[i] = (r[5] - r[0] - out_mean) / out_std;
  }
  // He-style initialization (seeded)
  std::mt19937_64 rng(seed);
  std::normal_distribution<float> nd(0.f, 1.f);
  std::vector<float> p(kMlpParams, 0.f);
  for (int i = 0; i < kMlpH * kMlpIn; ++i) p[i] = nd(rng) * std::sqrt(2.f / kMlpIn);
  for (int i = 0; i < kMlpH * kMlpH; ++i) p[kMlpH * kMlpIn + kMlpH + i] = nd(rng) * std::sqrt(2.f / kMlpH);
  for (int i = 0; i < kMlpH; ++i) p[kMlpH * kMlpIn + 2 * kMlpH + kMlpH * kMlpH + i] = nd(rng) * std::sqrt(1.f / kMlpH);
  const int B = std::min<int64_t>(batch, n);
  const int nblk = train_ctas(B);
  float *dp = nullptr, *dX = nullptr, *dt = nullptr, *part = nullptr, *m1 = nullptr, *m2 = nullptr;
  double* lp = nullptr;
  int* didx = nullptr;
  std::vector<int> perm(n);
  std::iota(perm.begin(), perm.end(), 0);
  int step = 0;
  double last = 0.0;
  std::vector<double> lh(nblk);
  MCK(cudaMalloc(&dp, sizeof(float) * kMlpParams));
  MCK(cudaMalloc(&m1, sizeof(float) * kMlpParams));
  MCK(cudaMalloc(&m2, sizeof(float) * kMlpParams));
  MCK(cudaMalloc(&dX, sizeof(float) * kMlpIn * n));
  MCK(cudaMalloc(&dt, sizeof(float) * n));
  MCK(cudaMalloc(&didx, sizeof(int) * n));
  MCK(cudaMalloc(&part, sizeof(float) * kMlpParams * nblk));
  MCK(cudaMalloc(&lp, sizeof(double) * nblk));
  MCK(cudaMemcpy(dp, p.data(), sizeof(float) * kMlpParams, cudaMemcpyHostToDevice));
  MCK(cudaMemset(m1, 0, sizeof(float) * kMlpParams));
  MCK(cudaMemset(m2, 0, sizeof(float) * kMlpParams));
  MCK(cudaMemcpy(dX, Xn.data(), sizeof(float) * kMlpIn * n, cudaMemcpyHostToDevice));
  MCK(cudaMemcpy(dt, tn.data(), sizeof(float) * n, cudaMemcpyHostToDevice));
  MCK(configure_train());
  for (int ep = 0; ep < epochs; ++ep) {
    std::shuffle(perm.begin(), perm.end(), rng);
    MCK(cudaMemcpy(didx, perm.data(), sizeof(int) * n, cudaMemcpyHostToDevice));
    double lsum = 0.0;
    int64_t lcnt = 0;
    for (int64_t b0 = 0; b0 + B <= n; b0 += B) {
      ++step;
      k_mlp_grad<<<nblk, kTrainThreads, sizeof(TrainSmem)>>>(dp, dX, dt, didx, b0, B, part, lp);
      k_mlp_reduce<<<kReduceCtas, 256>>>(part, nblk, nullptr, dp, m1, m2, lr, 0.9f, 0.999f, 1e-8f, step);
      if (b0 + 2 * B > n) {  // loss of the epoch's last batch
        MCK(cudaMemcpy(lh.data(), lp, sizeof(double) * nblk, cudaMemcpyDeviceToHost));
        for (double v : lh) lsum += v;
        lcnt += B;
      }
    }
    MCK(cudaGetLastError());
    if (lcnt) last = lsum / static_cast<double>(lcnt);
  }
  MCK(cudaMemcpy(params, dp, sizeof(float) * kMlpParams, cudaMemcpyDeviceToHost));
  for (int k = 0; k < kMlpIn; ++k) {
    params[kMlpParams + k] = in_mean[k];
    params[kMlpParams + kMlpIn + k] = in_std[k];
  }
  params[kMlpParams + 2 * kMlpIn] = out_mean;
  params[kMlpParams + 2 * kMlpIn + 1] = out_std;
  if (final_loss) *final_loss = static_cast<float>(last);
done:
  cudaFree(dp);
  cudaFree(m1);
  cudaFree(m2);
  cudaFree(dX);
  cudaFree(dt);
  cudaFree(didx);
  cudaFree(part);
  cudaFree(lp);
  return rc;
}

}  // extern "C"

namespace sbiem {
// Device copy of a deployed network (used by the handle).
int mlp_deploy(const float* params_host, MlpDev* dst, cudaStream_t st) {
  float* dp = nullptr;
  if (cudaMalloc(&dp, sizeof(float) * (kMlpParams + kMlpNorm)) != cudaSuccess) return SBIEM_ERR_NOMEM;
  cudaMemcpyAsync(dp, params_host, sizeof(float) * (kMlpParams + kMlpNorm), cudaMemcpyHostToDevice, st);
  k_mlp_pack<<<1, 256, 0, st>>>(dp, dst);
  cudaError_t e = cudaStreamSynchronize(st);
  cudaFree(dp);
  return e == cudaSuccess ? SBIEM_OK : SBIEM_ERR_CUDA;
}
}  // namespace sbiem
