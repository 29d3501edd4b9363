// Learned path cost model: a 3-layer MLP (hidden width h, BF16 weights, FP32
// master weights and accumulation) predicting the log time of a contraction
// step from its features; training and inference run in these kernels.
//
//   z1 = x W1 + b1, a1 = relu(z1); z2 = a1 W2 + b2, a2 = relu(z2); y = a2 W3 + b3
//   loss = mean (y - t)^2, gradients by the chain rule, Adam updates of the FP32
//   master weights followed by a refresh of their BF16 copies.
//
// The paper motivates such a model (a path with more flops ran faster on the
// hardware, Sec. 4.3) but defines none.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>
#include <new>
#include <random>
#include <string>
#include <vector>

#include "executor.h"
#include "kernels.cuh"
#include "mlp.h"
#include "rules.h"

namespace tnq {

namespace {

// ---------------------------------------------------------------- GEMM
// C[M][N] (+)= op(A)[M][K] * op(B)[K][N] (+ bias[N]); A float, B float or bf16.
// op(A)(i,k) = transA ? A[k*lda + i] : A[i*lda + k]; likewise B.
constexpr int MG_T = 64, MG_K = 16;

template <typename TB>
__global__ void __launch_bounds__(256) mlp_gemm_kernel(int M, int N, int K, const float* __restrict__ A, int lda,
                                                       int transA, const TB* __restrict__ B, int ldb, int transB,
                                                       float* __restrict__ C, int ldc, const float* __restrict__ bias,
                                                       int relu_into, float* __restrict__ R) {
  __shared__ float As[MG_K][MG_T + 1];
  __shared__ float Bs[MG_K][MG_T + 1];
  const int tid = threadIdx.x, tx = tid & 15, ty = tid >> 4;
  const int m0 = blockIdx.y * MG_T, n0 = blockIdx.x * MG_T;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  for (int k0 = 0; k0 < K; k0 += MG_K) {
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int idx = tid + 256 * l;
      // A tile: rows m0..m0+63, k0..k0+15
      {
        const int r = transA ? idx % MG_T : idx / MG_K, kk = transA ? idx / MG_T : idx % MG_K;
        float v = 0.f;
        if (m0 + r < M && k0 + kk < K) v = transA ? A[size_t(k0 + kk) * lda + m0 + r] : A[size_t(m0 + r) * lda + k0 + kk];
        As[kk][r] = v;
      }
      // B tile: k0..k0+15, columns n0..n0+63
      {
        const int c = transB ? idx / MG_K : idx % MG_T, kk = transB ? idx % MG_K : idx / MG_T;
        float v = 0.f;
        if (n0 + c < N && k0 + kk < K) {
          const TB b = transB ? B[size_t(n0 + c) * ldb + k0 + kk] : B[size_t(k0 + kk) * ldb + n0 + c];
          v = float(b);
        }
        Bs[kk][c] = v;
      }
    }
    __syncthreads();
#pragma unroll
    for (int kk = 0; kk < MG_K; ++kk) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int m = m0 + ty + 16 * i, n = n0 + tx + 16 * j;
      if (m < M && n < N) {
        float v = acc[i][j] + (bias ? bias[n] : 0.f);
        C[size_t(m) * ldc + n] = v;
        if (relu_into) R[size_t(m) * ldc + n] = fmaxf(v, 0.f);
      }
    }
}

template <typename TB>
cudaError_t gemm(cudaStream_t st, int M, int N, int K, const float* A, int lda, int tA, const TB* B, int ldb, int tB,
                 float* C, int ldc, const float* bias = nullptr, float* relu_out = nullptr) {
  dim3 grid((N + MG_T - 1) / MG_T, (M + MG_T - 1) / MG_T);
  mlp_gemm_kernel<TB><<<grid, 256, 0, st>>>(M, N, K, A, lda, tA, B, ldb, tB, C, ldc, bias, relu_out ? 1 : 0,
                                            relu_out);
  return cudaGetLastError();
}

// ---------------------------------------------------------------- elementwise
__global__ void dy_kernel(const float* y, const float* t, int B, float* dy, float* sq) {
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < B; i += gridDim.x * blockDim.x) {
    const float d = y[i] - t[i];
    dy[i] = 2.f * d / float(B);
    sq[i] = d * d;
  }
}

// g[i] *= (z[i] > 0)
__global__ void relu_mask_kernel(float* g, const float* z, size_t n) {
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x)
    if (!(z[i] > 0.f)) g[i] = 0.f;
}

// out[c] = sum over rows r < R of X[r*ld + c] (fixed row order); optionally / div
__global__ void colsum_kernel(const float* X, int R, int Cn, int ld, float* out, float scale) {
  for (int c = blockIdx.x * blockDim.x + threadIdx.x; c < Cn; c += gridDim.x * blockDim.x) {
    float s = 0.f;
    for (int r = 0; r < R; ++r) s += X[size_t(r) * ld + c];
    out[c] = s * scale;
  }
}

// BF16 copy of a weight matrix entry of the flat parameter vector (W1 b1 W2 b2
// W3 b3); biases have none.
struct Bf16Copies {
  size_t w1_end, w2, w2_end, w3, w3_end;
  __nv_bfloat16 *W1, *W2, *W3;
  __device__ __forceinline__ void set(size_t i, float v) const {
    const __nv_bfloat16 b = __float2bfloat16_rn(v);
    if (i < w1_end) W1[i] = b;
    else if (i >= w2 && i < w2_end) W2[i - w2] = b;
    else if (i >= w3 && i < w3_end) W3[i - w3] = b;
  }
};

__global__ void to_bf16_kernel(const float* p, size_t n, Bf16Copies c) {
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x)
    c.set(i, p[i]);
}

// Adam update of the FP32 parameters, their BF16 copies refreshed with it.
__global__ void adam_kernel(float* p, const float* g, float* m, float* v, size_t n, float lr, float b1, float b2,
                            float eps, float c1, float c2, Bf16Copies c) {
  for (size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x; i < n; i += size_t(gridDim.x) * blockDim.x) {
    const float gi = g[i];
    const float mi = b1 * m[i] + (1.f - b1) * gi;
    const float vi = b2 * v[i] + (1.f - b2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    const float pi = p[i] - lr * (mi / c1) / (sqrtf(vi / c2) + eps);
    p[i] = pi;
    c.set(i, pi);
  }
}

// ---------------------------------------------------------------- fused rows
// Everything of a training pass that is local to a row: z1, a1, z2, a2, y and,
// with BACK, dy, dz2, dz1.  A CTA takes MR_ROWS rows and keeps W2 (BF16, at most
// 256 x 256) in shared memory, where the forward pass reads its columns and the
// backward pass its rows; a thread owns a hidden unit for all rows of the CTA.
// The three layers and their gradients were ten launches of 64 x 64-tiled GEMMs
// and elementwise passes, each too small to fill the chip: 1024 rows of the
// 16-256-256-1 model took 466 us a call, now 87, most of it the call's host copies.
constexpr int MR_ROWS = 8, MR_THREADS = 256;

struct MlpRows {
  int B, d_in, h;
  const float *x, *t, *b1, *b2, *b3;
  const __nv_bfloat16 *W1, *W2, *W3;
  float *a1, *a2, *y, *dy, *sq, *dz1, *dz2;
};

__host__ __device__ inline int mr_pitch(int h) { return h + 8; }  // BF16 values a W2 row takes: 16-byte phases spread

__host__ __device__ inline size_t mr_smem(int d_in, int h) {
  return size_t(h) * mr_pitch(h) * 2 + sizeof(float) * MR_ROWS * (size_t(d_in) + 2 * h + MR_THREADS / 32 + 2);
}

__device__ __forceinline__ void fma_rows(float (&acc)[MR_ROWS], const float* v, float w) {
  const float4 p = *reinterpret_cast<const float4*>(v), q = *reinterpret_cast<const float4*>(v + 4);
  acc[0] = fmaf(p.x, w, acc[0]);
  acc[1] = fmaf(p.y, w, acc[1]);
  acc[2] = fmaf(p.z, w, acc[2]);
  acc[3] = fmaf(p.w, w, acc[3]);
  acc[4] = fmaf(q.x, w, acc[4]);
  acc[5] = fmaf(q.y, w, acc[5]);
  acc[6] = fmaf(q.z, w, acc[6]);
  acc[7] = fmaf(q.w, w, acc[7]);
}

template <bool BACK>
__global__ void __launch_bounds__(MR_THREADS) mlp_rows_kernel(const __grid_constant__ MlpRows P) {
  extern __shared__ __align__(16) unsigned char mr_raw[];
  const int h = P.h, d_in = P.d_in, pitch = mr_pitch(h);
  __nv_bfloat16* w2 = reinterpret_cast<__nv_bfloat16*>(mr_raw);     // [h][pitch]
  float* a1s = reinterpret_cast<float*>(w2 + size_t(h) * pitch);    // [h][MR_ROWS]
  float* dz2s = a1s + h * MR_ROWS;                                  // [h][MR_ROWS]
  float* xs = dz2s + h * MR_ROWS;                                   // [d_in][MR_ROWS]
  float* red = xs + d_in * MR_ROWS;                                 // [warps][MR_ROWS]
  float* dys = red + (MR_THREADS / 32) * MR_ROWS;                   // [MR_ROWS]
  const int t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int r0 = blockIdx.x * MR_ROWS, nr = min(MR_ROWS, P.B - r0);
  for (int i = t; i < h * (h / 8); i += MR_THREADS) {
    const int k = i / (h / 8), c8 = i % (h / 8);
    asm volatile("cp.async.cg.shared.global [%0], [%1], 16;" ::"r"(
                     static_cast<uint32_t>(__cvta_generic_to_shared(w2 + size_t(k) * pitch + 8 * c8))),
                 "l"(P.W2 + size_t(k) * h + 8 * c8)
                 : "memory");
  }
  asm volatile("cp.async.commit_group;" ::: "memory");
  for (int i = t; i < MR_ROWS * d_in; i += MR_THREADS) {
    const int r = i / d_in, d = i % d_in;
    xs[d * MR_ROWS + r] = r < nr ? P.x[size_t(r0 + r) * d_in + d] : 0.f;
  }
  __syncthreads();
  const bool on = t < h;
  float acc[MR_ROWS];
  if (on) {
    const float b = P.b1[t];
#pragma unroll
    for (int r = 0; r < MR_ROWS; ++r) acc[r] = 0.f;
#pragma unroll 4
    for (int d = 0; d < d_in; ++d) fma_rows(acc, xs + d * MR_ROWS, __bfloat162float(P.W1[size_t(d) * h + t]));
#pragma unroll
    for (int r = 0; r < MR_ROWS; ++r) {
      const float v = fmaxf(acc[r] + b, 0.f);
      a1s[t * MR_ROWS + r] = v;
      if (BACK && r < nr) P.a1[size_t(r0 + r) * h + t] = v;
    }
  }
  asm volatile("cp.async.wait_group 0;" ::: "memory");
  __syncthreads();
  float a2[MR_ROWS], yp[MR_ROWS];
  const float w3 = on ? __bfloat162float(P.W3[t]) : 0.f;
#pragma unroll
  for (int r = 0; r < MR_ROWS; ++r) acc[r] = a2[r] = yp[r] = 0.f;
  if (on) {
    const float b = P.b2[t];
#pragma unroll 8
    for (int k = 0; k < h; ++k) fma_rows(acc, a1s + k * MR_ROWS, __bfloat162float(w2[size_t(k) * pitch + t]));
#pragma unroll
    for (int r = 0; r < MR_ROWS; ++r) {
      a2[r] = fmaxf(acc[r] + b, 0.f);
      yp[r] = a2[r] * w3;
      if (BACK && r < nr) P.a2[size_t(r0 + r) * h + t] = a2[r];
    }
  }
#pragma unroll
  for (int r = 0; r < MR_ROWS; ++r) {
    for (int d = 16; d; d >>= 1) yp[r] += __shfl_xor_sync(0xffffffffu, yp[r], d);
    if (lane == 0) red[warp * MR_ROWS + r] = yp[r];
  }
  __syncthreads();
  if (t < MR_ROWS) {
    float y = 0.f;
    for (int w = 0; w < MR_THREADS / 32; ++w) y += red[w * MR_ROWS + t];
    y += P.b3[0];
    float dy = 0.f;
    if (t < nr) {
      P.y[r0 + t] = y;
      if (BACK) {
        const float e = y - P.t[r0 + t];
        dy = 2.f * e / float(P.B);
        P.dy[r0 + t] = dy;
        P.sq[r0 + t] = e * e;
      }
    }
    dys[t] = dy;
  }
  if (!BACK) return;
  __syncthreads();
  if (on) {
#pragma unroll
    for (int r = 0; r < MR_ROWS; ++r) {
      const float g = a2[r] > 0.f ? dys[r] * w3 : 0.f;
      dz2s[t * MR_ROWS + r] = g;
      if (r < nr) P.dz2[size_t(r0 + r) * h + t] = g;
    }
  }
  __syncthreads();
  if (on) {
#pragma unroll
    for (int r = 0; r < MR_ROWS; ++r) acc[r] = 0.f;
    for (int c = 0; c < h; c += 8) {
      const uint4 w = *reinterpret_cast<const uint4*>(w2 + size_t(t) * pitch + c);
      const uint32_t u[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        fma_rows(acc, dz2s + (c + 2 * j) * MR_ROWS, __uint_as_float(u[j] << 16));
        fma_rows(acc, dz2s + (c + 2 * j + 1) * MR_ROWS, __uint_as_float(u[j] & 0xffff0000u));
      }
    }
#pragma unroll
    for (int r = 0; r < MR_ROWS; ++r)
      if (r < nr) P.dz1[size_t(r0 + r) * h + t] = a1s[t * MR_ROWS + r] > 0.f ? acc[r] : 0.f;
  }
}

// Parameter gradients as partial sums over `rows` rows each (blockIdx.y):
// 64 x 64 tiles of W2 = a1^T dz2 and W1 = x^T dz1 (both operands are stored with
// the summed row index slowest, so a stage of 16 rows is two coalesced copies),
// then the column sums of W3, b2, b1 and the sums of b3 and the loss.  One CTA
// per tile over all rows would fill 20 of 152 SMs; the partials are added in
// order by mlp_reduce_kernel.
constexpr int MW_T = 64, MW_K = 16;

struct MlpGrads {
  int B, d_in, h, rows;
  const float *x, *a1, *a2, *dy, *sq, *dz1, *dz2;
  float* part;  // [splits][n_params + 1]; the last entry is the sum of squared errors
  size_t stride, w1, b1, w2, b2, w3, b3;
};

__global__ void __launch_bounds__(256) mlp_grads_kernel(const __grid_constant__ MlpGrads P) {
  __shared__ float As[MW_K][MW_T], Bs[MW_K][MW_T];
  const int tid = threadIdx.x, h = P.h;
  const int r0 = blockIdx.y * P.rows, r1 = min(P.B, r0 + P.rows);
  float* part = P.part + blockIdx.y * P.stride;
  const int tn = (h + MW_T - 1) / MW_T, t2 = tn * tn, t1 = ((P.d_in + MW_T - 1) / MW_T) * tn;
  int role = blockIdx.x;
  if (role >= t2 + t1) {
    role -= t2 + t1;
    if (role == 0) {  // b3 and the loss
      if (tid < 64) {
        const float* v = tid < 32 ? P.dy : P.sq;
        float s = 0.f;
        for (int r = r0 + (tid & 31); r < r1; r += 32) s += v[r];
        for (int d = 16; d; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
        if ((tid & 31) == 0) part[tid < 32 ? P.b3 : P.stride - 1] = s;
      }
      return;
    }
    const int c = (role - 1) * 64 + (tid & 63), g = tid >> 6;  // four row groups per column
    float s3 = 0.f, s2 = 0.f, s1 = 0.f;
    if (c < h) {
#pragma unroll 4
      for (int r = r0 + g; r < r1; r += 4) {
        s3 = fmaf(P.a2[size_t(r) * h + c], P.dy[r], s3);
        s2 += P.dz2[size_t(r) * h + c];
        s1 += P.dz1[size_t(r) * h + c];
      }
    }
    float* sh = &As[0][0];  // [3][4][64]
    sh[(0 + g) * 64 + (tid & 63)] = s3;
    sh[(4 + g) * 64 + (tid & 63)] = s2;
    sh[(8 + g) * 64 + (tid & 63)] = s1;
    __syncthreads();
    if (tid < 192) {
      const int q = tid >> 6, col = (role - 1) * 64 + (tid & 63);
      if (col < h) {
        float s = 0.f;
        for (int j = 0; j < 4; ++j) s += sh[(4 * q + j) * 64 + (tid & 63)];
        part[(q == 0 ? P.w3 : q == 1 ? P.b2 : P.b1) + col] = s;
      }
    }
    return;
  }
  const bool second = role < t2;
  if (!second) role -= t2;
  const float* A = second ? P.a1 : P.x;
  const float* Bm = second ? P.dz2 : P.dz1;
  const int M = second ? h : P.d_in;
  const int m0 = (role / tn) * MW_T, n0 = (role % tn) * MW_T;
  const int tx = tid & 15, ty = tid >> 4, lr = tid >> 6, lc = tid & 63;
  float acc[4][4];
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) acc[i][j] = 0.f;
  float pa[4], pb[4];
  auto fetch = [&](int k0) {
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      const int r = k0 + lr + 4 * l;
      pa[l] = r < r1 && m0 + lc < M ? A[size_t(r) * M + m0 + lc] : 0.f;
      pb[l] = r < r1 && n0 + lc < h ? Bm[size_t(r) * h + n0 + lc] : 0.f;
    }
  };
  fetch(r0);
  for (int k0 = r0; k0 < r1; k0 += MW_K) {
#pragma unroll
    for (int l = 0; l < 4; ++l) {
      As[lr + 4 * l][lc] = pa[l];
      Bs[lr + 4 * l][lc] = pb[l];
    }
    __syncthreads();
    if (k0 + MW_K < r1) fetch(k0 + MW_K);
#pragma unroll
    for (int kk = 0; kk < MW_K; ++kk) {
      float a[4], b[4];
#pragma unroll
      for (int i = 0; i < 4; ++i) a[i] = As[kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < 4; ++j) b[j] = Bs[kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < 4; ++i)
#pragma unroll
        for (int j = 0; j < 4; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    __syncthreads();
  }
  const size_t off = second ? P.w2 : P.w1;
#pragma unroll
  for (int i = 0; i < 4; ++i)
#pragma unroll
    for (int j = 0; j < 4; ++j) {
      const int m = m0 + ty + 16 * i, n = n0 + tx + 16 * j;
      if (m < M && n < h) part[off + size_t(m) * h + n] = acc[i][j];
    }
}

// grads = partials added in split order; the last entry becomes the mean loss.
__global__ void mlp_reduce_kernel(const float* __restrict__ part, int splits, size_t stride, float* grads, float* loss,
                                  float inv_b) {
  const size_t i = blockIdx.x * size_t(blockDim.x) + threadIdx.x;
  if (i >= stride) return;
  float s = 0.f;
#pragma unroll 8
  for (int k = 0; k < splits; ++k) s += part[size_t(k) * stride + i];
  if (i + 1 < stride) grads[i] = s;
  else *loss = s * inv_b;
}

unsigned nblk(size_t n) { return unsigned(std::max<size_t>(1, std::min<size_t>((n + 255) / 256, 2048))); }

}  // namespace

// ---------------------------------------------------------------- model
// partial gradients of a pass: at least 64 rows each, at most this many
constexpr int kGradSplits = 16;

size_t CostModel::n_params() const { return size_t(d_in) * h + h + size_t(h) * h + h + h + 1; }

void CostModel::layout() {
  const size_t P = n_params();
  size_t off = 0;
  auto take = [&](size_t bytes) {
    size_t o = off;
    off = (off + bytes + 255) / 256 * 256;
    return o;
  };
  o_params = take(4 * P);
  o_grads = take(4 * P);
  o_m = take(4 * P);
  o_v = take(4 * P);
  o_w1b = take(2 * size_t(d_in) * h);
  o_w2b = take(2 * size_t(h) * h);
  o_w3b = take(2 * size_t(h));
  const size_t B = size_t(max_batch);
  o_x = take(4 * B * d_in);
  o_t = take(4 * B);
  o_z1 = take(4 * B * h);
  o_a1 = take(4 * B * h);
  o_z2 = take(4 * B * h);
  o_a2 = take(4 * B * h);
  o_y = take(4 * B);
  o_dy = take(4 * B);
  o_sq = take(4 * B);
  o_dz1 = take(4 * B * h);
  o_dz2 = take(4 * B * h);
  o_loss = take(8);
  o_part = take(fused() ? 4 * (P + 1) * kGradSplits : 0);
  ws_bytes = off + kWorkspaceAlign;
}

// Parameter offsets (floats) inside the flat vector: W1, b1, W2, b2, W3, b3.
static void param_offsets(const CostModel& m, size_t* w1, size_t* b1, size_t* w2, size_t* b2, size_t* w3, size_t* b3) {
  *w1 = 0;
  *b1 = *w1 + size_t(m.d_in) * m.h;
  *w2 = *b1 + m.h;
  *b2 = *w2 + size_t(m.h) * m.h;
  *w3 = *b2 + m.h;
  *b3 = *w3 + m.h;
}

#define MLP_CUDA(call)                                  \
  do {                                                  \
    cudaError_t _e = (call);                            \
    if (_e != cudaSuccess) return cuda_fail(_e, #call); \
  } while (0)

static Bf16Copies bf16_copies(const CostModel& m) {
  char* ws = static_cast<char*>(m.ws);
  size_t w1, b1, w2, b2, w3, b3;
  param_offsets(m, &w1, &b1, &w2, &b2, &w3, &b3);
  Bf16Copies c;
  c.w1_end = b1;
  c.w2 = w2;
  c.w2_end = b2;
  c.w3 = w3;
  c.w3_end = b3;
  c.W1 = reinterpret_cast<__nv_bfloat16*>(ws + m.o_w1b);
  c.W2 = reinterpret_cast<__nv_bfloat16*>(ws + m.o_w2b);
  c.W3 = reinterpret_cast<__nv_bfloat16*>(ws + m.o_w3b);
  return c;
}

static tnq_status refresh_bf16(Ctx* ctx, CostModel* m) {
  const size_t P = m->n_params();
  to_bf16_kernel<<<nblk(P), 256, 0, ctx->stream>>>(
      reinterpret_cast<const float*>(static_cast<char*>(m->ws) + m->o_params), P, bf16_copies(*m));
  MLP_CUDA(cudaGetLastError());
  ctx->launches++;
  return TNQ_OK;
}

// The fused row kernel on B rows already in the x (and, with `back`, t) region:
// leaves y, or what the parameter gradients need as well.
static tnq_status rows_pass(Ctx* ctx, CostModel* m, int B, bool back) {
  char* ws = static_cast<char*>(m->ws);
  size_t w1, b1, w2, b2, w3, b3;
  param_offsets(*m, &w1, &b1, &w2, &b2, &w3, &b3);
  auto f = [&](size_t o) { return reinterpret_cast<float*>(ws + o); };
  const float* P = f(m->o_params);
  const Bf16Copies c = bf16_copies(*m);
  MlpRows a;
  a.B = B;
  a.d_in = m->d_in;
  a.h = m->h;
  a.x = f(m->o_x);
  a.t = f(m->o_t);
  a.b1 = P + b1;
  a.b2 = P + b2;
  a.b3 = P + b3;
  a.W1 = c.W1;
  a.W2 = c.W2;
  a.W3 = c.W3;
  a.a1 = f(m->o_a1);
  a.a2 = f(m->o_a2);
  a.y = f(m->o_y);
  a.dy = f(m->o_dy);
  a.sq = f(m->o_sq);
  a.dz1 = f(m->o_dz1);
  a.dz2 = f(m->o_dz2);
  const size_t smem = mr_smem(m->d_in, m->h);
  const unsigned grid = unsigned((B + MR_ROWS - 1) / MR_ROWS);
  auto k = back ? mlp_rows_kernel<true> : mlp_rows_kernel<false>;
  static std::atomic<uint64_t> done[2];
  MLP_CUDA(allow_smem(reinterpret_cast<const void*>(k), int(mr_smem(m->d_in, 256)), &done[back]));
  k<<<grid, MR_THREADS, smem, ctx->stream>>>(a);
  MLP_CUDA(cudaGetLastError());
  ctx->launches++;
  return TNQ_OK;
}

static tnq_status grads_pass(Ctx* ctx, CostModel* m, int B) {
  char* ws = static_cast<char*>(m->ws);
  auto f = [&](size_t o) { return reinterpret_cast<float*>(ws + o); };
  MlpGrads a;
  param_offsets(*m, &a.w1, &a.b1, &a.w2, &a.b2, &a.w3, &a.b3);
  a.B = B;
  a.d_in = m->d_in;
  a.h = m->h;
  a.rows = std::max(64, (B + kGradSplits - 1) / kGradSplits);
  a.x = f(m->o_x);
  a.a1 = f(m->o_a1);
  a.a2 = f(m->o_a2);
  a.dy = f(m->o_dy);
  a.sq = f(m->o_sq);
  a.dz1 = f(m->o_dz1);
  a.dz2 = f(m->o_dz2);
  a.part = f(m->o_part);
  a.stride = m->n_params() + 1;
  const int tn = (m->h + MW_T - 1) / MW_T, splits = (B + a.rows - 1) / a.rows;
  const dim3 grid{unsigned(tn * tn + ((m->d_in + MW_T - 1) / MW_T) * tn + 1 + tn), unsigned(splits), 1u};
  mlp_grads_kernel<<<grid, 256, 0, ctx->stream>>>(a);
  mlp_reduce_kernel<<<unsigned((a.stride + 255) / 256), 256, 0, ctx->stream>>>(a.part, splits, a.stride, f(m->o_grads),
                                                                             f(m->o_loss), 1.f / float(B));
  MLP_CUDA(cudaGetLastError());
  ctx->launches += 2;
  return TNQ_OK;
}

// Forward on B rows already in the x region; leaves y (and z/a for backward).
// Wider models than the fused kernel holds run layer by layer.
static tnq_status forward(Ctx* ctx, CostModel* m, int B, bool back) {
  if (m->fused()) return rows_pass(ctx, m, B, back);
  char* ws = static_cast<char*>(m->ws);
  size_t w1, b1, w2, b2, w3, b3;
  param_offsets(*m, &w1, &b1, &w2, &b2, &w3, &b3);
  const float* P = reinterpret_cast<const float*>(ws + m->o_params);
  auto f = [&](size_t o) { return reinterpret_cast<float*>(ws + o); };
  const __nv_bfloat16* W1 = reinterpret_cast<const __nv_bfloat16*>(ws + m->o_w1b);
  const __nv_bfloat16* W2 = reinterpret_cast<const __nv_bfloat16*>(ws + m->o_w2b);
  const __nv_bfloat16* W3 = reinterpret_cast<const __nv_bfloat16*>(ws + m->o_w3b);
  const int h = m->h;
  MLP_CUDA(gemm(ctx->stream, B, h, m->d_in, f(m->o_x), m->d_in, 0, W1, h, 0, f(m->o_z1), h, P + b1, f(m->o_a1)));
  MLP_CUDA(gemm(ctx->stream, B, h, h, f(m->o_a1), h, 0, W2, h, 0, f(m->o_z2), h, P + b2, f(m->o_a2)));
  MLP_CUDA(gemm(ctx->stream, B, 1, h, f(m->o_a2), h, 0, W3, 1, 0, f(m->o_y), 1, P + b3));
  ctx->launches += 3;
  return TNQ_OK;
}

// Backward for B rows with targets in the t region; writes the gradient vector.
static tnq_status backward(Ctx* ctx, CostModel* m, int B) {
  if (m->fused()) return grads_pass(ctx, m, B);
  char* ws = static_cast<char*>(m->ws);
  size_t w1, b1, w2, b2, w3, b3;
  param_offsets(*m, &w1, &b1, &w2, &b2, &w3, &b3);
  auto f = [&](size_t o) { return reinterpret_cast<float*>(ws + o); };
  float* G = f(m->o_grads);
  const __nv_bfloat16* W2 = reinterpret_cast<const __nv_bfloat16*>(ws + m->o_w2b);
  const __nv_bfloat16* W3 = reinterpret_cast<const __nv_bfloat16*>(ws + m->o_w3b);
  const int h = m->h;
  dy_kernel<<<nblk(B), 256, 0, ctx->stream>>>(f(m->o_y), f(m->o_t), B, f(m->o_dy), f(m->o_sq));
  // W3 grad = a2^T dy ; b3 grad = sum dy
  MLP_CUDA(gemm(ctx->stream, h, 1, B, f(m->o_a2), h, 1, f(m->o_dy), 1, 0, G + w3, 1));
  colsum_kernel<<<1, 32, 0, ctx->stream>>>(f(m->o_dy), B, 1, 1, G + b3, 1.f);
  // dz2 = (dy W3^T) * (z2 > 0)
  MLP_CUDA(gemm(ctx->stream, B, h, 1, f(m->o_dy), 1, 0, W3, 1, 1, f(m->o_dz2), h));
  relu_mask_kernel<<<nblk(size_t(B) * h), 256, 0, ctx->stream>>>(f(m->o_dz2), f(m->o_z2), size_t(B) * h);
  MLP_CUDA(gemm(ctx->stream, h, h, B, f(m->o_a1), h, 1, f(m->o_dz2), h, 0, G + w2, h));
  colsum_kernel<<<nblk(h), 256, 0, ctx->stream>>>(f(m->o_dz2), B, h, h, G + b2, 1.f);
  // dz1 = (dz2 W2^T) * (z1 > 0)
  MLP_CUDA(gemm(ctx->stream, B, h, h, f(m->o_dz2), h, 0, W2, h, 1, f(m->o_dz1), h));
  relu_mask_kernel<<<nblk(size_t(B) * h), 256, 0, ctx->stream>>>(f(m->o_dz1), f(m->o_z1), size_t(B) * h);
  MLP_CUDA(gemm(ctx->stream, m->d_in, h, B, f(m->o_x), m->d_in, 1, f(m->o_dz1), h, 0, G + w1, h));
  colsum_kernel<<<nblk(h), 256, 0, ctx->stream>>>(f(m->o_dz1), B, h, h, G + b1, 1.f);
  // loss = mean squared error (sum of squares in row order)
  colsum_kernel<<<1, 32, 0, ctx->stream>>>(f(m->o_sq), B, 1, 1, f(m->o_loss), 1.f / float(B));
  MLP_CUDA(cudaGetLastError());
  ctx->launches += 13;
  return TNQ_OK;
}

static tnq_status adam(Ctx* ctx, CostModel* m, float lr) {
  char* ws = static_cast<char*>(m->ws);
  m->adam_t += 1;
  const float c1 = float(1.0 - std::pow(0.9, m->adam_t)), c2 = float(1.0 - std::pow(0.999, m->adam_t));
  const size_t P = m->n_params();
  adam_kernel<<<nblk(P), 256, 0, ctx->stream>>>(reinterpret_cast<float*>(ws + m->o_params),
                                                reinterpret_cast<const float*>(ws + m->o_grads),
                                                reinterpret_cast<float*>(ws + m->o_m), reinterpret_cast<float*>(ws + m->o_v),
                                                P, lr, 0.9f, 0.999f, 1e-8f, c1, c2, bf16_copies(*m));
  MLP_CUDA(cudaGetLastError());
  ctx->launches++;
  return TNQ_OK;
}

tnq_status mlp_bind(Ctx* ctx, CostModel* m, void* ws, size_t bytes) {
  if (!ws || bytes < m->ws_bytes)
    return fail(TNQ_ERR_WORKSPACE, "cost-model workspace needs " + std::to_string(m->ws_bytes) + " bytes");
  MLP_CUDA(cudaSetDevice(ctx->device));
  m->ws = workspace_base(ws);
  return mlp_upload(ctx, m, m->host_params.data());
}

tnq_status mlp_upload(Ctx* ctx, CostModel* m, const float* params) {
  if (!m->ws) return fail(TNQ_ERR_WORKSPACE, "cost model has no bound workspace");
  char* ws = static_cast<char*>(m->ws);
  const size_t P = m->n_params();
  m->host_params.assign(params, params + P);
  MLP_CUDA(cudaMemcpyAsync(ws + m->o_params, params, 4 * P, cudaMemcpyHostToDevice, ctx->stream));
  MLP_CUDA(cudaMemsetAsync(ws + m->o_m, 0, 4 * P, ctx->stream));
  MLP_CUDA(cudaMemsetAsync(ws + m->o_v, 0, 4 * P, ctx->stream));
  m->adam_t = 0;
  tnq_status s = refresh_bf16(ctx, m);
  if (s != TNQ_OK) return s;
  MLP_CUDA(cudaStreamSynchronize(ctx->stream));
  return TNQ_OK;
}

tnq_status mlp_download(Ctx* ctx, CostModel* m, float* params) {
  if (!m->ws) return fail(TNQ_ERR_WORKSPACE, "cost model has no bound workspace");
  MLP_CUDA(cudaMemcpyAsync(params, static_cast<char*>(m->ws) + m->o_params, 4 * m->n_params(), cudaMemcpyDeviceToHost,
                           ctx->stream));
  MLP_CUDA(cudaStreamSynchronize(ctx->stream));
  return TNQ_OK;
}

tnq_status mlp_gradients(Ctx* ctx, CostModel* m, const float* X, const float* t, int64_t n, float* grads,
                         float* loss) {
  if (!m->ws) return fail(TNQ_ERR_WORKSPACE, "cost model has no bound workspace");
  if (n < 1 || n > m->max_batch) return fail(TNQ_ERR_INVALID_ARG, "row count must be in [1, max_batch]");
  char* ws = static_cast<char*>(m->ws);
  MLP_CUDA(cudaMemcpyAsync(ws + m->o_x, X, 4 * size_t(n) * m->d_in, cudaMemcpyHostToDevice, ctx->stream));
  MLP_CUDA(cudaMemcpyAsync(ws + m->o_t, t, 4 * size_t(n), cudaMemcpyHostToDevice, ctx->stream));
  tnq_status s = forward(ctx, m, int(n), true);
  if (s == TNQ_OK) s = backward(ctx, m, int(n));
  if (s != TNQ_OK) return s;
  if (grads)
    MLP_CUDA(cudaMemcpyAsync(grads, ws + m->o_grads, 4 * m->n_params(), cudaMemcpyDeviceToHost, ctx->stream));
  if (loss) MLP_CUDA(cudaMemcpyAsync(loss, ws + m->o_loss, 4, cudaMemcpyDeviceToHost, ctx->stream));
  MLP_CUDA(cudaStreamSynchronize(ctx->stream));
  return TNQ_OK;
}

tnq_status mlp_train(Ctx* ctx, CostModel* m, const float* X, const float* t, int64_t n, int epochs, int batch,
                     float lr, float* final_loss) {
  if (!m->ws) return fail(TNQ_ERR_WORKSPACE, "cost model has no bound workspace");
  if (n < 1 || epochs < 1 || batch < 1 || batch > m->max_batch)
    return fail(TNQ_ERR_INVALID_ARG, "bad training arguments (n >= 1, epochs >= 1, 1 <= batch <= max_batch)");
  char* ws = static_cast<char*>(m->ws);
  // minibatches in a seeded order per epoch; rows staged from the host per batch
  std::vector<int64_t> order(n);
  for (int64_t i = 0; i < n; ++i) order[i] = i;
  std::mt19937_64 g(m->seed ^ 0xC0FFEEULL);
  std::vector<float> xb(size_t(batch) * m->d_in), tb(batch);
  float last = 0.f;
  for (int e = 0; e < epochs; ++e) {
    std::shuffle(order.begin(), order.end(), g);
    for (int64_t s0 = 0; s0 < n; s0 += batch) {
      const int B = int(std::min<int64_t>(batch, n - s0));
      for (int r = 0; r < B; ++r) {
        const int64_t src = order[s0 + r];
        std::copy(X + src * m->d_in, X + (src + 1) * m->d_in, xb.begin() + size_t(r) * m->d_in);
        tb[r] = t[src];
      }
      MLP_CUDA(cudaMemcpyAsync(ws + m->o_x, xb.data(), 4 * size_t(B) * m->d_in, cudaMemcpyHostToDevice, ctx->stream));
      MLP_CUDA(cudaMemcpyAsync(ws + m->o_t, tb.data(), 4 * size_t(B), cudaMemcpyHostToDevice, ctx->stream));
      tnq_status s = forward(ctx, m, B, true);
      if (s == TNQ_OK) s = backward(ctx, m, B);
      if (s == TNQ_OK) s = adam(ctx, m, lr);
      if (s != TNQ_OK) return s;
      // the staging vectors are reused: wait for this batch's copies
      MLP_CUDA(cudaStreamSynchronize(ctx->stream));
    }
  }
  MLP_CUDA(cudaMemcpyAsync(&last, ws + m->o_loss, 4, cudaMemcpyDeviceToHost, ctx->stream));
  MLP_CUDA(cudaStreamSynchronize(ctx->stream));
  if (final_loss) *final_loss = last;
  return mlp_download(ctx, m, m->host_params.data());
}

tnq_status mlp_predict(Ctx* ctx, CostModel* m, const float* X, int64_t n, float* y) {
  if (!m->ws) return fail(TNQ_ERR_WORKSPACE, "cost model has no bound workspace");
  char* ws = static_cast<char*>(m->ws);
  const bool x_dev = false;
  (void)x_dev;
  for (int64_t s0 = 0; s0 < n; s0 += m->max_batch) {
    const int B = int(std::min<int64_t>(m->max_batch, n - s0));
    MLP_CUDA(cudaMemcpyAsync(ws + m->o_x, X + s0 * m->d_in, 4 * size_t(B) * m->d_in, cudaMemcpyHostToDevice,
                             ctx->stream));
    tnq_status s = forward(ctx, m, B, false);
    if (s != TNQ_OK) return s;
    MLP_CUDA(cudaMemcpyAsync(y + s0, ws + m->o_y, 4 * size_t(B), cudaMemcpyDeviceToHost, ctx->stream));
    MLP_CUDA(cudaStreamSynchronize(ctx->stream));
  }
  return TNQ_OK;
}

void mlp_init(CostModel* m) {
  // He-uniform initial weights from a seeded generator, zero biases
  const size_t P = m->n_params();
  m->host_params.assign(P, 0.f);
  size_t w1, b1, w2, b2, w3, b3;
  param_offsets(*m, &w1, &b1, &w2, &b2, &w3, &b3);
  std::mt19937_64 g(m->seed);
  auto fill = [&](size_t off, size_t count, int fan_in) {
    const double b = std::sqrt(6.0 / fan_in);
    for (size_t i = 0; i < count; ++i) m->host_params[off + i] = float((2.0 * ((g() >> 11) * (1.0 / 9007199254740992.0)) - 1.0) * b);
  };
  fill(w1, size_t(m->d_in) * m->h, m->d_in);
  fill(w2, size_t(m->h) * m->h, m->h);
  fill(w3, size_t(m->h), m->h);
}

}  // namespace tnq
