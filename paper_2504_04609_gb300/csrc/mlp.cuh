// Learned warm start: a 4-layer MLP mapping a target spectrum to initial potentials and weights.
//
//   features  x0 = [ n y / sum(y),  log sum(y) ]                        (n + 1)
//   hidden    h_l = GELU(h_{l-1} W_l^T + b_l),  l = 1..3, width H        (erf form of GELU)
//   output    z = h_3 W_4^T + b_4                                        (n + k)
//   targets   t = [ g / eps (n),  log w (k) ] of solved problems, normalised per output,
//             (t - mean) / std; bins whose target is not finite (g = -inf where y = 0 under the
//             KL datafit) are masked out of the loss.
//   loss      mean over unmasked entries of (z - t_norm)^2
// Weights are stored in BF16 for the forward pass (FP32 accumulation) with FP32 master copies
// updated by AdamW.  Inference runs on the tcgen05 GEMM (tc_gemm.cuh) with BF16 hi/lo activations;
// training contractions keep FP32 products and rounding (below).
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"

namespace otlm {
namespace mlp {

constexpr int LAYERS = 4;

__device__ __forceinline__ float gelu(float z) { return 0.5f * z * (1.f + erff(z * 0.70710678118654752f)); }
__device__ __forceinline__ float gelu_grad(float z) {
  return 0.5f * (1.f + erff(z * 0.70710678118654752f)) + z * 0.39894228040143268f * expf(-0.5f * z * z);
}

// ---- training ------------------------------------------------------------------------------------
// FP32 contractions C[m][n] = sum_k A(m,k) B(k,n) on the FP32 pipe: tiles of 128 x 64, 128 threads of
// 8 x 8 outputs (64 multiply-adds per four 16-byte shared loads), k blocks of 16 prefetched into
// registers while the previous block is used, and the reduction split over blockIdx.z so that two CTAs
// fit each SM (the layers' 512 x 512 outputs are 32 tiles).  The kernels that consume C add the
// partial-sum planes in order.  Operands are contiguous along k (AK, BK: rows of the batch, weights)
// or along m / n (the weight gradient reads dZ^T H without a transpose); row pitches are multiples of
// four floats (eight BF16) and padded with zeros.
//   n = 2048, width 512, batch 512, one step: 1615 us on 64 x 64 tiles of 4 x 4 outputs with neither
//   split nor prefetch. TF32 hi/lo operands on the tensor cores took 293 us, but their accumulator
//   truncates: the loss came out 1.3e-6 from the 64-bit value (FP32: 1.7e-7), so they were left out.
constexpr int GM = 128, GN = 64, GK = 16, GT = 128;

__device__ __forceinline__ void unpack8(const uint4& q, float (&v)[8]) {
  const uint32_t w[4] = {q.x, q.y, q.z, q.w};
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    v[2 * i] = __uint_as_float(w[i] << 16);
    v[2 * i + 1] = __uint_as_float(w[i] & 0xffff0000u);
  }
}

// TB: float or BF16 weights.  lda, ldb: row pitches (rows of m for AK, else of k; rows of n for BK,
// else of k).  C planes [z][M][ldc].
template <bool AK, bool BK, typename TB>
__global__ void __launch_bounds__(GT, 2) train_gemm_kernel(int M, int N, int K, const float* A, int lda, const TB* B,
                                                           int ldb, float* C, int ldc, size_t plane, int kper) {
  constexpr bool BH = sizeof(TB) == 2;
  __shared__ __align__(16) float As[2][GK][GM + 4];
  __shared__ __align__(16) float Bs[2][GK][GN + 4];
  const int t = threadIdx.x, tx = t % 8, ty = t / 8;
  const int m0 = blockIdx.y * GM, n0 = blockIdx.x * GN;
  const int k_beg = blockIdx.z * kper, k_end = min(K, k_beg + kper);
  float4 ra[4];
  float4 rb[2];
  uint4 rh;
  const float4 z4 = make_float4(0.f, 0.f, 0.f, 0.f);
  auto load = [&](int k0) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if constexpr (AK) {  // row m, four k
        const int m = m0 + t / 4 + 32 * q, k = k0 + (t % 4) * 4;
        ra[q] = (m < M && k < k_end) ? *reinterpret_cast<const float4*>(A + (size_t)m * lda + k) : z4;
      } else {  // row k, four m
        const int k = k0 + t / 32 + 4 * q, m = m0 + (t % 32) * 4;
        ra[q] = (k < k_end && m < M) ? *reinterpret_cast<const float4*>(A + (size_t)k * lda + m) : z4;
      }
    }
    if constexpr (BH) {
      if constexpr (BK) {  // row n, eight k
        const int n = n0 + t / 2, k = k0 + (t % 2) * 8;
        rh = (n < N && k < k_end) ? *reinterpret_cast<const uint4*>(B + (size_t)n * ldb + k) : make_uint4(0, 0, 0, 0);
      } else {  // row k, eight n
        const int k = k0 + t / 8, n = n0 + (t % 8) * 8;
        rh = (k < k_end && n < N) ? *reinterpret_cast<const uint4*>(B + (size_t)k * ldb + n) : make_uint4(0, 0, 0, 0);
      }
    } else {
#pragma unroll
      for (int q = 0; q < 2; ++q) {  // row k, four n
        const int k = k0 + t / 16 + 8 * q, n = n0 + (t % 16) * 4;
        rb[q] = (k < k_end && n < N) ? *reinterpret_cast<const float4*>(B + (size_t)k * ldb + n) : z4;
      }
    }
  };
  auto store = [&](int s) {
#pragma unroll
    for (int q = 0; q < 4; ++q) {
      if constexpr (AK) {
        const int m = t / 4 + 32 * q, k = (t % 4) * 4;
        As[s][k][m] = ra[q].x; As[s][k + 1][m] = ra[q].y; As[s][k + 2][m] = ra[q].z; As[s][k + 3][m] = ra[q].w;
      } else {
        *reinterpret_cast<float4*>(&As[s][t / 32 + 4 * q][(t % 32) * 4]) = ra[q];
      }
    }
    if constexpr (BH) {
      float v[8];
      unpack8(rh, v);
      if constexpr (BK) {
#pragma unroll
        for (int i = 0; i < 8; ++i) Bs[s][(t % 2) * 8 + i][t / 2] = v[i];
      } else {
        *reinterpret_cast<float4*>(&Bs[s][t / 8][(t % 8) * 8]) = make_float4(v[0], v[1], v[2], v[3]);
        *reinterpret_cast<float4*>(&Bs[s][t / 8][(t % 8) * 8 + 4]) = make_float4(v[4], v[5], v[6], v[7]);
      }
    } else {
#pragma unroll
      for (int q = 0; q < 2; ++q) *reinterpret_cast<float4*>(&Bs[s][t / 16 + 8 * q][(t % 16) * 4]) = rb[q];
    }
  };
  float acc[8][8] = {};
  load(k_beg);
  store(0);
  __syncthreads();
  int s = 0;
  for (int k0 = k_beg; k0 < k_end; k0 += GK, s ^= 1) {
    const bool more = k0 + GK < k_end;
    if (more) load(k0 + GK);
#pragma unroll
    for (int kk = 0; kk < GK; ++kk) {
      const float4 a0 = *reinterpret_cast<const float4*>(&As[s][kk][ty * 4]);
      const float4 a1 = *reinterpret_cast<const float4*>(&As[s][kk][64 + ty * 4]);
      const float4 b0 = *reinterpret_cast<const float4*>(&Bs[s][kk][tx * 4]);
      const float4 b1 = *reinterpret_cast<const float4*>(&Bs[s][kk][32 + tx * 4]);
      const float a[8] = {a0.x, a0.y, a0.z, a0.w, a1.x, a1.y, a1.z, a1.w};
      const float b[8] = {b0.x, b0.y, b0.z, b0.w, b1.x, b1.y, b1.z, b1.w};
#pragma unroll
      for (int i = 0; i < 8; ++i)
#pragma unroll
        for (int j = 0; j < 8; ++j) acc[i][j] = fmaf(a[i], b[j], acc[i][j]);
    }
    if (more) {
      store(s ^ 1);
      __syncthreads();
    }
  }
  float* out = C + blockIdx.z * plane;
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const int m = m0 + (i / 4) * 64 + ty * 4 + i % 4;
    if (m >= M) continue;
#pragma unroll
    for (int h = 0; h < 2; ++h) {
      const int n = n0 + h * 32 + tx * 4;
      if (n < ldc)  // the pitch's padding columns get sums of zero columns
        *reinterpret_cast<float4*>(out + (size_t)m * ldc + n) =
            make_float4(acc[i][4 * h], acc[i][4 * h + 1], acc[i][4 * h + 2], acc[i][4 * h + 3]);
    }
  }
}

__device__ __forceinline__ float plane_sum(const float* Z, int splits, size_t plane, size_t e) {
  float v = 0.f;
  for (int z = 0; z < splits; ++z) v += Z[z * plane + e];
  return v;
}
__device__ __forceinline__ float4 plane_sum4(const float* Z, int splits, size_t plane, size_t e) {
  float4 v = *reinterpret_cast<const float4*>(Z + e);
  for (int z = 1; z < splits; ++z) {
    const float4 u = *reinterpret_cast<const float4*>(Z + z * plane + e);
    v.x += u.x; v.y += u.y; v.z += u.z; v.w += u.w;
  }
  return v;
}

// features: x0[b] = [ n y_b / sum(y_b), log sum(y_b) ]  (one CTA per row, pitch ld)
__global__ void __launch_bounds__(256) features_kernel(const float* y, int n, float* x0, int ld) {
  __shared__ float red[32];
  const int b = blockIdx.x;
  float s = 0.f;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += y[(size_t)b * n + i];
  s = block_sum(s, red);
  const float inv = s > 0.f ? (float)n / s : 0.f;
  for (int i = threadIdx.x; i < n; i += blockDim.x) x0[(size_t)b * ld + i] = y[(size_t)b * n + i] * inv;
  if (threadIdx.x == 0) x0[(size_t)b * ld + n] = s > 0.f ? logf(s) : 0.f;
}

// Elementwise kernels over [rows][dout] in groups of four columns (pitch ld, a multiple of four;
// padding columns stay 0): grid.x = rows, grid.y covers ld / 4.
// hidden layer: pre = Z + bias (kept for the backward pass), h = GELU(pre)
__global__ void __launch_bounds__(128) act_train_kernel(const float* Z, int splits, size_t plane, int dout, int ld,
                                                        const float* bias, float* pre, float* h) {
  const int c = (blockIdx.y * 128 + threadIdx.x) * 4;
  if (c >= ld) return;
  const size_t e = (size_t)blockIdx.x * ld + c;
  const float4 v4 = plane_sum4(Z, splits, plane, e);
  float v[4] = {v4.x, v4.y, v4.z, v4.w}, g[4];
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    v[q] += c + q < dout ? bias[c + q] : 0.f;
    g[q] = c + q < dout ? gelu(v[q]) : 0.f;
  }
  *reinterpret_cast<float4*>(pre + e) = make_float4(v[0], v[1], v[2], v[3]);
  *reinterpret_cast<float4*>(h + e) = make_float4(g[0], g[1], g[2], g[3]);
}
// output layer and loss: z = Z + bias, dz = z - t_norm over unmasked entries (0 elsewhere; the scale
// 2 / count enters with the gradients); a row's sum of squares and count go to part[row]
__global__ void __launch_bounds__(256) loss_train_kernel(const float* Z, int splits, size_t plane, int dout, int ld,
                                                         const float* bias, const float* t, const float* mean,
                                                         const float* std_, float* dz, float2* part) {
  __shared__ float red[32];
  const int b = blockIdx.x;
  float l = 0.f, c = 0.f;
  for (int f = threadIdx.x; f < ld; f += 256) {
    const size_t e = (size_t)b * ld + f;
    if (f >= dout) {
      dz[e] = 0.f;
      continue;
    }
    const float v = plane_sum(Z, splits, plane, e) + bias[f], tv = t[(size_t)b * dout + f];
    const bool ok = isfinite(tv);
    const float r = ok ? v - (tv - mean[f]) / std_[f] : 0.f;
    dz[e] = r;
    l += r * r;
    c += ok ? 1.f : 0.f;
  }
  l = block_sum(l, red);
  c = block_sum(c, red);
  if (threadIdx.x == 0) part[b] = make_float2(l, c);
}
__global__ void __launch_bounds__(256) loss_finish_kernel(const float2* part, int parts, float* loss_scale) {
  __shared__ float red[32];
  float l = 0.f, c = 0.f;
  for (int i = threadIdx.x; i < parts; i += 256) {
    l += part[i].x;
    c += part[i].y;
  }
  l = block_sum(l, red);
  c = block_sum(c, red);
  if (threadIdx.x == 0) {
    loss_scale[0] = c > 0.f ? l / c : 0.f;    // loss
    loss_scale[1] = c > 0.f ? 2.f / c : 0.f;  // gradient scale
  }
}
// dZ of a hidden layer: (dZ W) * GELU'(pre)
__global__ void __launch_bounds__(128) gelu_back_kernel(const float* Z, int splits, size_t plane, int din, int ld,
                                                        const float* pre, float* dz) {
  const int c = (blockIdx.y * 128 + threadIdx.x) * 4;
  if (c >= ld) return;
  const size_t e = (size_t)blockIdx.x * ld + c;
  const float4 v = plane_sum4(Z, splits, plane, e), p = *reinterpret_cast<const float4*>(pre + e);
  *reinterpret_cast<float4*>(dz + e) =
      make_float4(v.x * gelu_grad(p.x), c + 1 < din ? v.y * gelu_grad(p.y) : 0.f, c + 2 < din ? v.z * gelu_grad(p.z) : 0.f,
                  c + 3 < din ? v.w * gelu_grad(p.w) : 0.f);
}

// A layer's gradient, 2 / count times: dW from its partial-sum planes [dout][pitch] (CTAs below
// wblocks) and db_o = sum_b dZ_bo (32 columns per CTA above).  With step == 0 it is written to G;
// otherwise AdamW runs on it directly: the FP32 master parameters, the moments, and the BF16 copy of
// the weights (row pitch inp) that the forward passes read.
struct LayerUpdate {
  const float* Z;
  int splits, pitch, dout, din, batch, ldz, wblocks, inp;
  size_t plane;
  const float* dz;
  const float* scale;
  float *G, *P, *M, *V;      // the layer's weights, then its biases
  __nv_bfloat16* w16;
  int step;                  // 0: write G; 1: AdamW
  float lr, b1, b2, eps, wd, bc1, bc2;
};
__device__ __forceinline__ float layer_step(const LayerUpdate& A, size_t e, float gr) {
  if (!A.step) {
    A.G[e] = gr;
    return 0.f;
  }
  const float mm = A.b1 * A.M[e] + (1.f - A.b1) * gr;
  const float vv = A.b2 * A.V[e] + (1.f - A.b2) * gr * gr;
  A.M[e] = mm;
  A.V[e] = vv;
  const float p = A.P[e], upd = (mm / A.bc1) / (sqrtf(vv / A.bc2) + A.eps);
  const float np = p - A.lr * (upd + A.wd * p);
  A.P[e] = np;
  return np;
}
__global__ void __launch_bounds__(256) layer_update_kernel(LayerUpdate A) {
  const float s = *A.scale;
  if ((int)blockIdx.x < A.wblocks) {
    for (int o = blockIdx.x; o < A.dout; o += A.wblocks)
      for (int i = threadIdx.x; i < A.din; i += 256) {
        const float np = layer_step(A, (size_t)o * A.din + i, s * plane_sum(A.Z, A.splits, A.plane, (size_t)o * A.pitch + i));
        if (A.step) A.w16[(size_t)o * A.inp + i] = __float2bfloat16_rn(np);
      }
    return;
  }
  __shared__ float red[8][33];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, o = ((int)blockIdx.x - A.wblocks) * 32 + lane;
  float a = 0.f;
  if (o < A.dout)
    for (int b = warp; b < A.batch; b += 8) a += A.dz[(size_t)b * A.ldz + o];
  red[warp][lane] = a;
  __syncthreads();
  if (warp == 0 && o < A.dout) {
    a = 0.f;
#pragma unroll
    for (int w = 0; w < 8; ++w) a += red[w][lane];
    (void)layer_step(A, (size_t)A.dout * A.din + o, s * a);
  }
}

__global__ void fill_kernel(float* p, size_t count, float v) {
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x)
    p[e] = v;
}

// Deterministic initialisation: uniform(-a, a) from a counter-based hash (splitmix64 of
// seed + index), a = sqrt(6 / (fan_in + fan_out)) for weights; biases 0.
__device__ __forceinline__ unsigned long long splitmix64(unsigned long long z) {
  z += 0x9E3779B97F4A7C15ull;
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}
__global__ void init_kernel(float* p, size_t count, float a, unsigned long long seed) {
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < count; e += (size_t)gridDim.x * blockDim.x) {
    const double u = (double)(splitmix64(seed + e) >> 11) * (1.0 / 9007199254740992.0);
    p[e] = (float)((2.0 * u - 1.0) * a);
  }
}

// ---- tensor-core forward pass (inference) ------------------------------------------------------
// Each layer is Z = H W^T on gemm3_kernel<KIND_BF16> with A = W (the BF16 weights, exact: two products
// give W times the activations to ~16 bits) and
// B = the activations as a BF16 hi/lo pair, K-major with a row pitch padded to 8 elements (TMA
// rows are 16-byte multiples).  Z may be split over the reduction (partial-sum planes); the
// activation kernel adds the planes in order, the bias and GELU, and writes the next operand.

// Weights of one layer, [out][in] FP32 -> BF16 with the row pitch inp.
__global__ void pad_bf16_kernel(const float* W, int dout, int din, int inp, __nv_bfloat16* out) {
  const size_t total = (size_t)dout * din;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int o = (int)(e / din), i = (int)(e - (size_t)o * din);
    out[(size_t)o * inp + i] = __float2bfloat16_rn(W[e]);
  }
}

__device__ __forceinline__ void split_bf16(float v, __nv_bfloat16* hi, __nv_bfloat16* lo) {
  const __nv_bfloat16 h = __float2bfloat16_rn(v);
  *hi = h;
  *lo = __float2bfloat16_rn(v - __bfloat162float(h));
}

// features as the first operand: [n y / sum(y), log sum(y)] as BF16 hi/lo, row pitch inp.
__global__ void features_split_kernel(const float* y, int n, int inp, __nv_bfloat16* hhi, __nv_bfloat16* hlo) {
  __shared__ float red[32];
  const int b = blockIdx.x;
  float s = 0.f;
  for (int i = threadIdx.x; i < n; i += blockDim.x) s += y[(size_t)b * n + i];
  s = block_sum(s, red);
  const float inv = s > 0.f ? (float)n / s : 0.f;
  const size_t row = (size_t)b * inp;
  for (int i = threadIdx.x; i < n; i += blockDim.x) split_bf16(y[(size_t)b * n + i] * inv, hhi + row + i, hlo + row + i);
  if (threadIdx.x == 0) split_bf16(s > 0.f ? logf(s) : 0.f, hhi + row + n, hlo + row + n);
}

// Hidden layer: v = sum over the `splits` planes of Z [rows][dout] + bias, GELU(v) as the next BF16
// hi/lo operand (row pitch outp, a multiple of eight). grid.x = row, four columns per thread.
__global__ void __launch_bounds__(256) act_split_kernel(const float* Z, int splits, size_t plane, int dout,
                                                        const float* bias, __nv_bfloat16* ohi, __nv_bfloat16* olo,
                                                        int outp) {
  const int f0 = (blockIdx.y * 256 + threadIdx.x) * 4;
  if (f0 >= dout) return;
  const size_t e = (size_t)blockIdx.x * dout + f0, o = (size_t)blockIdx.x * outp + f0;
  float v[4] = {0.f, 0.f, 0.f, 0.f};
  const bool vec = dout % 4 == 0 && plane % 4 == 0;  // 16-byte aligned rows and planes
  for (int z = 0; z < splits; ++z) {
    if (vec) {
      const float4 q = *reinterpret_cast<const float4*>(Z + z * plane + e);
      v[0] += q.x; v[1] += q.y; v[2] += q.z; v[3] += q.w;
    } else {
#pragma unroll
      for (int c = 0; c < 4; ++c)
        if (f0 + c < dout) v[c] += Z[z * plane + e + c];
    }
  }
  __align__(8) __nv_bfloat16 hi[4], lo[4];
#pragma unroll
  for (int c = 0; c < 4; ++c) split_bf16(f0 + c < dout ? gelu(v[c] + bias[f0 + c]) : 0.f, hi + c, lo + c);
  *reinterpret_cast<uint2*>(ohi + o) = *reinterpret_cast<uint2*>(hi);  // padding columns get zeros
  *reinterpret_cast<uint2*>(olo + o) = *reinterpret_cast<uint2*>(lo);
}

// Output layer -> warm start: z = sum over the planes + bias; g0 = eps * (z * std + mean) for the first
// n outputs (the potential g / eps), w0 = exp(z * std + mean) for the last k (log w); non-finite
// predictions fall back to the cold start (g0 = 0, w0 = cold_w) so that a bad network can only cost
// iterations, and so does every row when *fail is set (a GEMM of the forward pass gave up a wait).
// grid.x = row, 256 threads over 1024 outputs.
__global__ void __launch_bounds__(256) decode_kernel(const float* Z, int splits, size_t plane, const float* bias,
                                                     const float* mean, const float* std_, int n, int k, float eps,
                                                     const float* cold_w, float* g0, float* w0, const int* fail) {
  const int cols = n + k, b = blockIdx.x;
  const bool failed = fail && *fail;
#pragma unroll
  for (int q = 0; q < 4; ++q) {
    const int j = blockIdx.y * 1024 + q * 256 + threadIdx.x;
    if (j >= cols) continue;
    const float z = plane_sum(Z, splits, plane, (size_t)b * cols + j) + bias[j];
    const float v = failed ? CUDART_NAN_F : z * std_[j] + mean[j];
    if (j < n) {
      g0[(size_t)b * n + j] = isfinite(v) ? eps * v : 0.f;
    } else {
      const float wv = expf(v);
      w0[(size_t)b * k + (j - n)] = (isfinite(wv) && wv > 0.f) ? wv : cold_w[(size_t)b * k + (j - n)];
    }
  }
}


// ---- training data: targets of solved problems and their per-output normalisation ------------

// Target row [g / eps (n), log w (k)] of a solved problem: g / eps is clipped below at g_floor
// (far below any potential that matters: the prediction only seeds the iteration); a
// non-finite g (u1 = 0 where y = 0 under the KL datafit) and w <= 0 give -inf, which the loss
// masks out.
__global__ void make_targets_kernel(const float* g, const float* wts, int rows, int n, int k, float inv_eps,
                                    float g_floor, float* t) {
  const int cols = n + k;
  const size_t total = (size_t)rows * cols;
  for (size_t e = (size_t)blockIdx.x * blockDim.x + threadIdx.x; e < total; e += (size_t)gridDim.x * blockDim.x) {
    const int b = (int)(e / cols), j = (int)(e % cols);
    float v;
    if (j < n) {
      const float gv = g[(size_t)b * n + j];
      v = isfinite(gv) ? fmaxf(gv * inv_eps, g_floor) : -CUDART_INF_F;
    } else {
      const float wv = wts[(size_t)b * k + (j - n)];
      v = wv > 0.f ? logf(wv) : -CUDART_INF_F;
    }
    t[e] = v;
  }
}

// Per-output mean and standard deviation over the finite entries of targets [rows][cols], in two
// passes (sum and count, then squared deviations), FP64 partial sums per (row chunk, column) added
// in a fixed order; std is floored at 1e-3.  Thread = column (coalesced across a row), blockIdx.y =
// chunk of rows r = chunk, chunk + NORM_CHUNKS, ...
constexpr int NORM_CHUNKS = 128;
__global__ void norm_partial_kernel(const float* t, int rows, int cols, const float* mean, double* part,
                                    int* cnt) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x, z = blockIdx.y;
  if (c >= cols) return;
  double s = 0.0;
  int m = 0;
  const float mu = mean ? mean[c] : 0.f;
  for (int r = z; r < rows; r += NORM_CHUNKS) {
    const float v = t[(size_t)r * cols + c];
    if (isfinite(v)) {
      const double d = mean ? (double)v - (double)mu : (double)v;
      s += mean ? d * d : d;
      ++m;
    }
  }
  part[(size_t)z * cols + c] = s;
  if (cnt) cnt[(size_t)z * cols + c] = m;
}
// pass 1 (std_out == null): mean = sum / count; pass 2: std = sqrt(sum of squares / count)
__global__ void norm_finish_kernel(const double* part, const int* cnt, int cols, float* mean, float* std_out) {
  const int c = blockIdx.x * blockDim.x + threadIdx.x;
  if (c >= cols) return;
  double s = 0.0;
  long long m = 0;
  for (int z = 0; z < NORM_CHUNKS; ++z) {
    s += part[(size_t)z * cols + c];
    m += cnt[(size_t)z * cols + c];
  }
  const double q = s / (double)(m > 0 ? m : 1);
  if (!std_out) mean[c] = (float)q;
  else std_out[c] = fmaxf((float)sqrt(q), 1e-3f);
}

}  // namespace mlp
}  // namespace otlm
