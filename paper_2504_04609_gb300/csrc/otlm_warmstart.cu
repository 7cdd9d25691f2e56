// C ABI of the learned warm start (declared in include/otlm.h): a 4-layer MLP trained on solved
// problems to predict the initial target potential g / eps and log w (kernels in mlp.cuh).
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <cmath>
#include <new>

#include "../../include/otlm.h"
#include "mlp.cuh"
#include "tc_gemm.cuh"

using namespace otlm::mlp;

constexpr int TC_MAX_SPLITS = 16;

struct otlm_ws_ctx {
  int n = 0, k = 0, H = 0, batch_max = 0;
  cudaStream_t stream = nullptr;
  int d[LAYERS + 1] = {};
  size_t woff[LAYERS] = {}, boff[LAYERS] = {}, nparams = 0;
  void* mem = nullptr;
  float *P = nullptr, *G = nullptr, *M = nullptr, *V = nullptr;
  float* pre[LAYERS] = {};
  float *mean = nullptr, *stdv = nullptr, *loss_scale = nullptr;
  long long step = 0;
  // tensor-core forward pass (inference): padded BF16 weights, activations as BF16
  // hi/lo pairs (ping-pong), split partial sums, and the GEMMs' error flag
  int inp[LAYERS] = {};            // row pitch of layer l's input operand (d[l] rounded up to 8)
  int dmax = 0;                    // widest layer output
  __nv_bfloat16* W16p[LAYERS] = {};
  __nv_bfloat16 *Hhi[2] = {}, *Hlo[2] = {};
  float* Zs = nullptr;             // [TC_MAX_SPLITS][batch_max][dmax]
  int* tc_err = nullptr;
  bool dirty = true;               // W16p is stale (parameters set from outside since the last refresh)
  // training: the layers' inputs and the current dZ (ping-pong), row pitches of multiples of four with
  // zero padding, and the partial sums of a weight gradient
  int xp[LAYERS + 1] = {};
  float *X[LAYERS] = {}, *dZ[2] = {}, *Gs = nullptr;
  size_t gs_floats = 0;
  float2* lpart = nullptr;
  // per-output normalisation statistics: FP64 partial sums and counts per (row chunk, output)
  double* norm_part = nullptr;
  int* norm_cnt = nullptr;
};

namespace {

size_t align256(size_t v) { return (v + 255) & ~size_t(255); }

int pitch4(int v) { return (v + 3) / 4 * 4; }

// The BF16 weights of both passes after the parameters were set from outside.
void refresh_weights(otlm_ws_ctx* w) {
  if (!w->dirty) return;
  for (int l = 0; l < LAYERS; ++l)
    pad_bf16_kernel<<<1184, 256, 0, w->stream>>>(w->P + w->woff[l], w->d[l + 1], w->d[l], w->inp[l], w->W16p[l]);
  w->dirty = false;
}

// One training GEMM: partial-sum planes [splits][M][ldc], the reduction split so that two CTAs fit
// each SM, with at most `room` floats of planes.
template <bool AK, bool BK, typename TB>
void train_gemm(cudaStream_t s, int M, int N, int K, const float* A, int lda, const TB* B, int ldb, float* C, int ldc,
                size_t room, int* splits, size_t* plane) {
  const int tiles = ((M + GM - 1) / GM) * ((N + GN - 1) / GN), kb = (K + GK - 1) / GK;
  int z = 2 * otlm::tc::num_sms() / tiles;
  z = z > kb / 2 ? kb / 2 : z;
  z = z > TC_MAX_SPLITS ? TC_MAX_SPLITS : z;
  *plane = (size_t)M * ldc;
  while (z > 1 && z * *plane > room) --z;
  z = z < 1 ? 1 : z;
  const int per = (kb + z - 1) / z;
  z = (kb + per - 1) / per;
  *splits = z;
  train_gemm_kernel<AK, BK, TB><<<dim3((N + GN - 1) / GN, (M + GM - 1) / GM, z), GT, 0, s>>>(M, N, K, A, lda, B, ldb, C,
                                                                                            ldc, *plane, per * GK);
}

// forward, loss and gradients: into w->G (u.step == 0) or straight into AdamW's step; loss (and
// 2/count) in w->loss_scale.  u carries the optimiser's scalars.
cudaError_t backward(otlm_ws_ctx* w, int batch, const float* y, const float* target, LayerUpdate u) {
  cudaStream_t s = w->stream;
  const size_t zroom = (size_t)TC_MAX_SPLITS * w->batch_max * w->dmax;
  refresh_weights(w);
  features_kernel<<<batch, 256, 0, s>>>(y, w->n, w->X[0], w->xp[0]);
  int splits = 1;
  size_t plane = 0;
  for (int l = 0; l < LAYERS; ++l) {
    const int din = w->d[l], dout = w->d[l + 1], ld = w->xp[l + 1];
    train_gemm<true, true, __nv_bfloat16>(s, batch, dout, din, w->X[l], w->xp[l], w->W16p[l], w->inp[l], w->Zs, ld, zroom,
                                          &splits, &plane);
    const float* bias = w->P + w->boff[l];
    if (l < LAYERS - 1) {
      act_train_kernel<<<dim3(batch, (ld + 511) / 512), 128, 0, s>>>(w->Zs, splits, plane, dout, ld, bias, w->pre[l + 1],
                                                                     w->X[l + 1]);
    } else {
      loss_train_kernel<<<batch, 256, 0, s>>>(w->Zs, splits, plane, dout, ld, bias, target, w->mean, w->stdv, w->dZ[0],
                                              w->lpart);
      loss_finish_kernel<<<1, 256, 0, s>>>(w->lpart, batch, w->loss_scale);
    }
  }
  int cur = 0;
  for (int l = LAYERS - 1; l >= 0; --l) {
    const int din = w->d[l], dout = w->d[l + 1], ldz = w->xp[l + 1], ldx = w->xp[l];
    const float* dz = w->dZ[cur];
    if (l > 0) {  // dH[b][i] = sum_o dZ[b][o] W[o][i], before the layer's weights are stepped
      train_gemm<true, false, __nv_bfloat16>(s, batch, din, dout, dz, ldz, w->W16p[l], w->inp[l], w->Zs, ldx, zroom, &splits,
                                             &plane);
      gelu_back_kernel<<<dim3(batch, (ldx + 511) / 512), 128, 0, s>>>(w->Zs, splits, plane, din, ldx, w->pre[l],
                                                                      w->dZ[cur ^ 1]);
    }
    // dW[o][i] = sum_b dZ[b][o] X[b][i]
    train_gemm<false, false, float>(s, dout, din, batch, dz, ldz, w->X[l], ldx, w->Gs, ldx, w->gs_floats, &splits, &plane);
    u.Z = w->Gs; u.splits = splits; u.plane = plane; u.pitch = ldx; u.dout = dout; u.din = din; u.batch = batch;
    u.dz = dz; u.ldz = ldz; u.scale = w->loss_scale + 1; u.wblocks = dout < 1184 ? dout : 1184; u.inp = w->inp[l];
    u.G = w->G + w->woff[l]; u.P = w->P + w->woff[l]; u.M = w->M + w->woff[l]; u.V = w->V + w->woff[l];
    u.w16 = w->W16p[l];
    layer_update_kernel<<<u.wblocks + (dout + 31) / 32, 256, 0, s>>>(u);
    cur ^= 1;
  }
  return cudaGetLastError();
}

// Forward pass on the tensor cores, decoded into the warm start (inference only).
cudaError_t forward_tc(otlm_ws_ctx* w, int batch, const float* y, float eps, const float* cold_w, float* g0, float* w0) {
  cudaStream_t s = w->stream;
  refresh_weights(w);
  cudaError_t e = cudaMemsetAsync(w->tc_err, 0, sizeof(int), s);
  if (e != cudaSuccess) return e;
  features_split_kernel<<<batch, 256, 0, s>>>(y, w->n, w->inp[0], w->Hhi[0], w->Hlo[0]);
  const size_t plane = (size_t)w->batch_max * w->dmax;
  int cur = 0;
  for (int l = 0; l < LAYERS; ++l) {
    const int din = w->d[l], dout = w->d[l + 1];
    otlm::tc::GemmArgs g{};
    g.out = w->Zs; g.M = dout; g.N = batch; g.Kd = din; g.ld_out = dout; g.err = w->tc_err;
    // split the reduction only as far as the tiles leave SMs idle (every split is a plane of FP32 sums:
    // 4096 rows ran as seven planes of 8 MB in the input layer and eight of 35 MB in the output layer),
    // and drain the accumulators after every k block
    const int tiles = ((dout + otlm::tc::BM - 1) / otlm::tc::BM) * ((batch + otlm::tc::BN - 1) / otlm::tc::BN);
    const int want = otlm::tc::num_sms() / tiles, nkb = (din + 63) / 64;
    g.splits = want < 1 ? 1 : (want > nkb ? nkb : want);
    g.chunk = 1;
    g.pdl = true;
    if (g.splits > TC_MAX_SPLITS) g.splits = TC_MAX_SPLITS;
    g.a_exact = 1;  // BF16 weights: two products
    g.split_stride = plane;
    e = otlm::tc::launch_gemm3<otlm::tc::KIND_BF16>(w->W16p[l], w->W16p[l], w->inp[l], w->Hhi[cur], w->Hlo[cur],
                                                    w->inp[l], dout, batch, din, g, s);
    if (e != cudaSuccess) return e;
    if (l < LAYERS - 1)
      act_split_kernel<<<dim3(batch, (dout + 1023) / 1024), 256, 0, s>>>(w->Zs, g.splits, plane, dout, w->P + w->boff[l],
                                                                        w->Hhi[cur ^ 1], w->Hlo[cur ^ 1], w->inp[l + 1]);
    else
      decode_kernel<<<dim3(batch, (dout + 1023) / 1024), 256, 0, s>>>(w->Zs, g.splits, plane, w->P + w->boff[l], w->mean, w->stdv,
                                                                     w->n, w->k, eps, cold_w, g0, w0, w->tc_err);
    cur ^= 1;
  }
  return cudaGetLastError();
}

}  // namespace

extern "C" {

int otlm_ws_create(otlm_ws* out, int n, int k, int width, int batch_max, unsigned long long seed, void* stream) {
  if (!out) return OTLM_EINVAL;
  *out = nullptr;
  if (n < 2 || k < 1 || width < 1 || batch_max < 1) return OTLM_EINVAL;
  otlm_ws_ctx* w = new (std::nothrow) otlm_ws_ctx;
  if (!w) return OTLM_ENOMEM;
  w->n = n; w->k = k; w->H = width; w->batch_max = batch_max;
  w->stream = static_cast<cudaStream_t>(stream);
  const int d[LAYERS + 1] = {n + 1, width, width, width, n + k};
  size_t off = 0;
  for (int l = 0; l <= LAYERS; ++l) {
    w->d[l] = d[l];
  }
  for (int l = 0; l < LAYERS; ++l) {
    w->woff[l] = off;
    off += (size_t)d[l + 1] * d[l];
    w->boff[l] = off;
    off += d[l + 1];
  }
  w->nparams = off;
  size_t bytes = 4 * align256(4 * off);
  // training: layer inputs, pre-activations, dZ twice, partial sums of the largest weight gradient
  size_t trainb = 0;
  int dzp = 0;
  for (int l = 0; l <= LAYERS; ++l) w->xp[l] = pitch4(d[l]);
  for (int l = 0; l < LAYERS; ++l) {
    dzp = dzp > w->xp[l + 1] ? dzp : w->xp[l + 1];
    trainb += align256(4 * (size_t)batch_max * w->xp[l]);
    if (l > 0) trainb += align256(4 * (size_t)batch_max * w->xp[l]);
    const size_t g = 4 * (size_t)d[l + 1] * w->xp[l];
    w->gs_floats = w->gs_floats > g ? w->gs_floats : g;
  }
  trainb += 2 * align256(4 * (size_t)batch_max * dzp) + align256(4 * w->gs_floats) + align256(8 * (size_t)batch_max);
  bytes += trainb + 2 * align256(4 * (size_t)(n + k)) + 256;
  size_t w16b = 0;
  int maxp = 0;
  for (int l = 0; l < LAYERS; ++l) {
    w->inp[l] = (d[l] + 7) / 8 * 8;
    w16b += align256(2 * (size_t)d[l + 1] * w->inp[l]);
    maxp = maxp > w->inp[l] ? maxp : w->inp[l];
    w->dmax = w->dmax > w->xp[l + 1] ? w->dmax : w->xp[l + 1];
  }
  bytes += w16b + 4 * align256(2 * (size_t)batch_max * maxp) +
           align256(4 * (size_t)TC_MAX_SPLITS * batch_max * w->dmax) + 256;
  bytes += align256(8 * (size_t)NORM_CHUNKS * (n + k)) + align256(4 * (size_t)NORM_CHUNKS * (n + k));
  if (cudaMalloc(&w->mem, bytes) != cudaSuccess) {
    delete w;
    return OTLM_ENOMEM;
  }
  char* p = static_cast<char*>(w->mem);
  auto take = [&](size_t b) { char* r = p; p += align256(b); return r; };
  w->P = (float*)take(4 * off);
  w->G = (float*)take(4 * off);
  w->M = (float*)take(4 * off);
  w->V = (float*)take(4 * off);
  char* zeroed = p;  // the padded training buffers, cleared below
  for (int l = 1; l < LAYERS; ++l) w->pre[l] = (float*)take(4 * (size_t)batch_max * w->xp[l]);
  for (int l = 0; l < LAYERS; ++l) w->X[l] = (float*)take(4 * (size_t)batch_max * w->xp[l]);
  for (int c = 0; c < 2; ++c) w->dZ[c] = (float*)take(4 * (size_t)batch_max * dzp);
  const size_t zeroed_bytes = p - zeroed;
  w->Gs = (float*)take(4 * w->gs_floats);
  w->lpart = (float2*)take(8 * (size_t)batch_max);
  w->mean = (float*)take(4 * (size_t)(n + k));
  w->stdv = (float*)take(4 * (size_t)(n + k));
  w->loss_scale = (float*)take(256);
  for (int l = 0; l < LAYERS; ++l) w->W16p[l] = (__nv_bfloat16*)take(2 * (size_t)d[l + 1] * w->inp[l]);
  for (int c = 0; c < 2; ++c) {
    w->Hhi[c] = (__nv_bfloat16*)take(2 * (size_t)batch_max * maxp);
    w->Hlo[c] = (__nv_bfloat16*)take(2 * (size_t)batch_max * maxp);
  }
  w->Zs = (float*)take(4 * (size_t)TC_MAX_SPLITS * batch_max * w->dmax);
  w->tc_err = (int*)take(256);
  w->norm_part = (double*)take(8 * (size_t)NORM_CHUNKS * (n + k));
  w->norm_cnt = (int*)take(4 * (size_t)NORM_CHUNKS * (n + k));
  cudaStream_t s = w->stream;
  // zero padding columns of the weights and activations
  cudaError_t e = cudaMemsetAsync(w->W16p[0], 0, w16b + 4 * align256(2 * (size_t)batch_max * maxp), s);
  if (e == cudaSuccess) e = cudaMemsetAsync(zeroed, 0, zeroed_bytes, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(w->P, 0, 4 * off, s);
  for (int l = 0; l < LAYERS && e == cudaSuccess; ++l) {
    const float a = std::sqrt(6.f / (float)(d[l] + d[l + 1]));
    init_kernel<<<1184, 256, 0, s>>>(w->P + w->woff[l], (size_t)d[l + 1] * d[l], a, seed + 0x1000000ull * (l + 1));
    e = cudaGetLastError();
  }
  if (e == cudaSuccess) e = cudaMemsetAsync(w->M, 0, 4 * off, s);
  if (e == cudaSuccess) e = cudaMemsetAsync(w->V, 0, 4 * off, s);
  // identity normalisation (mean 0, std 1) until the caller sets one
  if (e == cudaSuccess) e = cudaMemsetAsync(w->mean, 0, 4 * (size_t)(n + k), s);
  if (e == cudaSuccess) {
    fill_kernel<<<(n + k + 255) / 256, 256, 0, s>>>(w->stdv, (size_t)(n + k), 1.f);
    e = cudaGetLastError();
  }
  if (e != cudaSuccess) {
    cudaFree(w->mem);
    delete w;
    return OTLM_ECUDA;
  }
  *out = w;
  return OTLM_OK;
}

void otlm_ws_destroy(otlm_ws w) {
  if (!w) return;
  cudaStreamSynchronize(w->stream);
  cudaFree(w->mem);
  delete w;
}

long long otlm_ws_num_params(otlm_ws w) { return w ? (long long)w->nparams : -1; }

int otlm_ws_set_normalization(otlm_ws w, const float* mean, const float* stdv) {
  if (!w || !mean || !stdv) return OTLM_EINVAL;
  const size_t b = 4 * (size_t)(w->n + w->k);
  if (cudaMemcpyAsync(w->mean, mean, b, cudaMemcpyDeviceToDevice, w->stream) != cudaSuccess ||
      cudaMemcpyAsync(w->stdv, stdv, b, cudaMemcpyDeviceToDevice, w->stream) != cudaSuccess)
    return OTLM_ECUDA;
  return OTLM_OK;
}

int otlm_ws_get_params(otlm_ws w, float* out) {
  if (!w || !out) return OTLM_EINVAL;
  return cudaMemcpyAsync(out, w->P, 4 * w->nparams, cudaMemcpyDeviceToDevice, w->stream) == cudaSuccess ? OTLM_OK
                                                                                                          : OTLM_ECUDA;
}

int otlm_ws_set_params(otlm_ws w, const float* in) {
  if (!w || !in) return OTLM_EINVAL;
  if (cudaMemcpyAsync(w->P, in, 4 * w->nparams, cudaMemcpyDeviceToDevice, w->stream) != cudaSuccess)
    return OTLM_ECUDA;
  w->dirty = true;
  return cudaGetLastError() == cudaSuccess ? OTLM_OK : OTLM_ECUDA;
}

int otlm_ws_gradients(otlm_ws w, int batch, const float* y, const float* target, float* grad_out, float* loss_out) {
  if (!w || !y || !target || batch < 1 || batch > w->batch_max) return OTLM_EINVAL;
  cudaError_t e = backward(w, batch, y, target, LayerUpdate{});
  if (e == cudaSuccess && grad_out)
    e = cudaMemcpyAsync(grad_out, w->G, 4 * w->nparams, cudaMemcpyDeviceToDevice, w->stream);
  if (e == cudaSuccess && loss_out) e = cudaMemcpyAsync(loss_out, w->loss_scale, 4, cudaMemcpyDeviceToDevice, w->stream);
  return e == cudaSuccess ? OTLM_OK : OTLM_ECUDA;
}

int otlm_ws_train_step(otlm_ws w, int batch, const float* y, const float* target, double lr, double weight_decay,
                       float* loss_out) {
  if (!w || !y || !target || batch < 1 || batch > w->batch_max || !(lr > 0) || !(weight_decay >= 0))
    return OTLM_EINVAL;
  w->step += 1;
  LayerUpdate u{};
  u.step = 1; u.lr = (float)lr; u.b1 = 0.9f; u.b2 = 0.999f; u.eps = 1e-8f; u.wd = (float)weight_decay;
  u.bc1 = 1.f - std::pow(u.b1, (float)w->step); u.bc2 = 1.f - std::pow(u.b2, (float)w->step);
  cudaError_t e = backward(w, batch, y, target, u);
  if (e == cudaSuccess && loss_out) e = cudaMemcpyAsync(loss_out, w->loss_scale, 4, cudaMemcpyDeviceToDevice, w->stream);
  return e == cudaSuccess ? OTLM_OK : OTLM_ECUDA;
}

int otlm_ws_predict(otlm_ws w, int batch, const float* y, double eps, const float* cold_w, float* g0, float* w0) {
  if (!w || !y || !cold_w || !g0 || !w0 || batch < 1 || batch > w->batch_max || !(eps > 0)) return OTLM_EINVAL;
  return forward_tc(w, batch, y, (float)eps, cold_w, g0, w0) == cudaSuccess ? OTLM_OK : OTLM_ECUDA;
}

int otlm_ws_make_targets(otlm_ws w, int batch, const float* g, const float* wts, double eps, double g_floor,
                         float* targets) {
  if (!w || !g || !wts || !targets || batch < 1 || !(eps > 0) || !std::isfinite(eps) || !(g_floor == g_floor))
    return OTLM_EINVAL;
  make_targets_kernel<<<1184, 256, 0, w->stream>>>(g, wts, batch, w->n, w->k, (float)(1.0 / eps), (float)g_floor,
                                                   targets);
  return cudaGetLastError() == cudaSuccess ? OTLM_OK : OTLM_ECUDA;
}

int otlm_ws_fit_normalization(otlm_ws w, int rows, const float* targets, float* mean_out, float* std_out) {
  if (!w || !targets || rows < 1) return OTLM_EINVAL;
  const int cols = w->n + w->k;
  const dim3 grid((cols + 255) / 256, NORM_CHUNKS);
  cudaStream_t s = w->stream;
  norm_partial_kernel<<<grid, 256, 0, s>>>(targets, rows, cols, nullptr, w->norm_part, w->norm_cnt);
  norm_finish_kernel<<<(cols + 255) / 256, 256, 0, s>>>(w->norm_part, w->norm_cnt, cols, w->mean, nullptr);
  norm_partial_kernel<<<grid, 256, 0, s>>>(targets, rows, cols, w->mean, w->norm_part, nullptr);
  norm_finish_kernel<<<(cols + 255) / 256, 256, 0, s>>>(w->norm_part, w->norm_cnt, cols, w->mean, w->stdv);
  cudaError_t e = cudaGetLastError();
  if (e == cudaSuccess && mean_out)
    e = cudaMemcpyAsync(mean_out, w->mean, 4 * (size_t)cols, cudaMemcpyDeviceToDevice, s);
  if (e == cudaSuccess && std_out) e = cudaMemcpyAsync(std_out, w->stdv, 4 * (size_t)cols, cudaMemcpyDeviceToDevice, s);
  return e == cudaSuccess ? OTLM_OK : OTLM_ECUDA;
}

}  // extern "C"
