// Learned T0 predictor: a 6 -> 128 -> 128 -> 2 multilayer perceptron (tanh hidden layers,
// linear output) with BF16 weights and FP32 accumulation, trained on the GPU by these
// kernels (forward, mean-squared-error loss, backward, Adam). The inputs are features of
// the linear system and the clock budget (Sec. VI: kappa, the eigenvalue bounds, N, Q_PE),
// the outputs the optimal Hamiltonian-simulation time T0* and the clock count, replacing the
// power-law fit T0* ~ kappa of Sec. VI where the network is available.
//
// Parameter vector (FP32 master copy, flat): W1 [128][6], b1 [128], W2 [128][128], b2 [128],
// W3 [2][128], b3 [2]. Forward and backward read the BF16 rounding of W1, W2, W3 (refreshed
// after every update); gradients and Adam moments are FP32.
#include <cuda_bf16.h>
#include <math.h>

#include <algorithm>
#include <vector>

#include "hhl_common.cuh"

namespace hhl {
namespace {

constexpr int kIn = HHL_MLP_IN, kH = HHL_MLP_HIDDEN, kOut = HHL_MLP_OUT;
constexpr int kOffW1 = 0, kOffB1 = kOffW1 + kH * kIn, kOffW2 = kOffB1 + kH, kOffB2 = kOffW2 + kH * kH,
              kOffW3 = kOffB2 + kH, kOffB3 = kOffW3 + kOut * kH, kParams = kOffB3 + kOut;
static_assert(kParams == HHL_MLP_PARAMS, "parameter layout");
constexpr int kRows = 4;         // rows per CTA of the row pass
constexpr int kThr = 128;        // one thread per hidden unit
constexpr int kGradThr = 1024;   // gradient pass: 2 units x 128 inputs x 4 row groups
constexpr int kGradUnits = 2;
constexpr int kGradRows = 1024;  // rows of one gradient chunk
// Rows that the activation buffers hold (0.5 GB): a longer batch goes through them slab by slab, its chunks'
// gradients added in the same order.
constexpr int kSlabRows = 1 << 18;
static_assert(kSlabRows % kGradRows == 0 && kSlabRows / kGradRows <= 65535, "chunks of a slab");
static_assert(kRows == 4 && kThr == kH && kGradThr == kGradUnits * kH * 4, "thread maps below");

__device__ __forceinline__ float bf_lo(uint32_t v) { return __uint_as_float(v << 16); }
__device__ __forceinline__ float bf_hi(uint32_t v) { return __uint_as_float(v & 0xffff0000u); }

// The rows of a batch, four per CTA, thread j = hidden unit j of both layers: forward, and with
// TRAIN the loss and the gradients with respect to the pre-activations (ga1, ga2), stored with the
// activations for the gradient pass. A thread keeps its row of W2 (128 BF16 values) in
// registers and reads the four rows' activations as one 16-byte broadcast per input. Bound by
// latency: a 256-row batch is 64 CTAs. (32 rows per CTA and W2 converted into shared memory filled
// 8 SMs: forward 41 us, loss and backward 96 us; this pass takes 6 and 9 us.)
template <bool TRAIN>
__global__ void __launch_bounds__(kThr) k_mlp_rows(const __nv_bfloat16* __restrict__ wb, const float* __restrict__ p,
                                                   const float* __restrict__ x, const float* __restrict__ target,
                                                   int rows, int total, float* __restrict__ y, float* __restrict__ act,
                                                   float* __restrict__ gy, float* __restrict__ loss_part) {
  __shared__ float4 h1s[kH], h2s[kH], g2s[kH];  // unit j of the four rows
  __shared__ float sx[kRows][kIn];
  __shared__ float sgy[kRows][kOut], sloss[kRows];
  const int j = threadIdx.x, lane = j & 31, warp = j >> 5;
  const int r0 = blockIdx.x * kRows;
  const int nr = min(kRows, rows - r0);
  uint32_t w2[kH / 2];
  {
    const uint4* src = reinterpret_cast<const uint4*>(wb + kOffW2 + j * kH);
#pragma unroll
    for (int q = 0; q < kH / 8; ++q) {
      const uint4 v = src[q];
      w2[4 * q] = v.x;
      w2[4 * q + 1] = v.y;
      w2[4 * q + 2] = v.z;
      w2[4 * q + 3] = v.w;
    }
  }
  if (j < kRows * kIn) sx[j / kIn][j % kIn] = j / kIn < nr ? x[(size_t)r0 * kIn + j] : 0.f;
  float w1[kIn];
#pragma unroll
  for (int i = 0; i < kIn; ++i) w1[i] = __bfloat162float(wb[kOffW1 + j * kIn + i]);
  const float bb1 = p[kOffB1 + j], bb2 = p[kOffB2 + j];
  __syncthreads();
  float h1[kRows], h2[kRows];
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    float a = bb1;
#pragma unroll
    for (int i = 0; i < kIn; ++i) a = fmaf(w1[i], sx[r][i], a);
    h1[r] = tanhf(a);
  }
  h1s[j] = make_float4(h1[0], h1[1], h1[2], h1[3]);
  __syncthreads();
  float a[kRows] = {bb2, bb2, bb2, bb2};
#pragma unroll
  for (int k = 0; k < kH; k += 2) {
    const float wl = bf_lo(w2[k / 2]), wh = bf_hi(w2[k / 2]);
    const float4 u = h1s[k], v = h1s[k + 1];
    a[0] = fmaf(wh, v.x, fmaf(wl, u.x, a[0]));
    a[1] = fmaf(wh, v.y, fmaf(wl, u.y, a[1]));
    a[2] = fmaf(wh, v.z, fmaf(wl, u.z, a[2]));
    a[3] = fmaf(wh, v.w, fmaf(wl, u.w, a[3]));
  }
#pragma unroll
  for (int r = 0; r < kRows; ++r) h2[r] = tanhf(a[r]);
  h2s[j] = make_float4(h2[0], h2[1], h2[2], h2[3]);
  __syncthreads();
  {  // output layer: warp r sums row r
    float o0 = 0.f, o1 = 0.f;
#pragma unroll
    for (int q = 0; q < kH / 32; ++q) {
      const int k = lane + 32 * q;
      const float h = reinterpret_cast<const float*>(&h2s[k])[warp];
      o0 = fmaf(__bfloat162float(wb[kOffW3 + k]), h, o0);
      o1 = fmaf(__bfloat162float(wb[kOffW3 + kH + k]), h, o1);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) {
      o0 += __shfl_xor_sync(0xffffffffu, o0, o);
      o1 += __shfl_xor_sync(0xffffffffu, o1, o);
    }
    if (lane < kOut) {
      const float v = (lane == 0 ? o0 : o1) + p[kOffB3 + lane];
      const bool ok = warp < nr;
      if (!TRAIN) {
        if (ok) y[(size_t)(r0 + warp) * kOut + lane] = v;
      } else {
        // loss = sum_{r,o} (y - t)^2 / (total * kOut), over the batch's slabs; gy = d loss / d y
        const float scale = 1.f / (float)(total * kOut);
        const float d = ok ? v - target[(size_t)(r0 + warp) * kOut + lane] : 0.f;
        sgy[warp][lane] = 2.f * d * scale;
        if (ok) gy[(size_t)(r0 + warp) * kOut + lane] = 2.f * d * scale;
        const float l = d * d * scale;
        const float l1 = __shfl_xor_sync(0x3u, l, 1);
        if (lane == 0) sloss[warp] = l + l1;
      }
    }
  }
  if (!TRAIN) return;
  __syncthreads();
  if (j == 0) loss_part[blockIdx.x] = (sloss[0] + sloss[1]) + (sloss[2] + sloss[3]);
  const float w30 = __bfloat162float(wb[kOffW3 + j]), w31 = __bfloat162float(wb[kOffW3 + kH + j]);
  const size_t plane = (size_t)rows * kH;  // act: h1, h2, ga1, ga2, rows x 128 each
  float g2[kRows];
#pragma unroll
  for (int r = 0; r < kRows; ++r) {
    g2[r] = (w30 * sgy[r][0] + w31 * sgy[r][1]) * (1.f - h2[r] * h2[r]);
    if (r < nr) {
      float* row = act + (size_t)(r0 + r) * kH + j;
      row[0] = h1[r];
      row[plane] = h2[r];
      row[3 * plane] = g2[r];
    }
  }
  g2s[j] = make_float4(g2[0], g2[1], g2[2], g2[3]);
  __syncthreads();
  float g1[kRows] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 16
  for (int k = 0; k < kH; ++k) {  // column j of W2
    const float w = __bfloat162float(wb[kOffW2 + k * kH + j]);
    const float4 u = g2s[k];
    g1[0] = fmaf(w, u.x, g1[0]);
    g1[1] = fmaf(w, u.y, g1[1]);
    g1[2] = fmaf(w, u.z, g1[2]);
    g1[3] = fmaf(w, u.w, g1[3]);
  }
#pragma unroll
  for (int r = 0; r < kRows; ++r)
    if (r < nr) act[2 * plane + (size_t)(r0 + r) * kH + j] = g1[r] * (1.f - h1[r] * h1[r]);
}

// Parameter gradients: CTA (u, chunk) sums kGradRows rows for two hidden units: 128 x 2 entries of
// gW2 by four row groups of threads (added in order), the other parameters of the two units by a
// warp each. Every entry is written once, so nothing is cleared and no atomics are needed; with
// one chunk g is the result, else chunk c goes to its own copy and k_mlp_chunks adds them.
__global__ void __launch_bounds__(kGradThr) k_mlp_grad(const float* __restrict__ x, const float* __restrict__ act,
                                                       const float* __restrict__ gy, int rows, float* __restrict__ g_all,
                                                       const float* __restrict__ loss_part, int loss_parts,
                                                       float* __restrict__ loss) {
  __shared__ float part[4][kGradUnits][kH];
  float* g = g_all + (size_t)blockIdx.y * kParams;
  const size_t plane = (size_t)rows * kH;
  const float *h1 = act, *h2 = act + plane, *ga1 = act + 2 * plane, *ga2 = act + 3 * plane;
  const int j0 = blockIdx.x * kGradUnits;
  const int ra = blockIdx.y * kGradRows, rb = min(rows, ra + kGradRows);
  const int k = threadIdx.x & (kH - 1), u = (threadIdx.x >> 7) & 1, grp = threadIdx.x >> 8;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  float a = 0.f;
#pragma unroll 16
  for (int r = ra + grp; r < rb; r += 4) a = fmaf(ga2[(size_t)r * kH + j0 + u], h1[(size_t)r * kH + k], a);
  part[grp][u][k] = a;
  // warps 0..19: bias, input and output weights of the units; 20, 21: output biases; 22: the loss
  if (warp < 20) {
    const int uu = warp / 10, item = warp % 10, j = j0 + uu;
    float s = 0.f;
    for (int r = ra + lane; r < rb; r += 32) {
      if (item < 6) s = fmaf(ga1[(size_t)r * kH + j], x[(size_t)r * kIn + item], s);
      else if (item == 6) s += ga1[(size_t)r * kH + j];
      else if (item == 7) s += ga2[(size_t)r * kH + j];
      else s = fmaf(gy[(size_t)r * kOut + item - 8], h2[(size_t)r * kH + j], s);
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) {
      const int at = item < 6 ? kOffW1 + j * kIn + item : item == 6 ? kOffB1 + j : item == 7 ? kOffB2 + j : kOffW3 + (item - 8) * kH + j;
      g[at] = s;
    }
  } else if (warp < 22 && blockIdx.x == 0) {
    float s = 0.f;
    for (int r = ra + lane; r < rb; r += 32) s += gy[(size_t)r * kOut + warp - 20];
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0) g[kOffB3 + warp - 20] = s;
  } else if (warp == 22 && blockIdx.x == 0 && blockIdx.y == 0 && loss != nullptr) {
    double s = 0.0;  // (a lane adds rows / 128 parts one after another)
    for (int q = lane; q < loss_parts; q += 32) s += (double)loss_part[q];
    s = warp_sum(s);
    if (lane == 0) loss[0] = (float)s;
  }
  __syncthreads();
  if (grp == 0)
    g[kOffW2 + (j0 + u) * kH + k] = (part[0][u][k] + part[1][u][k]) + (part[2][u][k] + part[3][u][k]);
}

// first: the batch's first slab (else g holds the sum of those before).
__global__ void k_mlp_chunks(const float* __restrict__ g_all, int chunks, bool first, float* __restrict__ g) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < kParams; e += gridDim.x * blockDim.x) {
    float s = first ? g_all[e] : g[e];
    for (int c = first ? 1 : 0; c < chunks; ++c) s += g_all[(size_t)c * kParams + e];
    g[e] = s;
  }
}

// Adam on the FP32 master parameters, then the BF16 copy.
__global__ void k_mlp_adam(float* __restrict__ p, float* __restrict__ m, float* __restrict__ v,
                           const float* __restrict__ g, __nv_bfloat16* __restrict__ wb, float lr, float b1c, float b2c) {
  const float beta1 = 0.9f, beta2 = 0.999f, eps = 1e-8f;
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < kParams; e += gridDim.x * blockDim.x) {
    const float gr = g[e];
    const float mm = beta1 * m[e] + (1.f - beta1) * gr;
    const float vv = beta2 * v[e] + (1.f - beta2) * gr * gr;
    m[e] = mm;
    v[e] = vv;
    const float upd = lr * (mm / b1c) / (sqrtf(vv / b2c) + eps);
    const float w = p[e] - upd;
    p[e] = w;
    wb[e] = __float2bfloat16_rn(w);
  }
}

__global__ void k_mlp_round(const float* __restrict__ p, __nv_bfloat16* __restrict__ wb) {
  for (int e = blockIdx.x * blockDim.x + threadIdx.x; e < kParams; e += gridDim.x * blockDim.x)
    wb[e] = __float2bfloat16_rn(p[e]);
}

}  // namespace
}  // namespace hhl

struct hhl_mlp_s {
  float* p = nullptr;           // FP32 master parameters
  float* m = nullptr;           // Adam moments
  float* v = nullptr;
  float* g = nullptr;           // gradients of a training step
  __nv_bfloat16* wb = nullptr;  // BF16 copy used by forward / backward
  float* act = nullptr;         // activations and their gradients (4 x cap x 128), gy (cap x 2) of one slab
  float* lp = nullptr;          // loss partials of the batch, one per four rows
  float* gc = nullptr;          // per-chunk gradients of batches over kGradRows rows, one slab's
  int cap = 0, cap_parts = 0, cap_chunks = 0;
  int64_t step = 0;
};

namespace hhl {
namespace {

hhl_status mlp_grow(float** buf, int* cap, int want, size_t each, const char* what) {
  if (want <= *cap) return HHL_OK;
  if (*buf) cudaFree(*buf);
  *buf = nullptr;
  *cap = 0;
  if (cudaMalloc(buf, (size_t)want * each * sizeof(float)) != cudaSuccess) {
    cudaGetLastError();
    return fail(HHL_ERR_OOM, what);
  }
  *cap = want;
  return HHL_OK;
}

hhl_status mlp_reserve(hhl_mlp_s* n, int rows) {
  const int slab = std::min(rows, kSlabRows), chunks = (slab + kGradRows - 1) / kGradRows;
  hhl_status s = mlp_grow(&n->act, &n->cap, slab, 4 * kH + kOut, "MLP activation buffers");
  if (s == HHL_OK) s = mlp_grow(&n->lp, &n->cap_parts, (rows - 1) / kRows + 1, 1, "MLP loss buffer");
  if (s == HHL_OK && chunks > 1) s = mlp_grow(&n->gc, &n->cap_chunks, chunks, kParams, "MLP gradient buffers");
  return s;
}

hhl_status mlp_grad(hhl_mlp_s* n, const float* x, const float* t, int rows, float* g, float* loss, cudaStream_t st) {
  hhl_status s = mlp_reserve(n, rows);
  if (s != HHL_OK) return s;
  const int parts = (rows - 1) / kRows + 1;
  for (int64_t r0 = 0; r0 < rows; r0 += kSlabRows) {
    const int nr = (int)std::min<int64_t>(rows - r0, kSlabRows), chunks = (nr + kGradRows - 1) / kGradRows;
    const bool last = r0 + nr == rows;
    float* gy = n->act + (size_t)nr * 4 * kH;
    HHL_PROF_BEGIN(st);
    k_mlp_rows<true><<<(nr + kRows - 1) / kRows, kThr, 0, st>>>(n->wb, n->p, x + r0 * kIn, t + r0 * kOut, nr, rows, nullptr,
                                                               n->act, gy, n->lp + r0 / kRows);
    HHL_LAUNCH_CHECK("k_mlp_rows");
    const bool whole = rows <= kGradRows;  // one chunk: its sums are the gradient
    HHL_PROF_BEGIN(st);
    k_mlp_grad<<<dim3(kH / kGradUnits, chunks), kGradThr, 0, st>>>(x + r0 * kIn, n->act, gy, nr, whole ? g : n->gc, n->lp, parts,
                                                                  last ? loss : nullptr);
    HHL_LAUNCH_CHECK("k_mlp_grad");
    if (!whole) {
      HHL_PROF_BEGIN(st);
      k_mlp_chunks<<<(kParams + 255) / 256, 256, 0, st>>>(n->gc, chunks, r0 == 0, g);
      HHL_LAUNCH_CHECK("k_mlp_chunks");
    }
  }
  return HHL_OK;
}

}  // namespace
}  // namespace hhl

extern "C" {

hhl_status hhl_mlp_create(hhl_mlp_t* out) {
  using namespace hhl;
  if (out == nullptr) return fail(HHL_ERR_INVALID_ARG, "NULL out");
  *out = nullptr;
  hhl_mlp_s* n = new hhl_mlp_s();
  if (cudaMalloc(&n->p, kParams * sizeof(float)) != cudaSuccess || cudaMalloc(&n->m, kParams * sizeof(float)) != cudaSuccess ||
      cudaMalloc(&n->v, kParams * sizeof(float)) != cudaSuccess || cudaMalloc(&n->g, kParams * sizeof(float)) != cudaSuccess ||
      cudaMalloc(&n->wb, kParams * sizeof(__nv_bfloat16)) != cudaSuccess) {
    cudaGetLastError();
    hhl_mlp_destroy(n);
    return fail(HHL_ERR_OOM, "MLP parameter buffers");
  }
  cudaMemset(n->p, 0, kParams * sizeof(float));
  cudaMemset(n->m, 0, kParams * sizeof(float));
  cudaMemset(n->v, 0, kParams * sizeof(float));
  cudaMemset(n->wb, 0, kParams * sizeof(__nv_bfloat16));
  *out = n;
  return HHL_OK;
}

void hhl_mlp_destroy(hhl_mlp_t n) {
  if (n == nullptr) return;
  void* ptrs[] = {n->p, n->m, n->v, n->g, n->wb, n->act, n->lp, n->gc};
  for (void* q : ptrs)
    if (q) cudaFree(q);
  delete n;
}

hhl_status hhl_mlp_set_params(hhl_mlp_t n, const float* host_params, void* stream) {
  using namespace hhl;
  if (n == nullptr || host_params == nullptr) return fail(HHL_ERR_INVALID_ARG, "NULL argument");
  cudaStream_t st = (cudaStream_t)stream;
  HHL_CUDA_TRY(cudaMemcpyAsync(n->p, host_params, kParams * sizeof(float), cudaMemcpyHostToDevice, st));
  HHL_CUDA_TRY(cudaMemsetAsync(n->m, 0, kParams * sizeof(float), st));
  HHL_CUDA_TRY(cudaMemsetAsync(n->v, 0, kParams * sizeof(float), st));
  n->step = 0;
  HHL_PROF_BEGIN(st);
  k_mlp_round<<<(kParams + 255) / 256, 256, 0, st>>>(n->p, n->wb);
  HHL_LAUNCH_CHECK("k_mlp_round");
  HHL_CUDA_TRY(cudaStreamSynchronize(st));
  return HHL_OK;
}

hhl_status hhl_mlp_get_params(hhl_mlp_t n, float* host_params, void* stream) {
  using namespace hhl;
  if (n == nullptr || host_params == nullptr) return fail(HHL_ERR_INVALID_ARG, "NULL argument");
  cudaStream_t st = (cudaStream_t)stream;
  HHL_CUDA_TRY(cudaMemcpyAsync(host_params, n->p, kParams * sizeof(float), cudaMemcpyDeviceToHost, st));
  HHL_CUDA_TRY(cudaStreamSynchronize(st));
  return HHL_OK;
}

hhl_status hhl_mlp_forward(hhl_mlp_t n, const float* x_dev, int32_t rows, float* y_dev, void* stream) {
  using namespace hhl;
  if (n == nullptr || x_dev == nullptr || y_dev == nullptr || rows < 1) return fail(HHL_ERR_INVALID_ARG, "bad argument");
  cudaStream_t st = (cudaStream_t)stream;
  HHL_PROF_BEGIN(st);
  k_mlp_rows<false><<<(rows + kRows - 1) / kRows, kThr, 0, st>>>(n->wb, n->p, x_dev, nullptr, rows, rows, y_dev, nullptr,
                                                                nullptr, nullptr);
  HHL_LAUNCH_CHECK("k_mlp_rows");
  return HHL_OK;
}

hhl_status hhl_t0_predict(hhl_mlp_t n, const float* features_dev, int32_t rows, float* out_dev, void* stream) {
  return hhl_mlp_forward(n, features_dev, rows, out_dev, stream);
}

hhl_status hhl_mlp_gradients(hhl_mlp_t n, const float* x_dev, const float* t_dev, int32_t rows, float* grad_dev,
                             float* loss_dev, void* stream) {
  using namespace hhl;
  if (n == nullptr || x_dev == nullptr || t_dev == nullptr || grad_dev == nullptr || loss_dev == nullptr || rows < 1)
    return fail(HHL_ERR_INVALID_ARG, "bad argument");
  cudaStream_t st = (cudaStream_t)stream;
  // the gradient pass still reads the rows while it writes: a gradient laid over them is formed beside
  auto over = [&](const float* in, size_t each) {
    return in < grad_dev + kParams && grad_dev < in + (size_t)rows * each;
  };
  if (!over(x_dev, kIn) && !over(t_dev, kOut)) return mlp_grad(n, x_dev, t_dev, rows, grad_dev, loss_dev, st);
  hhl_status s = mlp_grad(n, x_dev, t_dev, rows, n->g, loss_dev, st);
  if (s == HHL_OK) HHL_CUDA_TRY(cudaMemcpyAsync(grad_dev, n->g, kParams * sizeof(float), cudaMemcpyDeviceToDevice, st));
  return s;
}

hhl_status hhl_mlp_train_step(hhl_mlp_t n, const float* x_dev, const float* t_dev, int32_t rows, float lr,
                              float* loss_dev, void* stream) {
  using namespace hhl;
  if (n == nullptr || x_dev == nullptr || t_dev == nullptr || loss_dev == nullptr || rows < 1 || !(lr > 0.f))
    return fail(HHL_ERR_INVALID_ARG, "bad argument");
  cudaStream_t st = (cudaStream_t)stream;
  hhl_status s = mlp_grad(n, x_dev, t_dev, rows, n->g, loss_dev, st);
  if (s != HHL_OK) return s;
  n->step += 1;
  const float b1c = 1.f - powf(0.9f, (float)n->step), b2c = 1.f - powf(0.999f, (float)n->step);
  HHL_PROF_BEGIN(st);
  k_mlp_adam<<<(kParams + 255) / 256, 256, 0, st>>>(n->p, n->m, n->v, n->g, n->wb, lr, b1c, b2c);
  HHL_LAUNCH_CHECK("k_mlp_adam");
  return HHL_OK;
}

}  // extern "C"
