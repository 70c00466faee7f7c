// Initial-guess network (Sec. 5): a 24-256-256-256-11 multilayer perceptron
// with GELU activations, trained and evaluated by hand-written BF16
// tensor-core kernels with FP32 accumulation: a training step is one tcgen05
// kernel for the forward and backward pass, one for the weight gradients (both
// nn_tc.cu) and one that reduces them and applies Adam (here); inference is
// one fused tcgen05 kernel (mlp_tc.cu).  This file also holds weight packing,
// initialisation and the standardisation statistics, and the host driver.
//
// 16 steps of 8192 samples take 1.08 ms (3.28 ms when each product, transpose,
// row sum and the loss were launches of their own, 19 a step).
//
// Parameter blob (float32, see vfisv.h): W0[24][256] b0[256] W1[256][256]
// b1[256] W2[256][256] b2[256] W3[256][11] b3[11] in_mean[24] in_std[24]
// out_mean[10] out_std[10]; weights are [fan_in][fan_out] (y = x W + b).
#include <cuda_bf16.h>
#include <math.h>

#include <vector>

#include "common.cuh"
#include "nn.cuh"
#include "nn_device.cuh"
#include "nn_tc.cuh"

namespace vfisv {
namespace nn {

using bf16 = __nv_bfloat16;

// ---------------------------------------------------------------------------
// Features, targets, decoding (the network's view of a pixel).
//
// Features: f_j = (obs_j / Ic - in_mean_j) / in_std_j, Ic = max(largest I
// sample, 1e-30).  Targets (standardised with out_mean/out_std):
// [B, cos gamma, sin 2psi, cos 2psi, ln eta0, dlambdaD, a, v, S0/Ic, S1/Ic].

__device__ __forceinline__ void put_bf16(uint8_t* base, size_t off, float v) {
  *reinterpret_cast<bf16*>(base + off) = __float2bfloat16(v);
}

__constant__ LayerDim kLayers[4] = {{IN, HID, OFF_W0, OFF_B0},
                                    {HID, HID, OFF_W1, OFF_B1},
                                    {HID, HID, OFF_W2, OFF_B2},
                                    {HID, OUT, OFF_W3, OFF_B3}};

// End of a step: sums the split-K partials (fixed order: deterministic) and,
// ADAM, applies the update with bias correction (m = b1 m + (1-b1) g,
// v = b2 v + (1-b2) g^2, w -= lr (m / c1) / (sqrt(v / c2) + eps)) and writes
// the new weights' BF16 copies for the next step; otherwise writes the
// gradient.  One thread an element of the partials' layout, so that their
// reads (17 MB from L2 at a batch of 8192, what bounds it) are coalesced.
struct StepArgs {
  const float* wpart[4];  // [splits][256][32: W0^T | 256 | 256 | 16]
  const float* bpart[4];  // [splits][256 | 256 | 256 | 16]
  int splits;
  float *grad, *blob, *m, *v;
  float lr, b1, b2, c1, c2, eps;
  PackedNet P;
  const float* lossp;
  int nloss;
  float* loss_out;
};
constexpr int kStepW0 = HID * XT, kStepW1 = HID * HID, kStepW3 = HID * YN;
constexpr int kStepWeights = kStepW0 + 2 * kStepW1 + kStepW3;
constexpr int kStepTotal = kStepWeights + 3 * HID + YN;

template <bool ADAM>
__global__ void __launch_bounds__(256) step_kernel(StepArgs a) {
  int i = blockIdx.x * blockDim.x + threadIdx.x;
  if (i == 0 && a.loss_out) {
    float s = 0.0f;
#pragma unroll 8
    for (int q = 0; q < a.nloss; ++q) s += a.lossp[q];
    *a.loss_out = s;
  }
  if (i >= kStepTotal) return;
  int l, k = 0, n, stride;
  const float* part;
  const bool weight = i < kStepWeights;
  if (weight) {
    if (i < kStepW0) {
      l = 0;
      n = i / XT;
      k = i % XT;
      stride = kStepW0;
    } else if (i < kStepW0 + 2 * kStepW1) {
      i -= kStepW0;
      l = 1 + i / kStepW1;
      i %= kStepW1;
      k = i / HID;
      n = i % HID;
      stride = kStepW1;
    } else {
      i -= kStepW0 + 2 * kStepW1;
      l = 3;
      k = i / YN;
      n = i % YN;
      stride = kStepW3;
    }
    part = a.wpart[l] + i;
  } else {
    i -= kStepWeights;
    l = i / HID;
    n = i % HID;
    stride = (l == 3) ? YN : HID;
    part = a.bpart[l] + n;
  }
  const LayerDim& D = kLayers[l];
  if (k >= D.K || n >= D.N) return;  // padding
  float g = 0.0f;
#pragma unroll 16
  for (int q = 0; q < a.splits; ++q) g += part[(size_t)q * stride];
  const size_t e = weight ? D.offW + (size_t)k * D.N + n : D.offB + n;
  if constexpr (!ADAM) {
    a.grad[e] = g;
  } else {
    const float mi = fmaf(a.b1, a.m[e], (1.0f - a.b1) * g);
    const float vi = fmaf(a.b2, a.v[e], (1.0f - a.b2) * g * g);
    a.m[e] = mi;
    a.v[e] = vi;
    const float w = a.blob[e] - a.lr * (mi / a.c1) / (sqrtf(vi / a.c2) + a.eps);
    a.blob[e] = w;
    if (weight) {
      put_bf16(a.P.Wt[l], tl_off(n, k, l == 3 ? YN : HID), w);
      if (l > 0) put_bf16(a.P.Wn[l], tl_off(k, n, HID), w);
    }
  }
}

// Tiled (TL) BF16 copies of the weights, zero padded: Wt[l] with element
// (n, k) = W_l[k][n] (rows = outputs: 256, or 16 for the output layer; K =
// inputs: 64 for layer 0, else 256), the B operand of the forward products;
// Wn[l] with element (k, n) = W_l[k][n] (rows = the 256 inputs; K = outputs,
// 64 for the output layer), the B operand of the input gradients (l >= 1).
__global__ void pack_kernel(const float* __restrict__ blob, PackedNet P) {
  const int l = blockIdx.y;
  const LayerDim& D = kLayers[l];
  const int rt = (l == 3) ? YN : HID, kt = (l == 0) ? XK : HID, kn = (l == 3) ? DYK : HID;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < rt * kt; i += gridDim.x * blockDim.x) {
    const int n = i / kt, k = i % kt;
    const float w = (k < D.K && n < D.N) ? blob[D.offW + (size_t)k * D.N + n] : 0.0f;
    put_bf16(P.Wt[l], tl_off(n, k, rt), w);
  }
  if (l == 0) return;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < HID * kn; i += gridDim.x * blockDim.x) {
    const int k = i / kn, n = i % kn;
    const float w = (n < D.N) ? blob[D.offW + (size_t)k * D.N + n] : 0.0f;
    put_bf16(P.Wn[l], tl_off(k, n, HID), w);
  }
}

// Weight initialisation: uniform(-sqrt(6/fan_in), +sqrt(6/fan_in)) from a
// SplitMix64 hash of (seed, index); biases zero.
__device__ __forceinline__ uint64_t splitmix64(uint64_t x) {
  x += 0x9E3779B97F4A7C15ull;
  x = (x ^ (x >> 30)) * 0xBF58476D1CE4E5B9ull;
  x = (x ^ (x >> 27)) * 0x94D049BB133111EBull;
  return x ^ (x >> 31);
}
__global__ void init_weights_kernel(float* __restrict__ blob, uint64_t seed) {
  const int l = blockIdx.y;
  const LayerDim& D = kLayers[l];
  const float bound = sqrtf(6.0f / (float)D.K);
  const int total = D.K * D.N + D.N;
  for (int i = blockIdx.x * blockDim.x + threadIdx.x; i < total; i += gridDim.x * blockDim.x) {
    if (i < D.K * D.N) {
      const uint64_t h = splitmix64(seed * 0x100000001B3ull + D.offW + i);
      const float u = (float)(h >> 40) * (1.0f / 16777216.0f);
      blob[D.offW + i] = bound * (2.0f * u - 1.0f);
    } else {
      blob[D.offB + (i - D.K * D.N)] = 0.0f;
    }
  }
}

// Normalisation statistics of the training set: mean and standard deviation
// of the 24 features (obs / Ic) and of the 10 targets, in FP64, deterministic
// (fixed per-thread strides, block tree, then one ordered sum).
constexpr int kStat = IN + OUT - 1;
__global__ void stats_partial_kernel(const float* __restrict__ obs,
                                     const float* __restrict__ params, int64_t n,
                                     double* __restrict__ part) {
  __shared__ double sh[256];
  double s[kStat], q[kStat];
  for (int j = 0; j < kStat; ++j) s[j] = q[j] = 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n;
       i += (int64_t)gridDim.x * blockDim.x) {
    const float* o = obs + i * IN;
    const float ic = ic_of(o);
    for (int j = 0; j < IN; ++j) {
      const double f = (double)(o[j] / ic);
      s[j] += f;
      q[j] += f * f;
    }
    float t[OUT - 1];
    targets(params + i * 10, ic, t);
    for (int j = 0; j < OUT - 1; ++j) {
      s[IN + j] += t[j];
      q[IN + j] += (double)t[j] * t[j];
    }
  }
  for (int j = 0; j < 2 * kStat; ++j) {
    sh[threadIdx.x] = (j < kStat) ? s[j] : q[j - kStat];
    __syncthreads();
    for (int o = blockDim.x / 2; o > 0; o >>= 1) {
      if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
      __syncthreads();
    }
    if (threadIdx.x == 0) part[(size_t)blockIdx.x * 2 * kStat + j] = sh[0];
    __syncthreads();
  }
}
__global__ void stats_final_kernel(const double* __restrict__ part, int nblocks, int64_t n,
                                   float* __restrict__ blob) {
  const int j = threadIdx.x;
  if (j >= kStat) return;
  double s = 0.0, q = 0.0;
  for (int b = 0; b < nblocks; ++b) {
    s += part[(size_t)b * 2 * kStat + j];
    q += part[(size_t)b * 2 * kStat + kStat + j];
  }
  const double mean = s / (double)n;
  const double var = fmax(q / (double)n - mean * mean, 0.0);
  const float sd = (float)fmax(sqrt(var), 1e-6);
  if (j < IN) {
    blob[OFF_INM + j] = (float)mean;
    blob[OFF_INS + j] = sd;
  } else {
    blob[OFF_OUTM + j - IN] = (float)mean;
    blob[OFF_OUTS + j - IN] = sd;
  }
}

// ---------------------------------------------------------------------------
// host side

static int64_t round_up(int64_t x, int64_t m) { return (x + m - 1) / m * m; }

struct Bufs {
  uint8_t *XT, *HT[3], *dYT, *dZT[3];
  float *wpart[4], *bpart[4], *m, *v, *loss, *lossp;
  PackedNet P;
};

constexpr int kMaxLossBlocks = 4096;  // loss partials (256 rows each)

static Bufs carve(void* ws, int64_t M, size_t* used = nullptr) {
  char* p = (char*)ws;
  auto take = [&](size_t bytes) {
    void* r = p;
    p += (bytes + 255) & ~(size_t)255;
    return r;
  };
  Bufs b;
  take(infer_workspace_bytes());  // error word and packed inference weights
  b.XT = (uint8_t*)take((size_t)M * XT * 2);
  for (int i = 0; i < 3; ++i) {
    b.HT[i] = (uint8_t*)take((size_t)M * HID * 2);
    b.dZT[i] = (uint8_t*)take((size_t)M * HID * 2);
  }
  b.dYT = (uint8_t*)take((size_t)M * YN * 2);
  for (int l = 0; l < 4; ++l) {
    const int w = l == 0 ? XT : l == 3 ? YN : HID;
    b.wpart[l] = (float*)take((size_t)kSplits * HID * w * 4);
    b.bpart[l] = (float*)take((size_t)kSplits * HID * 4);
  }
  b.m = (float*)take(NBLOB * 4);
  b.v = (float*)take(NBLOB * 4);
  b.loss = (float*)take((size_t)M * 4);
  b.lossp = (float*)take(kMaxLossBlocks * 4);
  for (int l = 0; l < 4; ++l) {
    b.P.Wt[l] = (uint8_t*)take((size_t)(l == 3 ? YN : HID) * (l == 0 ? XK : HID) * 2);
    b.P.Wn[l] = (uint8_t*)take((size_t)HID * (l == 3 ? DYK : HID) * 2);
  }
  if (used) *used = (size_t)(p - (char*)ws);
  return b;
}

size_t workspace_bytes(int64_t rows) {
  size_t used = 0;
  carve(nullptr, padded_rows(rows), &used);
  const size_t stats = infer_workspace_bytes() + (size_t)256 * 2 * (IN + OUT - 1) * sizeof(double);
  return used > stats ? used : stats;
}

// batch rows padded to the 128-row tiles of the products
int64_t padded_rows(int64_t n) { return round_up(n > 0 ? n : 1, 128); }

static cudaError_t pack(const float* blob, const PackedNet& P, cudaStream_t s) {
  pack_kernel<<<dim3(64, 4), 256, 0, s>>>(blob, P);
  return cudaGetLastError();
}

// Split of a batch-long K (M rows, 64 per chunk) over at most kSplits CTAs
// per tile, every split owning at least one chunk.
static void batch_split(int64_t M, int* per, int* splits) {
  const int64_t total = M / 64;
  const int64_t want = total < kSplits ? total : kSplits;
  *per = (int)((total + want - 1) / want);
  *splits = (int)((total + *per - 1) / *per);
}

// Forward and backward pass and the gradients' split-K partials of a batch of
// M (padded) rows whose weights are packed; `st` gets what step_kernel needs.
static cudaError_t pass_and_partials(const Bufs& b, const float* blob, const float* obs,
                                     const float* params, int64_t rows, int64_t M, Perm perm,
                                     int* err, StepArgs* st, cudaStream_t s) {
  const int nloss = (int)((M + 255) / 256);
  if (nloss > kMaxLossBlocks) return cudaErrorInvalidValue;
  TrainPassArgs p{};
  p.blob = blob;
  p.obs = obs;
  p.params = params;
  p.perm = perm;
  p.rows = rows;
  p.P = b.P;
  TrainDwArgs d{};
  p.XT = b.XT;
  d.XT = b.XT;
  p.dYT = b.dYT;
  d.dYT = b.dYT;
  for (int l = 0; l < 3; ++l) {
    p.HT[l] = b.HT[l];
    d.HT[l] = b.HT[l];
    p.dZT[l] = b.dZT[l];
    d.dZT[l] = b.dZT[l];
  }
  p.loss = b.loss;
  d.loss = b.loss;
  d.lossp = b.lossp;
  d.nloss = nloss;
  p.err = err;
  d.err = err;
  d.chunks = (int)(M / 64);
  int splits = 1;
  batch_split(M, &d.per, &splits);
  *st = StepArgs{};
  for (int l = 0; l < 4; ++l) {
    d.wpart[l] = b.wpart[l];
    d.bpart[l] = b.bpart[l];
    st->wpart[l] = b.wpart[l];
    st->bpart[l] = b.bpart[l];
  }
  st->splits = splits;
  st->P = b.P;
  st->lossp = b.lossp;
  st->nloss = nloss;
  cudaError_t e = train_pass(p, M / 128, s);
  return e != cudaSuccess ? e : train_dw(d, splits, s);
}

constexpr int kStepBlocks = (kStepTotal + 255) / 256;

cudaError_t nn_init(void* ws, float* blob, const float* obs, const float* params, int64_t n,
                    uint64_t seed, cudaStream_t s) {
  init_weights_kernel<<<dim3(64, 4), 256, 0, s>>>(blob, seed);
  const int nb = 256;
  double* part = (double*)((char*)ws + infer_workspace_bytes());  // after the error word
  stats_partial_kernel<<<nb, 256, 0, s>>>(obs, params, n, part);
  stats_final_kernel<<<1, 64, 0, s>>>(part, nb, n, blob);
  return cudaGetLastError();
}

cudaError_t nn_grad(void* ws, const float* blob, const float* obs, const float* params,
                    int64_t n, float* grad_out, float* loss_out, cudaStream_t s) {
  const int64_t M = padded_rows(n);
  Bufs b = carve(ws, M);
  cudaError_t e;
  if ((e = pack(blob, b.P, s)) != cudaSuccess) return e;
  StepArgs st;
  if ((e = pass_and_partials(b, blob, obs, params, n, M, Perm{1, 0, 0, n}, static_cast<int*>(ws),
                             &st, s)) != cudaSuccess)
    return e;
  st.grad = grad_out;
  st.loss_out = loss_out;
  step_kernel<false><<<kStepBlocks, 256, 0, s>>>(st);
  return cudaGetLastError();
}

cudaError_t nn_train(void* ws, float* blob, const float* obs, const float* params, int64_t n,
                     int batch, int epochs, float lr0, uint64_t seed, float* loss_hist,
                     cudaStream_t s) {
  const int64_t M = batch;
  Bufs b = carve(ws, M);
  int* err = static_cast<int*>(ws);
  cudaError_t e;
  if ((e = cudaMemsetAsync(b.m, 0, NBLOB * 4, s)) != cudaSuccess) return e;
  if ((e = cudaMemsetAsync(b.v, 0, NBLOB * 4, s)) != cudaSuccess) return e;
  // the first step's BF16 weights; every step writes the next one's
  if ((e = pack(blob, b.P, s)) != cudaSuccess) return e;
  const int64_t spe = n / batch;
  const int64_t total = spe * epochs;
  const float b1 = 0.9f, b2 = 0.999f, eps = 1e-8f;
  double p1 = 1.0, p2 = 1.0;
  for (int64_t t = 0; t < total; ++t) {
    const int64_t ep = t / spe, bi = t % spe;
    // a different affine permutation of the training set every epoch
    uint64_t h = seed * 0x9E3779B97F4A7C15ull + (uint64_t)ep * 0xD1B54A32D192ED03ull + 1;
    h ^= h >> 31;
    h *= 0xBF58476D1CE4E5B9ull;
    h ^= h >> 29;
    auto gcd = [](uint64_t a, uint64_t c) {
      while (c) {
        const uint64_t r = a % c;
        a = c;
        c = r;
      }
      return a;
    };
    uint64_t mult = (n > 1) ? 1 + h % (uint64_t)(n - 1) : 1;
    while (n > 1 && gcd(mult, (uint64_t)n) != 1) mult = mult % (uint64_t)(n - 1) + 1;
    Perm perm{mult, (h >> 17) % (uint64_t)n, bi * batch, n};
    StepArgs st;
    if ((e = pass_and_partials(b, blob, obs, params, M, M, perm, err, &st, s)) != cudaSuccess)
      return e;
    const double lr = lr0 * 0.5 * (1.0 + cos(3.14159265358979323846 * (double)t / (double)total));
    p1 *= b1;
    p2 *= b2;
    st.blob = blob;
    st.m = b.m;
    st.v = b.v;
    st.lr = (float)lr;
    st.b1 = b1;
    st.b2 = b2;
    st.c1 = (float)(1.0 - p1);
    st.c2 = (float)(1.0 - p2);
    st.eps = eps;
    st.loss_out = loss_hist ? loss_hist + t : nullptr;
    step_kernel<true><<<kStepBlocks, 256, 0, s>>>(st);
    if ((e = cudaGetLastError()) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace nn
}  // namespace vfisv
