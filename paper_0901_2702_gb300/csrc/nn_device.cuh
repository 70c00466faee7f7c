// Per-pixel device pieces of the initial-guess network shared by the
// training kernels (nn.cu) and the fused tensor-memory inference kernel
// (mlp_tc.cu): the activation, the continuum estimate and the decoding of the
// network outputs into an initial model.
#pragma once

#include <math.h>

#include "f32x2.cuh"
#include "nn.cuh"

namespace vfisv {
namespace nn {

// GELU(x) = x Phi(x) = 0.5 x (1 + erf(x / sqrt(2))) and its derivative Phi(x) +
// x phi(x), two at a time: what surrounds the error function and the
// exponential in packed instructions (the scalar ones' roundings).
__device__ __forceinline__ f2 gelu2(f2 x) {
  const f2 t = f2_mul(x, f2_dup(0.70710678118654752f));
  const f2 e = f2_pack(erff(f2_lo(t)), erff(f2_hi(t)));
  return f2_mul(f2_mul(f2_dup(0.5f), x), f2_add(f2_dup(1.0f), e));
}
__device__ __forceinline__ f2 gelu_grad2(f2 x) {
  const f2 t = f2_mul(x, f2_dup(0.70710678118654752f));
  const f2 e = f2_pack(erff(f2_lo(t)), erff(f2_hi(t)));
  const f2 cdf = f2_mul(f2_dup(0.5f), f2_add(f2_dup(1.0f), e));
  const f2 q = f2_mul(f2_mul(f2_dup(-0.5f), x), x);
  const f2 pdf = f2_mul(f2_dup(0.39894228040143268f), f2_pack(expf(f2_lo(q)), expf(f2_hi(q))));
  return f2_fma(x, pdf, cdf);
}

// Continuum estimate: the largest of the six Stokes I samples (at least 1e-30).
__device__ __forceinline__ float ic_of(const float* o) {
  float ic = -INFINITY;
#pragma unroll
  for (int j = 0; j < 6; ++j) ic = fmaxf(ic, o[j]);
  return fmaxf(ic, 1e-30f);
}

// mult < n, offset + m < 2n and n < 2^31 keep the product inside 64 bits.
__device__ __forceinline__ int64_t sample_of(int64_t m, const Perm& p) {
  return (int64_t)((p.mult * (uint64_t)(p.offset + m) + p.add) % (uint64_t)p.n);
}

// Training targets of a parameter vector.
__device__ __forceinline__ void targets(const float* p, float ic, float (&t)[OUT - 1]) {
  const float g = p[1] * 0.017453292519943295f, ps = p[2] * 0.034906585039886591f;
  t[0] = p[0];
  t[1] = cosf(g);
  t[2] = sinf(ps);
  t[3] = cosf(ps);
  t[4] = logf(p[3]);
  t[5] = p[4];
  t[6] = p[5];
  t[7] = p[6];
  t[8] = p[7] / ic;
  t[9] = p[8] / ic;
}

// Loss of a sample (the regression of Sec. 5 plus the confidence output) with
// outputs y[0..10] and parameters p, and its gradient d = dL/dy for a batch of
// `rows` samples.
__device__ __forceinline__ float loss_row(const float* y, const float* p, float ic,
                                          const float* mean, const float* std, float rows,
                                          float* d) {
  float t[OUT - 1];
  targets(p, ic, t);
  const float invn = 1.0f / rows;
  float e[OUT - 1], mse = 0.0f;
#pragma unroll
  for (int o = 0; o < OUT - 1; ++o) {
    const float ts = (t[o] - mean[o]) / std[o];
    e[o] = y[o] - ts;
    mse = fmaf(e[o], e[o], mse);
  }
  const float c = logf(mse / (OUT - 1) + 1e-4f);
  const float ec = y[OUT - 1] - c;
#pragma unroll
  for (int o = 0; o < OUT - 1; ++o) d[o] = 2.0f * e[o] * invn / (OUT - 1);
  d[OUT - 1] = 2.0f * ec * invn;
  return mse * invn / (OUT - 1) + ec * ec * invn;
}

// Network outputs y[0..10] (standardised, bias included) -> initial model
// p[0..9]; the inverse of the training targets [B, cos gamma, sin 2psi,
// cos 2psi, ln eta0, dlambdaD, a, v, S0/Ic, S1/Ic].
__device__ __forceinline__ void decode_row(const float* y, float ic, float mu,
                                           const float* out_mean, const float* out_std,
                                           float* p) {
  float t[OUT - 1];
#pragma unroll
  for (int o = 0; o < OUT - 1; ++o) t[o] = fmaf(y[o], out_std[o], out_mean[o]);
  p[0] = fmaxf(t[0], 0.0f);
  p[1] = acosf(fminf(fmaxf(t[1], -1.0f), 1.0f)) * 57.295779513082321f;
  float ps = 0.5f * atan2f(t[2], t[3]) * 57.295779513082321f;
  if (ps < 0.0f) ps += 180.0f;
  p[2] = ps;
  p[3] = expf(t[4]);
  p[4] = t[5];
  p[5] = t[6];
  p[6] = t[7];
  p[7] = t[8] * ic;
  p[8] = t[9] * ic / mu;
  p[9] = 1.0f;
}

}  // namespace nn
}  // namespace vfisv
