// Wide-instrument path: inputs sampled by many narrow instrument profiles
// over a fine synthesis grid (spectrograph-shaped data, e.g. 112 samples x 4
// Stokes parameters from 448 grid points), where the filter-position kernels'
// register accumulators (rows x Stokes x filters per thread) cannot hold the
// whole convolution.  One pixel per warp:
//   1. the fine grid is walked in chunks of 64 points; each lane evaluates
//      two points, packed (synthesis and, for the inversion, the six Jacobian
//      rows of Secs. 3-4, the same per-point arithmetic as the filter
//      kernels);
//   2. the instrument profiles are applied.  In the inversion a lane owns one
//      of the 28 rows; where the samples' bands start one group of four points
//      after another (a uniform grid), it slides over the groups with the up
//      to eight samples that meet the current one in registers, each loaded
//      row value serving all of them.  Other instruments spread the samples
//      that meet a chunk over the lanes.  The synthesis, with four rows,
//      spreads the samples over the lanes too, over the whole grid at once;
//   3. the inversion forms chi2 (Eq. 1; compensated FP32 partial sums,
//      combined and compared in FP64) and, after an accepted step, J^T W J
//      and J^T W r, reduced across the warp;
//   4. the FP64 damped solve (Eqs. 4-5) runs spread over the warp's lanes;
//      the covariance is left to the batched covariance kernel.
// The instrument table is compacted on the device into bands (first point,
// length, weights) and, where they are regular, windows (the weights of the
// eight groups from a sample's first one), staged in shared memory by TMA.
#include "common.cuh"
#include "me_pair.cuh"
#include "solve.cuh"

namespace vfisv {

constexpr int kWMaxF = 128;          // samples per Stokes parameter
constexpr int kWBand = 32;           // fine points per instrument profile
constexpr int kWMaxLam = 1024;       // fine grid points
constexpr int kWChunk = 64;          // fine points per chunk: two per lane
constexpr int kWMaxChunks = kWMaxLam / kWChunk;
constexpr int kWWarps = 8;           // pixels in flight per CTA at most
constexpr int kWBand4 = kWBand + 4;  // a band starting on a multiple of 4, padded to 4
constexpr int kWBandStride = kWBand4 + 4;  // [lo4, n4, pad, pad, w[36]] per sample
constexpr int kWWin = 8;             // groups of four points a window holds
constexpr int kWWinStride = 4 * kWWin;

// Compacted table, in 16-byte pieces: header [window groups in use (0: not
// regular), first group of sample 0's window, 0, 0] (int); tau[nf]; the fine
// grid x[nlam]; windows, row sg + 7 the weights of the sample whose window
// starts with group sg (sg from -7 to the last group; zeros where there is
// none); bands [nf][kWBandStride]; the active sample range of each chunk
// [kWMaxChunks][2] (int).
__host__ __device__ inline int up4(int n) { return (n + 3) & ~3; }
__host__ __device__ inline int wide_groups(int nlam) { return (nlam + 3) / 4; }
__host__ __device__ inline int wide_x_at(int nf) { return 4 + up4(nf); }
__host__ __device__ inline int wide_common(int nf, int nlam) { return wide_x_at(nf) + up4(nlam); }
// (windows past the last group up to a whole half chunk of eight)
__host__ __device__ inline int wide_groups8(int nlam) { return (nlam + 31) / 32 * 8; }
__host__ __device__ inline int wide_win_floats(int nlam) {
  return (wide_groups8(nlam) + kWWin - 1) * kWWinStride;
}
__host__ __device__ inline int wide_band_floats(int nf) {
  return nf * kWBandStride + 2 * kWMaxChunks;
}
__host__ __device__ inline int wide_table_floats(int nf, int nlam) {
  return wide_common(nf, nlam) + wide_win_floats(nlam) + wide_band_floats(nf);
}

__global__ void wide_pack_kernel(const float* __restrict__ filters, int nf,
                                 const float* __restrict__ wl, int nlam,
                                 float* __restrict__ table, int* __restrict__ err) {
  __shared__ int slo[kWMaxF], shi[kWMaxF];
  __shared__ int start, width;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* win = table + wide_common(nf, nlam);
  float* bands = win + wide_win_floats(nlam);
  // a window reaches past its sample's band, with zero weights, and the points
  // there must not come out as NaN: no windows on a grid with NaN or far-off
  // values (padding; up to 1e12 mA the squares stay in range)
  bool near = true;
  for (int i = threadIdx.x; i < nlam; i += blockDim.x) near = near && fabsf(wl[i]) < 1e12f;
  for (int k = warp; k < nf; k += blockDim.x >> 5) {
    const float* row = filters + (size_t)k * nlam;
    // first and last non-zero point; tau in a fixed order (lane-strided
    // partial sums, then a shuffle tree)
    int lo = nlam, hi = -1;
    float s = 0.0f;
    for (int i = lane; i < nlam; i += 32) {
      const float t = row[i];
      if (t != 0.0f) {
        lo = min(lo, i);
        hi = max(hi, i);
      }
      s += t;
    }
    for (int o = 16; o > 0; o >>= 1) {
      lo = min(lo, __shfl_xor_sync(0xffffffffu, lo, o));
      hi = max(hi, __shfl_xor_sync(0xffffffffu, hi, o));
      s += __shfl_xor_sync(0xffffffffu, s, o);
    }
    const int n = (hi >= lo) ? hi - lo + 1 : 0;
    if (n > kWBand && lane == 0) atomicExch(err, VFISV_E_UNSUPPORTED);
    // the band starts on a multiple of 4 (aligned float4 reads) and its
    // length is padded to a multiple of 4 with the zeros around it
    const int lo4 = (n > 0) ? (lo & ~3) : 0;
    const int n4 = (n > 0 && n <= kWBand) ? ((hi - lo4 + 1) + 3) & ~3 : 0;
    float* b = bands + (size_t)k * kWBandStride;
    if (lane == 0) {
      b[0] = __int_as_float(lo4);
      b[1] = __int_as_float(n4);
      b[2] = b[3] = 0.0f;
      table[4 + k] = s;  // tau
      slo[k] = lo4;
      shi[k] = lo4 + n4;  // exclusive
    }
    for (int t = lane; t < kWBand4; t += 32)
      b[4 + t] = (t < n4 && lo4 + t < nlam) ? row[lo4 + t] : 0.0f;
  }
  const bool ordinary = __syncthreads_and(near);
  // regular bands: sample k's within the window of groups k + start, k +
  // start + width - 1, for every sample
  if (warp == 0) {
    int g0 = 1 << 20, g1 = -(1 << 20);
    for (int k = lane; k < nf; k += 32)
      if (shi[k] > slo[k]) g0 = min(g0, slo[k] / 4 - k);
    for (int o = 16; o > 0; o >>= 1) g0 = min(g0, __shfl_xor_sync(0xffffffffu, g0, o));
    for (int k = lane; k < nf; k += 32)
      if (shi[k] > slo[k]) g1 = max(g1, shi[k] / 4 - k);
    for (int o = 16; o > 0; o >>= 1) g1 = max(g1, __shfl_xor_sync(0xffffffffu, g1, o));
    if (lane == 0) {
      // (every sample's window meets the grid: kernels for 7 and 8 groups)
      const bool ok = ordinary && g1 > g0 && g1 - g0 <= kWWin &&
                      g0 > (g1 - g0 < kWWin ? -(kWWin - 1) : -kWWin) &&
                      g0 + nf <= wide_groups(nlam);
      start = g0;
      width = ok ? g1 - g0 : 0;
      int* h = reinterpret_cast<int*>(table);
      h[0] = width;
      h[1] = start;
      h[2] = h[3] = 0;
    }
  }
  __syncthreads();
  if (width)
    for (int t = threadIdx.x; t < wide_win_floats(nlam); t += blockDim.x) {
      const int sg = t / kWWinStride - (kWWin - 1), k = sg - start;
      const int i = 4 * sg + t % kWWinStride;  // fine point of this weight
      float w = 0.0f;
      if (k >= 0 && k < nf && i >= slo[k] && i < shi[k] && i < nlam)
        w = filters[(size_t)k * nlam + i];
      win[t] = w;
    }
  // samples whose band meets each chunk: [first, last] (their hull)
  int* ch = reinterpret_cast<int*>(bands + nf * kWBandStride);
  for (int c = warp; c < kWMaxChunks; c += blockDim.x >> 5) {
    const int c0 = c * kWChunk, c1 = c0 + kWChunk;
    int kf = 1 << 30, kl = -1;
    for (int k = lane; k < nf; k += 32)
      if (slo[k] < c1 && shi[k] > c0 && shi[k] > slo[k]) {
        kf = min(kf, k);
        kl = max(kl, k);
      }
    for (int o = 16; o > 0; o >>= 1) {
      kf = min(kf, __shfl_xor_sync(0xffffffffu, kf, o));
      kl = max(kl, __shfl_xor_sync(0xffffffffu, kl, o));
    }
    if (lane == 0) {
      ch[2 * c] = (kl >= 0) ? kf : 0;
      ch[2 * c + 1] = kl;
    }
  }
  for (int i = threadIdx.x; i < up4(nlam); i += blockDim.x)
    table[wide_x_at(nf) + i] = i < nlam ? wl[i] : 0.0f;
  for (int k = nf + threadIdx.x; k < up4(nf); k += blockDim.x) table[4 + k] = 0.0f;
}

// The inversion's buffer of a warp: one chunk of the 28 rows (row stride 68:
// the lanes' 16-byte reads of their rows meet different banks).
constexpr int kWRows = 4 * kRows;
constexpr int kWRowStride = kWChunk + 4;
constexpr int kWBuf = kWRows * kWRowStride;
// rows of the accumulators: an odd stride, for lanes owning rows and lanes
// owning samples alike
__host__ __device__ inline int wide_acc_stride(int nf) { return nf | 1; }

// Puts the 28 values of two points (columns i, i + 1 of the buffer) there.
struct WidePut {
  float* col;
  f2 iD;
  __device__ __forceinline__ void put(int v, f2 x) {
    *reinterpret_cast<unsigned long long*>(col + v * kWRowStride) = x.v;
  }
  __device__ __forceinline__ void unit(f2 yI, f2 yQ, f2 yU, f2 yV) {
    put(0, yI);
    put(1, yQ);
    put(2, yU);
    put(3, yV);
  }
  __device__ __forceinline__ void scale(f2 d) { iD = d; }
  __device__ __forceinline__ void rows(int S, f2 vB, f2 vG, f2 vE, f2 vD, f2 vA, f2 vV) {
    put(4 * kRowB + S, f2_mul(iD, vB));
    put(4 * kRowG + S, f2_mul(iD, vG));
    put(4 * kRowE + S, f2_mul(iD, vE));
    put(4 * kRowD + S, f2_mul(iD, vD));
    put(4 * kRowA + S, f2_mul(iD, vA));
    put(4 * kRowV + S, f2_mul(iD, vV));
  }
};

// The rows of the chunk at c0 into the buffer, two points a lane; zeros past
// the grid.
__device__ __forceinline__ void wide_chunk(const Weideman& W, const PixK& P, const float* xg,
                                           int c0, int nlam, float* buf, int lane) {
  __syncwarp();
  const int i = c0 + 2 * lane;
  WidePut put{buf + 2 * lane, {}};
  lambda_pair<true>(W, P, f2_pack(xg[min(i, nlam - 1)], xg[min(i + 1, nlam - 1)]), put);
  if (c0 + kWChunk > nlam) {
#pragma unroll 1
    for (int v = 0; v < kWRows; ++v) {
      float* row = buf + v * kWRowStride + 2 * lane;
      if (i >= nlam) row[0] = 0.0f;
      if (i + 1 >= nlam) row[1] = 0.0f;
    }
  }
  __syncwarp();
}

// Filtered rows of one pixel into accs[v * wide_acc_stride + k], v = 4 r +
// Stokes (row r: Stokes, then the six Jacobian rows before their per-pixel
// scale factors), for every sample k.  A sample's sum is formed chunk by
// chunk of 64 points, a chunk's part first.
//
// With windows of WD groups: lane v slides over the groups of its row.  The
// sample whose window starts with group sg sits in slot sg mod 8 of a[] and
// tot[] (static: a half chunk is eight groups).  A group of the row is loaded
// once for the WD samples that meet it, their weights are broadcasts: 40
// instructions a group, 4.5 k a pass against 10 k with a sample a lane, 28
// loads of four conflict-free rows for its 112 sums and a third of the lanes
// idle.  Instruction fetch bounds the kernel now (about one stall an issue:
// warps at different places of 20 KB of loop); rolling the pass' loops to
// half the code cost more instructions than it saved (43.3 -> 48.0 ms).
template <int WD>
__device__ __forceinline__ void wide_pass_windows(const Weideman& W, const PixK& P,
                                                  const float* xg, const float* win, int g0,
                                                  int nf, int nlam, float* buf, float* accs,
                                                  int lane) {
  const int v = min(lane, kWRows - 1);  // the last lanes follow along
  const int G = wide_groups8(nlam), AS = wide_acc_stride(nf);
  float* out = accs + v * AS;
  float a[kWWin], tot[kWWin];
#pragma unroll
  for (int u = 0; u < kWWin; ++u) a[u] = tot[u] = 0.0f;
  const float* wp = win + (kWWin - 1) * kWWinStride;  // window row of the current group
#pragma unroll 1
  for (int c0 = 0; c0 < nlam; c0 += kWChunk) {
    wide_chunk(W, P, xg, c0, nlam, buf, lane);
#pragma unroll 1
    for (int half = 0; half < 2; ++half) {
      const int gb = c0 / 4 + half * kWWin;  // first group
      if (gb >= G) break;
      const float* xb = buf + v * kWRowStride + 4 * kWWin * half;
      // (the block's results are stored behind it, so that nothing keeps the
      // next groups' loads from going ahead of the sums)
      float r[kWWin];
#pragma unroll
      for (int u = 0; u < kWWin; ++u) {
        const float4 x = *reinterpret_cast<const float4*>(xb + 4 * u);
        a[u] = tot[u] = 0.0f;
#pragma unroll
        for (int i = 0; i < WD; ++i) {
          const float4 w =
              *reinterpret_cast<const float4*>(wp + u * kWWinStride - i * (kWWinStride - 4));
          float& s = a[(u - i) & (kWWin - 1)];
          s = fmaf(w.x, x.x, fmaf(w.y, x.y, fmaf(w.z, x.z, fmaf(w.w, x.w, s))));
        }
        r[u] = tot[(u - WD + 1) & (kWWin - 1)] + a[(u - WD + 1) & (kWWin - 1)];
      }
      wp += kWWin * kWWinStride;
      const int k0 = gb - (WD - 1) - g0;  // the sample of r[0]
      if (lane < kWRows)
#pragma unroll
        for (int u = 0; u < kWWin; ++u)
          if (k0 + u >= 0 && k0 + u < nf) out[k0 + u] = r[u];
    }
#pragma unroll
    for (int u = 0; u < kWWin; ++u) {
      tot[u] += a[u];
      a[u] = 0.0f;
    }
  }
  // windows that reach past the last group
#pragma unroll
  for (int u = 0; u < kWWin; ++u) {
    // the last group that started slot u
    const int sg = G - 1 - ((G - 1 - u) & (kWWin - 1));
    const int k = sg - g0;
    if (sg > G - WD && lane < kWRows && k >= 0 && k < nf) out[k] = tot[u] + a[u];
  }
  __syncwarp();
}

// Any bands: the samples that meet a chunk are spread over the lanes.
__device__ __noinline__ void wide_pass_bands(const Weideman& W, const PixK& P, const float* xg,
                                             const float* bands, int nf, int nlam, float* buf,
                                             float* accs, int lane) {
  const int AS = wide_acc_stride(nf);
  for (int t = lane; t < kWRows * AS; t += 32) accs[t] = 0.0f;
  const int* ch = reinterpret_cast<const int*>(bands + nf * kWBandStride);
#pragma unroll 1
  for (int c0 = 0, c = 0; c0 < nlam; c0 += kWChunk, ++c) {
    wide_chunk(W, P, xg, c0, nlam, buf, lane);
    const int c1 = min(c0 + kWChunk, nlam);
    const int kf = ch[2 * c], kl = ch[2 * c + 1];
#pragma unroll 1
    for (int k = kf + lane; k <= kl; k += 32) {
      const float* b = bands + k * kWBandStride;
      const int lo4 = __float_as_int(b[0]), n4 = __float_as_int(b[1]);
      const int i0 = max(lo4, c0), i1 = min(lo4 + n4, (c1 + 3) & ~3);
      if (i0 >= i1) continue;
      float a[kWRows];
#pragma unroll
      for (int q = 0; q < kWRows; ++q) a[q] = 0.0f;
#pragma unroll 1
      for (int i = i0; i < i1; i += 4) {
        const float4 w = *reinterpret_cast<const float4*>(b + 4 + (i - lo4));
        const int col = i - c0;
#pragma unroll
        for (int q = 0; q < kWRows; ++q) {
          const float4 x = *reinterpret_cast<const float4*>(buf + q * kWRowStride + col);
          a[q] = fmaf(w.x, x.x, fmaf(w.y, x.y, fmaf(w.z, x.z, fmaf(w.w, x.w, a[q]))));
        }
      }
#pragma unroll
      for (int q = 0; q < kWRows; ++q) accs[q * AS + k] += a[q];
    }
  }
  __syncwarp();
}

constexpr int kWSynthWarps = 4;       // pixels in flight per CTA of the synthesis

struct WideSynthArgs {
  const float* params;
  int64_t npix;
  const float* table;
  int nf, nlam;
  float* stokes;
  int* err;
  Weideman W;
  LineK lk;
};

// Shared memory of a warp: the inversion's buffer and accumulators, or the
// synthesis' four rows over the whole grid.
__host__ __device__ inline int wide_warp_floats(int nf, int nlam, bool deriv) {
  return deriv ? kWBuf + up4(kWRows * wide_acc_stride(nf)) : 4 * (up4(nlam) + 4);
}

// Unit-S1 Stokes values of one model over the whole grid into rows[s][GS],
// two points a lane and round, packed; zeros past the grid.
__device__ __forceinline__ void wide_synth_rows(const Weideman& W, const PixK& P, const float* xg,
                                                int nlam, int GS, float* rows, int lane) {
  struct Take {
    f2 y[4];
    __device__ __forceinline__ void unit(f2 yI, f2 yQ, f2 yU, f2 yV) {
      y[0] = yI;
      y[1] = yQ;
      y[2] = yU;
      y[3] = yV;
    }
  } out;
  __syncwarp();
#pragma unroll 1
  for (int c0 = 0; c0 < up4(nlam); c0 += 64) {
    const int i = c0 + 2 * lane;
    lambda_pair<false>(W, P, f2_pack(xg[min(i, nlam - 1)], xg[min(i + 1, nlam - 1)]), out);
    if (i < up4(nlam))
#pragma unroll
      for (int s = 0; s < 4; ++s)
        *reinterpret_cast<float2*>(rows + s * GS + i) =
            make_float2(i < nlam ? f2_lo(out.y[s]) : 0.0f, i + 1 < nlam ? f2_hi(out.y[s]) : 0.0f);
  }
  __syncwarp();
}

// Rows 0 .. NR - 1 through sample k's band, chunk by chunk of 64 points.
template <int NR>
__device__ __forceinline__ void wide_synth_sample(const float* bands, int k, int nlam, int GS,
                                                  const float* rows, float (&y)[NR]) {
  const float* b = bands + k * kWBandStride;
  const int lo4 = __float_as_int(b[0]), n4 = __float_as_int(b[1]);
  const int hi = min(lo4 + n4, up4(nlam));
#pragma unroll
  for (int s = 0; s < NR; ++s) y[s] = 0.0f;
#pragma unroll 1
  for (int i = lo4; i < hi;) {
    const int end = min(hi, (i / kWChunk + 1) * kWChunk);
    float a[NR];
#pragma unroll
    for (int s = 0; s < NR; ++s) a[s] = 0.0f;
#pragma unroll 1
    for (; i < end; i += 4) {
      const float4 w = *reinterpret_cast<const float4*>(b + 4 + (i - lo4));
#pragma unroll
      for (int s = 0; s < NR; ++s) {
        const float4 x = *reinterpret_cast<const float4*>(rows + s * GS + i);
        a[s] = fmaf(w.x, x.x, fmaf(w.y, x.y, fmaf(w.z, x.z, fmaf(w.w, x.w, a[s]))));
      }
    }
#pragma unroll
    for (int s = 0; s < NR; ++s) y[s] += a[s];
  }
}

__global__ void __launch_bounds__(32 * kWSynthWarps) wide_synth_kernel(WideSynthArgs A) {
  extern __shared__ __align__(16) float smem[];
  const int nf = A.nf, nlam = A.nlam;
  const int cf = wide_common(nf, nlam), bf = wide_band_floats(nf);
  const int wf = wide_warp_floats(nf, nlam, false), GS = up4(nlam) + 4;
  float* tab = smem;
  float* bands = smem + cf;
  uint64_t* mbar = reinterpret_cast<uint64_t*>(bands + bf + kWSynthWarps * wf);
  if (!tma_load_table(tab, A.table, (uint32_t)(cf * sizeof(float)), mbar, A.err)) return;
  if (!tma_load_table(bands, A.table + cf + wide_win_floats(nlam),
                      (uint32_t)(bf * sizeof(float)), mbar + 1, A.err))
    return;
  if (*A.err) return;  // a band wider than the kernel takes
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* rows = bands + bf + warp * wf;
  const float* xg = tab + wide_x_at(nf);
  for (int64_t pix = (int64_t)blockIdx.x * kWSynthWarps + warp; pix < A.npix;
       pix += (int64_t)gridDim.x * kWSynthWarps) {
    const float* p = A.params + pix * 10;
    const float B = p[0], gam = p[1], psi = p[2], eta0 = p[3], dld = p[4], dmp = p[5],
                v = p[6], S0 = p[7], S1 = p[8], alpha = p[9];
    float c2, s2;
    sincosf(2.0f * psi * kDeg, &s2, &c2);
    const float mus1 = A.lk.mu * S1;
    float* out = A.stokes + pix * 4 * nf;
    // the non-magnetic component first (the same line with B = 0): its Stokes
    // I waits in the output
    if (alpha != 1.0f) {
      wide_synth_rows(A.W, make_pixk(A.lk, 0.0f, gam, eta0, dld, dmp, v), xg, nlam, GS, rows,
                      lane);
      for (int k = lane; k < nf; k += 32) {
        float y[1];
        wide_synth_sample<1>(bands, k, nlam, GS, rows, y);
        out[k] = y[0];
      }
    }
    wide_synth_rows(A.W, make_pixk(A.lk, B, gam, eta0, dld, dmp, v), xg, nlam, GS, rows, lane);
    for (int k = lane; k < nf; k += 32) {
      float a[4];
      wide_synth_sample<4>(bands, k, nlam, GS, rows, a);
      const float tau = tab[4 + k];
      const float In = (alpha != 1.0f) ? out[k] : 0.0f;
      const float yI = alpha * a[0] + (1.0f - alpha) * In;
      const float yQ = alpha * a[1], yU = alpha * a[2], yV = alpha * a[3];
      out[k] = fmaf(S0, tau, mus1 * yI);
      out[nf + k] = mus1 * fmaf(c2, yQ, -s2 * yU);
      out[2 * nf + k] = mus1 * fmaf(s2, yQ, c2 * yU);
      out[3 * nf + k] = mus1 * yV;
    }
  }
}

// Warp-wide sum: every lane gets the total (fixed butterfly order, the same
// on every lane because addition commutes).
__device__ __forceinline__ float warp_sum(float x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}
__device__ __forceinline__ double warp_sum(double x) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
  return x;
}

// The damped step of Eqs. 4-5 in FP64, spread over the warp.  An FP64
// instruction holds an SMSP's FP64 pipe ~80 cycles whatever the number of
// active lanes, so one lane solving alone (~600 instructions) would cost
// more than the wavelength pass; here lane l holds packed elements l and
// l + 32 of the Jacobi-scaled matrix and the factorisation, the two
// substitutions and the unscaling take ~130 FP64 instructions.  The
// factorisation and the forward substitution apply the same operations in
// the same order per element as the one-lane Cholesky (right-looking
// updates in increasing k) and give identical results; the back
// substitution accumulates its terms in the opposite order.
// Returns false (uniformly) when a pivot is not comfortably positive; the
// caller then runs the one-lane path with its eigen-decomposition fallback.
__device__ __forceinline__ void tri_ij(int e, int& i, int& j) {
  i = (int)((sqrtf(8.0f * (float)e + 1.0f) - 1.0f) * 0.5f);
  while ((i + 1) * (i + 2) / 2 <= e) ++i;
  while (i * (i + 1) / 2 > e) --i;
  j = e - i * (i + 1) / 2;
}

__device__ __forceinline__ double shfl_d(double v, int src) {
  return __shfl_sync(0xffffffffu, v, src);
}

// element e of the packed matrix from its owner lane (e & 31, register e >> 5)
__device__ __forceinline__ double fetch(double m0, double m1, int e) {
  const double a = shfl_d(m0, e & 31), b = shfl_d(m1, e & 31);
  return (e >> 5) ? b : a;
}

__device__ bool warp_damped_step(const float* Ash, uint32_t free_mask, double eps, int lane,
                                 double* delta /* shared [9] */) {
  int i0, j0, i1, j1;
  tri_ij(lane, i0, j0);
  const bool has1 = lane + 32 < kNPk;
  tri_ij(has1 ? lane + 32 : 0, i1, j1);
  // Jacobi scaling
  double sc = 0.0;
  bool held = true;
  if (lane < kNP) {
    const double d = (double)Ash[tri(lane, lane)];
    held = !((free_mask >> lane) & 1u) || !(d > 0.0) || !isfinite(d);
    sc = held ? 0.0 : rsqrt(d);
  }
  const uint32_t hmask = __ballot_sync(0xffffffffu, lane < kNP && held);
  // every lane runs the shuffles of both slots (uniform control flow)
  const double si0 = shfl_d(sc, i0), sj0 = shfl_d(sc, j0);
  const double si1 = shfl_d(sc, i1), sj1 = shfl_d(sc, j1);
  double m0, m1 = 0.0;
  {
    const bool hi = (hmask >> i0) & 1u, hj = (hmask >> j0) & 1u;
    m0 = (i0 == j0) ? (hi ? 1.0 : 1.0 + eps) : ((hi || hj) ? 0.0 : (double)Ash[lane] * si0 * sj0);
  }
  if (has1) {
    const bool hi = (hmask >> i1) & 1u, hj = (hmask >> j1) & 1u;
    m1 = (i1 == j1) ? (hi ? 1.0 : 1.0 + eps)
                    : ((hi || hj) ? 0.0 : (double)Ash[lane + 32] * si1 * sj1);
  }
  double b = 0.0;  // right-hand side on lanes 0..8
  if (lane < kNP && !((hmask >> lane) & 1u)) b = (double)Ash[kNPk + lane] * sc;
  double rown = 0.0;  // reciprocal pivot of row `lane`
  // right-looking factorisation
#pragma unroll 1
  for (int j = 0; j < kNP; ++j) {
    const int ejj = tri(j, j);
    const double p = shfl_d((ejj >> 5) ? m1 : m0, ejj & 31);
    if (!(p > 1e-10)) return false;
    const double r = rsqrt(p);
    if (lane == j) rown = r;
    // column j below the diagonal
    if (j0 == j && i0 > j) m0 *= r;
    if (has1 && j1 == j && i1 > j) m1 *= r;
    // trailing update of elements (i, k), i >= k > j
    const double lij0 = fetch(m0, m1, tri(max(i0, j), j)), lkj0 = fetch(m0, m1, tri(max(j0, j), j));
    const double lij1 = fetch(m0, m1, tri(max(i1, j), j)), lkj1 = fetch(m0, m1, tri(max(j1, j), j));
    if (j0 > j) m0 = fma(-lij0, lkj0, m0);
    if (has1 && j1 > j) m1 = fma(-lij1, lkj1, m1);
  }
  // forward substitution L y = b (b_i on lane i)
#pragma unroll 1
  for (int i = 0; i < kNP; ++i) {
    if (lane == i) b *= rown;
    const double yi = shfl_d(b, i);
    const double lmi = fetch(m0, m1, tri(max(lane, i), min(lane, i)));
    if (lane > i && lane < kNP) b = fma(-lmi, yi, b);
  }
  // back substitution L^T x = y
#pragma unroll 1
  for (int i = kNP - 1; i >= 0; --i) {
    if (lane == i) b *= rown;
    const double xi = shfl_d(b, i);
    const double lim = fetch(m0, m1, tri(max(lane, i), min(lane, i)));
    if (lane < i) b = fma(-lim, xi, b);
  }
  if (lane < kNP) delta[lane] = ((hmask >> lane) & 1u) ? 0.0 : sc * b;
  __syncwarp();
  return true;
}

// Per-warp LM state in shared memory (written by lane 0, read by all).
struct WideWarpState {
  float A[kScratchPerSlot];  // packed J^T W J and J^T W r at the best model
  float M[10], Mt[10];
  double delta[kNP];
  double chi2b, eps;
  long long pix;
  int it;
};

// windows or bands, whichever the instrument has
__host__ __device__ inline int wide_part_floats(int nf, int nlam) {
  return max(wide_win_floats(nlam), wide_band_floats(nf));
}

__global__ void __launch_bounds__(32 * kWWarps, 1) wide_invert_kernel(InvertArgs A, int nf) {
  extern __shared__ __align__(16) float smem[];
  const int nlam = A.nlam, nwarps = blockDim.x >> 5;
  const int cf = wide_common(nf, nlam);
  const int pf = wide_part_floats(nf, nlam);
  const int wf = wide_warp_floats(nf, nlam, true);
  float* tab = smem;
  float* part = smem + cf;  // windows or bands
  WideWarpState* states = reinterpret_cast<WideWarpState*>(part + pf + nwarps * wf);
  uint64_t* mbar = reinterpret_cast<uint64_t*>(states + nwarps);
  if (!tma_load_table(tab, A.table, (uint32_t)(cf * sizeof(float)), mbar, A.err)) return;
  if (*A.err) return;
  const int width = reinterpret_cast<const int*>(tab)[0];
  const int start = reinterpret_cast<const int*>(tab)[1];
  if (!tma_load_table(part, A.table + cf + (width ? 0 : wide_win_floats(nlam)),
                      (uint32_t)((width ? wide_win_floats(nlam) : wide_band_floats(nf)) *
                                 sizeof(float)),
                      mbar + 1, A.err))
    return;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  float* buf = part + pf + warp * wf;
  float* accs = buf + kWBuf;
  const int AS = wide_acc_stride(nf);
  const float* taus = tab + 4;
  WideWarpState& S = states[warp];
  const int nobs = 4 * nf;
  const int dof = nobs - A.nfree;
  const int64_t npix = A.npix_dev ? *A.npix_dev : A.npix;
  const float mu = A.lk.mu;

  if (lane == 0) S.pix = -1;
  __syncwarp();
  while (true) {
    bool fresh = false;
    if (S.pix < 0) {
      long long pix = 0;
      if (lane == 0) pix = (long long)atomicAdd(A.queue, 1ull);
      pix = __shfl_sync(0xffffffffu, pix, 0);
      if (pix >= npix) break;
      fresh = true;
      const float* o = A.obs + pix * nobs;
      const float* wv = weight_row(A, pix, nobs);
      bool bad = false;
      float wsum = 0.0f, ic = -INFINITY;
      for (int j = lane; j < nobs; j += 32) {
        const float ov = o[j], ww = wv[j];
        bad |= !isfinite(ov) || !isfinite(ww);
        wsum += isfinite(ww) ? ww : 0.0f;
        if (j < nf) ic = fmaxf(ic, isfinite(ov) ? ov : 0.0f);
      }
      bad = __any_sync(0xffffffffu, bad);
      wsum = warp_sum(wsum);
      for (int o2 = 16; o2 > 0; o2 >>= 1) ic = fmaxf(ic, __shfl_xor_sync(0xffffffffu, ic, o2));
      bad |= !(wsum > 0.0f);
      if (lane == 0) {
        float Mt[10];
        if (A.init) {
          const float guess[10] = {500.f, 60.f, 45.f, 10.f, 35.f, 0.25f, 0.f, 0.25f, 0.75f, 1.f};
          for (int j = 0; j < 10; ++j) {
            const float v = A.init[pix * 10 + j];
            bad |= !isfinite(v);
            Mt[j] = isfinite(v) ? v : guess[j];
          }
        } else {
          Mt[0] = 500.f; Mt[1] = 60.f; Mt[2] = 45.f; Mt[3] = 10.f; Mt[4] = 35.f;
          Mt[5] = 0.25f; Mt[6] = 0.f;
          Mt[7] = 0.25f * ic;
          Mt[8] = 0.75f * ic / mu;
        }
        Mt[9] = 1.0f;
        apply_bounds(Mt);
        for (int j = 0; j < 10; ++j) S.Mt[j] = Mt[j];
        S.it = 0;
        S.eps = A.eps0;
        S.pix = pix;
      }
      bad = __shfl_sync(0xffffffffu, (int)bad, 0) != 0;
      __syncwarp();
      if (bad) {
        if (lane < 10) A.params_out[pix * 10 + lane] = S.Mt[lane];
        if (lane == 0) {
          A.chi2_out[pix] = 0.0f;
          A.iters_out[pix] = 0;
          A.status_out[pix] = VFISV_PIX_BAD_INPUT;
          map_retired(A, pix);
        }
        if (A.cov_out)
          for (int j = lane; j < 100; j += 32) A.cov_out[pix * 100 + j] = 0.0f;
        __syncwarp();
        if (lane == 0) S.pix = -1;
        __syncwarp();
        continue;
      }
    } else {
      // ---- damped step (Eqs. 4-5), FP64 over the warp ----
      const double eps = S.eps;
      const bool ok = warp_damped_step(S.A, A.free_mask, eps, lane, S.delta);
      if (!ok && lane == 0) damped_step_fp64(S.A, 1, A.free_mask, eps, S.delta);  // eigen fallback
      __syncwarp();
      // parameter j on lane j: the FP64 sums side by side
      if (lane < kNP) S.Mt[lane] = (float)((double)S.M[lane] + S.delta[lane]);
      __syncwarp();
      if (lane == 0) {
        float Mt[10];
        for (int j = 0; j < kNP; ++j) Mt[j] = S.Mt[j];
        Mt[9] = 1.0f;
        apply_bounds(Mt);
        for (int j = 0; j < 10; ++j) S.Mt[j] = Mt[j];
      }
      __syncwarp();
    }

    // ---- fused synthesis + Jacobian at the trial model ----
    float Mt[10];
#pragma unroll
    for (int j = 0; j < 10; ++j) Mt[j] = S.Mt[j];
    {
      const PixK P = make_pixk(A.lk, Mt[0], Mt[1], Mt[3], Mt[4], Mt[5], Mt[6]);
      const float* xg = tab + wide_x_at(nf);
      if (width == kWWin)
        wide_pass_windows<kWWin>(A.W, P, xg, part, start, nf, nlam, buf, accs, lane);
      else if (width)
        wide_pass_windows<kWWin - 1>(A.W, P, xg, part, start, nf, nlam, buf, accs, lane);
      else
        wide_pass_bands(A.W, P, xg, part, nf, nlam, buf, accs, lane);
    }
    const long long pix = S.pix;
    const float* o = A.obs + pix * nobs;
    const float* wv = weight_row(A, pix, nobs);
    float c2p, s2p;
    sincosf(2.0f * Mt[2] * kDeg, &s2p, &c2p);
    const float mus1 = mu * Mt[8];
    const float s0 = Mt[7];
    // ---- chi2 (Eq. 1): compensated FP32 partial sums per lane (TwoProduct
    // and TwoSum: exact to ~1e-14 relative for a lane's few terms), combined
    // and compared in FP64 ----
    double c2l;
    {
      float qs = 0.0f, qc = 0.0f;
#pragma unroll 1
      for (int k = lane; k < nf; k += 32) {
        const float tau = taus[k];
        const float* a = accs + k;
        const float q0 = a[AS], u0 = a[2 * AS];
        const float syn[4] = {fmaf(s0, tau, mus1 * a[0]), mus1 * fmaf(c2p, q0, -s2p * u0),
                              mus1 * fmaf(s2p, q0, c2p * u0), mus1 * a[3 * AS]};
#pragma unroll
        for (int st = 0; st < 4; ++st) {
          const float r = o[st * nf + k] - syn[st];
          const float wr = wv[st * nf + k] * r;
          const float ew = fmaf(wv[st * nf + k], r, -wr);  // wr + ew = w r exactly
          const float p = wr * r;
          const float ep = fmaf(wr, r, -p) + ew * r;
          const float t = qs + p;
          const float bp = t - qs;
          qc += ((qs - (t - bp)) + (p - bp)) + ep;
          qs = t;
        }
      }
      c2l = (double)qs + (double)qc;
    }
    const double c2 = warp_sum(c2l) / (double)dof;

    // ---- accept / converge (uniform across the warp) ----
    bool accept, retire = false;
    int status = VFISV_PIX_MAXITER;
    int it = S.it;
    if (fresh) {
      accept = isfinite(c2);
      if (!accept) {
        retire = true;
        status = VFISV_PIX_NAN_STATE;
      }
    } else {
      ++it;
      const double chi2b = S.chi2b;
      accept = isfinite(c2) && c2 < chi2b;
      const double eps_used = S.eps;
      const double eps = eps_update(eps_used, accept);
      if (accept) {
        const double rel = (chi2b - c2) / chi2b;
        if (rel < A.conv_rtol && eps_used <= A.conv_eps) {
          retire = true;
          status = VFISV_PIX_CONVERGED;
        }
      } else if (eps >= 1e12) {
        retire = true;
        status = VFISV_PIX_STALLED;
      }
      __syncwarp();
      if (lane == 0) S.eps = eps;
    }

    if (accept) {
      // ---- J^T W J and J^T W r at the new best model ----
      constexpr int rowOf[kNP] = {kRowB, kRowG, -1, kRowE, kRowD, kRowA, kRowV, -1, -1};
      const RowScale Rs = row_scale(A.lk, Mt[3], Mt[4]);
      float am[kNPk], g[kNP];
#pragma unroll
      for (int i = 0; i < kNPk; ++i) am[i] = 0.0f;
#pragma unroll
      for (int i = 0; i < kNP; ++i) g[i] = 0.0f;
#pragma unroll 1
      for (int k = lane; k < nf; k += 32) {
        const float tau = taus[k];
        const float* a = accs + k;
        const float q0 = a[AS], u0 = a[2 * AS];
        const float Qk = mus1 * fmaf(c2p, q0, -s2p * u0);
        const float Uk = mus1 * fmaf(s2p, q0, c2p * u0);
#pragma unroll 1
        for (int st = 0; st < 4; ++st) {
          const int sa = (st == 0) ? 0 : (st == 3 ? 3 : 1);
          const int sb = (st == 0) ? 0 : (st == 3 ? 3 : 2);
          const float cA = (st == 1) ? c2p : (st == 2 ? s2p : 1.0f);
          const float cB = (st == 1) ? -s2p : (st == 2 ? c2p : 0.0f);
          float J[kNP];
#pragma unroll
          for (int pp = 0; pp < kNP; ++pp)
            if (rowOf[pp] >= 0)
              J[pp] = (mus1 * Rs.s[rowOf[pp]]) *
                      fmaf(cA, a[(rowOf[pp] * 4 + sa) * AS], cB * a[(rowOf[pp] * 4 + sb) * AS]);
          J[2] = (st == 1) ? -2.0f * kDeg * Uk : (st == 2 ? 2.0f * kDeg * Qk : 0.0f);
          J[7] = (st == 0) ? tau : 0.0f;
          const float lin = fmaf(cA, a[sa * AS], cB * a[sb * AS]);
          J[8] = mu * lin;
          const float sv = (st == 0) ? fmaf(s0, tau, mus1 * lin) : mus1 * lin;
          const float ww = wv[st * nf + k];
          const float rr = o[st * nf + k] - sv;
#pragma unroll
          for (int pp = 0; pp < kNP; ++pp) {
            const float wj = ww * J[pp];
            g[pp] = fmaf(wj, rr, g[pp]);
#pragma unroll
            for (int q = 0; q <= pp; ++q) am[tri(pp, q)] = fmaf(wj, J[q], am[tri(pp, q)]);
          }
        }
      }
      // sums over the lanes: the butterfly of warp_sum(), halving the values a
      // lane carries at every step (54 exchanges instead of 270); lane l ends
      // with elements l and l + 32
      float v[64];
#pragma unroll
      for (int i = 0; i < 64; ++i)
        v[i] = (i < kNPk) ? am[i] : (i < kNPk + kNP ? g[i < kNPk ? 0 : i - kNPk] : 0.0f);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        const bool up = lane & o;
#pragma unroll
        for (int i = 0; i < 64; ++i)
          if (!(i & (32 - o))) {  // elements i (kept by the lower lanes) and i + o
            const float keep = up ? v[i + o] : v[i], give = up ? v[i] : v[i + o];
            v[i] = keep + __shfl_xor_sync(0xffffffffu, give, o);
          }
      }
      __syncwarp();
      S.A[lane] = v[0];
      if (lane + 32 < kNPk + kNP) S.A[lane + 32] = v[32];
      if (lane == 0) {
        for (int j = 0; j < 10; ++j) S.M[j] = Mt[j];
        S.chi2b = c2;
      }
      __syncwarp();
    }
    if (!retire && it >= A.max_iter) retire = true;
    __syncwarp();
    if (lane == 0) S.it = it;
    __syncwarp();

    if (retire) {
      if (lane == 0) {
        double chi2b = S.chi2b;
        float Mo[10];
        for (int j = 0; j < 10; ++j) Mo[j] = (status == VFISV_PIX_NAN_STATE) ? S.Mt[j] : S.M[j];
        if (status == VFISV_PIX_NAN_STATE) chi2b = c2;
        for (int j = 0; j < 10; ++j) A.params_out[pix * 10 + j] = Mo[j];
        A.chi2_out[pix] = (float)chi2b;
        A.iters_out[pix] = it;
        A.status_out[pix] = status;
      }
      if (A.cov_out) {
        // parked for the batched covariance kernel, as in the filter path
        float* cv = A.cov_out + pix * 100;
        for (int j = lane; j < 100; j += 32)
          cv[j] = (status == VFISV_PIX_NAN_STATE || j >= kNPk) ? 0.0f : S.A[j];
      }
      __syncwarp();
      if (lane == 0) {
        map_retired(A, pix);
        S.pix = -1;
      }
      __syncwarp();
    }
  }
}

size_t wide_table_bytes(int nf, int nlam) { return (size_t)wide_table_floats(nf, nlam) * 4; }

static size_t wide_smem(int nf, int nlam, bool invert, int warps) {
  const int part = invert ? wide_part_floats(nf, nlam) : wide_band_floats(nf);
  size_t b = (size_t)(wide_common(nf, nlam) + part + warps * wide_warp_floats(nf, nlam, invert)) * 4;
  if (invert) b += warps * sizeof(WideWarpState);
  return ((b + 15) & ~(size_t)15) + 16;
}

bool wide_supported(int nf, int nlam) {
  return nf >= 1 && nf <= kWMaxF && nlam >= 1 && nlam <= kWMaxLam;
}

cudaError_t launch_wide_pack(const float* filters, int nf, const float* wl, int nlam,
                             float* table, int* err, cudaStream_t s) {
  // one warp per sample and round: 32 warps take 112 samples in four rounds
  // (8 warps took 36 us, 32 take 13)
  wide_pack_kernel<<<1, 1024, 0, s>>>(filters, nf, wl, nlam, table, err);
  return cudaGetLastError();
}

cudaError_t launch_wide_synth(const float* params, int64_t npix, const float* table, int nf,
                              int nlam, float* stokes, int* err, const Weideman& W,
                              const LineK& lk, cudaStream_t s) {
  const size_t smem = wide_smem(nf, nlam, false, kWSynthWarps);
  cudaError_t e = cudaFuncSetAttribute(wide_synth_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       shared_memory_limit());
  if (e != cudaSuccess) return e;
  int dev = 0, nsm = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  nsm = sm_budget(nsm);
  cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, wide_synth_kernel, 32 * kWSynthWarps, smem);
  if (per < 1) per = 1;
  int64_t g = (int64_t)nsm * per;
  const int64_t need = (npix + kWSynthWarps - 1) / kWSynthWarps;
  if (need < g) g = need;
  if (g < 1) g = 1;
  WideSynthArgs a{params, npix, table, nf, nlam, stokes, err, W, lk};
  wide_synth_kernel<<<(int)g, 32 * kWSynthWarps, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_wide_invert(const InvertArgs& a, int nf, cudaStream_t s) {
  int dev = 0, nsm = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  const int most = shared_memory_limit();
  nsm = sm_budget(nsm);
  // one CTA per SM, a pixel a warp: up to 8 warps (65,536 pixels of 112
  // samples 43.0 ms; with 9, what the shared memory holds, 43.3; halving the
  // chunk's buffer made room for 12, 43.1), fewer when a long instrument table
  // leaves no room or the map does not fill them, so that its pixels spread
  // over all SMs
  int64_t warps = (a.npix + nsm - 1) / nsm;
  if (warps > kWWarps) warps = kWWarps;
  if (warps < 1) warps = 1;
  while (warps > 1 && wide_smem(nf, a.nlam, true, (int)warps) > (size_t)most) --warps;
  const size_t smem = wide_smem(nf, a.nlam, true, (int)warps);
  cudaError_t e = cudaFuncSetAttribute(wide_invert_kernel,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  if (e != cudaSuccess) return e;
  int64_t g = (a.npix + warps - 1) / warps;
  if (g > nsm) g = nsm;
  wide_invert_kernel<<<(int)(g < 1 ? 1 : g), 32 * (int)warps, smem, s>>>(a, nf);
  return cudaGetLastError();
}

}  // namespace vfisv
