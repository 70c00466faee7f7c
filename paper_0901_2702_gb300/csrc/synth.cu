// Milne-Eddington synthesis through the instrument filters (Secs. 3.1-3.2):
// one pixel per thread, the filter/wavelength table in shared memory.
#include "common.cuh"
#include "me_pair.cuh"

namespace vfisv {

// Pack filters [nf][nlam] and offsets [nlam] into the row-major table and
// append tau_k = sum_i T_k(x_i).  One block; threads stride over rows.
//
// Grid points that carry almost none of any filter's weight are left out
// (kept rows stay in grid order).  With M_k = sum_i |T_k(x_i)| and a point's
// relative weight r_i = max_k |T_k(x_i)| / M_k, the points of least r are
// dropped as long as, for every filter, the dropped |weights| sum to at most
// kMassDrop * M_k.  A filtered value S_k = sum_i T_k(x_i) y(x_i) then moves
// by at most 2^-24 M_k max|y|: the size of one FP32 rounding of a sum of that
// magnitude, so the sums are those over the whole grid to working precision.
// For the HMI-like filters (Gaussian FWHM 76 mA x sinc^2, six positions
// 69 mA apart) on the 149-point grid 63 points remain, the central
// -310 ... +310 mA; the oracle's Stokes through the cut grid differ from the
// full-grid ones by 1e-8 of the continuum.  The largest dropped set is found
// by a 32-way search over the bit patterns of r (non-negative floats order
// like their bits).  tau_k still sums every row; a NaN or infinite weight, or a
// grid longer than kMassGrid points, keeps every row.  The number of kept
// rows goes to the last float of the tau row (as int bits).
constexpr float kMassDrop = 0x1p-24f;
constexpr int kMassGrid = 4096;
constexpr int kMassMaxNF = 128;
constexpr int kPackThreads = 1024;
constexpr int kPackStage = 6144;  // floats of |T| kept in shared memory
constexpr int kCand = 32, kCandWarp = 8;  // candidate thresholds a round, and of one warp

__global__ void __launch_bounds__(kPackThreads) pack_table_kernel(
    const float* __restrict__ filters, int nf, const float* __restrict__ wl, int nlam,
    float* __restrict__ table, unsigned long long* queues, int rows) {
  const int S = table_stride(nf);
  __shared__ float rbuf[kMassGrid];  // relative weight r_i of each point
  __shared__ float mass[kMassMaxNF];  // M_k
  __shared__ float tbuf[kPackStage];  // |T| when it fits
  __shared__ int wsum[32];
  __shared__ int base, hi_s;
  __shared__ unsigned bad_s[2];  // candidates that drop too much (two rounds' worth)
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31, nw = blockDim.x >> 5;
  const bool staged = (int64_t)nf * nlam <= kPackStage;
  // M_k: one warp per filter, lane-strided then a shuffle tree
  for (int k = warp; k < nf && k < kMassMaxNF; k += nw) {
    float m = 0.0f;
#pragma unroll 4
    for (int i = lane; i < nlam; i += 32) {
      const float t = fabsf(filters[(size_t)k * nlam + i]);
      if (staged) tbuf[k * nlam + i] = t;
      m += t;
    }
    for (int o = 16; o > 0; o >>= 1) m += __shfl_xor_sync(0xffffffffu, m, o);
    if (lane == 0) mass[k] = m;
  }
  if (threadIdx.x == 0) {
    base = 0;
    hi_s = 0;
    bad_s[0] = bad_s[1] = 0u;
  }
  __syncthreads();
  bool usable = nlam <= kMassGrid && nf <= kMassMaxNF;
  for (int k = 0; k < nf && usable; ++k) usable = isfinite(mass[k]);
  int lo = -1;  // bits of the largest r dropped (-1: none); the same in every thread
  if (usable) {
    int rmax = 0;
    for (int i = threadIdx.x; i < nlam; i += blockDim.x) {
      float r = 0.0f;
      for (int k = 0; k < nf; ++k)
        if (mass[k] > 0.0f)
          r = fmaxf(r, (staged ? tbuf[k * nlam + i] : fabsf(filters[(size_t)k * nlam + i])) / mass[k]);
      rbuf[i] = r;
      rmax = max(rmax, __float_as_int(r));
    }
    for (int o = 16; o > 0; o >>= 1) rmax = max(rmax, __shfl_xor_sync(0xffffffffu, rmax, o));
    if (lane == 0) atomicMax(&hi_s, rmax);
    __syncthreads();
    // invariant: dropping r <= lo is within bounds; hi is not known to be.
    // The interval is cut into kCand parts a round (7 rounds for 31 bits,
    // halving it took 31: 25 -> 18 us with 6 filters x 149 points): a warp
    // takes one filter and kCandWarp candidates, reading each weight once for
    // them.
    int hi = hi_s;
    for (int round = 0; hi - lo > 1; ++round) {
      const long long d = (long long)hi - lo;
      for (int t = warp; t < nf * (kCand / kCandWarp); t += nw) {
        const int k = t / (kCand / kCandWarp), c0 = (t % (kCand / kCandWarp)) * kCandWarp;
        float drop[kCandWarp];
        int mid[kCandWarp];
#pragma unroll
        for (int c = 0; c < kCandWarp; ++c) {
          drop[c] = 0.0f;
          mid[c] = (int)(lo + d * (c0 + c) / kCand);
        }
        for (int i = lane; i < nlam; i += 32) {
          const int r = __float_as_int(rbuf[i]);
          const float w = staged ? tbuf[k * nlam + i] : fabsf(filters[(size_t)k * nlam + i]);
#pragma unroll
          for (int c = 0; c < kCandWarp; ++c)
            if (r <= mid[c]) drop[c] += w;
        }
        for (int o = 16; o > 0; o >>= 1)
#pragma unroll
          for (int c = 0; c < kCandWarp; ++c)
            drop[c] += __shfl_xor_sync(0xffffffffu, drop[c], o);
        unsigned bad = 0u;
#pragma unroll
        for (int c = 0; c < kCandWarp; ++c)
          if (!(drop[c] <= kMassDrop * mass[k])) bad |= 1u << (c0 + c);
        if (lane == 0 && bad) atomicOr(&bad_s[round & 1], bad);
      }
      __syncthreads();
      // the dropped sum grows with the candidate: the good ones come first
      // (candidate 0 is lo itself, good by the invariant or, at -1, empty)
      const unsigned bad = bad_s[round & 1] & ~1u;
      const int first = bad ? __ffs(bad) - 1 : kCand;
      if (threadIdx.x == 0) bad_s[(round + 1) & 1] = 0u;
      if (first < kCand) hi = (int)(lo + d * first / kCand);
      lo = (int)(lo + d * (first - 1) / kCand);
      __syncthreads();
    }
  }
  __syncthreads();
  // ordered compaction, blockDim rows at a time
  for (int i0 = 0; i0 < nlam; i0 += blockDim.x) {
    const int i = i0 + threadIdx.x;
    const bool keep = i < nlam && (!usable || __float_as_int(rbuf[i]) > lo);
    const unsigned b = __ballot_sync(0xffffffffu, keep);
    if (lane == 0) wsum[warp] = __popc(b);
    __syncthreads();
    if (warp == 0) {  // exclusive prefix over the warps, total into base
      const int c = lane < nw ? wsum[lane] : 0;
      int x = c;
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      const int b0 = base;
      __syncwarp();
      wsum[lane] = b0 + x - c;
      if (lane == 31) base = b0 + x;
    }
    __syncthreads();
    const int off = wsum[warp];
    if (keep) {
      float* row = table + (size_t)(off + __popc(b & ((1u << lane) - 1u))) * S;
      for (int k = 0; k < nf; ++k) row[k] = filters[(size_t)k * nlam + i];
      row[nf] = wl[i];
      for (int j = nf + 1; j < S; ++j) row[j] = 0.0f;
    }
    __syncthreads();
  }
  // tau: one warp per filter, fixed summation order (lane-strided, then a
  // shuffle tree) so the result does not depend on the launch.
  for (int k = warp; k < S; k += nw) {
    float s = 0.0f;
    if (k < nf)
#pragma unroll 4
      for (int i = lane; i < nlam; i += 32) s += filters[(size_t)k * nlam + i];
    for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
    if (lane == 0)
      table[(size_t)nlam * S + k] = (k < nf) ? s : (k == S - 1 ? __int_as_float(base) : 0.0f);
  }
  if (queues && threadIdx.x == 0) queues[base > rows ? 0 : 1] = 1ull << 62;
}

cudaError_t launch_pack_table(const float* filters, int nf, const float* wl, int nlam,
                              float* table, cudaStream_t s, unsigned long long* queues,
                              int rows) {
  pack_table_kernel<<<1, kPackThreads, 0, s>>>(filters, nf, wl, nlam, table, queues, rows);
  return cudaGetLastError();
}

// Filtered unit-S1 Stokes values of one model.  Two wavelength points per
// round, packed: the scalar loop issued 327 instructions a point and stalled
// on dispatch with the FMA pipe 73 % active (1,048,576 pixels, 63 points:
// 710 us); packed it issues 185 and the FMA pipe, 81 % active and throttling,
// bounds it (627 us).  The sums still take the points one by one in grid
// order.
template <int NF>
__device__ __forceinline__ void synth_pixel(const Weideman& W, const PixK& P,
                                            const float* __restrict__ tab, int nl,
                                            float (&acc)[4][NF]) {
  constexpr int S = ((NF + 1) + 3) & ~3;
#pragma unroll 1
  for (int i = 0; i < nl; i += 2) {
    const bool both = i + 1 < nl;
    float T0[NF], T1[NF];
    const float x0 = load_row<NF>(tab + (size_t)i * S, T0);
    const float x1 = load_row<NF>(tab + (size_t)(both ? i + 1 : i) * S, T1);
    struct Take {
      f2 y[4];
      __device__ __forceinline__ void unit(f2 yI, f2 yQ, f2 yU, f2 yV) {
        y[0] = yI;
        y[1] = yQ;
        y[2] = yU;
        y[3] = yV;
      }
    } out;
    lambda_pair<false>(W, P, f2_pack(x0, x1), out);
    const f2 (&y)[4] = out.y;
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int k = 0; k < NF; ++k) acc[s][k] = fmaf(T0[k], f2_lo(y[s]), acc[s][k]);
    if (both)
#pragma unroll
      for (int s = 0; s < 4; ++s)
#pragma unroll
        for (int k = 0; k < NF; ++k) acc[s][k] = fmaf(T1[k], f2_hi(y[s]), acc[s][k]);
  }
}

template <int NF>
__global__ void __launch_bounds__(128) synth_kernel(SynthArgs A) {
  extern __shared__ __align__(16) float smem[];
  const int S = table_stride(NF);
  float* tab = smem;
  uint64_t* mbar = reinterpret_cast<uint64_t*>(smem + table_floats(NF, A.nlam));
  if (!tma_load_table(tab, A.table, (uint32_t)(table_floats(NF, A.nlam) * sizeof(float)),
                      mbar, A.err))
    return;
  const float* tau = tab + (size_t)A.nlam * S;
  const int nl = table_rows(tab, NF, A.nlam);

  for (int64_t pix = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; pix < A.npix;
       pix += (int64_t)gridDim.x * blockDim.x) {
    const float* p = A.params + pix * 10;
    const float B = p[0], gam = p[1], psi = p[2], eta0 = p[3], dld = p[4], dmp = p[5],
                v = p[6], S0 = p[7], S1 = p[8], alpha = p[9];
    float acc[4][NF];
    float accn[4][NF];
#pragma unroll
    for (int s = 0; s < 4; ++s)
#pragma unroll
      for (int k = 0; k < NF; ++k) acc[s][k] = accn[s][k] = 0.0f;
    synth_pixel<NF>(A.W, make_pixk(A.lk, B, gam, eta0, dld, dmp, v), tab, nl, acc);
    if (alpha != 1.0f)  // non-magnetic component: the same line with B = 0
      synth_pixel<NF>(A.W, make_pixk(A.lk, 0.0f, gam, eta0, dld, dmp, v), tab, nl, accn);
    float c2, s2;
    sincosf(2.0f * psi * kDeg, &s2, &c2);
    const float mus1 = A.lk.mu * S1;
    float* out = A.stokes + pix * 4 * NF;
#pragma unroll
    for (int k = 0; k < NF; ++k) {
      const float yI = alpha * acc[0][k] + (1.0f - alpha) * accn[0][k];
      const float yQ = alpha * acc[1][k];
      const float yU = alpha * acc[2][k];
      const float yV = alpha * acc[3][k];
      out[k] = fmaf(S0, tau[k], mus1 * yI);
      out[NF + k] = mus1 * fmaf(c2, yQ, -s2 * yU);
      out[2 * NF + k] = mus1 * fmaf(s2, yQ, c2 * yU);
      out[3 * NF + k] = mus1 * yV;
    }
  }
}

template <int NF>
static cudaError_t launch_synth_nf(const SynthArgs& a, cudaStream_t s) {
  const size_t smem = table_floats(NF, a.nlam) * sizeof(float) + 16;
  auto kern = synth_kernel<NF>;
  if (smem > 48 * 1024) {
    cudaError_t e =
        cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, shared_memory_limit());
    if (e != cudaSuccess) return e;
  }
  // one CTA per 128 pixels: with a grid of resident CTAs striding over the
  // map the warps drifted apart (oldest first) and the last ones ran alone
  // (1,048,576 pixels: 654 us, 24 % of the warps active on average against
  // 36 % here, 627 us)
  int64_t grid = (a.npix + 127) / 128;
  if (grid > (1 << 20)) grid = 1 << 20;
  kern<<<(int)grid, 128, smem, s>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_synth(const SynthArgs& a, int nf, cudaStream_t s) {
  switch (nf) {
    case 1: return launch_synth_nf<1>(a, s);
    case 2: return launch_synth_nf<2>(a, s);
    case 3: return launch_synth_nf<3>(a, s);
    case 4: return launch_synth_nf<4>(a, s);
    case 5: return launch_synth_nf<5>(a, s);
    case 6: return launch_synth_nf<6>(a, s);
    case 7: return launch_synth_nf<7>(a, s);
    case 8: return launch_synth_nf<8>(a, s);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace vfisv
