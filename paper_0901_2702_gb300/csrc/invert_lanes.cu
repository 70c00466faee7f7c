// Levenberg-Marquardt kernel for maps too small to fill the chip one pixel a
// thread (Secs. 2 and 4; default configuration: 6 filter positions, FP64
// damped solve and chi2, filling factor held, no restarts).  T consecutive
// lanes share a pixel, a CTA is one warp, and a call's time is the latency of
// its longest chain of iterations; the lanes shorten every part of it:
//   pass      a step takes 2 T grid points: lane q evaluates points 2 q and
//             2 q + 1 (packed) and puts their 28 values and 1/Delta into
//             shared memory; then each lane adds the step's points, in grid
//             order, to its own share of the 168 filtered sums (one Stokes
//             parameter, 24 / T filters, 7 rows);
//   chi2      a lane forms the FP64 products of its observables, every lane
//             adds the 24 of them in order;
//   normal    the lanes put the Jacobian rows of their observables into
//   equations shared memory, then each adds all 24 in order to its share of
//             the 54 compensated sums;
//   solve     lane l holds rows of the 9 x 9 system: a column's eliminations
//             run side by side (about 230 FP64 instructions on the chain
//             instead of 550, each holding the pipe 64 cycles).
// Every sum takes its terms in the order, and every element its operations,
// of invert_kernel with one thread per pixel, so results are the same bits.
// A 300-pixel map (51 passes) takes 1.16 ms against 3.82 ms of invert_kernel,
// 4,096 pixels 1.64 against 4.06; about 43 k cycles an iteration, a good
// third of them FP64 instructions in a chain.  On maps that fill the chip the
// FP64 pipe bounds it (300 instructions serve four pixels, 550 serve 32 in
// the other kernels) and it loses: 1,048,576 pixels 204 ms against 85.
#include <math.h>

#include "common.cuh"
#include "lm_device.cuh"
#include "me_pair.cuh"
#include "solve.cuh"

namespace vfisv {

// Weideman coefficients of this translation unit (set by invert_set_constants).
__constant__ Weideman c_Wln;

namespace {

constexpr int kLnNF = 6, kLnObs = 4 * kLnNF;
constexpr int kLnVals = 4 * kRows + 1;  // values a point hands over: 7 rows x 4 Stokes, 1/Delta
constexpr int kLnRec = 12;              // floats of an observable's record: r, J_0 .. J_8, w, pad
constexpr uint32_t kFull = 0xffffffffu;

template <int T>
struct LnSmem {
  static constexpr int P = 32 / T;  // pixels of a warp
  static constexpr int kPixRec = kLnObs * kLnRec + kLnRec;  // padded: no bank conflicts
  static constexpr int kBuf = (kLnVals * 64 > P * kPixRec) ? kLnVals * 64 : P * kPixRec;
  float buf[kBuf];              // point values, chi2 terms, observables' records (in turn)
  float scr[P][kNPk + kNP];     // normal equations of the best model
  float m[P][10], mt[P][10];    // best and trial model
  double x[P][kNP];             // the one-lane solve's step
  uint64_t bar;
  uint64_t pad;
};

// Position of value v of the step's point j (of 2 T) of pixel p in the
// buffer: row v of 64 floats, its 16-byte pieces permuted so that lanes
// reading the same piece of the rows of different Stokes parameters (v mod 4)
// meet different banks.
template <int T>
__device__ __forceinline__ int ln_at(int v, int p, int j) {
  const int c = (p * 2 * T + j) >> 2;
  return v * 64 + (((c ^ (v & 3)) << 2) | (j & 3));
}

// Puts the values of lambda_pair() (points j, j + 1) into the buffer.
template <int T>
struct LnPut {
  float* buf;
  int p, j;
  __device__ __forceinline__ void put(int v, f2 x) {
    *reinterpret_cast<unsigned long long*>(buf + ln_at<T>(v, p, j)) = x.v;
  }
  __device__ __forceinline__ void unit(f2 yI, f2 yQ, f2 yU, f2 yV) {
    put(0, yI);
    put(1, yQ);
    put(2, yU);
    put(3, yV);
  }
  __device__ __forceinline__ void scale(f2 iD) { put(4 * kRows, iD); }
  __device__ __forceinline__ void rows(int S, f2 vB, f2 vG, f2 vE, f2 vD, f2 vA, f2 vV) {
    put(4 * kRowB + S, vB);
    put(4 * kRowG + S, vG);
    put(4 * kRowE + S, vE);
    put(4 * kRowD + S, vD);
    put(4 * kRowA + S, vA);
    put(4 * kRowV + S, vV);
  }
};

// The fused pass: acc[r][i] = filtered row r of Stokes s, filter k0 + i.
template <int T, int KPL>
__device__ __forceinline__ void ln_pass(const PixK& P, const float* __restrict__ tab, int nrows,
                                        float* buf, int p, int q, int s, int k0,
                                        float (&acc)[kRows][KPL]) {
  constexpr int S = ((kLnNF + 1) + 3) & ~3;
#pragma unroll
  for (int r = 0; r < kRows; ++r)
#pragma unroll
    for (int i = 0; i < KPL; ++i) acc[r][i] = 0.0f;
  LnPut<T> put{buf, p, 2 * q};
#pragma unroll 1
  for (int base = 0; base < nrows; base += 2 * T) {
    // past the last point: its values again, which nothing adds
    const int i0 = min(base + 2 * q, nrows - 1), i1 = min(base + 2 * q + 1, nrows - 1);
    lambda_pair<true>(c_Wln, P, f2_pack(tab[(size_t)i0 * S + kLnNF], tab[(size_t)i1 * S + kLnNF]),
                      put);
    __syncwarp();
#pragma unroll 1
    for (int h = 0; h < 2 * T; h += 4) {
      float v[kRows][4], d[4];
#pragma unroll
      for (int r = 0; r < kRows; ++r)
        *reinterpret_cast<float4*>(v[r]) =
            *reinterpret_cast<const float4*>(buf + ln_at<T>(4 * r + s, p, h));
      *reinterpret_cast<float4*>(d) =
          *reinterpret_cast<const float4*>(buf + ln_at<T>(4 * kRows, p, h));
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        if (base + h + j >= nrows) break;  // the same for the whole warp
        const float* row = tab + (size_t)(base + h + j) * S + k0;
#pragma unroll
        for (int i = 0; i < KPL; ++i) {
          const float t = row[i], td = t * d[j];
          acc[0][i] = fmaf(t, v[0][j], acc[0][i]);
#pragma unroll
          for (int r = 1; r < kRows; ++r) acc[r][i] = fmaf(td, v[r][j], acc[r][i]);
        }
      }
    }
    __syncwarp();
  }
}

// damped_step_fp64() on the T lanes of a pixel: lane l eliminates rows l + 1,
// l + 1 + T, ... of the balanced system (row 0 is its diagonal alone).  Each
// element takes the operations of the one-lane factorisation and
// substitutions in their order.  Every lane gets the solution x (before the
// scaling exponents ex); false, for the pixel's lanes alike, when a pivot is
// not comfortably positive.
template <int T>
__device__ __forceinline__ bool ln_solve(const float* scr, uint32_t free_mask, double eps, int q,
                                         double (&x)[kNP], int (&ex)[kNP], uint32_t& hm) {
  constexpr int R = (kNP - 1 + T - 1) / T;  // rows of a lane
  const int l0 = threadIdx.x & 31 & ~(T - 1);  // the pixel's first lane
  hm = 0;
  float pw[kNP];
#pragma unroll
  for (int i = 0; i < kNP; ++i) {
    const float d = scr[tri(i, i)];
    const bool h = !((free_mask >> i) & 1u) || !(d > 0.0f) || !isfinite(d);
    hm |= (h ? 1u : 0u) << i;
    int k = 0;
    frexpf(h ? 1.0f : d, &k);
    ex[i] = (k + 1) >> 1;
    pw[i] = pow2f(-ex[i]);
  }
  const double one_eps = 1.0 + eps;
  auto diag = [&](int i, float p) {
    return ((hm >> i) & 1u) ? 1.0 : (double)(scr[tri(i, i)] * p * p) * one_eps;
  };
  auto rhs = [&](int i, float p) {
    return ((hm >> i) & 1u) ? 0.0 : (double)(scr[kNPk + i] * p);
  };
  // a lane's rows i = q + 1 + g T: elements j < i, the diagonal apart
  double a[R][kNP], b[R];
  int row[R];
#pragma unroll
  for (int g = 0; g < R; ++g) {
    const int i = min(q + 1 + g * T, kNP - 1);
    row[g] = q + 1 + g * T;  // past the last row: a copy that nothing reads
    float pi = pw[1];
#pragma unroll
    for (int e = 2; e < kNP; ++e) pi = (e == i) ? pw[e] : pi;
    const bool hi = (hm >> i) & 1u;
#pragma unroll
    for (int j = 0; j < kNP; ++j) {
      const bool h = hi || ((hm >> j) & 1u);
      const int e = (j < i) ? tri(i, j) : tri(i, i);
      double m = h ? 0.0 : (double)(scr[e] * pi * pw[j]);
      if (j == i) m = diag(i, pi);
      a[g][j] = (j <= i) ? m : 0.0;
    }
    b[g] = rhs(i, pi);
  }
  auto from = [&](double v, int i) {  // a value of row i (>= 1) from its lane
    return __shfl_sync(kFull, v, l0 + (i - 1) % T);
  };
  bool ok = true;
  double inv[kNP];
#pragma unroll
  for (int j = 0; j < kNP; ++j) {
    double d;
    if (j == 0) {
      d = diag(0, pw[0]);
    } else {
      // column j of the rows from j on: subtract the products of the columns before
#pragma unroll
      for (int k = 0; k < j; ++k) {
        const double ljk = from(a[(j - 1) / T][k], j);
#pragma unroll
        for (int g = 0; g < R; ++g)
          if (g * T + T >= j) a[g][j] = fma(-a[g][k], ljk, a[g][j]);
      }
      d = from(a[(j - 1) / T][j], j);
    }
    ok = ok && (d > 1e-10);
    const double r = rsqrt(ok ? d : 1.0);
    inv[j] = r;
#pragma unroll
    for (int g = 0; g < R; ++g)
      if (g * T + T > j) a[g][j] = (row[g] == j) ? r : a[g][j] * r;
  }
  // forward substitution
  double y[kNP];
  y[0] = rhs(0, pw[0]) * inv[0];
#pragma unroll
  for (int k = 0; k < kNP; ++k) {
    if (k > 0) y[k] = from(b[(k - 1) / T], k) * inv[k];
#pragma unroll
    for (int g = 0; g < R; ++g)
      if (g * T + T > k) b[g] = (row[g] > k) ? fma(-a[g][k], y[k], b[g]) : b[g];
  }
  // back substitution, on every lane
#pragma unroll
  for (int i = kNP - 1; i >= 0; --i) {
    double s = y[i];
#pragma unroll
    for (int k = i + 1; k < kNP; ++k) s = fma(-from(a[(k - 1) / T][i], k), x[k], s);
    x[i] = s * inv[i];
  }
  return ok;
}

// The share of the normal equations a lane sums: units (p, m) of the pairs
// (J^T W r_p, A_p0) for m = 0, (A_p,2m-1, A_p,2m) for m > 0.
constexpr int kLnUnits = 29;
__host__ __device__ constexpr int ln_unit_p(int u) {
  int p = 0;
  while (u >= (p + 3) / 2) u -= (p + 3) / 2, ++p;
  return p;
}
__host__ __device__ constexpr int ln_unit_m(int u) {
  for (int p = 0; u >= (p + 3) / 2; ++p) u -= (p + 3) / 2;
  return u;
}

template <int T>
__global__ void __launch_bounds__(32, 16) invert_lanes_kernel(InvertArgs A) {
  static_assert(T == 4 || T == 8, "lanes of a pixel");
  constexpr int NF = kLnNF, NOBS = kLnObs, NP = kNP, NPK = kNPk;
  constexpr int KPL = NF * 4 / T;                     // filters of a lane
  constexpr int UPL = (kLnUnits + T - 1) / T;         // normal-equation units of a lane
  extern __shared__ __align__(16) float smem[];
  const int tabf = table_floats(NF, A.nlam);
  float* tab = smem;
  LnSmem<T>& B = *reinterpret_cast<LnSmem<T>*>(smem + tabf);
  if (!tma_load_table(tab, A.table, (uint32_t)(tabf * sizeof(float)), &B.bar, A.err)) return;
  const float* tau = tab + (size_t)A.nlam * table_stride(NF);
  const int nrows = table_rows(tab, NF, A.nlam);
  const int lane = threadIdx.x;
  const int p = lane / T, q = lane % T, l0 = p * T;
  const uint32_t gmask = ((1u << T) - 1u) << l0;  // the pixel's lanes
  const int s = q / (T / 4), k0 = (q % (T / 4)) * KPL;  // this lane's Stokes parameter, filters
  const int dof = NOBS - A.nfree;
  const int64_t npix = A.npix_dev ? *A.npix_dev : A.npix;
  float* scr = B.scr[p];
  float* M = B.m[p];
  float* Mt = B.mt[p];
  // units of this lane: record offsets of J_p and of the pair
  int up[UPL], um[UPL];
#pragma unroll
  for (int i = 0; i < UPL; ++i) {
    up[i] = 0;
    um[i] = 0;
#pragma unroll
    for (int l = 0; l < T; ++l)
      if (l * UPL + i < kLnUnits && q == l) {
        up[i] = ln_unit_p(l * UPL + i);
        um[i] = ln_unit_m(l * UPL + i);
      }
  }
  unsigned long long n_pass = 0, n_acc = 0, n_ret = 0;
  // LM state of the pixel, the same on all its lanes
  long long pix = -1;
  bool drained = false, fresh = false, near_in = false;
  int it = 0;
  double eps = 0.0, chi2b = 0.0;
  float ob[KPL], wt[KPL];  // this lane's observables and weights
#pragma unroll
  for (int i = 0; i < KPL; ++i) ob[i] = wt[i] = 0.0f;
#pragma unroll
  for (int j = 0; j < 10; ++j) Mt[j] = 1.0f;
  for (int e = q; e < NPK + NP; e += T) scr[e] = 0.0f;

  for (;;) {
    // ---- the next pixel of the queue, for pixels' lanes that have none ----
    fresh = false;
    while (pix < 0 && !drained) {
      unsigned long long qp = 0;
      if (q == 0) qp = atomicAdd(A.queue, 1ull);
      qp = __shfl_sync(gmask, qp, l0);
      if ((long long)qp >= npix) {
        drained = true;
        break;
      }
      const long long pq = A.pix_list ? A.pix_list[qp] : (long long)qp;
      const float* o = A.obs + pq * NOBS;
      const float* wv = weight_row(A, pq, NOBS);
      bool bad = false;
      float wsum = 0.0f, ic = -INFINITY;
#pragma unroll
      for (int j = 0; j < NOBS; ++j) {
        const float ov = o[j], ww = wv[j];
        bad |= !isfinite(ov) || !isfinite(ww);
        wsum += isfinite(ww) ? ww : 0.0f;
        if (j < NF) ic = fmaxf(ic, isfinite(ov) ? ov : 0.0f);
      }
      bad |= !(wsum > 0.0f);
      float m[10];
      if (A.init) {
        const float guess[10] = {500.f, 60.f, 45.f, 10.f, 35.f, 0.25f, 0.f, 0.25f, 0.75f, 1.f};
#pragma unroll
        for (int j = 0; j < 10; ++j) {
          const float v = A.init[pq * 10 + j];
          bad |= !isfinite(v);
          m[j] = isfinite(v) ? v : guess[j];
        }
      } else {
        m[0] = 500.f; m[1] = 60.f; m[2] = 45.f; m[3] = 10.f; m[4] = 35.f;
        m[5] = 0.25f; m[6] = 0.f;
        m[7] = 0.25f * ic;
        m[8] = 0.75f * ic / A.lk.mu;
      }
      m[9] = 1.0f;
      apply_bounds(m);
      if (bad) {
        if (q == 0) {
          for (int j = 0; j < 10; ++j) A.params_out[pq * 10 + j] = m[j];
          A.chi2_out[pq] = 0.0f;
          A.iters_out[pq] = 0;
          A.status_out[pq] = VFISV_PIX_BAD_INPUT;
          map_retired(A, pq);
        }
        if (A.cov_out)
          for (int j = q; j < 100; j += T) A.cov_out[pq * 100 + j] = 0.0f;
        continue;
      }
      pix = pq;
      fresh = true;
      it = 0;
      eps = A.eps0;
      near_in = false;
      if (q == 0)
#pragma unroll
        for (int j = 0; j < 10; ++j) Mt[j] = m[j];
#pragma unroll
      for (int i = 0; i < KPL; ++i) {
        ob[i] = o[s * NF + k0 + i];
        wt[i] = wv[s * NF + k0 + i];
      }
    }
    __syncwarp();
    if (!__any_sync(kFull, pix >= 0)) break;
    const bool live = pix >= 0;

    // ---- next trial model: FP64 damped solve (Eqs. 3-5) ----
    if (__any_sync(kFull, live && !fresh)) {
      double x[NP];
      int ex[NP];
      uint32_t hm;
      const bool ok = ln_solve<T>(scr, A.free_mask, eps, q, x, ex, hm);
      if (live && !fresh && !ok && q == 0) {  // numerically singular
        double d[NP];
        damped_step_fp64<NP>(scr, 1, A.free_mask, eps, d);
#pragma unroll
        for (int j = 0; j < NP; ++j) B.x[p][j] = d[j];
      }
      __syncwarp();
      if (live && !fresh) {
        // parameters j = q, q + T, ...: their model on this lane
#pragma unroll
        for (int g = 0; g < (NP + T - 1) / T; ++g) {
          const int j = q + g * T;
          double xj = x[g * T < NP ? g * T : 0];
          int ej = ex[g * T < NP ? g * T : 0];
#pragma unroll
          for (int l = 1; l < T; ++l)
            if (g * T + l < NP && q == l) {
              xj = x[g * T + l];
              ej = ex[g * T + l];
            }
          if (j < NP) {
            const double d = ok ? (((hm >> j) & 1u) ? 0.0 : xj * pow2d(-ej)) : B.x[p][j];
            Mt[j] = (float)((double)M[j] + d);
          }
        }
      }
      __syncwarp();
      if (live && !fresh) {
        float m[10];
#pragma unroll
        for (int j = 0; j < NP; ++j) m[j] = Mt[j];
        m[9] = 1.0f;
        apply_bounds(m);
        __syncwarp(gmask);
        if (q == 0)
#pragma unroll
          for (int j = 0; j < 10; ++j) Mt[j] = m[j];
      }
      __syncwarp();
    }

    // ---- fused synthesis + Jacobian at the trial model (Secs. 3 and 4.4) ----
    float acc[kRows][KPL];
    ln_pass<T, KPL>(make_pixk(A.lk, Mt[0], Mt[1], Mt[3], Mt[4], Mt[5], Mt[6]), tab, nrows, B.buf,
                    p, q, s, k0, acc);

    // ---- residuals and chi-square (Eq. 1, FP64) ----
    float c2p, s2p;
    sincosf(2.0f * Mt[2] * kDeg, &s2p, &c2p);
    const float mus1 = A.lk.mu * Mt[8], s0 = Mt[7];
    // row r of an observable: fmaf(cA, a[r], cB * b[r]), the psi rotation of
    // (Q0, U0); a and b are the rows of Stokes 1 and 2 for s = 1, 2, else own
    const float cA = (s == 1) ? c2p : (s == 2 ? s2p : 1.0f);
    const float cB = (s == 1) ? -s2p : (s == 2 ? c2p : 0.0f);
    constexpr int kPartner = (T == 4) ? 3 : 6;  // lanes of Stokes 1 <-> 2, same filters
    double* terms = reinterpret_cast<double*>(B.buf) + p * (2 * NOBS + 2);
#pragma unroll
    for (int i = 0; i < KPL; ++i) {
      const float other = __shfl_xor_sync(kFull, acc[0][i], kPartner);
      const float a = (s == 2) ? other : acc[0][i], b = (s == 1) ? other : acc[0][i];
      const float lin = fmaf(cA, a, cB * b);
      const float r = (s == 0) ? ob[i] - fmaf(s0, tau[k0 + i], mus1 * acc[0][i])
                               : fmaf(-mus1, (s == 3) ? acc[0][i] : lin, ob[i]);
      terms[2 * (s * NF + k0 + i)] = (double)wt[i] * (double)r;
      terms[2 * (s * NF + k0 + i) + 1] = (double)r;
    }
    __syncwarp();
    double c2 = 0.0;
#pragma unroll
    for (int j = 0; j < NOBS; ++j) c2 = fma(terms[2 * j], terms[2 * j + 1], c2);
    c2 /= (double)dof;
    __syncwarp();

    // ---- acceptance test (Fig. 6) ----
    bool accept = false, retire = false, keepA = false;
    int status = VFISV_PIX_MAXITER;
    if (live) {
      ++n_pass;
      double rel_acc = INFINITY;
      if (fresh) {
        accept = isfinite(c2);
        if (!accept) {
          retire = true;
          status = VFISV_PIX_NAN_STATE;
        }
      } else {
        ++it;
        accept = isfinite(c2) && c2 < chi2b;
        const double eps_used = eps;
        eps = eps_update(eps_used, accept);
        bool conv = false, stall = false;
        if (accept) {
          const double rel = (chi2b - c2) / chi2b;
          rel_acc = rel;
          conv = rel < A.conv_rtol && eps_used <= A.conv_eps;
        } else {
          stall = eps >= 1e12;
        }
        if (conv || stall) {
          retire = true;
          status = conv ? VFISV_PIX_CONVERGED : VFISV_PIX_STALLED;
        }
        if (accept) ++n_acc;
      }
      if (accept) {
        // Hessian reuse (Sec. 4.4): this and the previous accepted step both
        // close to the minimum -> keep J^T W J, rebuild J^T W r only
        const bool nr = rel_acc < A.hess_reuse;
        keepA = nr && near_in;
        near_in = nr;
        chi2b = c2;
      }
      if (!retire && it >= A.max_iter) retire = true;  // status stays MAXITER
    }

    // ---- J^T W J and J^T W r at an accepted model (compensated FP32) ----
    if (__any_sync(kFull, accept)) {
      const RowScale R = row_scale(A.lk, Mt[3], Mt[4]);
      float* recs = B.buf + p * LnSmem<T>::kPixRec;
      constexpr int rowOf[NP] = {kRowB, kRowG, -1, kRowE, kRowD, kRowA, kRowV, -1, -1};
#pragma unroll
      for (int i = 0; i < KPL; ++i) {
        float a[kRows], b[kRows];
#pragma unroll
        for (int r = 0; r < kRows; ++r) {
          const float other = __shfl_xor_sync(kFull, acc[r][i], kPartner);
          a[r] = (s == 2) ? other : acc[r][i];
          b[r] = (s == 1) ? other : acc[r][i];
        }
        float J[NP];
#pragma unroll
        for (int pp = 0; pp < NP; ++pp)
          if (rowOf[pp] >= 0)
            J[pp] = (mus1 * R.s[rowOf[pp]]) * fmaf(cA, a[rowOf[pp]], cB * b[rowOf[pp]]);
        J[2] = 0.0f;  // psi only rotates Q and U
        if (s == 1 || s == 2) {
          const float Qk = mus1 * fmaf(c2p, a[0], -s2p * b[0]);
          const float Uk = mus1 * fmaf(s2p, a[0], c2p * b[0]);
          J[2] = (s == 1) ? -2.0f * kDeg * Uk : 2.0f * kDeg * Qk;
        }
        J[7] = (s == 0) ? tau[k0 + i] : 0.0f;
        const float lin = fmaf(cA, a[0], cB * b[0]);
        J[8] = A.lk.mu * lin;
        const float sv = (s == 0) ? fmaf(s0, tau[k0 + i], mus1 * lin) : __fmul_rn(mus1, lin);
        float4* rec = reinterpret_cast<float4*>(recs + (4 * (k0 + i) + s) * kLnRec);
        rec[0] = make_float4(ob[i] - sv, J[0], J[1], J[2]);
        rec[1] = make_float4(J[3], J[4], J[5], J[6]);
        rec[2] = make_float4(J[7], J[8], wt[i], 0.0f);
      }
      __syncwarp();
      Dot2x2 sum[UPL];
#pragma unroll
      for (int i = 0; i < UPL; ++i)
        sum[i] = Dot2x2{make_float2(0.0f, 0.0f), make_float2(0.0f, 0.0f)};
#pragma unroll 2
      for (int j = 0; j < NOBS; ++j) {  // filter-major, Stokes inner
        const float* rec = recs + j * kLnRec;
        const float ww = rec[10];
#pragma unroll
        for (int i = 0; i < UPL; ++i) {
          const float wj = ww * rec[1 + up[i]];
          const float2 b = *reinterpret_cast<const float2*>(rec + 2 * um[i]);
          sum[i].add(make_float2(wj, wj), make_float2(-wj, -wj), b);
        }
      }
      if (accept) {
#pragma unroll
        for (int i = 0; i < UPL; ++i) {
          if (q * UPL + i >= kLnUnits) break;
          const int pp = up[i], m = um[i];
          const float vx = sum[i].s.x + sum[i].c.x, vy = sum[i].s.y + sum[i].c.y;
          if (m == 0)
            scr[NPK + pp] = vx;
          else if (!keepA)
            scr[tri(pp, 2 * m - 1)] = vx;
          if (2 * m <= pp && !keepA) scr[tri(pp, 2 * m)] = vy;
        }
        for (int j = q; j < 10; j += T) M[j] = Mt[j];
      }
      __syncwarp();
    }

    if (live && retire) {
      const bool nan = status == VFISV_PIX_NAN_STATE;
      const float* src = nan ? Mt : M;
      for (int j = q; j < 10; j += T) A.params_out[pix * 10 + j] = src[j];
      if (A.cov_out) {
        // the covariance itself is computed by covariance_kernel for all
        // pixels at once; here the pixel's J^T W J is parked in its row
        float* cv = A.cov_out + pix * 100;
        for (int j = q; j < 100; j += T)
          if (nan || j < NPK) cv[j] = nan ? 0.0f : scr[j];
      }
      if (q == 0) {
        A.chi2_out[pix] = (float)(nan ? c2 : chi2b);
        A.iters_out[pix] = it;
        A.status_out[pix] = status;
        map_retired(A, pix);
      }
      ++n_ret;
      pix = -1;
    }
    __syncwarp();
  }
  if (A.counters && q == 0) {
    atomicAdd(A.counters + 0, n_pass);
    atomicAdd(A.counters + 1, n_acc);
    atomicAdd(A.counters + 2, n_ret);
    atomicAdd(A.counters + 3, n_pass * (unsigned long long)nrows);
  }
}

template <int T>
size_t lanes_smem(int nlam) {
  return (size_t)table_floats(kLnNF, nlam) * 4 + sizeof(LnSmem<T>);
}

}  // namespace

cudaError_t invert_lanes_set_constants(const Weideman& W) {
  return cudaMemcpyToSymbol(c_Wln, &W, sizeof(W));
}

cudaError_t invert_lanes_slots(int nlam, int64_t npix, int64_t* nslots, int* grid, size_t* smem) {
  constexpr int T = kInvLanes;
  const size_t sm = lanes_smem<T>(nlam);
  cudaError_t e = cudaFuncSetAttribute(invert_lanes_kernel<T>,
                                       cudaFuncAttributeMaxDynamicSharedMemorySize,
                                       shared_memory_limit());
  if (e != cudaSuccess) return e;
  int dev = 0, nsm = 0, per = 0;
  cudaGetDevice(&dev);
  cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
  nsm = sm_budget(nsm);
  e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&per, invert_lanes_kernel<T>, 32, sm);
  if (e != cudaSuccess) return e;
  if (per < 1) return cudaErrorLaunchOutOfResources;
  int64_t g = (int64_t)nsm * per;
  const int64_t need = (npix + 32 / T - 1) / (32 / T);
  if (need < g) g = need;
  if (g < 1) g = 1;
  *grid = (int)g;
  *smem = sm;
  *nslots = g * (32 / T);
  return cudaSuccess;
}

cudaError_t launch_invert_lanes(const InvertArgs& a, int grid, size_t smem, cudaStream_t s) {
  invert_lanes_kernel<kInvLanes><<<grid, 32, smem, s>>>(a);
  return cudaGetLastError();
}

}  // namespace vfisv
