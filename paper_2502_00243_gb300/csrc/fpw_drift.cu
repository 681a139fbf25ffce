// FPW with the baseline drift marginalised (Appendix A.1-A.2) for a ragged
// batch: the covariance of the data is C_B + C_sigma, C_B = B B^T with a
// Chebyshev basis B[i, k] = beta T_k(tau_i), k < K (tau: the curve's times
// mapped to [-1, 1]), and the statistic is
//
//   S = u^T (I / alpha^2 + E^T W E)^-1 u,   u = E^T W x,   W = (C_B + C_sigma)^-1.
//
// With D = diag(w), H0 = I + B^T D B and g = H0^-1 B^T D x (per curve, once),
// Woodbury twice reduces it to per-bin sums over the observations in bin m,
//
//   Y_m = sum w x,   Bw_m = sum w,   Q_mk = sum w B_ik,
//
// and a K x K system per frequency:
//
//   z_m = Y_m - Q_m . g,  L_m = Bw_m + 1/alpha^2,
//   S = sum_m z_m^2 / L_m + v^T H^-1 v,  v = sum_m Q_m z_m / L_m,
//   H = H0 - sum_m Q_m Q_m^T / L_m   (symmetric positive definite, >= I).
//
// Bins with no observation and 1/alpha^2 = 0 are dropped (their rows vanish).
// Since z_m = sum over bin m of w (x - B g), the bins accumulate the residuals
// of the baseline fit (formed per observation in binary64) and hold z_m
// itself: a drift far above the noise never enters an FP32 sum. B_0 = beta T_0
// = beta is constant, so Q_m0 = beta Bw_m needs no sum of its own: a bin holds
// z, Bw and Q_m1..Q_m(K-1), 1 + max(K, 1) floats; the row of H and the entry of
// v that belong to B_0 take closed forms in the bin sums.
// The sums accumulate in FP32 in thread-private shared-memory bins (one, two or
// four frequencies per thread, packed as float2 / float4 / float4 + float), phases
// are the exact 64-bit anchors of the tile kernels stepped across a span of
// frequencies; the per-frequency reduction (one reciprocal per bin, the lower
// triangle of the symmetric H) and the K x K Cholesky solve run in FP32 pairs, or
// in binary64 for curves outside the pairs' range.
#include <math.h>

#include <type_traits>

#include "fpw_shared.cuh"

namespace fpw {
namespace {

constexpr int kDrMaxK = 4;
constexpr int kDrStage = 128;  // observations the staging area has room for
constexpr int kDrChunk = 120;  // staged at a time; the block's constants lie behind them

// Per observation, written once by the prep kernel.
struct DriftObs {
  float4 q;                // w (x - B g) (w x for K = 0), w, w B_1, w B_2
  unsigned long long D;    // frac(t df) as 64-bit fixed point (linear grids)
  float q3;                // w B_3
  float pad;
};
static_assert(sizeof(DriftObs) == 32, "32-byte records");

// Bytes of the staged copy of one observation: {Phi, D}, q and, for K = 4, q3.
__host__ __device__ constexpr int drift_stage_bytes(int K) { return 16 + 16 + (K > 3 ? 4 : 0); }
// Bytes of one (frequency, bin) slot: (Y, Bw), then Q_1, Q_2 in the same
// float4 for K = 2, 3, and Q_3 in a float of its own for K = 4.
__host__ __device__ constexpr int drift_bin_bytes(int K) { return K <= 1 ? 8 : (K <= 3 ? 16 : 20); }

// float -> double from the IEEE 754 layouts with integer operations (exact for
// normal numbers and zero; subnormal, infinite and NaN inputs take the
// hardware conversion).
__device__ __forceinline__ double widen(float f) {
  const unsigned u = __float_as_uint(f);
  const unsigned e = (u >> 23) & 0xFFu;
  if (e == 0u || e == 0xFFu) {
    if ((u & 0x7FFFFFFFu) == 0u) return __hiloint2double((int)(u & 0x80000000u), 0);
    return (double)f;
  }
  const unsigned hi = ((u & 0x80000000u) | ((u & 0x7FFFFFFFu) >> 3)) + (896u << 20);
  return __hiloint2double((int)hi, (int)(u << 29));
}

// 1/L in binary64 from the FP32 reciprocal of Lf (L formed in FP32) and one
// Newton-Raphson step (r <- r + r (1 - L r)), which squares the FP32
// estimate's relative error to ~2^-45; an exact division where Lf lies
// outside [2^-100, 2^100].
__device__ __forceinline__ double recip(double L, float Lf) {
  if (!(Lf > 0x1p-100f && Lf < 0x1p100f)) return 1.0 / L;
  const double r0 = widen(__frcp_rn(Lf));
  return fma(r0, fma(-L, r0, 1.0), r0);
}

// B[k] = beta T_k(tau), k < kDrMaxK (Chebyshev polynomials of the first kind).
__device__ __forceinline__ void chebyshev(double tau, double beta, double (&Bk)[kDrMaxK]) {
  double tkm1 = 1.0, tk = tau;
#pragma unroll
  for (int k = 0; k < kDrMaxK; ++k) {
    double T;
    if (k == 0) {
      T = 1.0;
    } else if (k == 1) {
      T = tau;
    } else {
      const double tn = 2.0 * tau * tk - tkm1;
      tkm1 = tk;
      tk = tn;
      T = tn;
    }
    Bk[k] = beta * T;
  }
}

__device__ __forceinline__ double warp_sum(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v += __shfl_xor_sync(0xffffffffu, v, o);
  return v;
}

// Per curve (one block of kDrPrep threads): validation, the time span, the payload
// of every observation, H0 = I + B^T D B and g = H0^-1 B^T D x.
//
// Bound by the binary64 instructions of one SM per curve (about 20 clocks each
// and warp): a weight and a mapped time are formed once for a thread's first
// kDrKeep observations, the sums are those of a lower triangle, 97 us -> 59
// us for 64 curves of 1000, K = 3.
constexpr int kDrPrep = 512, kDrPrepWarps = kDrPrep / 32, kDrKeep = 4;

__global__ void __launch_bounds__(kDrPrep) drift_prep_kernel(const DriftArgs a) {
  __shared__ double red[kDrPrepWarps][kDrMaxK * kDrMaxK + kDrMaxK + 3];
  __shared__ double tl[2];
  __shared__ double sg[kDrMaxK];
  const int64_t c = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int K = a.K;
  const int64_t o0 = a.offsets[c], n = a.offsets[c + 1] - o0;
  // validation and the time span
  double tmin = INFINITY, tmax = -INFINITY;
  int bad = 0;
  for (int64_t i = tid; i < n; i += blockDim.x) {
    const double s = a.sigma[o0 + i], x = a.x[o0 + i], t = a.t[o0 + i];
    if (!(isfinite(s) && isfinite(x) && isfinite(t) && s > 0.0)) bad = 1;
    if (isfinite(t)) {
      tmin = fmin(tmin, t);
      tmax = fmax(tmax, t);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    tmin = fmin(tmin, __shfl_xor_sync(0xffffffffu, tmin, o));
    tmax = fmax(tmax, __shfl_xor_sync(0xffffffffu, tmax, o));
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
  }
  if (lane == 0) {
    red[warp][0] = tmin;
    red[warp][1] = tmax;
    red[warp][2] = (double)bad;
  }
  __syncthreads();
  if (tid == 0) {
    double a0 = INFINITY, a1 = -INFINITY, b = 0.0;
    for (int q = 0; q < kDrPrepWarps; ++q) {
      a0 = fmin(a0, red[q][0]);
      a1 = fmax(a1, red[q][1]);
      b = fmax(b, red[q][2]);
    }
    tl[0] = a0;
    tl[1] = a1;
    a.tabs[c] = (a1 >= a0) ? fmax(fabs(a0), fabs(a1)) : 0.0;  // max |t| (0 with no finite time)
    a.curve_bad[c] = b > 0.0 ? kCurveBad : 0;
    if (b > 0.0) atomicOr(a.status, kStatusData);
  }
  __syncthreads();
  const bool cbad = a.curve_bad[c] != 0;
  const double lo = tl[0], span = tl[1] - tl[0];
  // payload and the curve sums B^T D B (K x K) and B^T D x (K)
  double acc[kDrMaxK * kDrMaxK + kDrMaxK];
#pragma unroll
  for (int q = 0; q < kDrMaxK * kDrMaxK + kDrMaxK; ++q) acc[q] = 0.0;
  const double df = (a.nfreq > 1) ? (a.freqs[a.nfreq - 1] - a.freqs[0]) / (double)(a.nfreq - 1) : 0.0;
  double kw[kDrKeep], kt[kDrKeep];  // w and tau of the thread's first observations
  auto weigh = [&](int64_t i, double& w, double& tau) {
    const double s = cbad ? 1.0 : a.sigma[o0 + i];
    w = cbad ? 0.0 : 1.0 / (s * s);
    tau = (span > 0.0) ? 2.0 * (a.t[o0 + i] - lo) / span - 1.0 : 0.0;
  };
  auto payload = [&](int64_t i, double w, double tau) {
    DriftObs* const pay = reinterpret_cast<DriftObs*>(a.payload) + (o0 + i);
    const double x = cbad ? 0.0 : a.x[o0 + i];
    double Bk[kDrMaxK];
    chebyshev(tau, a.beta, Bk);
    float wb[kDrMaxK];
#pragma unroll
    for (int k = 0; k < kDrMaxK; ++k) {
      const double wB = w * Bk[k];
      wb[k] = k < K ? (float)wB : 0.f;
      if (k < K) {
#pragma unroll
        for (int l = 0; l <= k; ++l) acc[k * kDrMaxK + l] += wB * Bk[l];
        acc[kDrMaxK * kDrMaxK + k] += wB * x;
      }
    }
    DriftObs ob;
    ob.q = make_float4((float)(w * x), (float)w, wb[1], wb[2]);
    ob.D = isfinite(a.t[o0 + i]) ? phase_fixed64(a.t[o0 + i], df) : 0ull;
    ob.q3 = wb[3];
    ob.pad = 0.f;
    *pay = ob;
  };
#pragma unroll
  for (int q = 0; q < kDrKeep; ++q) {
    const int64_t i = tid + (int64_t)q * kDrPrep;
    if (i < n) {
      weigh(i, kw[q], kt[q]);
      payload(i, kw[q], kt[q]);
    }
  }
  for (int64_t i = tid + (int64_t)kDrKeep * kDrPrep; i < n; i += kDrPrep) {
    double w, tau;
    weigh(i, w, tau);
    payload(i, w, tau);
  }
  __syncthreads();
#pragma unroll
  for (int q = 0; q < kDrMaxK * kDrMaxK + kDrMaxK; ++q) {
    const double v = warp_sum(acc[q]);
    if (lane == 0) red[warp][q] = v;
  }
  __syncthreads();
  if (tid < kDrMaxK * kDrMaxK + kDrMaxK) {
    double s = 0.0;
    for (int q = 0; q < kDrPrepWarps; ++q) s += red[q][tid];
    red[0][tid] = s;  // (only this thread reads the column)
  }
  __syncthreads();
  if (tid == 0) {
    double H[kDrMaxK][kDrMaxK], r[kDrMaxK];
    for (int k = 0; k < K; ++k) {
      r[k] = red[0][kDrMaxK * kDrMaxK + k];
      for (int l = 0; l <= k; ++l) H[k][l] = H[l][k] = red[0][k * kDrMaxK + l] + (k == l ? 1.0 : 0.0);
    }
    double* h0 = a.H0 + c * kDrMaxK * kDrMaxK;
    for (int k = 0; k < kDrMaxK * kDrMaxK; ++k) h0[k] = (k / kDrMaxK < K && k % kDrMaxK < K) ? H[k / kDrMaxK][k % kDrMaxK] : 0.0;
    // g = H0^-1 B^T D x by Cholesky (H0 >= I is positive definite)
    double Lc[kDrMaxK][kDrMaxK];
    for (int k = 0; k < K; ++k)
      for (int l = 0; l <= k; ++l) {
        double s = H[k][l];
        for (int q = 0; q < l; ++q) s -= Lc[k][q] * Lc[l][q];
        Lc[k][l] = (k == l) ? sqrt(s) : s / Lc[l][l];
      }
    double y[kDrMaxK];
    for (int k = 0; k < K; ++k) {
      double s = r[k];
      for (int q = 0; q < k; ++q) s -= Lc[k][q] * y[q];
      y[k] = s / Lc[k][k];
    }
    double* g = a.g + c * kDrMaxK;
    for (int k = K - 1; k >= 0; --k) {
      double s = y[k];
      for (int q = k + 1; q < K; ++q) s -= Lc[q][k] * g[q];
      g[k] = s / Lc[k][k];
    }
    for (int k = K; k < kDrMaxK; ++k) g[k] = 0.0;
    for (int k = 0; k < kDrMaxK; ++k) sg[k] = g[k];
  }
  __syncthreads();
  // The bins sum w (x - B g), the residuals of the curve's baseline fit: their
  // bin sums are z_m = Y_m - Q_m . g itself, so a drift far above the noise
  // does not cancel inside FP32 sums of w x.
  // The pair reduction's range: H0 with a trace of at most 2^25, which bounds
  // its condition: a pair's 2^-46 then costs S up to 5e-7, where 2^-24 of the FP32
  // bins leaves it no digit (against 64 bits, K = 0-4, beta = 1, 3 and 30, 20-3000
  // observations: the largest, mean and RMS error of S are those of a binary64
  // reduction to five digits, 1e-7 RMS with beta = 1); with
  // weights in [2^-30, 2^30], residuals at most 2^30 and not all below 2^-25,
  // beta <= 2^20, 1/alpha^2 zero or in [2^-60, 2^30] and under 2^20
  // observations, no product leaves FP32 and none that matters loses its low part.
  double trace = 0.0;
  for (int k = 0; k < K; ++k) trace += a.H0[c * kDrMaxK * kDrMaxK + k * (kDrMaxK + 1)];
  bool wide = !cbad && (n >= (1 << 20) || !a.pairs || !(trace <= 0x1p25));
  double rmax = 0.0;
  auto residual = [&](int64_t i, double w, double tau) {
    double Bk[kDrMaxK];
    chebyshev(tau, a.beta, Bk);
    double r = a.x[o0 + i];
#pragma unroll
    for (int k = 0; k < kDrMaxK; ++k)
      if (k < K) r -= Bk[k] * sg[k];
    if (K > 0) reinterpret_cast<DriftObs*>(a.payload)[o0 + i].q.x = (float)(r * w);
    wide = wide || !(w >= 0x1p-30 && w <= 0x1p30) || !(fabs(r) <= 0x1p30);
    rmax = fmax(rmax, fabs(r));
  };
  if (!cbad) {
#pragma unroll
    for (int q = 0; q < kDrKeep; ++q) {
      const int64_t i = tid + (int64_t)q * kDrPrep;
      if (i < n) residual(i, kw[q], kt[q]);
    }
    for (int64_t i = tid + (int64_t)kDrKeep * kDrPrep; i < n; i += kDrPrep) {
      double w, tau;
      weigh(i, w, tau);
      residual(i, w, tau);
    }
  }
  wide = __syncthreads_or(wide);
  const bool small = !__syncthreads_or(rmax >= 0x1p-25);
  if (tid == 0 && !cbad && (wide || small)) a.curve_bad[c] = kCurveWide;
  for (int64_t q = (int64_t)blockIdx.x * kDrPrep + tid; q < a.nfreq; q += (int64_t)gridDim.x * kDrPrep)
    if (!isfinite(a.freqs[q])) atomicOr(a.status, kStatusGrid);
}

// FP32 pairs (value h + l, |l| a few ulp of h). Products are rounded once
// (2^-47 relative), sums carry the exact error of the leading parts in l.
// mul_rn / fma_rn: the exact error of a product must not be contracted away.
static_assert((kDrStage - kDrChunk) * 32 >= kDrMaxK * kDrMaxK * 8 + 8, "room for H0 and df");

struct Pair {
  float h, l;
};
__device__ __forceinline__ Pair pmul(float a, float b) {
  const float p = __fmul_rn(a, b);
  return Pair{p, __fmaf_rn(a, b, -p)};
}
__device__ __forceinline__ Pair pmul(Pair a, float b) {
  const float p = __fmul_rn(a.h, b);
  return Pair{p, __fmaf_rn(a.l, b, __fmaf_rn(a.h, b, -p))};
}
__device__ __forceinline__ Pair pmul(Pair a, Pair b) {
  const float p = __fmul_rn(a.h, b.h);
  return Pair{p, __fmaf_rn(a.l, b.h, __fmaf_rn(a.h, b.l, __fmaf_rn(a.h, b.h, -p)))};
}
__device__ __forceinline__ void padd(Pair& s, Pair p) {
  const float t = __fadd_rn(s.h, p.h), z = __fsub_rn(t, s.h);
  const float e = __fadd_rn(__fsub_rn(s.h, __fsub_rn(t, z)), __fsub_rn(p.h, z));
  s.h = t;
  s.l = __fadd_rn(s.l, __fadd_rn(p.l, e));
}
__device__ __forceinline__ void psub(Pair& s, Pair p) { padd(s, Pair{-p.h, -p.l}); }
__device__ __forceinline__ Pair pnorm(Pair s) {
  const float t = __fadd_rn(s.h, s.l);
  return Pair{t, __fsub_rn(s.l, __fsub_rn(t, s.h))};
}

// The reduction of one frequency from its bins (slots slot0 + m T), in FP32
// pairs; drift_reduce below is the same in binary64 and holds the formulas.
// The bins are FP32 sums (2^-24 relative), so a pair's 2^-46 is as far below
// them as binary64 for every S; a binary64 instruction of a warp occupies the
// SM for about 20 clocks, an FP32 one for a quarter: the 310 of a K = 3, M = 20
// frequency were 6200 clocks beside about 10000 of bin updates at N = 1000.
// Taken where no product leaves FP32 (kCurveWide clear).
template <int K>
__device__ __forceinline__ Pair drift_reduce_pairs(const DriftArgs& a, const unsigned char* bins, const float* bQ3,
                                                   int slot0, int T, const float2* h0) {
  constexpr bool kWide = K >= 2;
  constexpr int KK = K > 0 ? K : 1;
  const int M = a.M;
  Pair H[KK][KK], v[KK];
#pragma unroll
  for (int p = 0; p < K; ++p) {
    v[p] = Pair{0.f, 0.f};
#pragma unroll
    for (int q = 0; q <= p; ++q) H[p][q] = q == 0 ? Pair{0.f, 0.f} : Pair{h0[p * kDrMaxK + q].x, h0[p * kDrMaxK + q].y};
  }
  const Pair cal{a.cal.x, a.cal.y};
  const bool finite_alpha = a.inv_alpha2 != 0.0;
  Pair S{0.f, 0.f};
#pragma unroll 1
  for (int m = 0; m < M; ++m) {
    const int sl = slot0 + m * T;
    float z, bw, Q[kDrMaxK];
    if (kWide) {
      const float4 b = reinterpret_cast<const float4*>(bins)[sl];
      z = b.x;
      bw = b.y;
      Q[1] = b.z;
      if (K > 2) Q[2] = b.w;
    } else {
      const float2 b = reinterpret_cast<const float2*>(bins)[sl];
      z = b.x;
      bw = b.y;
    }
    if (K > 3) Q[3] = bQ3[sl];
    Pair L = cal;
    padd(L, Pair{bw, 0.f});
    if (!(L.h > 0.f)) continue;  // empty bin with 1/alpha^2 = 0: dropped
    Pair rL;
    rL.h = __frcp_rn(L.h);
    rL.l = __fmul_rn(rL.h, __fmaf_rn(-L.l, rL.h, __fmaf_rn(-L.h, rL.h, 1.f)));
    const Pair zl = pmul(rL, z);
    padd(S, pmul(zl, z));
    if (K > 0) {
      padd(v[0], pmul(zl, bw));
      if (finite_alpha) padd(H[0][0], pmul(rL, bw));
    }
#pragma unroll
    for (int p = 1; p < K; ++p) {
      padd(v[p], pmul(zl, Q[p]));
      const Pair qs = pmul(rL, Q[p]);
      if (finite_alpha) padd(H[p][0], qs);
#pragma unroll
      for (int q = 1; q <= p; ++q) psub(H[p][q], pmul(qs, Q[q]));
    }
  }
  if (K > 0) {
    v[0] = pmul(pnorm(v[0]), Pair{a.beta_p.x, a.beta_p.y});
    Pair h{1.f, 0.f};
    padd(h, pmul(pnorm(H[0][0]), Pair{a.b2cal.x, a.b2cal.y}));
    H[0][0] = h;
#pragma unroll
    for (int p = 1; p < K; ++p) H[p][0] = pmul(pnorm(H[p][0]), Pair{a.bcal.x, a.bcal.y});
  }
  Pair Lc[KK][KK], di[KK], y[KK];
#pragma unroll
  for (int p = 0; p < K; ++p)
#pragma unroll
    for (int q = 0; q <= p; ++q) {
      Pair s = H[p][q];
#pragma unroll
      for (int r = 0; r < q; ++r) psub(s, pmul(Lc[p][r], Lc[q][r]));
      s = pnorm(s);
      if (p == q) {
        // 1 / sqrt(s): the FP32 estimate u and one Newton step, u + u (1 - s u^2) / 2
        const float u = rsqrtf(s.h);
        const Pair u2 = pmul(u, u);
        const Pair su = pmul(s, u2);
        const float d = __fsub_rn(__fsub_rn(1.f, su.h), su.l);
        di[p] = s.h > 0.f ? Pair{u, 0.5f * u * d} : Pair{0.f, 0.f};
      } else {
        Lc[p][q] = pnorm(pmul(s, di[q]));
      }
    }
#pragma unroll
  for (int p = 0; p < K; ++p) {
    Pair s = v[p];
#pragma unroll
    for (int r = 0; r < p; ++r) psub(s, pmul(Lc[p][r], y[r]));
    y[p] = pnorm(pmul(pnorm(s), di[p]));
    padd(S, pmul(y[p], y[p]));
  }
  return pnorm(S);
}

// The binary64 reduction of one frequency from its bins (slots slot0 + m T):
// S = sum z^2 / L + v^T H^-1 v, H kept as its lower triangle. The constant
// basis function B_0 = beta has Q_m0 = beta Bw_m, and sum_i w_i B_ip =
// sum_m Q_mp, so its row of H and its entry of v take closed forms in the bin
// sums,
//   H_00 = 1 + beta^2 (1/alpha^2) sum_m Bw_m / L_m,
//   H_p0 = beta (1/alpha^2) sum_m Q_mp / L_m   (p >= 1),
//   v_0  = beta sum_m Bw_m z_m / L_m,
// (1 and 0 when 1/alpha^2 = 0) instead of H0 minus sums that cancel it.
template <int K>
__device__ __noinline__ double drift_reduce(const DriftArgs& a, const unsigned char* bins, const float* bQ3,
                                               int slot0, int T, int64_t c) {
  constexpr bool kWide = K >= 2;
  const int M = a.M;
  double H[kDrMaxK][kDrMaxK], v[kDrMaxK];
  const double* h0 = a.H0 + c * kDrMaxK * kDrMaxK;
#pragma unroll
  for (int p = 0; p < K; ++p) {
    v[p] = 0.0;
#pragma unroll
    for (int q = 0; q <= p; ++q) H[p][q] = q == 0 ? 0.0 : h0[p * kDrMaxK + q];  // column 0: sums of 1/L terms
  }
  const double cal = a.inv_alpha2, beta = a.beta;
  const float calf = (float)cal;
  const bool finite_alpha = cal != 0.0;
  double S = 0.0;
  for (int m = 0; m < M; ++m) {
    const int sl = slot0 + m * T;
    double Y, Bw, Q[kDrMaxK];
    float bwf;
    if (kWide) {
      const float4 b = reinterpret_cast<const float4*>(bins)[sl];
      Y = widen(b.x);
      bwf = b.y;
      Q[1] = widen(b.z);
      if (K > 2) Q[2] = widen(b.w);
    } else {
      const float2 b = reinterpret_cast<const float2*>(bins)[sl];
      Y = widen(b.x);
      bwf = b.y;
    }
    Bw = widen(bwf);
    if (K > 3) Q[3] = widen(bQ3[sl]);
    const double L = Bw + cal;
    if (!(L > 0.0)) continue;  // empty bin with 1/alpha^2 = 0: dropped
    const double rL = recip(L, bwf + calf);
    const double z = Y;  // the bin's sum of w (x - B g)
    const double zl = z * rL;
    S += z * zl;
    if (K > 0) {
      v[0] += Bw * zl;
      if (finite_alpha) H[0][0] += Bw * rL;
    }
#pragma unroll
    for (int p = 1; p < K; ++p) {
      v[p] += Q[p] * zl;
      const double qs = Q[p] * rL;
      if (finite_alpha) H[p][0] += qs;
#pragma unroll
      for (int q = 1; q <= p; ++q) H[p][q] -= qs * Q[q];
    }
  }
  if (K > 0) {
    v[0] *= beta;
    H[0][0] = 1.0 + beta * beta * cal * H[0][0];
#pragma unroll
    for (int p = 1; p < K; ++p) H[p][0] *= beta * cal;
  }
  // v^T H^-1 v by Cholesky (H >= I): off-diagonal factors and the forward
  // substitution multiply by the reciprocal square roots of the pivots
  double Lc[kDrMaxK][kDrMaxK], di[kDrMaxK], y[kDrMaxK];
#pragma unroll
  for (int p = 0; p < K; ++p)
#pragma unroll
    for (int q = 0; q <= p; ++q) {
      double s = H[p][q];
#pragma unroll
      for (int r = 0; r < q; ++r) s -= Lc[p][r] * Lc[q][r];
      if (p == q)
        di[p] = s > 0.0 ? rsqrt(s) : 0.0;
      else
        Lc[p][q] = s * di[q];
    }
#pragma unroll
  for (int p = 0; p < K; ++p) {
    double s = v[p];
#pragma unroll
    for (int r = 0; r < p; ++r) s -= Lc[p][r] * y[r];
    y[p] = s * di[p];
    S += y[p] * y[p];
  }
  return S;
}

// One block per (tile of T R frequencies, curve), R consecutive frequencies per
// thread. Bins thread-private (bank = lane), [R][M][T] slots of
// drift_bin_bytes(K): one packed read-modify-write per evaluation for K <= 3
// (two for K = 4). The slots of the next observation are formed while this
// one's bins are loaded. An anchor per a.span frequencies, which one block holds
// as T threads of R: phases do not depend on how the span is divided.
//
// Bound by shared memory: 8 passes per 16-byte update of a warp and 4 / R for
// the staged record. With one frequency per thread, two observations per trip
// and a binary64 reduction, 64 curves of 1000 observations x 20000 frequencies,
// K = 3, M = 20 took 1846 us; with the pair reduction and the slots ahead 1668;
// R = 2 1456 (M = 10: R = 4 1295; M = 50: R = 1 2185, R = 2 2543).
template <int K, int R>
__global__ void __launch_bounds__(128) drift_kernel(const DriftArgs a) {
  constexpr bool kWide = K >= 2;  // (Y, Bw, Q_1, Q_2) as float4, else (Y, Bw) as float2
  constexpr int kUnroll = kWide && R > 1 ? 2 : 4;  // the longer body of the others ran up to 3 % slower at 4
  using Bin = std::conditional_t<kWide, float4, float2>;
  extern __shared__ __align__(16) unsigned char smem[];
  const int T = blockDim.x, tid = threadIdx.x;
  const int M = a.M, MT = M * T;
  const int64_t c = blockIdx.y, F = a.nfreq;
  const int64_t f0 = (int64_t)blockIdx.x * (T * R);
  const int64_t fanchor = (int64_t)((unsigned)f0 / (unsigned)a.span) * a.span;  // f0 < 2^31
  const int j0 = (int)(f0 - fanchor) + tid * R;  // the thread's first frequency past the anchor
  Bin* const bins = reinterpret_cast<Bin*>(smem);                                           // [R][M][T] main slots
  float* const bQ3 = reinterpret_cast<float*>(bins + (size_t)R * MT);                       // [R][M][T] (K = 4)
  ulonglong2* const sPD = reinterpret_cast<ulonglong2*>(smem + (size_t)R * MT * drift_bin_bytes(K));  // [chunk]
  float4* const sQ = reinterpret_cast<float4*>(sPD + kDrChunk);                             // [chunk]
  float* const sQ3 = reinterpret_cast<float*>(sQ + kDrChunk);                               // [chunk] (K = 4)
  float2* const s_h0 = reinterpret_cast<float2*>(sQ3 + (K > 3 ? kDrChunk : 0));             // [16] H0 as pairs
  double& s_df = *reinterpret_cast<double*>(s_h0 + kDrMaxK * kDrMaxK);
  const bool grid_bad = (*(volatile unsigned*)a.status & kStatusGrid) != 0u;
  if (grid_bad) return;
  const unsigned flags = a.curve_bad[c];
  const bool cbad = flags & kCurveBad;
  const int64_t o0 = a.offsets[c], n = a.offsets[c + 1] - o0;
  const double fa = a.freqs[fanchor];
  // linear grid over this tile (the tile kernels' bound on the phase error)?
  const double tm = a.tabs[c];
  double fk[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t k = fanchor + j0 + r;
    fk[r] = k < F ? a.freqs[k] : fa;
  }
  if (tid < 32) {  // one warp's binary64 work for the block
    if (tid == 0) s_df = (F > 1) ? (a.freqs[F - 1] - a.freqs[0]) / (double)(F - 1) : 0.0;
    if (tid < kDrMaxK * kDrMaxK) {
      const double h = a.H0[c * kDrMaxK * kDrMaxK + tid];
      s_h0[tid] = make_float2((float)h, (float)(h - (double)(float)h));
    }
  }
#pragma unroll 4
  for (int q = 0; q < R * M; ++q) {
    bins[q * T + tid] = Bin{};
    if (K > 3) bQ3[q * T + tid] = 0.f;
  }
  __syncthreads();
  const double df = s_df;
  bool nonlin = false;
#pragma unroll
  for (int r = 0; r < R; ++r)
    if (fanchor + j0 + r < F && fabs(fk[r] - fma((double)(j0 + r), df, fa)) * tm > kGridTolCycles) nonlin = true;
  const bool lin = !__syncthreads_or(nonlin);
  const DriftObs* const obs = reinterpret_cast<const DriftObs*>(a.payload) + o0;
  for (int64_t oc = 0; oc < n; oc += kDrChunk) {
    const int cnt = (int)((n - oc) < kDrChunk ? (n - oc) : kDrChunk);
    if (oc > 0) __syncthreads();
    for (int i = tid; i < cnt; i += T) {
      const double ti = a.t[o0 + oc + i];
      const DriftObs ob = obs[oc + i];
      sPD[i] = lin ? make_ulonglong2(phase_fixed64(ti, fa), ob.D)
                   : make_ulonglong2((unsigned long long)__double_as_longlong(ti), 0ull);
      sQ[i] = ob.q;
      if (K > 3) sQ3[i] = ob.q3;
    }
    __syncthreads();
    if (cbad) continue;
    // the observation's slot for each of the thread's R frequencies
    auto slots = [&](const ulonglong2 pd, int (&sl)[R]) {
      const unsigned long long phi = pd.x + (unsigned long long)j0 * pd.y;
#pragma unroll
      for (int r = 0; r < R; ++r)
        sl[r] = r * MT + (int)bin_of_phase(phi + (unsigned long long)r * pd.y, (unsigned)M) * T + tid;
    };
    auto update = [&](const Bin (&b)[R], const int (&sl)[R], const float4 q) {
#pragma unroll
      for (int r = 0; r < R; ++r) {
        if constexpr (kWide)
          bins[sl[r]] = make_float4(b[r].x + q.x, b[r].y + q.y, b[r].z + q.z, b[r].w + q.w);
        else
          bins[sl[r]] = make_float2(b[r].x + q.x, b[r].y + q.y);
      }
    };
    if (lin) {
      int sl[R];
      slots(sPD[0], sl);
#pragma unroll(kUnroll)
      for (int i = 0; i < cnt; ++i) {
        Bin b[R];
        float b3[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
          b[r] = bins[sl[r]];
          if (K > 3) b3[r] = bQ3[sl[r]];
        }
        const float4 q = sQ[i];
        const float q3 = K > 3 ? sQ3[i] : 0.f;
        int sn[R];
        slots(sPD[i + 1 < cnt ? i + 1 : i], sn);
        update(b, sl, q);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          if (K > 3) bQ3[sl[r]] = b3[r] + q3;
          sl[r] = sn[r];
        }
      }
    } else {
      for (int i = 0; i < cnt; ++i) {
        const double ti = __longlong_as_double((long long)sPD[i].x);
        int sl[R];
        Bin b[R];
#pragma unroll
        for (int r = 0; r < R; ++r) {
          sl[r] = r * MT + (int)bin_of_phase(phase_fixed64(ti, fk[r]), (unsigned)M) * T + tid;
          b[r] = bins[sl[r]];
        }
        update(b, sl, sQ[i]);
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (K > 3) bQ3[sl[r]] += sQ3[i];
      }
    }
  }
#pragma unroll 1
  for (int r = 0; r < R; ++r) {
    const int64_t k = fanchor + j0 + r;
    if (k >= F) break;
    float Sf;
    double S;
    if (cbad) {
      Sf = __int_as_float(0x7fc00000);
      S = (double)Sf;
    } else if (flags & kCurveWide) {
      S = drift_reduce<K>(a, smem, bQ3, r * MT + tid, T, c);
      Sf = (float)S;
    } else {
      const Pair s = drift_reduce_pairs<K>(a, smem, bQ3, r * MT + tid, T, s_h0);
      Sf = s.h;
      S = a.S_out ? (double)s.h + (double)s.l : 0.0;
    }
    if (a.S32) a.S32[c * F + k] = Sf;
    if (a.S_out) a.S_out[c * F + k] = S;
  }
}

template <int K>
const void* drift_fn_k(int R) {
  return R == 4 ? reinterpret_cast<const void*>(&drift_kernel<K, 4>)
                : (R == 2 ? reinterpret_cast<const void*>(&drift_kernel<K, 2>)
                          : reinterpret_cast<const void*>(&drift_kernel<K, 1>));
}

const void* drift_fn(int K, int R) {
  switch (K) {
    case 0: return drift_fn_k<0>(R);
    case 1: return drift_fn_k<1>(R);
    case 2: return drift_fn_k<2>(R);
    case 3: return drift_fn_k<3>(R);
    default: return drift_fn_k<4>(R);
  }
}

}  // namespace

// Dynamic shared memory the drift kernel may use: the opt-in limit minus its
// static shared memory.
static size_t drift_dynamic_limit(int smem_optin) {
  cudaFuncAttributes fa{};
  if (cudaFuncGetAttributes(&fa, drift_fn(4, 4)) != cudaSuccess) return 0;
  return smem_optin > (int)fa.sharedSizeBytes ? (size_t)(smem_optin - (int)fa.sharedSizeBytes) : 0;
}

int drift_threads(int M, int K, int smem_optin) {
  const size_t lim = drift_dynamic_limit(smem_optin);
  for (int T = 128; T >= 32; T >>= 1)
    if (drift_smem_bytes(M, K, T, 1) <= lim) return T;
  return 0;
}

// The span's frequencies as T threads of R: the record read for an observation
// is shared by R evaluations, so the largest R that leaves eight warps on an SM
// (the bins of a span take the same room however it is divided), else R = 1
// (measured at 8 warps against 4: M = 50, K = 3 2185 us against 2543, K = 4, M =
// 20 1971 at R = 2, 8 warps, against 2412 at R = 4; at 10 against 20: M = 20,
// K = 3 1456 against 1668) and eight per SM in the whole call: fewer spans than
// that are over sooner the more threads each has.
void drift_split(int M, int K, int span, int64_t nspans, int nsm, int smem_optin, int* T, int* R) {
  const size_t block = drift_smem_bytes(M, K, span, 1) + 1024;
  for (int r = 4; r >= 1; r >>= 1) {
    const int t = span / r;
    if (span % r || t % 32 || t > 128) continue;
    *T = t;
    *R = r;
    if ((smem_optin + 1024) / block * (size_t)(t / 32) >= 8 && nspans * (t / 32) >= 8 * (int64_t)nsm) return;
  }
}

bool drift_fits(int M, int K, int T, int R, int smem_optin) {
  return drift_smem_bytes(M, K, T, R) <= drift_dynamic_limit(smem_optin);
}

size_t drift_smem_bytes(int M, int K, int T, int R) {
  return (size_t)R * M * T * drift_bin_bytes(K) + (size_t)kDrStage * drift_stage_bytes(K);
}

int drift_max_basis() { return kDrMaxK; }

size_t drift_payload_bytes() { return sizeof(DriftObs); }

cudaError_t drift_init_attributes(int max_smem) {
  const int lim = (int)drift_dynamic_limit(max_smem);
  for (int K = 0; K <= kDrMaxK; ++K)
    for (int R = 1; R <= 4; R *= 2) {
      const cudaError_t e = cudaFuncSetAttribute(drift_fn(K, R), cudaFuncAttributeMaxDynamicSharedMemorySize, lim);
      if (e != cudaSuccess) return e;
    }
  return cudaSuccess;
}

cudaError_t launch_drift(const DriftArgs& a, int T, int R, cudaStream_t st) {
  if (a.ncurves <= 0) return cudaSuccess;
  drift_prep_kernel<<<(unsigned)a.ncurves, kDrPrep, 0, st>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess || a.nfreq <= 0) return e;
  const int64_t tiles = (a.nfreq + (int64_t)T * R - 1) / ((int64_t)T * R);
  if (a.timing_start) cudaEventRecord(a.timing_start, st);
  void* params[] = {const_cast<DriftArgs*>(&a)};
  e = cudaLaunchKernel(drift_fn(a.K, R), dim3((unsigned)tiles, (unsigned)a.ncurves), dim3(T), params,
                       drift_smem_bytes(a.M, a.K, T, R), st);
  if (e != cudaSuccess) return e;
  if (a.timing_stop) cudaEventRecord(a.timing_stop, st);
  if (a.k > 0) {
    DenseTopk32Args t{};
    t.S32 = a.S32;
    t.nfreq = a.nfreq;
    t.k = a.k;
    t.peak_raw = a.peak_raw;
    t.curve_bad = a.curve_bad;
    t.status = a.status;
    t.topk_idx = a.topk_idx;
    t.topk_S = a.topk_S;
    e = launch_dense_topk32(t, a.ncurves, st);
  }
  return e;
}

}  // namespace fpw
