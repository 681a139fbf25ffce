// Auxiliary FPW kernels:
//   prep         w_i = 1/sigma_i^2, a_i = x_i w_i (Eq. 1's weights), the time as
//                a fixed-point number and the phase step per observation, once
//                per call; input validation; the grid's deviation from a line
//                per anchor block
//   merge        per-curve top-k peaks from the per-item candidates (Section 3.5)
//   plain        the binary64 reference form: fl(t f) per evaluation, binary64
//                bins (Appendix A.1) and sums (Eq. 1), one curve per launch
//   dense_topk   top-k peaks of one dense periodogram (for the plain form)
#include <math.h>

#include "fpw_internal.cuh"

namespace fpw {
namespace {

__device__ __forceinline__ int64_t curve_of(const int64_t* offsets, int64_t ncurves, int64_t i) {
  // largest c with offsets[c] <= i (binary search; only used on the error path)
  int64_t lo = 0, hi = ncurves - 1;
  while (lo < hi) {
    const int64_t mid = (lo + hi + 1) >> 1;
    if (offsets[mid] <= i)
      lo = mid;
    else
      hi = mid - 1;
  }
  return lo;
}

__device__ __forceinline__ void report(const PrepArgs& a, unsigned bit) {
  atomicOr(a.status, bit);
  if (a.latch) atomicOr(a.latch, bit);
}

__global__ void prep_kernel(const PrepArgs a) {
  const int64_t stride = (int64_t)gridDim.x * blockDim.x;
  const double f0 = a.freqs[0];
  // one division a block: a binary64 operation takes a warp 50 clocks, a division
  // 25 of them
  __shared__ double s_df;
  __shared__ int s_bits;
  if (threadIdx.x == 0) {
    s_df = (a.nfreq > 1) ? (a.freqs[a.nfreq - 1] - f0) / (double)(a.nfreq - 1) : 0.0;
    if (a.df && blockIdx.x == 0) *a.df = s_df;
    if (a.rec) {
      s_bits = a.nobs > 0 ? fixed_time_bits(a.t[0], a.t[a.nobs - 1]) : 0;
      if (blockIdx.x == 0) *a.time_bits = s_bits;
    }
  }
  __syncthreads();
  const double df = s_df;
  float tmax = 0.f;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.nobs; i += stride) {
    const double s = a.sigma[i], x = a.x[i], t = a.t[i];
    const bool ok = isfinite(s) && isfinite(x) && isfinite(t) && s > 0.0;
    const double w = ok ? 1.0 / (s * s) : 0.0;
    const double xa = ok ? x * w : 0.0;
    if (ok) tmax = fmaxf(tmax, __double2float_ru(fabs(t)));
    bool fits = true;
    if (a.rec) {
      unsigned long long p = 0ull;
      unsigned top = 0u;
      const bool phases = ok && isfinite(df);
      if (phases) fits = fixed_time(t, s_bits, p, top);
      a.rec[i] = make_ulonglong2(p, phases ? phase_fixed64(t, df) : 0ull);
      a.rec_top[i] = top;
    }
    if (a.aw == nullptr) {
    } else if (a.accum == FPW_ACCUM_FP64) {
      reinterpret_cast<double2*>(a.aw)[i] = make_double2(xa, w);
    } else if (a.accum == FPW_ACCUM_FP32_COMP) {
      // hi + lo FP32 pairs: the compensated sums add the low parts too
      const float ah = (float)xa, wh = (float)w;
      reinterpret_cast<float4*>(a.aw)[i] = make_float4(ah, wh, (float)(xa - (double)ah), (float)(w - (double)wh));
    } else {
      reinterpret_cast<float2*>(a.aw)[i] = make_float2((float)xa, (float)w);
    }
    const bool wide = !(w > 0x1p-60 && w < 0x1p+60);
    if (!ok || wide || !fits) {
      const int64_t c = a.offsets ? curve_of(a.offsets, a.ncurves, i) : 0;
      const unsigned flags = ok ? (wide ? kCurveWide : 0u) | (fits ? 0u : kCurveUnfit) : kCurveBad;
      atomicOr(reinterpret_cast<unsigned*>(a.curve_bad) + (c >> 2), flags << (8 * (c & 3)));
      if (!ok) report(a, kStatusData);
    }
  }
  for (int64_t q = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; q < a.nfreq; q += stride)
    if (!isfinite(a.freqs[q])) report(a, kStatusGrid);
  if (!a.rec) return;
  // (maxima of non-negative binary64 numbers as FP32 rounded up: their bits order
  // as integers, and binary64 compares run at 2 lanes/clk/SM)
  if (__any_sync(0xffffffffu, tmax > 0.f)) {
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(tmax));
    if ((threadIdx.x & 31) == 0 && m > *(volatile unsigned*)(a.grid_dev + 1)) atomicMax(a.grid_dev + 1, m);
  }
  // per anchor block: the largest deviation of its frequencies (and one more on
  // either side) from the line through its anchor with the mean spacing. From the
  // last block of threads on: the first ones have the observations.
  __shared__ unsigned wd[8];
  const int64_t A = a.anchor_span, blocks = (a.nfreq + A - 1) / A;
  for (int64_t q = gridDim.x - 1 - blockIdx.x; q < blocks; q += gridDim.x) {
    const int64_t s = q * A - 1, an = s < 0 ? 0 : s;
    const double fa = a.freqs[an];
    float dev = 0.f;
    for (int j = threadIdx.x; j < (int)A + 2; j += blockDim.x) {
      const int64_t k = s + j;
      if (k >= 0 && k < a.nfreq) dev = fmaxf(dev, fabsf(__double2float_ru(fabs(a.freqs[k] - fma((double)(int)(k - an), df, fa)))));
    }
    const unsigned m = __reduce_max_sync(0xffffffffu, __float_as_uint(dev));
    __syncthreads();
    if ((threadIdx.x & 31) == 0) wd[threadIdx.x >> 5] = m;
    __syncthreads();
    if (threadIdx.x < 32) {
      const unsigned d = __reduce_max_sync(0xffffffffu, threadIdx.x < 8 ? wd[threadIdx.x] : 0u);
      if (threadIdx.x == 0) {
        a.block_dev[q] = __uint_as_float(d);
        if (d > *(volatile unsigned*)a.grid_dev) atomicMax(a.grid_dev, d);
        if (!fixed_anchor(fa, s_bits).ok) a.grid_dev[2] = 1u;
      }
    }
  }
}

__device__ __forceinline__ void warp_best(double& bs, int& bi, int& bp) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double os = __shfl_xor_sync(0xffffffffu, bs, o);
    const int oi = __shfl_xor_sync(0xffffffffu, bi, o);
    const int op = __shfl_xor_sync(0xffffffffu, bp, o);
    if (op >= 0 && (bp < 0 || ranks_before(os, oi, bs, bi))) {
      bs = os;
      bi = oi;
      bp = op;
    }
  }
}

// One warp per curve: the k best of its candidate rows. A candidate ranks after
// the previously selected one iff it is strictly worse in the (S desc, idx asc)
// order, so no marking is needed.
__device__ __forceinline__ MergeArgs merge_group(MergeArgs a) {
  const int64_t g = blockIdx.y;
  a.cand_S += g * a.group_rows * a.k;
  a.cand_idx += g * a.group_rows * a.k;
  a.topk_idx += g * a.k;
  a.topk_S += g * a.k;
  if (a.topk_off) a.topk_off += g * a.k;
  return a;
}

__global__ void merge_kernel(const MergeArgs all) {
  const MergeArgs a = merge_group(all);
  const int lane = threadIdx.x & 31;
  const int64_t warps = (int64_t)gridDim.x * (blockDim.x >> 5);
  const bool grid_bad = (*a.status & kStatusGrid) != 0u;
  const int64_t stride = a.out_stride > 0 ? a.out_stride : a.k;
  for (int64_t c = (int64_t)blockIdx.x * (blockDim.x >> 5) + (threadIdx.x >> 5); c < a.ncurves; c += warps) {
    int32_t* oi = a.topk_idx + c * stride;
    float* os = a.topk_S + c * stride;
    int32_t* oo = a.topk_off ? a.topk_off + c * stride : nullptr;
    if (grid_bad || (a.curve_bad[c] & kCurveBad)) {
      for (int q = lane; q < a.k; q += 32) {
        oi[q] = -1;
        os[q] = __int_as_float(0x7fc00000);
        if (oo) oo[q] = -1;
      }
      continue;
    }
    const int64_t e0 = (int64_t)a.cand_base[c] * a.k, e1 = (int64_t)a.cand_base[c + 1] * a.k;
    double ps = INFINITY;
    int pi = -1;
    for (int q = 0; q < a.k; ++q) {
      double bs = -INFINITY;
      int bi = -1, bp = -1;
      for (int64_t e = e0 + lane; e < e1; e += 32) {
        const int i = a.cand_idx[e];
        if (i < 0) continue;
        const double s = a.cand_S[e];
        const bool after_prev = (q == 0) || ranks_before(ps, pi, s, i);
        if (after_prev && (bp < 0 || ranks_before(s, i, bs, bi))) {
          bs = s;
          bi = i;
          bp = 1;
        }
      }
      warp_best(bs, bi, bp);
      if (lane == 0) {
        if (oo) {
          oi[q] = (bp >= 0) ? (bi >> 6) : -1;
          oo[q] = (bp >= 0) ? (bi & 63) : -1;
        } else {
          oi[q] = (bp >= 0) ? bi : -1;
        }
        os[q] = (bp >= 0) ? (float)bs : __int_as_float(0x7fc00000);
      }
      if (bp < 0) {
        for (int r = q + 1 + lane; r < a.k; r += 32) {
          oi[r] = -1;
          os[r] = __int_as_float(0x7fc00000);
          if (oo) oo[r] = -1;
        }
        break;
      }
      ps = bs;
      pi = bi;
    }
  }
}

// The same selection with one block per curve, for curves with many candidate
// rows (one long curve cut into thousands of work items). A row is sorted, so
// only its first entry not yet taken can be the next best: every thread holds
// the heads of its rows in registers, as order-preserving integers (binary64
// compares run at 2 lanes/clk/SM: they took 40 us for 3000 rows where reading
// and ranking integers takes 13), and replaces the one that was taken.
// More rows than kMergeRows go through in several passes, the list so far as
// entries of thread 0's.
constexpr int kMergeBlock = 1024, kMergeHeads = 6, kMergeRows = kMergeBlock * kMergeHeads;

// The best (largest r, then lowest key) of the warp's entries; r = 0: none.
__device__ __forceinline__ void warp_rank(unsigned long long& r, unsigned& key, int& place) {
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(r >> 32));
  const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(r >> 32) == hi ? (unsigned)r : 0u);
  const unsigned long long m = ((unsigned long long)hi << 32) | lo;
  const unsigned k = __reduce_min_sync(0xffffffffu, r == m ? key : 0xffffffffu);
  const unsigned who = __ballot_sync(0xffffffffu, r == m && key == k);
  place = __shfl_sync(0xffffffffu, place, __ffs(who) - 1);
  r = m;
  key = k;
}

__global__ void __launch_bounds__(kMergeBlock) merge_block_kernel(const MergeArgs all) {
  const MergeArgs a = merge_group(all);
  __shared__ unsigned long long wr[32];
  __shared__ unsigned wk[32];
  __shared__ int wp[32];  // the head's place: thread * kMergeHeads + number
  __shared__ unsigned long long resR[2][FPW_MAX_TOPK];
  __shared__ unsigned resK[2][FPW_MAX_TOPK];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const bool grid_bad = (*a.status & kStatusGrid) != 0u;
  const int64_t stride = a.out_stride > 0 ? a.out_stride : a.k;
  for (int64_t c = blockIdx.x; c < a.ncurves; c += gridDim.x) {
    int32_t* oi = a.topk_idx + c * stride;
    float* os = a.topk_S + c * stride;
    int32_t* oo = a.topk_off ? a.topk_off + c * stride : nullptr;
    if (grid_bad || (a.curve_bad[c] & kCurveBad)) {
      for (int q = tid; q < a.k; q += kMergeBlock) {
        oi[q] = -1;
        os[q] = __int_as_float(0x7fc00000);
        if (oo) oo[q] = -1;
      }
      continue;
    }
    const int64_t r0 = a.cand_base[c], r1 = a.cand_base[c + 1];
    int pass = 0;
    for (int64_t rp = r0; rp < r1; rp += kMergeRows, ++pass) {
      unsigned long long hr[kMergeHeads];
      unsigned hk[kMergeHeads];
      int hq[kMergeHeads];
#pragma unroll
      for (int h = 0; h < kMergeHeads; ++h) {
        const int64_t r = rp + tid + h * kMergeBlock;
        const int i = r < r1 ? a.cand_idx[r * a.k] : -1;
        const double s = r < r1 ? a.cand_S[r * a.k] : 0.0;
        hr[h] = i >= 0 ? rank_bits(s) : 0ull;
        hk[h] = (unsigned)i;
        hq[h] = 0;
      }
      int lq = 0;  // thread 0: the first entry not yet taken of the list of the passes before
      for (int q = 0; q < a.k; ++q) {
        unsigned long long br = 0ull;
        unsigned bk = 0xffffffffu;
        int bp = -1;
#pragma unroll
        for (int h = 0; h < kMergeHeads; ++h)
          if (hr[h] > br || (hr[h] == br && hr[h] != 0ull && hk[h] < bk)) {
            br = hr[h];
            bk = hk[h];
            bp = tid * kMergeHeads + h;
          }
        if (tid == 0 && pass > 0 && lq < a.k) {
          const unsigned long long r = resR[(pass - 1) & 1][lq];
          const unsigned k = resK[(pass - 1) & 1][lq];
          if (r > br || (r == br && r != 0ull && k < bk)) {
            br = r;
            bk = k;
            bp = kMergeRows;
          }
        }
        warp_rank(br, bk, bp);
        if (lane == 0) {
          wr[warp] = br;
          wk[warp] = bk;
          wp[warp] = bp;
        }
        __syncthreads();
        br = wr[lane];
        bk = wk[lane];
        bp = wp[lane];
        warp_rank(br, bk, bp);  // every warp: the block's best
        if (br == 0ull) bp = -1;
        if (tid == 0) {
          resR[pass & 1][q] = br;
          resK[pass & 1][q] = bk;
          if (bp == kMergeRows) ++lq;
        }
#pragma unroll
        for (int h = 0; h < kMergeHeads; ++h)
          if (bp == tid * kMergeHeads + h) {  // this head was taken: its row's next entry
            const int64_t e = (rp + tid + h * kMergeBlock) * a.k + ++hq[h];
            const int i = hq[h] < a.k ? a.cand_idx[e] : -1;
            const double s = hq[h] < a.k ? a.cand_S[e] : 0.0;
            hr[h] = i >= 0 ? rank_bits(s) : 0ull;
            hk[h] = (unsigned)i;
          }
        __syncthreads();
      }
    }
    for (int q = tid; q < a.k; q += kMergeBlock) {
      const unsigned long long r = pass > 0 ? resR[(pass - 1) & 1][q] : 0ull;
      const int i = r != 0ull ? (int)resK[(pass - 1) & 1][q] : -1;
      os[q] = i >= 0 ? (float)from_rank_bits(r) : __int_as_float(0x7fc00000);
      oi[q] = oo && i >= 0 ? i >> 6 : i;
      if (oo) oo[q] = i >= 0 ? i & 63 : -1;
    }
    __syncthreads();
  }
}

// Plain binary64 form. One thread per trial frequency; observations staged in
// shared memory in chunks; per-thread bins [m][thread] as {A, B} binary64.
// DUMP: also writes the bin of every (observation, frequency) in the window.
constexpr int kPlainThreads = 128;
constexpr int kPlainChunk = 256;

template <bool DUMP>
__global__ void __launch_bounds__(kPlainThreads) plain_kernel(const PlainArgs a) {
  extern __shared__ __align__(16) unsigned char smem[];
  double* st = reinterpret_cast<double*>(smem);
  double* sa = st + kPlainChunk;
  double* sw = sa + kPlainChunk;
  double2* bins = reinterpret_cast<double2*>(sw + kPlainChunk);
  const int tid = threadIdx.x;
  const int64_t k = (int64_t)blockIdx.x * kPlainThreads + tid;
  const double f = a.freqs[k < a.nfreq ? k : a.nfreq - 1];
  const int M = a.M;
  for (int m = 0; m < M; ++m) bins[m * kPlainThreads + tid] = make_double2(0.0, 0.0);
  bool bad = false;
  for (int64_t o = 0; o < a.n; o += kPlainChunk) {
    const int cnt = (int)((a.n - o) < kPlainChunk ? (a.n - o) : kPlainChunk);
    __syncthreads();
    for (int i = tid; i < cnt; i += kPlainThreads) {
      const double s = a.sigma[o + i], x = a.x[o + i], t = a.t[o + i];
      if (!(isfinite(s) && isfinite(x) && isfinite(t) && s > 0.0)) bad = true;
      const double w = 1.0 / (s * s);
      st[i] = t;
      sa[i] = x * w;
      sw[i] = w;
    }
    __syncthreads();
    for (int i = 0; i < cnt; ++i) {
      const double p = __dmul_rn(st[i], f);
      const double ph = __dsub_rn(p, floor(p));
      int m = (int)floor(__dmul_rn((double)M, ph));
      m = m > M - 1 ? M - 1 : (m < 0 ? 0 : m);
      if (DUMP && k < a.nfreq && k >= a.bins_k0 && k < a.bins_k1)
        a.bins_out[(k - a.bins_k0) * a.bins_nobs + a.bins_base + o + i] = m;
      double2* b = &bins[m * kPlainThreads + tid];
      double2 v = *b;
      v.x = __dadd_rn(v.x, sa[i]);
      v.y = __dadd_rn(v.y, sw[i]);
      *b = v;
    }
  }
  bad = __syncthreads_or(bad);
  if (bad && tid == 0) atomicOr(a.status, kStatusData);
  if (k < a.nfreq) {
    double S = 0.0;
    for (int m = 0; m < M; ++m) {
      const double2 v = bins[m * kPlainThreads + tid];
      const double den = __dadd_rn(v.y, a.inv_alpha2);
      if (den > 0.0) S = __dadd_rn(S, __ddiv_rn(__dmul_rn(v.x, v.x), den));
    }
    a.S_out[k] = bad ? __longlong_as_double(0x7ff8000000000000ll) : S;
  }
}

// Top-k peaks of one dense periodogram, one block: k rounds of a block-wide
// arg-max restricted to entries ranked strictly after the previous pick.
constexpr int kTopkThreads = 1024;

__global__ void __launch_bounds__(kTopkThreads) dense_topk_kernel(const DenseTopkArgs a) {
  __shared__ double ws[32];
  __shared__ int wi[32];
  __shared__ int wp[32];
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t F = a.nfreq;
  const bool bad = F > 0 && isnan(a.S[0]);  // the plain kernel writes NaN for invalid curves
  double ps = INFINITY;
  int pi = -1;
  for (int q = 0; q < a.k; ++q) {
    double bs = -INFINITY;
    int bi = -1, bp = -1;
    if (!bad) {
      for (int64_t e = tid; e < F; e += kTopkThreads) {
        const double s = a.S[e];
        bool peak = true;
        if (!a.peak_raw) {
          const double l = (e > 0) ? a.S[e - 1] : -INFINITY;
          const double r = (e + 1 < F) ? a.S[e + 1] : -INFINITY;
          peak = s > l && s >= r;
        }
        if (!peak) continue;
        const bool after_prev = (q == 0) || ranks_before(ps, pi, s, (int)e);
        if (after_prev && (bp < 0 || ranks_before(s, (int)e, bs, bi))) {
          bs = s;
          bi = (int)e;
          bp = 1;
        }
      }
    }
    warp_best(bs, bi, bp);
    if (lane == 0) {
      ws[warp] = bs;
      wi[warp] = bi;
      wp[warp] = bp;
    }
    __syncthreads();
    if (warp == 0) {
      bs = ws[lane];
      bi = wi[lane];
      bp = wp[lane];
      warp_best(bs, bi, bp);
      if (lane == 0) {
        a.topk_idx[q] = (bp >= 0) ? bi : -1;
        a.topk_S[q] = (bp >= 0) ? (float)bs : __int_as_float(0x7fc00000);
        wi[0] = bi;
        wp[0] = bp;
        ws[0] = bs;
      }
    }
    __syncthreads();
    ps = ws[0];
    pi = wi[0];
    if (wp[0] < 0) {
      for (int r = q + 1 + tid; r < a.k; r += kTopkThreads) {
        a.topk_idx[r] = -1;
        a.topk_S[r] = __int_as_float(0x7fc00000);
      }
      break;
    }
    __syncthreads();
  }
}

__global__ void latch_kernel(unsigned* words) { words[kWordLatch] |= words[1]; }

__global__ void fill_topk_kernel(int32_t* idx, float* S, int64_t n) {
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (int64_t)gridDim.x * blockDim.x) {
    idx[i] = -1;
    S[i] = __int_as_float(0x7fc00000);
  }
}

}  // namespace

cudaError_t launch_latch(unsigned* words, cudaStream_t st) {
  latch_kernel<<<1, 1, 0, st>>>(words);
  return cudaGetLastError();
}

cudaError_t allow_shared_memory(const void* fn, int static_smem) {
  int dev = 0, limit = 0;
  cudaError_t e = cudaGetDevice(&dev);
  if (e == cudaSuccess) e = cudaDeviceGetAttribute(&limit, cudaDevAttrMaxSharedMemoryPerBlockOptin, dev);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(fn, cudaFuncAttributeMaxDynamicSharedMemorySize, limit - static_smem);
}

cudaError_t launch_fill_topk(int32_t* idx, float* S, int64_t n, cudaStream_t st) {
  if (n <= 0) return cudaSuccess;
  int64_t blocks = (n + 255) / 256;
  blocks = blocks > 4096 ? 4096 : blocks;
  fill_topk_kernel<<<(unsigned)blocks, 256, 0, st>>>(idx, S, n);
  return cudaGetLastError();
}

cudaError_t launch_prep(const PrepArgs& a, cudaStream_t st) {
  const int64_t work = a.nobs > a.nfreq ? a.nobs : a.nfreq;
  int blocks = (int)((work + 255) / 256);
  blocks = blocks < 1 ? 1 : (blocks > 1216 ? 1216 : blocks);  // 8 a SM
  prep_kernel<<<blocks, 256, 0, st>>>(a);  // 8 warps (prep_kernel's wd)
  return cudaGetLastError();
}

cudaError_t launch_merge(const MergeArgs& a, cudaStream_t st) {
  if (a.ncurves <= 0 || a.k <= 0) return cudaSuccess;
  const unsigned groups = a.ngroups > 1 ? (unsigned)a.ngroups : 1u;
  // A block per curve where that is over sooner, in microseconds as measured on 152
  // SMs: a block fills an SM and takes 5 + k; the curves' warps run at once, k
  // rounds through the longest one's candidates. 20 curves, k = 5, 100 rows: 10
  // against 33; 304 curves, 80 rows: 19 against 27; 608 curves, 45 rows: 35 against
  // 18; 4000 curves, k = 20: 660 against 140; k = 64 2000 against 800.
  const int64_t rounds = ((a.ncurves * groups) + 151) / 152, entries = (int64_t)a.max_rows * a.k;
  if (rounds * (5 + a.k) < 5 + a.k + a.k * entries / 90) {
    const int64_t blocks = a.ncurves < 65535 ? a.ncurves : 65535;
    merge_block_kernel<<<dim3((unsigned)blocks, groups), kMergeBlock, 0, st>>>(a);
    return cudaGetLastError();
  }
  int blocks = (int)((a.ncurves + 7) / 8);
  blocks = blocks > 65535 ? 65535 : blocks;
  merge_kernel<<<dim3((unsigned)blocks, groups), 256, 0, st>>>(a);
  return cudaGetLastError();
}

size_t plain_smem_bytes(int M) { return (size_t)3 * kPlainChunk * 8 + (size_t)M * kPlainThreads * 16; }

cudaError_t plain_init_attributes(int max_smem) {
  cudaError_t e = cudaFuncSetAttribute(plain_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(plain_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, max_smem);
}

cudaError_t launch_plain(const PlainArgs& a, cudaStream_t st) {
  if (a.nfreq <= 0) return cudaSuccess;
  const size_t smem = plain_smem_bytes(a.M);
  const int64_t blocks = (a.nfreq + kPlainThreads - 1) / kPlainThreads;
  if (a.bins_out)
    plain_kernel<true><<<(unsigned)blocks, kPlainThreads, smem, st>>>(a);
  else
    plain_kernel<false><<<(unsigned)blocks, kPlainThreads, smem, st>>>(a);
  return cudaGetLastError();
}

cudaError_t launch_dense_topk(const DenseTopkArgs& a, cudaStream_t st) {
  if (a.k <= 0) return cudaSuccess;
  dense_topk_kernel<<<1, kTopkThreads, 0, st>>>(a);
  return cudaGetLastError();
}

}  // namespace fpw
