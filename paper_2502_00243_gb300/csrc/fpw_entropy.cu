// Phase entropy of the observation times (Appendix C):
//   H(f) = -sum_m (N_m / N) log(N_m / N),  N_m observations in phase bin m,
// with Hutcheson's expectation and variance for equally likely bins,
//   E(H)   = log M - (M - 1) / (2 N) - (M - 1)(M + 1) / (12 N^2),
//   Var(H) = (M - 1) / (2 N^2) + (M^2 - 1) / (6 N^3),
// used to flag periodogram peaks whose phase coverage is anomalously uneven
// (z = (H - E) / sqrt(Var) strongly negative).
//
// Bins use the exact anchors and 64-bit stepping of the periodogram kernels,
// so they equal floor(M frac(t f)) except within 2e-10 cycles of an edge.
#include <math.h>

#include "fpw_internal.cuh"

namespace fpw {
namespace {

constexpr int kEntThreads = 128;
constexpr int kEntChunk = 256;
constexpr unsigned kEntTable = 256;  // counts whose logarithm is read from a table

// H from bin counts: log N - (1/N) sum_m N_m log N_m, in FP32 (the count
// terms are exact integers; the logarithms carry the rounding).
__device__ __forceinline__ float entropy_from_counts_sum(float sum_clogc, float N) {
  return N > 0.f ? logf(N) - sum_clogc / N : 0.f;
}

// One more in a count of this thread's, and its value.
__device__ __forceinline__ void count_up(unsigned a) { asm volatile("red.shared.add.u32 [%0], 1;" ::"r"(a) : "memory"); }
__device__ __forceinline__ unsigned read_count(unsigned a) {
  unsigned v;
  asm volatile("ld.shared.u32 %0, [%1];" : "=r"(v) : "r"(a) : "memory");
  return v;
}

// R consecutive frequencies per thread, blocks of kEntThreads R frequencies;
// counts per (bin, frequency slot, thread) as 32-bit integers, [m][r][thread]
// (conflict-free). Anchors lie every `span` frequencies (a multiple of the
// block's: the phases, and with them the counts, do not depend on the launch).
// Per staged observation the block holds the exact anchor phase P_i = frac(t_i
// f_a) and the step D_i = frac(t_i df) as 64-bit fixed point; where all of the
// span's frequencies lie on the linear grid (the tile kernels' bound on the
// phase error) frequency j past the anchor has phase P_i + j D_i (mod 2^64),
// else the exact anchor at its own frequency.
//
// Bound by the instructions and the shared-memory pipe together, about 2.8
// clocks per SM and 32 counts. A count is one red.shared.add: nothing comes
// back, so an observation's R counts wait for nothing (load, add and store ran
// M = 20 at 2.49e12 counts/s, this at 3.05e12; 1000 times x 1e6 frequencies).
// With the slots inside the bin, r T is an offset of the instruction; outside
// it the address cost one more (2.87e12). Two 16-bit counts to a word, for
// twice the blocks per SM, cost three more (2.10e12), phases by a tree of
// 64-bit adds the shifts (2.74e12), the bin from a 32 x 32 -> 64 product
// instead of its upper half 2.77e12. Four observations a trip against two: 6 %.
template <int R>
__global__ void __launch_bounds__(kEntThreads) entropy_dense_kernel(const double* t, int64_t n, const double* freqs,
                                                            int64_t nfreq, int M, int span, float* H_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  ulonglong2* const sPD = reinterpret_cast<ulonglong2*>(smem);
  float* const logq = reinterpret_cast<float*>(sPD + kEntChunk + 1);  // one record of padding after the chunk
  unsigned* const cnt = reinterpret_cast<unsigned*>(logq + kEntTable);
  __shared__ unsigned long long s_tm[kEntThreads / 32];
  __shared__ double s_df;
  constexpr int T = kEntThreads;
  const int tid = threadIdx.x;
  const int64_t f0 = (int64_t)blockIdx.x * (T * R);
  const int64_t fanchor = f0 & -(int64_t)span;
  const int j0 = (int)(f0 - fanchor) + tid * R;  // the thread's first frequency past the anchor
  const double fa = freqs[fanchor];
  // max |t| as the largest bit pattern (NaN left out), and one division a block: a warp's binary64
  // instruction occupies the SM for about 20 clocks
  unsigned long long tb = 0ull;
  for (int64_t i = tid; i < n; i += T) {
    const unsigned long long v = (unsigned long long)__double_as_longlong(t[i]) & 0x7fffffffffffffffull;
    if (v <= 0x7ff0000000000000ull && v > tb) tb = v;
  }
  if (tid == 0) s_df = (nfreq > 1) ? (freqs[nfreq - 1] - freqs[0]) / (double)(nfreq - 1) : 0.0;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(0xffffffffu, tb, o);
    tb = v > tb ? v : tb;
  }
  if ((tid & 31) == 0) s_tm[tid >> 5] = tb;
  for (int q = tid; q < (int)kEntTable; q += T) logq[q] = q > 1 ? logf((float)q) : 0.f;
  unsigned* const mine = cnt + tid;  // this thread's column of the [r][m][thread] counts
  for (int q = 0; q < R * M; ++q) mine[q * T] = 0u;
  __syncthreads();
  tb = s_tm[0];
  for (int q = 1; q < T / 32; ++q) tb = s_tm[q] > tb ? s_tm[q] : tb;
  const double tm = __longlong_as_double((long long)tb), df = s_df;
  bool nonlin = false;  // of the whole span, whichever of its blocks this is
#pragma unroll R
  for (int j = tid; j < span; j += T)
    if (fanchor + j < nfreq && fabs(freqs[fanchor + j] - fma((double)j, df, fa)) * tm > kGridTolCycles) nonlin = true;
  const bool lin = !__syncthreads_or(nonlin);
  const unsigned col = (unsigned)__cvta_generic_to_shared(mine);
  constexpr unsigned step = 4u * (unsigned)(T * R);
  for (int64_t o = 0; o < n; o += kEntChunk) {
    const int c = (int)((n - o) < kEntChunk ? (n - o) : kEntChunk);
    if (o > 0) __syncthreads();
    for (int i = tid; i < c; i += T) {
      const double ti = t[o + i];
      sPD[i] = lin ? make_ulonglong2(phase_fixed64(ti, fa), phase_fixed64(ti, df))
                   : make_ulonglong2((unsigned long long)__double_as_longlong(ti), 0ull);
    }
    if (tid == 0) sPD[c] = make_ulonglong2(0ull, 0ull);  // read by the last iteration's prefetch, never used
    __syncthreads();
    if (lin) {
      ulonglong2 pd = sPD[0];
#pragma unroll 4
      for (int i = 0; i < c; ++i) {
        const ulonglong2 pdn = sPD[i + 1];  // i + 1 <= c <= kEntChunk: staged or the zeroed record
        // the R phases are independent multiply-adds (no serial chain of 64-bit adds)
        unsigned long long phi[R];
        phi[0] = pd.x + (unsigned long long)j0 * pd.y;
#pragma unroll
        for (int r = 1; r < R; ++r) phi[r] = phi[0] + (unsigned long long)r * pd.y;
#pragma unroll
        for (int r = 0; r < R; ++r) count_up(col + 4u * (unsigned)(r * T) + bin_of_phase(phi[r], (unsigned)M) * step);
        pd = pdn;
      }
    } else {
      for (int i = 0; i < c; ++i) {
        const double ti = __longlong_as_double((long long)sPD[i].x);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int64_t k = fanchor + j0 + r;
          count_up(col + 4u * (unsigned)(r * T) + bin_of_phase(phase_fixed64(ti, freqs[k < nfreq ? k : nfreq - 1]), (unsigned)M) * step);
        }
      }
    }
  }
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t k = fanchor + j0 + r;
    if (k < nfreq) {
      float s = 0.f;
      for (int m = 0; m < M; ++m) {
        const unsigned q = read_count(col + 4u * (unsigned)(r * T) + (unsigned)m * step);
        if (q > 1u) s += (float)q * (q < kEntTable ? logq[q] : logf((float)q));
      }
      H_out[k] = entropy_from_counts_sum(s, (float)n);
    }
  }
}

// One warp per (curve, peak): counts in shared memory, H, then the z-score.
constexpr int kPeakWarps = 4;

__global__ void __launch_bounds__(kPeakWarps * 32) entropy_peaks_kernel(const int64_t* offsets, int64_t ncurves,
                                                                        const double* t, const double* freqs,
                                                                        int64_t nfreq, int M, int k,
                                                                        const int32_t* topk_idx, float* H_out,
                                                                        float* z_out) {
  extern __shared__ __align__(16) unsigned char smem[];
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  unsigned* cnt = reinterpret_cast<unsigned*>(smem) + warp * M;
  const int64_t total = ncurves * k;
  for (int64_t e = (int64_t)blockIdx.x * kPeakWarps + warp; e < total; e += (int64_t)gridDim.x * kPeakWarps) {
    const int64_t c = e / k;
    const int32_t fi = topk_idx[e];
    if (fi < 0 || fi >= nfreq) {
      if (lane == 0) {
        H_out[e] = __int_as_float(0x7fc00000);
        z_out[e] = __int_as_float(0x7fc00000);
      }
      continue;
    }
    for (int m = lane; m < M; m += 32) cnt[m] = 0u;
    __syncwarp();
    const double f = freqs[fi];
    const int64_t o0 = offsets[c], n = offsets[c + 1] - o0;
    for (int64_t i = lane; i < n; i += 32) atomicAdd(&cnt[bin_of_phase(phase_fixed64(t[o0 + i], f), (unsigned)M)], 1u);
    __syncwarp();
    float s = 0.f;
    for (int m = lane; m < M; m += 32) {
      const unsigned q = cnt[m];
      if (q > 1u) s += (float)q * logf((float)q);
    }
#pragma unroll
    for (int d = 16; d > 0; d >>= 1) s += __shfl_xor_sync(0xffffffffu, s, d);
    if (lane == 0) {
      const float N = (float)n;
      const float H = entropy_from_counts_sum(s, N);
      const double Md = (double)M, Nd = (double)n;
      float z = __int_as_float(0x7fc00000);
      if (n > 0 && M > 1) {
        const double E = log(Md) - (Md - 1.0) / (2.0 * Nd) - (Md - 1.0) * (Md + 1.0) / (12.0 * Nd * Nd);
        const double V = (Md - 1.0) / (2.0 * Nd * Nd) + (Md * Md - 1.0) / (6.0 * Nd * Nd * Nd);
        z = (float)(((double)H - E) / sqrt(V));
      }
      H_out[e] = H;
      z_out[e] = z;
    }
    __syncwarp();
  }
}

}  // namespace

cudaError_t launch_entropy_dense(const double* t, int64_t n, const double* freqs, int64_t nfreq, int M, int nsm,
                                 float* H_out, cudaStream_t st) {
  if (nfreq <= 0) return cudaSuccess;
  // Frequencies between anchors: the counts of one span fill about 48 KB (four
  // blocks per SM). A thread takes as many frequencies as that leaves it, the
  // staged record and the loop being shared by them (1000 times x 1e6
  // frequencies, counts/s at R = 8, 4, 2, 1: M = 10 3.32e12, 3.11e12, 2.51e12,
  // 1.72e12; M = 20 2.51e12 (two blocks per SM), 3.05e12, 2.49e12, 1.72e12;
  // M = 50 R = 4 2.07e12, R = 2 2.31e12), and fewer while that leaves under two
  // blocks per SM (1e5 frequencies, M = 10: 1.21e12, 1.38e12, 1.45e12, 1.10e12),
  // under one from R = 2 on (6e4 frequencies, M = 31: R = 1 2 % slower; 1e4: 10 % faster).
  const int span = M <= 12 ? 1024 : (M <= 24 ? 512 : (M <= 96 ? 256 : 128));
  int R = span / kEntThreads;
  while (R > 1 && (nfreq + R * kEntThreads - 1) / (R * kEntThreads) < (R > 2 ? 2 : 1) * nsm) R >>= 1;
  const void* fn = R == 8   ? reinterpret_cast<const void*>(&entropy_dense_kernel<8>)
                   : R == 4 ? reinterpret_cast<const void*>(&entropy_dense_kernel<4>)
                   : R == 2 ? reinterpret_cast<const void*>(&entropy_dense_kernel<2>)
                            : reinterpret_cast<const void*>(&entropy_dense_kernel<1>);
  const size_t smem = (size_t)(kEntChunk + 1) * 16 + kEntTable * 4 + (size_t)R * M * kEntThreads * 4;
  const cudaError_t e = allow_shared_memory(fn, 64);  // s_tm, s_df
  if (e != cudaSuccess) return e;
  const int64_t per_block = (int64_t)kEntThreads * R;
  const int64_t blocks = (nfreq + per_block - 1) / per_block;
  void* args[] = {const_cast<double**>(&t), &n, const_cast<double**>(&freqs), &nfreq, &M, const_cast<int*>(&span), &H_out};
  return cudaLaunchKernel(fn, dim3((unsigned)blocks), dim3(kEntThreads), args, smem, st);
}

cudaError_t launch_entropy_peaks(const int64_t* offsets, int64_t ncurves, const double* t, const double* freqs,
                                 int64_t nfreq, int M, int k, const int32_t* topk_idx, float* H_out, float* z_out,
                                 cudaStream_t st) {
  const int64_t total = ncurves * k;
  if (total <= 0) return cudaSuccess;
  const size_t smem = (size_t)kPeakWarps * M * 4;
  const cudaError_t e = allow_shared_memory(reinterpret_cast<const void*>(&entropy_peaks_kernel), 0);
  if (e != cudaSuccess) return e;
  int64_t blocks = (total + kPeakWarps - 1) / kPeakWarps;
  blocks = blocks > 65535 ? 65535 : blocks;
  entropy_peaks_kernel<<<(unsigned)blocks, kPeakWarps * 32, smem, st>>>(
      offsets, ncurves, t, freqs, nfreq, M, k, topk_idx, H_out, z_out);
  return cudaGetLastError();
}

}  // namespace fpw
