// Curves that share their observation times (Section 4 and the batch routine of
// Appendix D): the bins of every (observation, frequency) pair are the same for
// all curves, so per frequency the bin sums of a whole group of curves are one
// matrix product
//
//   D[(curve, part), (frequency, bin)] = sum_i  V[(curve, part), i] * H[i, (frequency, bin)]
//
// with V the per-observation values (part 0: a_i = x_i / sigma_i^2, part 1:
// w_i = 1 / sigma_i^2) and H the one-hot bin matrix (H[i, (f, m)] = 1 iff
// observation i falls in bin m at frequency f). That product runs on the
// tensor cores (tcgen05.mma kind::f16, FP32 accumulators in tensor memory):
//
// * V in fp16 with FP32-level precision: each value is scaled by a power of two
//   per curve and part (exact), then split v = hi + lo into two fp16 numbers;
//   hi and lo are adjacent entries of the K dimension, and the one-hot row of
//   the observation is duplicated for both, so the tensor core adds hi + lo
//   itself. Products with the one-hot entries are exact; sums are FP32.
// * H is built in shared memory for each chunk of 32 observations from exact
//   phases (phase_fixed64: the integer product of the binary64 significands),
//   so bins equal floor(M frac(t f)) except within 2^-32 of a cycle below an edge.
// * Groups of 64 curves are taken two at a time, one accumulator for part 0 and
//   one for part 1 of their 128 curves; a group left over (or every group, where
//   few items make pairs the slower way) is taken by itself,
//   parts in neighbouring rows, an accumulator for each half of the pass.
// * One CTA per SM (persistent over (groups, frequency pass) work items) holds
//   two accumulators of 128 x N (N = frequencies per accumulator x M <= 256) in
//   512 TMEM columns; V chunks arrive by bulk copy (TMA) into a
//   double buffer, H is double-buffered too, and the single issuing thread's
//   MMAs signal an mbarrier per buffer (tcgen05.commit).
// * The epilogue reads D with tcgen05.ld (a pair of groups: lane = curve; one
//   group: lane = (curve, part), paired with one shuffle), and reduces S = sum_m A_m^2 / (B_m +
//   1/alpha^2) per frequency into a dense FP32 array; a per-curve top-k pass
//   follows.
//
// Every wait (mbarrier) is bounded by a clock limit; on expiry the kernel sets
// kStatusTimeout, waits (bounded) for its own copies and MMAs, frees its tensor
// memory and returns.
#include <cuda_fp16.h>
#include <math.h>

#include "fpw_shared.cuh"

namespace fpw {
namespace {

constexpr int kShCurves = 64;                   // curves per group
constexpr int kShRows = 128;                    // MMA M: (curve, part) rows
constexpr int kShObs = 32;                      // observations per chunk
constexpr int kShK = 2 * kShObs;                // K entries per chunk (hi, lo)
constexpr int kShKSteps = kShK / 16;            // MMA k-steps per chunk
constexpr int kShChunkBytes = kShRows * kShK * 2;  // V image of one chunk: 16 KB
constexpr int kShThreads = 576;  // 16 builder/epilogue warps + 2 issuer warps
constexpr int kShNMax = 256;                    // MMA N limit (M = 128)
constexpr int kShMaxFpm = 64;                   // frequencies per accumulator, at most
constexpr int kShHOperandMax = kShNMax * kShK * 2;   // one H operand of a chunk: 32 KB
constexpr int kShHSlotBytes = 2 * kShHOperandMax;    // two H operands (two accumulators of one group)
constexpr int kShTmemCols = 512;
constexpr unsigned kOneOne = 0x3C003C00u;       // two fp16 1.0
constexpr long long kWaitClocks = 4000000000LL; // default wait limit, ~2 s at 2 GHz
// A waiting thread is suspended in mbarrier.try_wait until the phase completes
// or this many nanoseconds pass (so waiting warps do not take issue slots).
constexpr uint32_t kSuspendNs = 20000u;
constexpr int kMaxPassFreqs = 2 * kShMaxFpm;
constexpr int kMaxPairs = kMaxPassFreqs * kShObs;
constexpr int kShVSlots = 4;                    // V chunks in flight: loads run two chunks ahead
constexpr int kShStage = 1024;                  // observations staged at a time (t, anchor P, step D)
constexpr int kShStageChunks = kShStage / kShObs;

// Shared-memory carve-up (bytes).
constexpr int kOffV = 0;                                   // V chunks: 4 x 16 KB, or 4 x 32 KB for two groups
constexpr int kOffOld = kOffV + kShVSlots * kShChunkBytes + 2 * kShHSlotBytes;  // (H chunks: 2 x 64 KB, or 2 x 32 KB) bin of every (frequency, observation) pair in H, per slot
constexpr int kOffF = kOffOld + 2 * kMaxPairs;             // the pass's frequencies (binary64)
constexpr int kOffStage = kOffF + kMaxPassFreqs * 8;       // t, P, D of kShStage observations
constexpr int kOffPart = kOffStage + 3 * kShStage * 8;    // epilogue: partial S of a frequency split between warps
constexpr int kOffBar = kOffPart + 2 * 128 * 4;
constexpr int kSmemBytes = kOffBar + 128;

// Byte offset of element (row r, k-entry q) of a K-major, unswizzled operand
// with R rows and kShK columns: one 16-column k-step after another; inside a
// k-step, 8-row x 16-byte core matrices, the two of a row group adjacent (the
// K-direction stride, 128 B) and row groups 256 B apart.
__host__ __device__ __forceinline__ uint32_t km_off(uint32_t r, uint32_t q, uint32_t R) {
  return (q >> 4) * (R * 32u) + (r >> 3) * 256u + ((q >> 3) & 1u) * 128u + (r & 7u) * 16u + (q & 7u) * 2u;
}

// Approximate reciprocal (one special-function instruction, relative error
// about 2^-23), subnormal inputs and results flushed to zero: the epilogue
// drops denominators below FLT_MIN, and a reciprocal that flushes (a
// denominator above 2^126) leaves a term far below the absolute tolerance.
__device__ __forceinline__ float rcp_approx(float x) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(x));
  return r;
}

__device__ __forceinline__ uint32_t smem_addr(const void* p) { return (uint32_t)__cvta_generic_to_shared(p); }

// tcgen05 shared-memory matrix descriptor: unswizzled, K-direction core-matrix
// stride 128 B (leading byte offset), row-group stride 256 B (stride byte offset).
__device__ __forceinline__ uint64_t smem_desc(uint32_t saddr) {
  uint64_t d = (uint64_t)((saddr & 0x3FFFFu) >> 4);
  d |= (uint64_t)(128u >> 4) << 16;
  d |= (uint64_t)(256u >> 4) << 32;
  d |= (uint64_t)1 << 46;  // descriptor version
  return d;
}

// Instruction descriptor, kind::f16: fp16 A and B (K-major), FP32 D, M x N.
__device__ __forceinline__ uint32_t mma_idesc(int M, int N) {
  return (1u << 4) | ((uint32_t)(N >> 3) << 17) | ((uint32_t)(M >> 4) << 24);
}

// Bounded wait for completion of phase `parity` of an mbarrier.
__device__ __forceinline__ bool mbar_wait(uint64_t* bar, uint32_t parity) {
  const long long t0 = clock64();
  while (true) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity), "r"(kSuspendNs)
        : "memory");
    if (done) return true;
    if (clock64() - t0 > kWaitClocks) return false;
  }
}

// mbarrier wait of the chunk pipeline: gives up after `limit` clocks or when
// another role of the CTA set *abort; `suspend_ns` is the longest time one
// try_wait may suspend the thread.
__device__ __forceinline__ bool mbar_wait_ab(uint64_t* bar, uint32_t parity, volatile int* abort, long long limit,
                                             uint32_t suspend_ns) {
  const long long t0 = clock64();
  while (true) {
    uint32_t done;
    asm volatile(
        "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\tselp.u32 %0, 1, 0, p;\n\t}\n"
        : "=r"(done)
        : "r"(smem_addr(bar)), "r"(parity), "r"(suspend_ns)
        : "memory");
    if (done) return true;
    if (*abort || clock64() - t0 > limit) return false;
  }
}

__device__ __forceinline__ void mbar_init_n(uint64_t* bar, uint32_t count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;" ::"r"(smem_addr(bar)), "r"(count) : "memory");
}

__device__ __forceinline__ void mbar_arrive(uint64_t* bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];" ::"r"(smem_addr(bar)) : "memory");
}

// Named barrier among the builder warps only (the issuer warp never joins).
__device__ __forceinline__ void builders_sync(int nthreads) {
  asm volatile("bar.sync 1, %0;" ::"r"(nthreads) : "memory");
}

__device__ __forceinline__ bool builders_or(bool v, int nthreads) {
  uint32_t r;
  asm volatile(
      "{\n\t.reg .pred p, q;\n\tsetp.ne.u32 p, %1, 0;\n\tbar.red.or.pred q, 1, %2, p;\n\tselp.u32 %0, 1, 0, q;\n\t}\n"
      : "=r"(r)
      : "r"((uint32_t)v), "r"(nthreads)
      : "memory");
  return r != 0u;
}

__device__ __forceinline__ void mbar_expect(uint64_t* bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;" ::"r"(smem_addr(bar)), "r"(bytes) : "memory");
}

__device__ __forceinline__ void bulk_load(void* dst, const void* src, uint32_t bytes, uint64_t* bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];" ::"r"(
                   smem_addr(dst)),
               "l"(src), "r"(bytes), "r"(smem_addr(bar))
               : "memory");
}

__device__ __forceinline__ void mma_f16(uint32_t d_tmem, uint64_t da, uint64_t db, uint32_t idesc, uint32_t acc) {
  asm volatile(
      "{\n\t.reg .pred p;\n\tsetp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f16 [%0], %1, %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "l"(da), "l"(db), "r"(idesc), "r"(acc)
      : "memory");
}

__device__ __forceinline__ void mma_commit(uint64_t* bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];" ::"r"(smem_addr(bar))
               : "memory");
}

// tcgen05.ld of 8 columns without the wait; the registers are valid only after
// tmem_wait_ld8 on the same array, which names them as operands so that no
// use of them can be scheduled before the wait.
__device__ __forceinline__ void tmem_ld8_issue(uint32_t taddr, uint32_t (&v)[8]) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x8.b32 {%0, %1, %2, %3, %4, %5, %6, %7}, [%8];"
               : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7])
               : "r"(taddr));
}

__device__ __forceinline__ void tmem_wait_ld8(uint32_t (&v)[8]) {
  asm volatile("tcgen05.wait::ld.sync.aligned;"
               : "+r"(v[0]), "+r"(v[1]), "+r"(v[2]), "+r"(v[3]), "+r"(v[4]), "+r"(v[5]), "+r"(v[6]), "+r"(v[7])
               :
               : "memory");
}

__device__ __forceinline__ void fence_before_sync() { asm volatile("tcgen05.fence::before_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_after_sync() { asm volatile("tcgen05.fence::after_thread_sync;" ::: "memory"); }
__device__ __forceinline__ void fence_async_smem() { asm volatile("fence.proxy.async.shared::cta;" ::: "memory"); }

// ---------------------------------------------------------------- prep
// One block per curve slot of the padded groups: validation, per-curve
// power-of-two scales, and the fp16 hi/lo image of (a, w) in the operand
// layout, one 16 KB chunk per (group, 32 observations). Bound by the binary64
// division of every observation (a warp's binary64 instruction occupies the SM
// for about 20 clocks): one, not one a pass, and integer maxima, 143 us ->
// 32 us for 512 curves of 1000.
constexpr int kShPrepKeep = 4;
__global__ void __launch_bounds__(256) shared_prep_kernel(const SharedArgs a) {
  __shared__ unsigned long long red_a[8], red_w[8];
  __shared__ int red_bad[8];
  const int64_t c = blockIdx.x;  // padded curve slot
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int64_t n = a.n;
  const bool real = c < a.ncurves;
  // maxima as bit patterns (the values are not negative); a thread's first
  // kShPrepKeep observations stay in registers for the second pass
  unsigned long long amax = 0ull, wmax = 0ull;
  int bad = 0;
  double kw[kShPrepKeep] = {}, ka[kShPrepKeep] = {};
  auto weigh = [&](int64_t i, double& w, double& v) {
    const double s = a.sigma[c * n + i], x = a.x[c * n + i], t = a.t[i];
    const bool ok = isfinite(s) && isfinite(x) && isfinite(t) && s > 0.0;
    w = ok ? 1.0 / (s * s) : 0.0;
    v = ok ? x * w : 0.0;
    if (!ok) bad = 1;
    const unsigned long long av = (unsigned long long)__double_as_longlong(v) & 0x7fffffffffffffffull;
    const unsigned long long wv = (unsigned long long)__double_as_longlong(w);
    if (av > amax && av <= 0x7ff0000000000000ull) amax = av;  // NaN left out
    if (wv > wmax) wmax = wv;
  };
  if (real) {
#pragma unroll
    for (int q = 0; q < kShPrepKeep; ++q) {
      const int64_t i = tid + (int64_t)q * 256;
      if (i < n) weigh(i, kw[q], ka[q]);
    }
    for (int64_t i = tid + (int64_t)kShPrepKeep * 256; i < n; i += 256) {
      double w, v;
      weigh(i, w, v);
    }
  }
  auto larger = [](unsigned long long p, unsigned long long q) { return p > q ? p : q; };
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    amax = larger(amax, __shfl_xor_sync(0xffffffffu, amax, o));
    wmax = larger(wmax, __shfl_xor_sync(0xffffffffu, wmax, o));
    bad |= __shfl_xor_sync(0xffffffffu, bad, o);
  }
  if (lane == 0) {
    red_a[warp] = amax;
    red_w[warp] = wmax;
    red_bad[warp] = bad;
  }
  __syncthreads();
  amax = wmax = 0ull;
  bad = 0;
  for (int q = 0; q < (int)(blockDim.x >> 5); ++q) {
    amax = larger(amax, red_a[q]);
    wmax = larger(wmax, red_w[q]);
    bad |= red_bad[q];
  }
  // scale so that the largest magnitude lies in [2^14, 2^15): fp16 holds it
  // with room for the hi + lo split; an all-zero part keeps scale 1
  const int ea = amax > 0ull ? 14 - ilogb(__longlong_as_double((long long)amax)) : 0;
  const int ew = wmax > 0ull ? 14 - ilogb(__longlong_as_double((long long)wmax)) : 0;
  if (tid == 0) {
    a.inv_scale[2 * c] = real ? ldexpf(1.0f, -ea) : 0.0f;
    a.inv_scale[2 * c + 1] = real ? ldexpf(1.0f, -ew) : 0.0f;
    a.curve_bad[c] = (uint8_t)(real && bad);
    if (real && bad) atomicOr(a.status, kStatusData);
  }
  // rows of the curve's parts: in a pair of groups one image holds a, the other
  // w of the pair's 128 curves; in a group by itself the parts are neighbours
  const int64_t g = c / kShCurves;
  const size_t gbytes = (size_t)a.nchunks * kShChunkBytes;
  const bool paired = g < a.pair_groups;
  const uint32_t row = paired ? (uint32_t)(c % (2 * kShCurves)) : (uint32_t)(c % kShCurves) * 2u;
  unsigned char* const img = a.image + (size_t)(paired ? (g & ~(int64_t)1) : g) * gbytes;
  const size_t wpart = paired ? gbytes : 0;
  const uint32_t wrow = paired ? row : row + 1u;
  const bool zero = !real || bad;
  const int64_t npad = a.nchunks * kShObs;
  auto put = [&](int64_t i, double w, double v) {
    const float av = zero ? 0.f : (float)ldexp(v, ea), wv = zero ? 0.f : (float)ldexp(w, ew);
    const __half ah = __float2half_rn(av), wh = __float2half_rn(wv);
    const __half al = __float2half_rn(av - __half2float(ah)), wl = __float2half_rn(wv - __half2float(wh));
    unsigned char* ch = img + (size_t)(i / kShObs) * kShChunkBytes;
    const uint32_t q = 2u * (uint32_t)(i % kShObs);
    *reinterpret_cast<__half2*>(ch + km_off(row, q, kShRows)) = __halves2half2(ah, al);
    *reinterpret_cast<__half2*>(ch + wpart + km_off(wrow, q, kShRows)) = __halves2half2(wh, wl);
  };
#pragma unroll
  for (int q = 0; q < kShPrepKeep; ++q) {
    const int64_t i = tid + (int64_t)q * 256;
    if (i < npad) put(i, kw[q], ka[q]);
  }
  for (int64_t i = tid + (int64_t)kShPrepKeep * 256; i < npad; i += 256) {
    double w = 0.0, v = 0.0;
    if (!zero && i < n) {
      const double s = a.sigma[c * n + i];
      w = 1.0 / (s * s);
      v = a.x[c * n + i] * w;
    }
    put(i, w, v);
  }
  for (int64_t q = (int64_t)blockIdx.x * 256 + tid; q < a.nfreq; q += (int64_t)gridDim.x * 256)
    if (!isfinite(a.freqs[q])) atomicOr(a.status, kStatusGrid);
}

// ---------------------------------------------------------------- phase steps
// Per observation: the 64-bit phase step D_i = frac(t_i df) for the grid's
// mean spacing df, and max |t| (for the grid-linearity bound).
__global__ void shared_steps_kernel(const SharedArgs a) {
  const int64_t F = a.nfreq;
  const double df = (F > 1) ? (a.freqs[F - 1] - a.freqs[0]) / (double)(F - 1) : 0.0;
  for (int64_t i = (int64_t)blockIdx.x * blockDim.x + threadIdx.x; i < a.n; i += (int64_t)gridDim.x * blockDim.x) {
    const double t = a.t[i];
    const bool ok = isfinite(t) && isfinite(df);
    a.step[i] = ok ? phase_fixed64(t, df) : 0ull;
    if (ok) atomicMax(a.tmax_bits, (unsigned long long)__double_as_longlong(fabs(t)));
  }
}

// ---------------------------------------------------------------- MMA kernel
// Warp-specialised pipeline over this CTA's stream of chunks (32 observations
// of one item each; gc counts them across items):
//  * builder warps (0-14): for chunk gc, wait until the MMAs of gc - 2 have
//    released H slot gc & 1 (mbarrier `empty`), then each (frequency,
//    observation) pair clears its previous one in that slot and sets its new
//    one (pairs own disjoint 4-byte words; phases step from staged anchors,
//    Phi = P_i + j D_i, when the pass lies on the linear grid, else exact
//    anchors per pair); each warp then arrives on `full`. At an item's end
//    warps 0-7 read the accumulators (after `acc`) and arrive on `tfree`.
//  * issuer warp (15, one lane): waits for `full`, starts the bulk copy of the
//    V chunk two chunks ahead (its slot was last read by the MMAs of gc - 2,
//    complete once `full` of gc has completed), waits for V of gc (and, on an
//    item's first chunk, for `tfree`), issues the 2 x 4 MMAs and commits them
//    to `empty` (and to `acc` after an item's last chunk).
// No block-wide barrier inside the loop; every wait is bounded and gives up
// when another role has set the abort flag.
constexpr int kShBuilderWarps = 16;
constexpr int kShBuilders = kShBuilderWarps * 32;
constexpr int kShIssuers = kShThreads / 32 - kShBuilderWarps;  // one per accumulator

// Epilogue of a pair of groups: accumulator 0 holds the sums of a, accumulator 1
// those of w, of the pair's 128 curves (TMEM lane = curve) at fpm frequencies,
// so a lane reads both sums of a bin and forms S by itself. Warp w takes lanes
// 32 (w % 4) .. + 31 and the (w / 4)-th quarter of the frequencies; 8 columns
// per step, the next step's loads in flight. The terms are added in the order of
// the epilogue of one group (even and odd columns of a step apart from M = 8 on,
// a frequency in two parts where it holds that epilogue's split column), so S does
// not depend on how a call's groups are taken (512 curves x 1000 times x 50000
// frequencies, M = 20: 3050 us a call, 3037 with an order of its own).
__device__ __forceinline__ void pair_epilogue(const SharedArgs& a, uint32_t tmem, int64_t c, int64_t f0, bool cbad, float2 scale,
                                              int warp, int lane) {
  const int M = a.M, quarter = warp & 3, seg = warp >> 2;
  const int64_t F = a.nfreq;
  const bool cvalid = c < a.ncurves;
  const float sa = scale.x, sw = scale.y, cal = (float)a.inv_alpha2;
  int jl = seg * a.fpm / 4;
  const int jend = (seg + 1) * a.fpm / 4;
  if (jl >= jend) return;
  const int cb = jl * M, ce = jend * M;
  const int jmax = (int)((F - f0) < jend ? (F - f0) : jend);
  float* const s32 = a.S32 ? (cvalid ? a.S32 + c * F + f0 : a.scratch32 + lane * kShMaxFpm) : nullptr;
  double* const s64 = a.S_out ? (cvalid ? a.S_out + c * F + f0 : a.scratch64 + lane * kShMaxFpm) : nullptr;
  const float nan = __int_as_float(0x7fc00000);
  const uint32_t ta = tmem + ((uint32_t)(quarter * 32) << 16), tb = ta + 256u;
  const int split = ((a.fpm * M + 15) >> 4) << 3;
  float acc0 = 0.f, acc1 = 0.f, part = 0.f;  // even and odd columns; the sum up to the split column
  int fend = cb + M;             // where frequency jl ends (warp-uniform)
  auto term = [&](uint32_t va, uint32_t vb) {
    const float A = __uint_as_float(va) * sa, den = __uint_as_float(vb) * sw + cal;
    return den >= 1.17549435e-38f ? (A * A) * rcp_approx(den) : 0.f;
  };
  if (a.nchunks == 0) {  // no observations: no MMA has written the accumulators
    for (; jl < jmax; ++jl) {
      if (s32) s32[jl] = 0.f;
      if (s64) s64[jl] = 0.0;
    }
    return;
  }
  uint32_t na[8], nb[8];
  int c0 = cb & ~7;
  const int clast = (ce - 1) & ~7;
  tmem_ld8_issue(ta + (uint32_t)c0, na);
  tmem_ld8_issue(tb + (uint32_t)c0, nb);
#pragma unroll 1
  for (; c0 < ce; c0 += 8) {
    uint32_t va[8], vb[8];
    tmem_wait_ld8(na);
    tmem_wait_ld8(nb);
#pragma unroll
    for (int u = 0; u < 8; ++u) {
      va[u] = na[u];
      vb[u] = nb[u];
    }
    // (the last step loads its own columns again: no load is conditional, so none is moved before its wait)
    const uint32_t cn = (uint32_t)(c0 < clast ? c0 + 8 : clast);
    tmem_ld8_issue(ta + cn, na);
    tmem_ld8_issue(tb + cn, nb);
    if (c0 == split) {
      part = acc0 + acc1;
      acc0 = acc1 = 0.f;
    }
    auto emit = [&]() {  // frequency jl complete
      if (jl < jmax) {
        const float S = cbad ? nan : acc0 + acc1 + part;
        if (s32) s32[jl] = S;
        if (s64) s64[jl] = (double)S;
      }
      acc0 = acc1 = part = 0.f;
      ++jl;
      fend += M;
    };
    // (all conditions on columns are warp-uniform)
    if (c0 >= cb && fend > c0 + 8) {
      float lo0 = term(va[0], vb[0]), lo1 = term(va[1], vb[1]);
#pragma unroll
      for (int u = 2; u < 8; u += 2) {
        lo0 += term(va[u], vb[u]);
        lo1 += term(va[u + 1], vb[u + 1]);
      }
      acc0 += lo0;
      acc1 += lo1;
    } else if (M >= 8) {  // one frequency end at most
      float lo0 = 0.f, lo1 = 0.f, hi0 = 0.f, hi1 = 0.f;
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int col = c0 + u;
        if (col >= cb && col < ce) (u & 1 ? (col < fend ? lo1 : hi1) : (col < fend ? lo0 : hi0)) += term(va[u], vb[u]);
      }
      acc0 += lo0;
      acc1 += lo1;
      if (fend <= c0 + 8 && fend <= ce) {
        emit();
        acc0 = hi0;
        acc1 = hi1;
      }
    } else {
#pragma unroll
      for (int u = 0; u < 8; ++u) {
        const int col = c0 + u;
        if (col >= cb && col < ce) {
          acc0 += term(va[u], vb[u]);
          if (col + 1 == fend) emit();
        }
      }
    }
  }
  tmem_wait_ld8(na);
  tmem_wait_ld8(nb);
}

// kPaired: the two accumulators hold the two parts of two groups of curves at
// fpm frequencies: both multiply one H operand, and the epilogue finds a
// curve's sums in one lane. Else both parts of one group, rows side by side, at
// 2 fpm frequencies, two operands. A chunk's MMAs are the same, its one-hot
// stores halve; V, read from L2, doubles. A chunk takes 0.69 us either way, the
// MMAs' own time (1.76e15 FLOP/s with what the padding leaves); what the pair
// saves is the epilogue, without shuffles: 512 curves x 50000 frequencies, M =
// 20, 100 times 1133 us -> 895 with the epilogue below, 805 with it deferred;
// 1000 times 3187 -> 2930; M = 50 7219 -> 6927.
template <bool kPaired>
__global__ void __launch_bounds__(kShThreads, 1) shared_mma_kernel(const SharedArgs a) {
  constexpr int kVSlot = (kPaired ? 2 : 1) * kShChunkBytes, kHSlot = kShHSlotBytes / (kPaired ? 2 : 1);
  static_assert(kShVSlots * kVSlot + 2 * kHSlot <= kShVSlots * kShChunkBytes + 2 * kShHSlotBytes, "same area");
  extern __shared__ __align__(1024) unsigned char smem[];
  unsigned char* sV = smem + kOffV;
  unsigned char* sH = sV + kShVSlots * kVSlot;
  uint8_t* sOld = smem + kOffOld;
  double* sF = reinterpret_cast<double*>(smem + kOffF);
  double* sT = reinterpret_cast<double*>(smem + kOffStage);
  unsigned long long* sP = reinterpret_cast<unsigned long long*>(sT + kShStage);
  unsigned long long* sD = sP + kShStage;
  uint64_t* bar_full = reinterpret_cast<uint64_t*>(smem + kOffBar);  // [2]
  uint64_t* bar_empty = bar_full + 2;                                 // [2]
  uint64_t* bar_v = bar_empty + 2;                                    // [kShVSlots]
  uint64_t* bar_acc = bar_v + kShVSlots;
  uint64_t* bar_tfree = bar_acc + 1;
  uint32_t* tslot = reinterpret_cast<uint32_t*>(bar_tfree + 1);
  volatile int* s_abort = reinterpret_cast<volatile int*>(tslot + 1);

  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int M = a.M, fpm = a.fpm, Nm = a.n_mma, FP = kPaired ? fpm : 2 * fpm, rows_used = fpm * M;
  const int npairs = FP * kShObs;
  const int64_t F = a.nfreq, n = a.n, nch = a.nchunks;
  const bool resident = n <= kShStage;
  const bool grid_bad = (*(volatile unsigned*)a.status & kStatusGrid) != 0u;
  const int64_t items = grid_bad ? 0 : a.units * a.npass;
  const int64_t my_items = (int64_t)blockIdx.x < items ? (items - 1 - blockIdx.x) / gridDim.x + 1 : 0;
  const float cal = (float)a.inv_alpha2;
  const double df = (F > 1) ? (a.freqs[F - 1] - a.freqs[0]) / (double)(F - 1) : 0.0;
  const double tmax = __longlong_as_double((long long)*a.tmax_bits);
  const uint32_t op_bytes = (uint32_t)(Nm * kShK * 2);  // one H operand
  // byte offset of this lane's observation (hi, lo) word inside a row of H
  const uint32_t lane_off = (uint32_t)(lane >> 3) * (uint32_t)(Nm * 32) + (uint32_t)((lane >> 2) & 1) * 128u +
                            (uint32_t)(lane & 3) * 4u;

  if (tid == 0) {
    for (int q = 0; q < 2; ++q) {
      mbar_init_n(&bar_full[q], kShBuilderWarps);
      mbar_init_n(&bar_empty[q], kShIssuers);
    }
    for (int v = 0; v < kShVSlots; ++v) mbar_init_n(&bar_v[v], 1);
    mbar_init_n(bar_acc, kShIssuers);
    mbar_init_n(bar_tfree, kShBuilderWarps);
    *s_abort = 0;
    asm volatile("fence.mbarrier_init.release.cluster;" ::: "memory");
  }
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;" ::"r"(smem_addr(tslot)),
                 "r"(kShTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;" ::: "memory");
  }
  // H starts as all pairs in bin 0 (rows beyond fpm * M stay zero for good)
  for (int e = tid; e < 2 * kHSlot / 16; e += kShThreads)
    reinterpret_cast<uint4*>(sH)[e] = make_uint4(0u, 0u, 0u, 0u);
  __syncthreads();
  for (int e = tid; e < npairs; e += kShThreads) {
    const int j = e >> 5;
    const int op = j >= fpm ? 1 : 0;
    const uint32_t r = (uint32_t)((j - op * fpm) * M);
    const uint32_t w = lane_off + (uint32_t)op * op_bytes + (r >> 3) * 256u + (r & 7u) * 16u;
    for (int q = 0; q < 2; ++q) {
      *reinterpret_cast<uint32_t*>(sH + q * kHSlot + w) = kOneOne;
      sOld[q * kMaxPairs + e] = 0;
    }
  }
  fence_async_smem();
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tslot;
  bool fail = false;
  // limit of the pipeline's waits (the drain after a failure keeps the
  // default); a limit far below one suspension also stops each try_wait from
  // suspending, so that a wait whose phase is not complete gives up at once
  const long long wait_limit = a.wait_clocks > 0 ? a.wait_clocks : kWaitClocks;
  const uint32_t suspend_ns = wait_limit < 100000 ? 0u : kSuspendNs;

  if (warp >= kShBuilderWarps) {
    // ------------------------------------------------------------ issuers: warp 16 drives accumulator 0 and
    // the V loads, warp 17 accumulator 1; both commit to `empty` and `acc` (count 2)
    const int iop = warp - kShBuilderWarps;
    if (lane == 0 && my_items > 0 && nch > 0) {
      const uint32_t idesc = mma_idesc(kShRows, Nm);
      // descriptors of chunk operands: a base descriptor plus the byte offset / 16
      // in the start-address field (all offsets stay inside shared memory)
      const uint64_t dv0 = smem_desc(smem_addr(sV)), dh0 = smem_desc(smem_addr(sH));
      const int64_t total = my_items * nch;
      // the V-load cursor (item lk of this CTA, chunk lch) runs two chunks ahead
      // of the MMA cursor; both advance incrementally (no 64-bit division per chunk)
      int64_t lk = 0, lch = 0;
      const size_t gbytes = (size_t)nch * kShChunkBytes;  // one group's image
      auto unit_image = [&](int64_t it) {
        return a.image + (size_t)(a.group0 + (it / a.npass) * (kPaired ? 2 : 1)) * gbytes;
      };
      const unsigned char* limg = unit_image(blockIdx.x);
      auto load_next = [&](int slot) {
        mbar_expect(&bar_v[slot], kVSlot);
        bulk_load(sV + slot * kVSlot, limg + (size_t)lch * kShChunkBytes, kShChunkBytes, &bar_v[slot]);
        if (kPaired)
          bulk_load(sV + slot * kVSlot + kShChunkBytes, limg + gbytes + (size_t)lch * kShChunkBytes, kShChunkBytes,
                    &bar_v[slot]);
        if (++lch == nch) {
          lch = 0;
          ++lk;
          limg = unit_image(blockIdx.x + lk * gridDim.x);  // past the last item: formed, not read
        }
      };
      if (iop == 0)
        for (int64_t c = 0; c < 2 && c < total; ++c) load_next((int)c);
      // per-slot phase parities and flags as bit masks in registers (a
      // run-time-indexed array would live in local memory)
      uint32_t ph_full = 0u, ph_v = 0u, ph_tfree = 0u;
      uint32_t commits0 = 0u, commits1 = 0u;
      uint32_t v_out = iop == 0 ? ((total > 0 ? 1u : 0u) | (total > 1 ? 2u : 0u)) : 0u;  // own loads in flight
      int64_t ch = 0;
      for (int64_t gc = 0; gc < total && !fail; ++gc, ch = (ch + 1 == nch) ? 0 : ch + 1) {
        const int s = (int)(gc & 1), vs = (int)(gc & (kShVSlots - 1));
        if (!mbar_wait_ab(&bar_full[s], (ph_full >> s) & 1u, s_abort, wait_limit, suspend_ns)) { fail = true; break; }
        ph_full ^= 1u << s;
        if (iop == 0 && gc + 2 < total) {  // its slot was last read by the MMAs of gc - 2, done before `full` of gc
          const int v2 = (int)((gc + 2) & (kShVSlots - 1));
          load_next(v2);
          v_out |= 1u << v2;
        }
        if (!mbar_wait_ab(&bar_v[vs], (ph_v >> vs) & 1u, s_abort, wait_limit, suspend_ns)) { fail = true; break; }
        ph_v ^= 1u << vs;
        v_out &= ~(1u << vs);
        if (ch == 0 && gc > 0) {  // the previous item's accumulators have been read
          if (!mbar_wait_ab(bar_tfree, ph_tfree, s_abort, wait_limit, suspend_ns)) { fail = true; break; }
          ph_tfree ^= 1u;
        }
        fence_after_sync();
        const uint64_t dvs = dv0 + (uint64_t)((vs * kVSlot + (kPaired ? iop * kShChunkBytes : 0)) >> 4);
        const uint64_t dhs = dh0 + (uint64_t)((s * kHSlot + (kPaired ? 0 : iop * (int)op_bytes)) >> 4);
#pragma unroll
        for (int ks = 0; ks < kShKSteps; ++ks) {
          const uint32_t acc = (ch > 0 || ks > 0) ? 1u : 0u;
          mma_f16(tmem + (uint32_t)iop * 256u, dvs + (uint64_t)((ks * kShRows * 32) >> 4),
                  dhs + (uint64_t)(((uint32_t)ks * (uint32_t)(Nm * 32)) >> 4), idesc, acc);
        }
        mma_commit(&bar_empty[s]);
        if (s == 0) ++commits0; else ++commits1;
        if (ch == nch - 1) mma_commit(bar_acc);
      }
      if (fail) {
        *s_abort = 1;
        atomicOr(a.status, kStatusTimeout);
        // nothing may be in flight when the CTA frees TMEM and exits: bounded
        // waits for the last commit of each slot and for outstanding V loads
        for (int q = 0; q < 2; ++q)
          if ((q == 0 ? commits0 : commits1) > 0u) mbar_wait(&bar_empty[q], ((q == 0 ? commits0 : commits1) - 1u) & 1u);
        for (int v = 0; v < kShVSlots; ++v)
          if ((v_out >> v) & 1u) mbar_wait(&bar_v[v], (ph_v >> v) & 1u);
      }
    }
  } else {
    // ------------------------------------------------------------ builders (+ epilogue in warps 0-7)
    // Every builder runs the same loops to the end and passes every named
    // barrier even after a failure (it then skips the work), so no builder
    // can wait at a barrier for one that left; failure decisions are made
    // warp-uniform before any warp-collective instruction.
    uint32_t ph_empty = 0u, ph_acc = 0u;  // per-slot parities as bits
    bool staged = false;
    int64_t gc = 0;
    // a pair's epilogue runs once the next item's first chunk is built, so that
    // staging and building overlap the last MMAs
    int64_t gprev = 0, fprev = 0;
    auto finish_pair = [&]() {
      const int64_t c = gprev * kShCurves + (warp & 3) * 32 + lane;  // loads before the wait
      const bool cbad = c < a.ncurves && a.curve_bad[c];
      const float2 scale = reinterpret_cast<const float2*>(a.inv_scale)[c];
      if (!fail && nch > 0) {
        fail = !mbar_wait_ab(bar_acc, ph_acc, s_abort, wait_limit, suspend_ns);
        fence_after_sync();
      }
      fail = __any_sync(0xffffffffu, fail);
      if (fail && lane == 0) *s_abort = 1;
      if (!fail) pair_epilogue(a, tmem, c, fprev, cbad, scale, warp, lane);
      fence_before_sync();
      __syncwarp();
      if (!fail && nch > 0 && lane == 0) mbar_arrive(bar_tfree);
      ph_acc ^= 1u;
    };
    for (int64_t k = 0; k < my_items; ++k) {
      const int64_t item = blockIdx.x + k * gridDim.x;
      const int64_t g = a.group0 + (item / a.npass) * (kPaired ? 2 : 1), p = item % a.npass;
      const int64_t f0 = p * FP;
      // anchors every 2 fpm frequencies, whichever way a pass takes them
      const int jo = kPaired && (p & 1) ? fpm : 0;
      const double fa = a.freqs[f0 - jo];
      if (k > 0) builders_sync(kShBuilders);  // every builder is done with the previous item's sF and stage
      // on the line, all of them or none, whichever part of them is this pass
      bool nonlin = false;
      for (int j = tid; j < 2 * fpm; j += kShBuilders) {
        const int64_t fi = f0 - jo + j;
        const double f = fi < F ? a.freqs[fi] : 0.0;
        if (j >= jo && j < jo + FP) sF[j - jo] = f;
        if (fi < F && fabs(f - fma((double)j, df, fa)) * tmax > kGridTolCycles) nonlin = true;
      }
      const bool lin = !builders_or(nonlin, kShBuilders);
      for (int64_t ch = 0; ch < nch; ++ch, ++gc) {
        const int s = (int)(gc & 1);
        if (ch % kShStageChunks == 0) {  // stage a block of observations (same thread per entry throughout)
          if (ch > 0) builders_sync(kShBuilders);
          const int64_t o0 = ch * kShObs;
          for (int i = tid; i < kShStage; i += kShBuilders) {
            const int64_t oi = o0 + i;
            if (!resident || !staged) {
              sT[i] = oi < n ? a.t[oi] : 0.0;
              sD[i] = oi < n ? a.step[oi] : 0ull;
            }
            sP[i] = phase_fixed64(sT[i], fa);
          }
          staged = true;
          builders_sync(kShBuilders);
        }
        if (!fail && gc >= 2) {  // the MMAs of gc - 2 read H slot s
          fail = !mbar_wait_ab(&bar_empty[s], (ph_empty >> s) & 1u, s_abort, wait_limit, suspend_ns);
          ph_empty ^= 1u << s;
        }
        fail = __any_sync(0xffffffffu, fail);
        if (fail && lane == 0) *s_abort = 1;  // the other roles stop waiting
        if (!fail) {
          unsigned char* hs = sH + s * kHSlot;
          uint8_t* old = sOld + s * kMaxPairs;
          const int ib = (int)(ch % kShStageChunks) * kShObs + lane;
          const bool obs_ok = ch * kShObs + lane < n;
          const unsigned long long P = sP[ib], D = sD[ib];
          const double tl = sT[ib];
          // pair e = (frequency e / 32, this lane's observation): clear its
          // previous one and set its new one; two pairs at a time, both bins
          // and both previous bins read before any store (the pairs' rows are
          // disjoint)
          auto put = [&](int e, unsigned m, unsigned mo) {
            const int j = e >> 5;  // warp-uniform
            const int op = j >= fpm ? 1 : 0;
            const uint32_t r0 = (uint32_t)((j - op * fpm) * M);
            const uint32_t base = lane_off + (uint32_t)op * op_bytes;
            const uint32_t ro = r0 + mo, rn = r0 + m;
            *reinterpret_cast<uint32_t*>(hs + base + (ro >> 3) * 256u + (ro & 7u) * 16u) = 0u;
            *reinterpret_cast<uint32_t*>(hs + base + (rn >> 3) * 256u + (rn & 7u) * 16u) = kOneOne;
            old[e] = (uint8_t)m;
          };
          if (lin) {
            for (int e = tid; e < npairs; e += 2 * kShBuilders) {
              const int e2 = e + kShBuilders;
              const bool two = e2 < npairs;  // warp-uniform
              const int ja = e >> 5, jb = e2 >> 5;
              const unsigned ma = (obs_ok && f0 + ja < F) ? bin_of_phase(P + (unsigned long long)(jo + ja) * D, (unsigned)M) : 0u;
              const unsigned mb =
                  (two && obs_ok && f0 + jb < F) ? bin_of_phase(P + (unsigned long long)(jo + jb) * D, (unsigned)M) : 0u;
              const unsigned oa = old[e], ob = two ? old[e2] : 0u;
              put(e, ma, oa);
              if (two) put(e2, mb, ob);
            }
          } else {
            for (int e = tid; e < npairs; e += kShBuilders) {
              const int j = e >> 5;
              const unsigned m = (obs_ok && f0 + j < F) ? bin_of_phase(phase_fixed64(tl, sF[j]), (unsigned)M) : 0u;
              put(e, m, old[e]);
            }
          }
          fence_async_smem();
          __syncwarp();
          if (lane == 0) mbar_arrive(&bar_full[s]);
        }
        if (kPaired && ch == 0 && k > 0) finish_pair();
      }
      if constexpr (kPaired) {
        gprev = g;
        fprev = f0;
        if (nch == 0 || k + 1 == my_items) finish_pair();
        continue;
      }
      if (!fail && nch > 0) {
        fail = !mbar_wait_ab(bar_acc, ph_acc, s_abort, wait_limit, suspend_ns);
        fence_after_sync();
      }
      fail = __any_sync(0xffffffffu, fail);
      if (fail && lane == 0) *s_abort = 1;
      // epilogue: all builder warps. Warp w reads TMEM lanes 32 (w % 4) .. + 31
      // of accumulator (w / 4) % 2, columns [0, split) for w < 8 and
      // [split, fpm M) above (split a multiple of 8 near the middle); the
      // partial sum of a frequency that straddles the split is handed over
      // through shared memory.
      float* sPart = reinterpret_cast<float*>(smem + kOffPart);
      const int quarter = warp & 3, op = (warp >> 2) & 1, half = warp >> 3;
      const int row = quarter * 32 + lane;
      const int64_t c = g * kShCurves + (row >> 1);
      const bool cvalid = c < a.ncurves;
      const int split = ((rows_used + 15) >> 4) << 3;
      const int js = split / M;                          // frequency holding column `split`
      const bool straddle = split < rows_used && split % M != 0;
      const int64_t fbase = f0 + (int64_t)op * fpm;
      const int jmax = (int)((F - fbase) < fpm ? (F - fbase) : fpm);
      const bool cbad = cvalid && a.curve_bad[c];
      // both lanes of a pair store the pair's sum to the same address
      // (one transaction, no divergent branch before the next shuffle); lanes
      // of padding curves write into a scratch area instead
      float* const s32 = a.S32 ? (cvalid ? a.S32 + c * F + fbase : a.scratch32 + lane * kShMaxFpm) : nullptr;
      double* const s64 = a.S_out ? (cvalid ? a.S_out + c * F + fbase : a.scratch64 + lane * kShMaxFpm) : nullptr;
      const float nan = __int_as_float(0x7fc00000);
      // this lane's part of the running frequency sum; the two lanes of a
      // curve's pair add up to the sum
      float acc = 0.f;
      if (!fail) {
        // lanes 2c and 2c + 1 hold the A and B rows of curve c. For M >= 8 the
        // pair splits each block of 8 columns: one shuffle per two columns gives
        // the even lane B of an even column and the odd lane A of an odd one, so
        // each lane forms the terms A^2 / (B + 1/alpha^2) of its own columns, and
        // a block holds at most one frequency end. Below 8 bins the even lane
        // forms every term.
        const float sa = cvalid ? a.inv_scale[2 * c] : 0.f, sw = cvalid ? a.inv_scale[2 * c + 1] : 0.f;
        const int cb = half == 0 ? 0 : split, ce = half == 0 ? split : rows_used;
        const int par = lane & 1;
        int jl = cb / M;
        int fend = (jl + 1) * M;  // the column where frequency jl ends (warp-uniform)
        auto emit = [&](float S) {  // frequency jl complete
          if (half == 1 && straddle && jl == js) {
            sPart[op * 128 + row] = S;  // the second part of the straddling frequency
          } else if (jl < jmax) {
            if (s32) s32[jl] = cbad ? nan : S;
            if (s64) s64[jl] = cbad ? (double)nan : (double)S;
          }
        };
        const uint32_t tbase = tmem + ((uint32_t)(quarter * 32) << 16) + (uint32_t)op * 256u;
        // 8 columns per step; the next step's TMEM load is in flight while
        // this step's columns are reduced
        uint32_t nx[8];
        if (nch > 0 && cb < ce) tmem_ld8_issue(tbase + (uint32_t)cb, nx);
        for (int c0 = cb; c0 < ce; c0 += 8) {
          uint32_t v[8];
          if (nch > 0) {
            tmem_wait_ld8(nx);
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = nx[u];
            if (c0 + 8 < ce) tmem_ld8_issue(tbase + (uint32_t)(c0 + 8), nx);
          } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) v[u] = 0u;
          }
          if (M >= 8) {
            float lo = 0.f, hi = 0.f;  // this lane's terms before / after the frequency end
#pragma unroll
            for (int q = 0; q < 4; ++q) {
              const float ev = __uint_as_float(v[2 * q]), od = __uint_as_float(v[2 * q + 1]);
              const float recv = __shfl_xor_sync(0xffffffffu, par ? ev : od, 1);
              const float A = (par ? recv : ev) * sa;
              const float den = (par ? od : recv) * sw + cal;
              const int col = c0 + 2 * q + par;
              const float term = (den >= 1.17549435e-38f && col < ce) ? (A * A) * rcp_approx(den) : 0.f;
              lo += col < fend ? term : 0.f;
              hi += col < fend ? 0.f : term;
            }
            acc += lo;
            if (fend <= c0 + 8 && fend <= ce) {
              emit(acc + __shfl_xor_sync(0xffffffffu, acc, 1));
              acc = hi;
              ++jl;
              fend += M;
            }
          } else {
#pragma unroll
            for (int u = 0; u < 8; ++u) {
              const float val = __uint_as_float(v[u]);
              const float other = __shfl_xor_sync(0xffffffffu, val, 1);
              const float A = val * sa;
              const float den = other * sw + cal;
              acc += (par == 0 && den >= 1.17549435e-38f && c0 + u < ce) ? (A * A) * rcp_approx(den) : 0.f;
              if (c0 + u < ce && c0 + u + 1 == fend) {  // warp-uniform
                emit(acc + __shfl_xor_sync(0xffffffffu, acc, 1));
                acc = 0.f;
                ++jl;
                fend += M;
              }
            }
          }
        }
      }
      fence_before_sync();
      builders_sync(kShBuilders);  // partial sums visible; every TMEM read of this item done
      if (!fail && half == 0 && straddle && js < jmax) {
        const float S = acc + __shfl_xor_sync(0xffffffffu, acc, 1) + sPart[op * 128 + (row & ~1)];
        if (s32) s32[js] = cbad ? nan : S;
        if (s64) s64[js] = cbad ? (double)nan : (double)S;
      }
      if (!fail && nch > 0 && lane == 0) mbar_arrive(bar_tfree);
      ph_acc ^= 1u;
    }
    if (fail) {
      *s_abort = 1;
      atomicOr(a.status, kStatusTimeout);
    }
  }
  // teardown: on success the last epilogue waited for `acc`, which covers
  // every MMA, and every V load was waited for; after a failure the issuer
  // drained its own work above
  fence_before_sync();
  __syncthreads();
  if (warp == 0)
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;" ::"r"(tmem), "r"(kShTmemCols) : "memory");
}

// ---------------------------------------------------------------- top-k
// One block per curve, one pass over its dense FP32 periodogram: every warp
// keeps the k best peaks of its part sorted in registers (entries lane and lane
// + 32), an element is looked at again only where it beats the warp's k-th,
// and the warps' lists are merged at the end. Peaks are integer keys, larger S
// first, then the lower index (0: no entry). Bound by the one read from L2 and
// memory. With a binary64 comparison a peak and a pass over the periodogram for
// each of the k picks, the call on 512 curves x 1000 times x 50000 frequencies,
// k = 5, took 3603 us in all; with this pass 3437.
constexpr int kShTopkThreads = 512;
constexpr int kShTopkWarps = kShTopkThreads / 32;
constexpr int kShTopkSteps = 4;  // loads in flight per lane

// Greater for what ranks first; a NaN (a peak only when every value is one) ranks last.
__device__ __forceinline__ unsigned long long topk_key(float s, unsigned e) {
  const unsigned u = __float_as_uint(s == 0.f ? 0.f : s);
  const unsigned r = s != s ? 1u : ((u >> 31) ? ~u : (u | 0x80000000u));
  return (unsigned long long)r << 32 | (0xFFFFFFFFu - e);
}

__global__ void __launch_bounds__(kShTopkThreads) dense_topk32_kernel(const DenseTopk32Args a) {
  __shared__ unsigned long long lists[kShTopkWarps][FPW_MAX_TOPK];
  const int64_t c = blockIdx.x;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5, k = a.k;
  const int64_t F = a.nfreq;
  const float* S = a.S32 + c * F;
  const bool grid_bad = (*(volatile unsigned*)a.status & kStatusGrid) != 0u;
  const bool bad = grid_bad || (a.curve_bad[c] & kCurveBad);
  unsigned long long k0 = 0ull, k1 = 0ull, tail = 0ull;  // entries lane, lane + 32; the k-th
  if (!bad) {
    for (int64_t base = (int64_t)warp * 32 * kShTopkSteps; base < F; base += kShTopkThreads * kShTopkSteps) {
      float s[kShTopkSteps], l[kShTopkSteps], r[kShTopkSteps];
#pragma unroll
      for (int u = 0; u < kShTopkSteps; ++u) {
        const int64_t e = base + 32 * u + lane;
        s[u] = e < F ? S[e] : 0.f;
        l[u] = (!a.peak_raw && e > 0 && e < F) ? S[e - 1] : -INFINITY;
        r[u] = (!a.peak_raw && e + 1 < F) ? S[e + 1] : -INFINITY;
      }
#pragma unroll
      for (int u = 0; u < kShTopkSteps; ++u) {
        const int64_t e = base + 32 * u + lane;
        bool peak = e < F;
        if (!a.peak_raw)
          peak = peak && (e == 0 ? (F == 1 || s[u] >= r[u]) : (e + 1 == F ? s[u] > l[u] : (s[u] > l[u] && s[u] >= r[u])));
        const unsigned long long key = peak ? topk_key(s[u], (unsigned)e) : 0ull;
        unsigned todo = __ballot_sync(0xffffffffu, key > tail);
        while (todo) {
          const unsigned long long x = __shfl_sync(0xffffffffu, key, __ffs(todo) - 1);
          const int p = __popc(__ballot_sync(0xffffffffu, k0 > x)) + __popc(__ballot_sync(0xffffffffu, k1 > x));
          const unsigned long long u0 = __shfl_up_sync(0xffffffffu, k0, 1), u1 = __shfl_up_sync(0xffffffffu, k1, 1);
          const unsigned long long last0 = __shfl_sync(0xffffffffu, k0, 31);
          k1 = lane + 32 < p ? k1 : (lane + 32 == p ? x : (lane == 0 ? last0 : u1));
          k0 = lane < p ? k0 : (lane == p ? x : u0);
          tail = __shfl_sync(0xffffffffu, k <= 32 ? k0 : k1, (k - 1) & 31);
          todo &= todo - 1;
          todo &= __ballot_sync(0xffffffffu, key > tail);
        }
      }
    }
  }
  if (lane < k) lists[warp][lane] = k0;
  if (lane + 32 < k) lists[warp][lane + 32] = k1;
  __syncthreads();
  if (warp != 0) return;
  static_assert(kShTopkWarps == 16 && FPW_MAX_TOPK == 64, "lanes 0-15 hold the heads, two entries a lane");
  int32_t* oi = a.topk_idx + c * k;
  float* os = a.topk_S + c * k;
  int h = 0;  // this lane's position in the list of warp `lane`
  unsigned long long head = lane < kShTopkWarps ? lists[lane][0] : 0ull;
  for (int q = 0; q < k; ++q) {
    unsigned long long best = head;
#pragma unroll
    for (int o = 8; o > 0; o >>= 1) {
      const unsigned long long v = __shfl_xor_sync(0xffffffffu, best, o);
      best = v > best ? v : best;
    }
    if (lane == 0) {
      const unsigned rank = (unsigned)(best >> 32);
      oi[q] = best ? (int32_t)(0xFFFFFFFFu - (unsigned)best) : -1;
      os[q] = __uint_as_float(rank <= 1u ? 0x7fc00000u : ((rank >> 31) ? rank & 0x7FFFFFFFu : ~rank));
    }
    best = __shfl_sync(0xffffffffu, best, 0);
    if (best && head == best) head = ++h < k ? lists[lane][h] : 0ull;
  }
}

}  // namespace

size_t shared_image_bytes(int64_t ncurves, int64_t n) {
  const int64_t groups = (ncurves + kShCurves - 1) / kShCurves;
  const int64_t nch = (n + kShObs - 1) / kShObs;
  return (size_t)groups * (size_t)nch * kShChunkBytes;
}

int shared_curves_per_group() { return kShCurves; }

// Frequencies per accumulator and the MMA's N for M bins (0 if M is too large).
int shared_freqs_per_mma(int M, int* n_mma) {
  if (M < 1 || M > kShNMax) return 0;
  const int fpm = kShNMax / M < kShMaxFpm ? kShNMax / M : kShMaxFpm;
  *n_mma = ((fpm * M + 15) / 16) * 16;
  return fpm;
}

cudaError_t launch_dense_topk32(const DenseTopk32Args& t, int64_t ncurves, cudaStream_t st) {
  if (t.k <= 0 || ncurves <= 0) return cudaSuccess;
  dense_topk32_kernel<<<(unsigned)ncurves, kShTopkThreads, 0, st>>>(t);
  return cudaGetLastError();
}

cudaError_t shared_init_attributes() {
  const cudaError_t e = cudaFuncSetAttribute(shared_mma_kernel<true>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
  if (e != cudaSuccess) return e;
  return cudaFuncSetAttribute(shared_mma_kernel<false>, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemBytes);
}

size_t shared_smem_bytes() { return kSmemBytes; }

// Groups taken in pairs: all but an odd one, where that is over sooner than
// group by group, in rounds of items over the SMs (a pair's item takes 0.9 of a
// group's, and the odd group's launch fills rounds of its own: 130 curves, M =
// 35, 2449 frequencies took 110 us in pairs, 3 + 2 rounds, and 100 in 4).
static int64_t shared_pair_groups(int64_t ngroups, int64_t nfreq, int fpm, int nsm) {
  const int64_t np = (nfreq + fpm - 1) / fpm, ns = (nfreq + 2 * fpm - 1) / (2 * fpm);
  auto rounds = [&](int64_t items) { return (items + nsm - 1) / nsm; };
  const int64_t pairs = 9 * rounds(ngroups / 2 * np) + 10 * rounds(ngroups % 2 * ns);
  return pairs <= 10 * rounds(ngroups * ns) ? (ngroups & ~(int64_t)1) : 0;
}

cudaError_t launch_shared(const SharedArgs& args, int nsm, cudaStream_t st) {
  const int64_t slots = args.ngroups * kShCurves;
  if (slots <= 0) return cudaSuccess;
  SharedArgs a = args;
  a.pair_groups = shared_pair_groups(a.ngroups, a.nfreq, a.fpm, nsm);
  shared_prep_kernel<<<(unsigned)slots, 256, 0, st>>>(a);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  e = cudaMemsetAsync(a.tmax_bits, 0, sizeof(unsigned long long), st);
  if (e != cudaSuccess) return e;
  if (a.n > 0) {
    const int64_t blocks = (a.n + 255) / 256;
    shared_steps_kernel<<<(unsigned)(blocks < 1024 ? blocks : 1024), 256, 0, st>>>(a);
    e = cudaGetLastError();
    if (e != cudaSuccess) return e;
  }
  if (a.ngroups > 0 && a.nfreq > 0) {
    if (a.timing_start) cudaEventRecord(a.timing_start, st);
    SharedArgs b = a;
    b.group0 = 0;
    b.units = a.pair_groups / 2;
    b.npass = (a.nfreq + a.fpm - 1) / a.fpm;
    if (b.units > 0) {
      const int64_t items = b.units * b.npass;
      shared_mma_kernel<true><<<(int)(items < nsm ? items : nsm), kShThreads, kSmemBytes, st>>>(b);
      e = cudaGetLastError();
      if (e != cudaSuccess) return e;
    }
    b.group0 = a.pair_groups;
    b.units = a.ngroups - a.pair_groups;
    b.npass = (a.nfreq + 2 * a.fpm - 1) / (2 * a.fpm);
    if (b.units > 0) {
      const int64_t items = b.units * b.npass;
      shared_mma_kernel<false><<<(int)(items < nsm ? items : nsm), kShThreads, kSmemBytes, st>>>(b);
      e = cudaGetLastError();
      if (e != cudaSuccess) return e;
    }
    if (a.timing_stop) cudaEventRecord(a.timing_stop, st);
  }
  if (a.k > 0 && a.ncurves > 0) {
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
