// Device templates of the persistent FPW tile kernels: Eq. 1 (Section 2) for
// every (curve, frequency) of a work list, with the per-curve top-k peaks of
// Section 3.5; and the same with several bin counts M = M_max / g derived from
// one M_max pass (Section 3.4). The kernels are instantiated in several
// translation units (fpw_tile_*.cu) so that they compile in parallel; the host
// side (shapes, launches) is fpw_tile.cu.
//
// Work decomposition
//   A work item is (curve c, frequency segment [f_lo, f_hi)), swept by ONE WARP
//   in tiles of W = 32 R consecutive frequencies: lane l owns tile positions
//   l R + r (r < R). The first item of a warp is fixed by its index (so that a
//   short list spreads over every SM), the next ones come from a global counter
//   (items are sorted by cost, longest first). Warps share nothing: no barrier
//   wider than a warp runs, so one warp's staging, reduction and peaks overlap
//   the other warps' bin updates. (A block per item, its four warps meeting at
//   barriers around every chunk and tile, ran the same loop at 1.93e12
//   evaluations/s where warps of their own run 2.05e12, M = 20, N = 1000.)
//   Phases are anchored every anchor_span frequencies, and a tile lies in one
//   anchor block, whose frequencies with one more on either side (the
//   local-maximum test needs both neighbours) are a whole number of tiles. Tiles
//   do not overlap, the last two values of a tile are carried to the next; items
//   that meet inside a block leave each other the values at their ends (Meeting).
//
// Per tile
//   1. Stage (per 32 observations, lane = observation, a ring of two chunks in
//      shared memory, the next chunk's inputs already in registers): the phase
//      Phi_s = frac(t_i * f_s) at the tile's first frequency as a 64-bit
//      fixed-point fraction, the step D_i = frac(t_i * df) (df = grid spacing) and
//      the weights (a_i = x_i w_i, w_i). Phi_s steps from the exact phase at the
//      block's anchor frequency, the integer product of the significands, for
//      which the prep kernel leaves the times as fixed-point numbers (about 20
//      operations an observation and tile; 60 with both numbers taken apart held
//      up the hot loops for 5-10 % of the time).
//   2. Hot loop (per observation, per lane, per r): Phi = Phi_s + (l R + r) D_i
//      (mod 2^64), bin m = floor(M * Phi_hi / 2^32), A_m += a_i, B_m += w_i in a
//      lane-private [r][m][lane] bin array in shared memory (bank = lane, so
//      conflict-free). Software-pipelined: the addresses of observation i + 1
//      are formed while the bins of observation i are on their way, from a
//      record loaded one observation earlier, across chunk boundaries too.
//   3. Reduce: S = sum_m A_m^2 / (B_m + 1/alpha^2), empty bins contribute 0.
//      Several-M kernel: in-place prefix sums of the M_max bins, then for each
//      group g the windows of g consecutive bins (circularly) for every offset;
//      S_g(f) is the largest S over the g offsets, and that offset is kept.
//   4. Peaks: local maxima among owned frequencies that beat the k-th best so
//      far are inserted into the item's sorted list (shared memory), written as
//      candidates at the item's end.
//
// Grids that are not linear to within kGridTolCycles over a tile: the phase is
// frac(t_i f_b) (exact, f_b the tile's middle frequency) plus t_i (f_k - f_b) from
// FP32 pairs, correct to 2^-36 cycles (NlTile), and the exact product where that
// leaves the bin open: the bins are those of frac(t_i f_k), whatever the tile. A
// tile whose frequencies spread over more than 2^7 cycles either side takes a
// direct exact anchor per (observation, frequency).
//
// Bin sums (policy P): FP32 pairs (A, B); binary64 pairs; or FP32 pairs with
// compensation terms (A, B, cA, cB), where each addition is an exact two-sum
// whose rounding error, plus the low part of the staged term, goes to the
// compensation term (the weights are staged as hi + lo FP32 pairs), so the
// sums carry about 48 significant bits; each bin's term is then taken from
// hi + lo rounded once to FP32, and S is accumulated in binary64.
//
// DUMP instantiations additionally write the bin m of every (observation,
// owned frequency k) with bins_k0 <= k < bins_k1 to args.bins_out, in the loop that
// forms the sums (bin-identity checks of the product kernel).
#pragma once
#include <math.h>

#include "fpw_internal.cuh"

namespace fpw {

// Per-translation-unit kernel getters (fpw_tile_*.cu).
const void* tile_fn_f32(int R, int phase_mode, bool dump);
const void* tile_fn_f32_odd(int R, int phase_mode, bool dump);  // R = 3, 5, 6
const void* tile_fn_f64(int R, int phase_mode, bool dump);
const void* tile_fn_comp(int R, int phase_mode, bool dump);
const void* tile_fn_multi(int R, int phase_mode, int spec);  // spec: multi_spec_of(), 0 = any groups

struct WarpLayout {
  size_t pd, aw, topS, topI, total;
};

__host__ __device__ inline size_t align16(size_t x) { return (x + 15) & ~(size_t)15; }

// Staged observations of a warp: a ring of two chunks of 32, plus copies of the
// first two slots after the last (the hot loop prefetches two records ahead
// without wrapping the index).
constexpr int kSlots = 64;
constexpr int kRing = kSlots + 2;

// Shared memory of one warp: bins [R][M][32] of bin_bytes, the ring of staged
// {Phi, D} (16 B) and weights (bin_bytes), the top-k lists of every group.
__host__ __device__ inline WarpLayout warp_layout(int R, int M, size_t bin_bytes, int kk, int ngroups) {
  const size_t tops = (size_t)(ngroups > 1 ? ngroups : 1) * (size_t)kk;
  WarpLayout L;
  size_t o = (size_t)R * M * 32 * bin_bytes;
  L.pd = o;
  o += (size_t)kRing * 16;
  L.aw = o;
  o = align16(o + (size_t)kRing * bin_bytes);
  L.topS = o;
  o += tops * 8;
  L.topI = o;
  o = align16(o + tops * 4);
  L.total = o;
  return L;
}

// Threads of a launched block: FP32 sums of one M and the other sum modes; several M.
constexpr int kTileMaxThreads = 384, kMultiMaxThreads = 256;

#ifdef __CUDACC__
namespace {

// ---- accumulation policies ----------------------------------------------
struct AccF32 {  // FP32 (A, B)
  using Bin = float2;
  using In = float2;  // (a, w)
  using S = float;
};
struct AccF64 {  // binary64 (A, B)
  using Bin = double2;
  using In = double2;
  using S = double;
};
struct AccComp {  // FP32 (A, B) with compensation (cA, cB): float4 {A, B, cA, cB}
  using Bin = float4;
  using In = float4;  // {a_hi, w_hi, a_lo, w_lo}
  using S = double;
};

__device__ __forceinline__ unsigned long long pack2(float2 a) {
  unsigned long long x;
  asm("mov.b64 %0, {%1, %2};" : "=l"(x) : "f"(a.x), "f"(a.y));
  return x;
}
__device__ __forceinline__ float2 unpack2(unsigned long long z) {
  float2 r;
  asm("mov.b64 {%0, %1}, %2;" : "=f"(r.x), "=f"(r.y) : "l"(z));
  return r;
}

__device__ __forceinline__ float2 bin_add(float2 v, float2 x) { return f2add(v, x); }
__device__ __forceinline__ double2 bin_add(double2 v, double2 x) { return make_double2(v.x + x.x, v.y + x.y); }
// Compensated: (s, e) = TwoSum(v.AB, x.hi) exactly (s + e = v.AB + x.hi), then
// c += e + x.lo. Packed FP32 pairs handle A and B together.
__device__ __forceinline__ float4 bin_add(float4 v, float4 x) {
  const unsigned long long a = pack2(make_float2(v.x, v.y)), b = pack2(make_float2(x.x, x.y));
  const unsigned long long c = pack2(make_float2(v.z, v.w)), lo = pack2(make_float2(x.z, x.w));
  unsigned long long s, bb, t1, t2, t3, e, c1, c2;
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(s) : "l"(a), "l"(b));
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(bb) : "l"(s), "l"(a));
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(t1) : "l"(s), "l"(bb));
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(t2) : "l"(a), "l"(t1));
  asm("sub.rn.f32x2 %0, %1, %2;" : "=l"(t3) : "l"(b), "l"(bb));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(e) : "l"(t2), "l"(t3));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(c1) : "l"(e), "l"(lo));
  asm("add.rn.f32x2 %0, %1, %2;" : "=l"(c2) : "l"(c), "l"(c1));
  const float2 sv = unpack2(s), cv = unpack2(c2);
  return make_float4(sv.x, sv.y, cv.x, cv.y);
}

__device__ __forceinline__ void bin_zero(float2& v) { v = make_float2(0.f, 0.f); }
__device__ __forceinline__ void bin_zero(double2& v) { v = make_double2(0.0, 0.0); }
__device__ __forceinline__ void bin_zero(float4& v) { v = make_float4(0.f, 0.f, 0.f, 0.f); }

// One bin's term A^2 / (B + 1/alpha^2) of Eq. 1; a bin whose denominator is 0 contributes 0.
// FP32: the reciprocal-based quotient (2 ulp), branch-free (a branch to a
// correctly rounded division for out-of-range denominators kept the compiler
// from overlapping the terms of the reduce); a denominator outside
// [2^-100, 2^100] is scaled by 2^-+64 into that range first, the numerator
// alike, so the reciprocal stays accurate. Binary64: correctly rounded.
__device__ __forceinline__ float bin_term(float2 v, float cal) {
  const float den = v.y + cal;
  const float sc = den > 0x1p+100f ? 0x1p-64f : (den < 0x1p-100f ? 0x1p+64f : 1.0f);
  const float q = __fdividef((v.x * v.x) * sc, den * sc);
  return (den > 0.f) ? q : 0.f;
}
// The same where every denominator is known to be 0 or inside [2^-100, 2^100]
// (the curve's weights and 1/alpha^2 lie well inside, Warp::plain): the same
// value, about half the instructions.
__device__ __forceinline__ float bin_term_plain(float2 v, float cal) {
  const float den = v.y + cal;
  const float q = __fdividef(v.x * v.x, den);
  return (den > 0.f) ? q : 0.f;
}
__device__ __forceinline__ double bin_term(double2 v, double cal) {
  const double den = v.y + cal;
  return (den > 0.0) ? v.x * v.x / den : 0.0;
}
// Compensated: the sums' value hi + lo rounded once to FP32 (the compensation
// already holds their rounding error), the term as in the FP32 policy (about
// 3e-7 relative), S accumulated in binary64. A binary64 division per bin took
// 28 % of the kernel's time at M = 20 and 44 % at M = 50.
__device__ __forceinline__ double bin_term(float4 v, double cal) {
  return (double)bin_term(make_float2(v.x + v.z, v.y + v.w), (float)cal);
}

__device__ __forceinline__ double bin_term_plain(double2 v, double cal) { return bin_term(v, cal); }
__device__ __forceinline__ double bin_term_plain(float4 v, double cal) {
  return (double)bin_term_plain(make_float2(v.x + v.z, v.y + v.w), (float)cal);
}

__device__ __forceinline__ float2 f2sub(float2 a, float2 b) { return make_float2(a.x - b.x, a.y - b.y); }

__device__ __forceinline__ double warp_max(double v) {
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) v = fmax(v, __shfl_xor_sync(0xffffffffu, v, o));
  return v;
}

// The largest s among the lanes with k >= 0 (one at least), and whether the
// lane holds it.
__device__ __forceinline__ bool warp_best(float s, int k, float& best) {
  const unsigned u = __float_as_uint(s), r = k >= 0 ? ((u >> 31) ? ~u : (u | 0x80000000u)) : 0u;
  const unsigned m = __reduce_max_sync(0xffffffffu, r);
  best = __uint_as_float((m >> 31) ? (m & 0x7fffffffu) : ~m);
  return k >= 0 && r == m;
}
__device__ __forceinline__ bool warp_best(double s, int k, double& best) {
  const unsigned long long r = k >= 0 ? rank_bits(s) : 0ull;
  const unsigned hi = __reduce_max_sync(0xffffffffu, (unsigned)(r >> 32));
  const unsigned lo = __reduce_max_sync(0xffffffffu, (unsigned)(r >> 32) == hi ? (unsigned)r : 0u);
  const unsigned long long m = ((unsigned long long)hi << 32) | lo;
  best = from_rank_bits(m);
  return k >= 0 && r == m;
}

// The k-th best S that some item of curve row `row` has found so far (0: none):
// items of the curve skip what lies below it. Nothing depends on when a value
// arrives: k peaks at least as high are then in that item's list.
__device__ __forceinline__ unsigned long long curve_floor(const TileArgs& args, int64_t row) {
  return args.floors ? *(volatile unsigned long long*)(args.floors + row) : 0ull;
}
template <class A>
__device__ __forceinline__ A floor_value(unsigned long long f) {
  return f != 0ull ? (A)from_rank_bits(f) : (A)-INFINITY;
}
__device__ __forceinline__ void raise_floor(const TileArgs& args, int64_t row, const double* topS, const int* topI,
                                            int kk, int lane) {
  if (args.floors && lane == 0 && topI[kk - 1] >= 0) atomicMax(args.floors + row, rank_bits(topS[kk - 1]));
}

// Shared-memory bin access by 32-bit address. volatile: their order is the
// program's (the next observation's bin loads follow this one's stores).
__device__ __forceinline__ unsigned smem_u32(const void* p) { return (unsigned)__cvta_generic_to_shared(p); }
__device__ __forceinline__ void lds(unsigned a, float2& v) {
  asm volatile("ld.shared.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(a) : "memory");
}
__device__ __forceinline__ void lds(unsigned a, float4& v) {
  asm volatile("ld.shared.v4.f32 {%0, %1, %2, %3}, [%4];"
               : "=f"(v.x), "=f"(v.y), "=f"(v.z), "=f"(v.w)
               : "r"(a)
               : "memory");
}
__device__ __forceinline__ void lds(unsigned a, double2& v) {
  asm volatile("ld.shared.v2.f64 {%0, %1}, [%2];" : "=d"(v.x), "=d"(v.y) : "r"(a) : "memory");
}
__device__ __forceinline__ void lds(unsigned a, ulonglong2& v) {
  asm volatile("ld.shared.v2.u64 {%0, %1}, [%2];" : "=l"(v.x), "=l"(v.y) : "r"(a) : "memory");
}
__device__ __forceinline__ void sts(unsigned a, float2 v) {
  asm volatile("st.shared.v2.f32 [%0], {%1, %2};" ::"r"(a), "f"(v.x), "f"(v.y) : "memory");
}
__device__ __forceinline__ void sts(unsigned a, float4 v) {
  asm volatile("st.shared.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w) : "memory");
}
__device__ __forceinline__ void sts(unsigned a, double2 v) {
  asm volatile("st.shared.v2.f64 [%0], {%1, %2};" ::"r"(a), "d"(v.x), "d"(v.y) : "memory");
}

// Per-warp view of shared memory and the constants every stage needs.
template <class P>
struct Warp {
  using A = typename P::S;
  unsigned char* bins;       // this lane's column of the [r][m][lane] bin array
  ulonglong2* pd;            // ring of staged {Phi, D} (or {P, T}, NlTile; or {t, 0})
  typename P::In* aw;        // ring of staged weights
  double* topS;              // [groups][kk], sorted
  int* topI;
  int lane, M, kk;
  int64_t F;
  double df;
  int tbits;                 // binary places of the prep kernel's times
  static constexpr unsigned kBinStride = 32u * (unsigned)sizeof(typename P::Bin);  // bytes between bins of a column
};

template <int R, class P>
__device__ __forceinline__ Warp<P> make_warp(unsigned char* smem, const TileArgs& args) {
  Warp<P> w;
  w.lane = threadIdx.x & 31;
  w.M = args.M;
  w.kk = args.k;
  const WarpLayout L = warp_layout(R, w.M, sizeof(typename P::Bin), w.kk, args.ngroups);
  unsigned char* const mine = smem + (size_t)(threadIdx.x >> 5) * L.total;
  w.bins = mine + (size_t)w.lane * sizeof(typename P::Bin);
  w.pd = reinterpret_cast<ulonglong2*>(mine + L.pd);
  w.aw = reinterpret_cast<typename P::In*>(mine + L.aw);
  w.topS = reinterpret_cast<double*>(mine + L.topS);
  w.topI = reinterpret_cast<int*>(mine + L.topI);
  w.F = args.nfreq;
  w.df = args.df ? *args.df : (w.F > 1) ? (args.freqs[w.F - 1] - args.freqs[0]) / (double)(w.F - 1) : 0.0;
  w.tbits = args.rec ? *args.time_bits : 0;
  // bins start at zero (every reduce leaves them zero again), and so does the
  // ring (the prefetch past a curve's last observation reads slots not staged)
  for (int q = 0; q < R * w.M; ++q)
    bin_zero(*reinterpret_cast<typename P::Bin*>(w.bins + (size_t)q * Warp<P>::kBinStride));
  for (int q = w.lane; q < kRing; q += 32) {
    w.pd[q] = make_ulonglong2(0ull, 0ull);
    bin_zero(w.aw[q]);
  }
  return w;
}

// v as the unevaluated sum of two FP32 numbers, by integer operations: to 2^-48
// relative for 2^-74 <= |v| < 2^100, to 2^-98 for smaller |v|.
__device__ __forceinline__ float2 split_f32(double v) {
  const unsigned long long b = (unsigned long long)__double_as_longlong(v);
  const unsigned hi = (unsigned)(b >> 32), e = (hi >> 20) & 0x7ffu, sign = hi & 0x80000000u;
  if (e < 949u) return make_float2((e < 924u) ? 0.f : __uint_as_float(sign | (e - 896u) << 23 | ((unsigned)(b >> 29) & 0x7fffffu)), 0.f);
  // the leading 24 significand bits are one float, the other 29 become one
  return make_float2(__uint_as_float(sign | (e - 896u) << 23 | ((unsigned)(b >> 29) & 0x7fffffu)),
                     __uint2float_rn((unsigned)b & 0x1fffffffu) * __uint_as_float(sign | (e - 948u) << 23));
}

__device__ __forceinline__ int exponent_of(double v) {  // floor(log2 |v|) for normal v; -1023 for 0 and subnormals
  return (int)(((unsigned long long)__double_as_longlong(v) >> 52) & 0x7ffull) - 1023;
}

// How a tile's phases are formed: stepped from the exact phase at the anchor of
// the tile's block (the block on a line), which kRecord takes from the prep
// kernel's fixed-point times and kAnchor from the general product (the same
// number, where a time or the anchor is not of that form); products with the
// distance from an exact phase (NlTile); the exact phase of every pair. kStep32: the bins of kRecord or kAnchor's records by
// FPW_PHASE_FP32's rule, an FP32 phase every K frequencies and FP32 steps.
enum TileMode { kRecord, kAnchor, kFixed, kExact, kStep32 };

// The frequencies of a tile off the linear grid, as FP32 pairs of f_k - f_b (f_b:
// the tile's middle frequency). An observation's phase at f_k is its exact phase
// at f_b plus t (f_k - f_b), |t (f_k - f_b)| < 2^7 cycles, with t an FP32 pair
// too: the product's multiple of 2^-14 cycles comes off the mantissa of one
// fused multiply-add (kMagic), the rest is a sum of the exact remainder and the
// cross terms, in units of 2^-36. Off by less than a unit either way; the staged
// phase is rounded up and carries one unit more, so the sum is never below the
// exact phase (a phase on a bin edge stays in the upper bin) and at most 3 units
// above it. FP32 multiply-adds because integer products are slow: mul.hi runs at
// 30 lanes/clk/SM, fma at 110 (measured); the same sum from 61-bit integer
// factors (three mul.hi more than the linear step) ran 1.04e12 evaluations/s at
// M = 20.
// The bin is that of the exact phase's leading 32 bits. The sum's are the same or
// one more, and the bin another one only where the last one is the first of its
// bin, the low word of M times it below M: M in 2^32 pairs, which take the exact
// product (exact_bin). Times of 0 would all do: their phase is staged as a unit of
// 2^-32 and a half, which is as well in bin 0. Asked per observation: 24 curves x
// 100003 frequencies 1440 us -> 1760 (6600 with the exact product of every pair);
// asked once a tile, which then starts over, 2100, its warps end so much later.
template <int R>
struct NlTile {
  float dh[R], dl[R];
};
constexpr float kMagic = 768.f;               // 1.5 * 2^9: sums keep multiples of 2^-14 in the low mantissa bits
constexpr unsigned kMagicLow = 0x4B400000u;   // bits of 1.5 * 2^23

// pd: {P's 32 bits below the binary point | its next four and -kMagicLow, th | tl}
__device__ __forceinline__ unsigned nl_phase(const ulonglong2& pd, float dh, float dl) {
  const float th = __uint_as_float((unsigned)pd.y), tl = __uint_as_float((unsigned)(pd.y >> 32));
  const float m = __fmaf_rn(th, dh, kMagic);
  float e = __fmaf_rn(th, dh, -__fsub_rn(m, kMagic));
  e = __fmaf_rn(th, dl, e);
  e = __fmaf_rn(tl, dh, e);
  e = __fmaf_rn(e, 0x1p36f, 0x1.8p23f);
  const int low = (int)(__float_as_uint(e) + (unsigned)(pd.x >> 32));
  return (__float_as_uint(m) << 18) + (unsigned)pd.x + (unsigned)(low >> 4);
}

__device__ __noinline__ unsigned exact_bin(double t, double f, unsigned M) { return bin_of_phase(phase_fixed64(t, f), M); }

// Geometry of one tile: first frequency s (-1 possible), its anchor block's first
// position sq and anchor frequency fa (index max(sq, 0)), and how its phases are
// formed.
struct Tile {
  int64_t s, sq;
  double fa;
  TileMode mode;
};

// The tile at s in anchor block q.
template <int R, class P>
__device__ __forceinline__ Tile make_tile(const TileArgs& args, const Warp<P>& w, int64_t s, int64_t q, double tm,
                                          bool every_lin, bool unfit, NlTile<R>& nl) {
  Tile g;
  g.s = s;
  g.sq = q * args.anchor_span - 1;
  const int64_t a = g.sq < 0 ? 0 : g.sq;
  g.fa = args.freqs[a];
  bool lin = every_lin;
  if (every_lin) {
  } else if (args.block_dev) {
    lin = (double)args.block_dev[q] * tm <= kGridTolCycles;
  } else {
    bool off = false;
    for (int64_t j = w.lane; j < args.anchor_span + 2; j += 32) {
      const int64_t k = g.sq + j;
      if (k >= 0 && k < w.F && fabs(args.freqs[k] - fma((double)(k - a), w.df, g.fa)) * tm > kGridTolCycles) off = true;
    }
    lin = !__any_sync(0xffffffffu, off);
  }
  if (lin) {
    g.mode = args.rec && !unfit && (every_lin || fixed_anchor(g.fa, w.tbits).ok) ? kRecord : kAnchor;
    return g;
  }
  const int64_t s0 = s < 0 ? 0 : (s < w.F ? s : w.F - 1), mid = s + 16 * R;
  const double fb = args.freqs[mid < w.F ? mid : s0];
  double f[R];
  int de = -1023;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t k = s + (int64_t)(w.lane * R + r);
    f[r] = k >= 0 && k < w.F ? args.freqs[k] - fb : 0.0;
    de = max(de, exponent_of(f[r]));
  }
  de = __reduce_max_sync(0xffffffffu, de);
  const int te = exponent_of(tm);
  if (te < -20 || te > 40 || te + de + 2 > 7) {  // |t (f_k - f_b)| may reach 2^7 cycles (or split_f32's range ends)
    g.mode = kExact;
    return g;
  }
  g.mode = kFixed;
  g.fa = fb;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const float2 d = split_f32(f[r]);
    nl.dh[r] = d.x;
    nl.dl[r] = d.y;
  }
  return g;
}

// One observation's inputs on their way from global memory to the ring.
template <class P>
struct Obs {
  ulonglong2 rec;  // the prep kernel's record (kRecord), {t, 0} else
  unsigned top;    // kRecord: the time's top word
  typename P::In aw;
};

template <class P>
__device__ __forceinline__ Obs<P> fetch(const TileArgs& args, TileMode mode, int64_t base, int64_t n, int64_t i) {
  Obs<P> o;
  o.rec = make_ulonglong2(0ull, 0ull);  // past the curve's end: t = 0 and zero weights, which add 0 to some bin
  o.top = 0u;
  bin_zero(o.aw);
  if (i < n) {
    if (mode == kRecord) {
      o.rec = args.rec[base + i];
      o.top = args.rec_top[base + i];
    } else {
      o.rec.x = (unsigned long long)__double_as_longlong(args.t[base + i]);
    }
    o.aw = reinterpret_cast<const typename P::In*>(args.aw)[base + i];
  }
  return o;
}

// The staged phase record: {phase, step D}, {P, T} (NlTile) or {t, 0}. The phase is
// that of the tile's first frequency: the exact phase at the block's anchor,
// rounded up at 2^-64, plus s - sq steps (one less in block 0, which starts one
// step before its anchor). Nothing shorter than the exact anchor will do: visits
// a round fraction of a day apart put phases within 10^-15 cycles of bin edges at
// round frequencies, where a step rounded once and summed over the grid, or an
// anchor to 2^-54, moves observations to other bins.
template <class P>
__device__ __forceinline__ ulonglong2 record(const TileArgs& args, const Warp<P>& w, const Tile& g, TileMode mode,
                                             const FixedAnchor& anchor, const Obs<P>& o) {
  if (mode == kExact) return o.rec;
  const unsigned long long steps = (unsigned long long)(g.s - g.sq - (g.sq < 0 ? 1 : 0));
  if (mode == kRecord) {
    return make_ulonglong2(fixed_phase(o.rec.x, o.top, anchor) + steps * o.rec.y, o.rec.y);
  }
  const double t = __longlong_as_double((long long)o.rec.x);
  unsigned long long Pa = phase_fixed64(t, g.fa);
  if (mode == kFixed) {
    const float2 tt = split_f32(t);
    const unsigned long long p = t == 0.0 ? 24ull : ((Pa + 0xfffffffull) >> 28) + 1ull;  // units of 2^-36, rounded up, one more
    const unsigned c = (unsigned)(p & 15ull) - kMagicLow;
    return make_ulonglong2(((unsigned long long)c << 32) | (unsigned)(p >> 4),
                           ((unsigned long long)__float_as_uint(tt.y) << 32) | __float_as_uint(tt.x));
  }
  const unsigned long long D = phase_fixed64(t, w.df);
  return make_ulonglong2(Pa + steps * D, D);
}

// Chunk c of 32 observations into its half of the ring.
template <class P>
__device__ __forceinline__ void put(const Warp<P>& w, int64_t c, const ulonglong2& pd, const typename P::In& aw) {
  const int slot = (int)(c & 1) * 32 + w.lane;
  w.pd[slot] = pd;
  w.aw[slot] = aw;
  if (slot < 2) {
    w.pd[slot + kSlots] = pd;
    w.aw[slot + kSlots] = aw;
  }
}

// Steps 1 and 2 for one tile. The R phases of an observation are independent
// multiply-adds, its R bin loads precede its R stores, and the addresses of the
// next observation are formed in between; four observations per trip rename the
// pipelined registers instead of moving them. Against the loop that formed and
// used an observation's bins in the same trip (probe, loop alone): M = 20, R =
// 5, 8 warps per SM 1.85 -> 2.08e12 evaluations/s; M = 60, R = 3, 4 warps 1.15
// -> 1.5e12. One loop for every way of forming the bins, with and without the
// dump (FPW_PHASE_FP32 and the exact phase of every pair ran 0.16e12 and 0.26e12
// evaluations/s at M = 20 in a plain loop of their own, 1.35e12 and 0.30e12 in
// this one). MODE kRecord serves kAnchor too (mode).
template <int R, class P, TileMode MODE, bool DUMP>
__device__ __forceinline__ void accumulate(const TileArgs& args, const Warp<P>& w, const Tile& g, const NlTile<R>& nl,
                                           int64_t base, int64_t n, const WorkItem& wi, TileMode mode) {
  using Bin = typename P::Bin;
  using In = typename P::In;
  constexpr int U = MODE == kExact ? 1 : 4, kChunk = 32;  // (the product of a pair is long enough by itself)
  const unsigned M = (unsigned)w.M;
  const unsigned j0 = (unsigned)w.lane * R;
  const unsigned col = smem_u32(w.bins), rstride = M * Warp<P>::kBinStride;
  const int64_t npad = (n + U - 1) / U * U, nchunk = (n + kChunk - 1) / kChunk;
  const auto freq = [&](int r) { return args.freqs[max((int64_t)0, min(w.F - 1, g.s + j0 + r))]; };
  double f[MODE == kExact ? R : 1];
  float past[MODE == kStep32 ? R : 1];  // steps past the frequency's FP32 anchor, and from the tile's first to that
  int anchor32[MODE == kStep32 ? R : 1];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    if (MODE == kExact) f[r] = freq(r);
    if (MODE == kStep32) {
      const int k = (int)(g.s + j0 + r), ak = k >= 0 ? k - k % args.K : 0;
      past[r] = (float)(k - ak);
      anchor32[r] = ak - (int)g.s;
    }
  }
  const int64_t dump_hi = min((int64_t)wi.f_hi, g.sq + 1 + args.anchor_span);
  // the addresses of the bins of observation i, whose record is p
  const auto addresses = [&](const ulonglong2& p, int64_t i, unsigned (&ad)[R]) {
    unsigned m[R];
    if (MODE == kFixed) {
      unsigned low = ~0u;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const unsigned ph = nl_phase(p, nl.dh[r], nl.dl[r]);
        low = min(low, ph * M);
        m[r] = __umulhi(ph, M);
      }
      if (low < M && i < n) {
#pragma unroll
        for (int r = 0; r < R; ++r)
          if (nl_phase(p, nl.dh[r], nl.dl[r]) * M < M) m[r] = exact_bin(args.t[base + i], freq(r), M);
      }
    } else if (MODE == kExact) {
#pragma unroll
      for (int r = 0; r < R; ++r) m[r] = bin_of_phase(phase_fixed64(__longlong_as_double((long long)p.x), f[r]), M);
    } else if (MODE == kStep32) {
      const float d32 = (float)(unsigned)(p.y >> 32) * 0x1p-32f;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const unsigned long long pa = p.x + (unsigned long long)(long long)anchor32[r] * p.y;
        float ph = fmaf(past[r], d32, (float)(unsigned)(pa >> 32) * 0x1p-32f);
        ph = ph - floorf(ph);
        const unsigned b = (unsigned)(ph * (float)M);
        m[r] = b < M ? b : M - 1u;
      }
    } else {
      const unsigned long long phi = p.x + (unsigned long long)j0 * p.y;
#pragma unroll
      for (int r = 0; r < R; ++r) m[r] = bin_of_phase(phi + (unsigned long long)r * p.y, M);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      ad[r] = col + (unsigned)r * rstride + m[r] * Warp<P>::kBinStride;
      if (DUMP) {
        const int64_t k = g.s + j0 + r;
        if (i < n && k >= wi.f_lo && k < dump_hi && k >= args.bins_k0 && k < args.bins_k1)
          args.bins_out[(k - args.bins_k0) * args.bins_nobs + base + i] = (int32_t)m[r];
      }
    }
  };
  Obs<P> o = fetch<P>(args, mode, base, n, w.lane);
  const Obs<P> o1 = fetch<P>(args, mode, base, n, 32 + w.lane);
  const FixedAnchor anchor = fixed_anchor(g.fa, w.tbits);  // (after the loads: it waits for its own)
  __syncwarp();  // every lane is done with the previous tile's ring
  put<P>(w, 0, record<P>(args, w, g, mode, anchor, o), o.aw);
  put<P>(w, 1, record<P>(args, w, g, mode, anchor, o1), o1.aw);
  o = fetch<P>(args, mode, base, n, 64 + w.lane);
  __syncwarp();
  const unsigned pd0 = smem_u32(w.pd), aw0 = smem_u32(w.aw);
  ulonglong2 p1;
  In x0, x1;
  unsigned ad[R];
  lds(pd0, p1);
  addresses(p1, 0, ad);
  lds(aw0, x0);
  lds(pd0 + 16u, p1);
  lds(aw0 + (unsigned)sizeof(In), x1);
  for (int64_t c = 0; c < nchunk; ++c) {
    const int lim = (int)((npad - c * kChunk) < kChunk ? (npad - c * kChunk) : kChunk);
    const unsigned first = (unsigned)(c & 1) * kChunk + 2u;
    unsigned pa = pd0 + first * 16u, xa = aw0 + first * (unsigned)sizeof(In);
#pragma unroll 1
    for (int i = 0; i < lim; i += U) {
#pragma unroll
      for (int u = 0; u < U; ++u) {
        Bin v[R];
#pragma unroll
        for (int r = 0; r < R; ++r) lds(ad[r], v[r]);
        ulonglong2 p2;
        In x2;
        lds(pa + (unsigned)u * 16u, p2);  // two records ahead: staged, a copy, or a slot whose value is not used
        lds(xa + (unsigned)u * (unsigned)sizeof(In), x2);
        unsigned an[R];
        addresses(p1, c * kChunk + i + u + 1, an);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          sts(ad[r], bin_add(v[r], x0));
          ad[r] = an[r];
        }
        x0 = x1;
        x1 = x2;
        p1 = p2;
      }
      pa += U * 16u;
      xa += U * (unsigned)sizeof(In);
    }
    if (c + 2 < nchunk) {  // this chunk's half of the ring is free: the next but one
      __syncwarp();
      put<P>(w, c + 2, record<P>(args, w, g, mode, anchor, o), o.aw);
      o = fetch<P>(args, mode, base, n, (c + 3) * kChunk + w.lane);
      __syncwarp();
    }
  }
}

template <int R, int PHASE, class P, bool DUMP>
__device__ __forceinline__ void accumulate_tile(const TileArgs& args, const Warp<P>& w, const Tile& g,
                                                const NlTile<R>& nl, int64_t base, int64_t n, const WorkItem& wi) {
  if (g.mode == kExact)
    accumulate<R, P, kExact, DUMP>(args, w, g, nl, base, n, wi, kExact);
  else if (g.mode == kFixed)
    accumulate<R, P, kFixed, DUMP>(args, w, g, nl, base, n, wi, kFixed);
  else
    accumulate<R, P, PHASE == FPW_PHASE_FP32 ? kStep32 : kRecord, DUMP>(args, w, g, nl, base, n, wi, g.mode);
}

// Inserts (s, key) into the list topS/topI (kk entries sorted by S descending,
// then key ascending; key < 0: empty) if it ranks there. One warp, all lanes
// with the same s and key.
__device__ __noinline__ void list_insert(double* topS, int* topI, int kk, double s, int key, int lane) {
  int pos = 0;
  double up[2];
  int ui[2];
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int q = lane + 32 * h;
    const bool in = q < kk;
    const bool ahead = in && topI[q] >= 0 && ranks_before(topS[q], topI[q], s, key);
    pos += __popc(__ballot_sync(0xffffffffu, ahead));
    up[h] = in && q > 0 ? topS[q - 1] : 0.0;
    ui[h] = in && q > 0 ? topI[q - 1] : 0;
  }
  __syncwarp();
#pragma unroll
  for (int h = 0; h < 2; ++h) {
    const int q = lane + 32 * h;
    if (q < kk && q >= pos) {
      topS[q] = q == pos ? s : up[h];
      topI[q] = q == pos ? key : ui[h];
    }
  }
  __syncwarp();
}

// Two values of S and, in single precision, a bin offset as 128 bits that are not zero.
__device__ __forceinline__ ulonglong2 pack_ends(float a, float b, int off) {
  return make_ulonglong2((unsigned long long)__float_as_uint(b) << 32 | __float_as_uint(a), (unsigned long long)off + 1ull);
}
__device__ __forceinline__ ulonglong2 pack_ends(double a, double b, int) {  // (no sum is the NaN of all ones)
  return make_ulonglong2((unsigned long long)__double_as_longlong(a) + 1ull, (unsigned long long)__double_as_longlong(b) + 1ull);
}
__device__ __forceinline__ void unpack_ends(ulonglong2 v, float& a, float& b, int& off) {
  a = __uint_as_float((unsigned)v.x);
  b = __uint_as_float((unsigned)(v.x >> 32));
  off = (int)(v.y - 1ull);
}
__device__ __forceinline__ void unpack_ends(ulonglong2 v, double& a, double& b, int& off) {
  a = __longlong_as_double((long long)(v.x - 1ull));
  b = __longlong_as_double((long long)(v.y - 1ull));
  off = 0;
}
__device__ __forceinline__ ulonglong2 exchange128(ulonglong2* p, ulonglong2 v) {
  ulonglong2 r;
  asm volatile(
      "{\n\t.reg .b128 a, b;\n\tmov.b128 b, {%2, %3};\n\tatom.global.exch.b128 a, [%4], b;\n\t"
      "mov.b128 {%0, %1}, a;\n\t}"
      : "=l"(r.x), "=l"(r.y)
      : "l"(v.x), "l"(v.y), "l"(p)
      : "memory");
  return r;
}

// Where two items of a curve meet inside an anchor block, the left one's last
// frequency k and the right one's first, k + 1, lack a neighbour. Each item
// exchanges the S at its end (of k - 1, k or k + 1, k + 2) with what is at the
// meeting's place: the first finds nothing there, the second the other's values,
// and ranks k and k + 1 into its list. left: the item's beginning (S of its first
// two frequencies, the first one's bin offset), place row; right: its end (S of its
// last two, the last one's offset), place row + 1. Returns whether the list changed.
template <class A>
__device__ __noinline__ bool meet(const TileArgs& args, int64_t row, bool left, bool right, int f_lo, int f_hi, A b0,
                                  A b1, int boff, A e0, A e1, int eoff, int key_shift, double* topS, int* topI, int kk,
                                  int lane) {
  ulonglong2 v = make_ulonglong2(0ull, 0ull);
  if (lane == 0 && left) v = exchange128(args.meetings + row, pack_ends(b0, b1, boff));
  if (lane == 1 && right) v = exchange128(args.meetings + row + 1, pack_ends(e0, e1, eoff));
  const unsigned found = __ballot_sync(0xffffffffu, (v.x | v.y) != 0ull);
  bool changed = false;
  for (int side = 0; side < 2; ++side) {
    if (!(found >> side & 1u)) continue;
    A o0, o1;
    int off;
    unpack_ends(make_ulonglong2(__shfl_sync(0xffffffffu, v.x, side), __shfl_sync(0xffffffffu, v.y, side)), o0, o1, off);
    const A S[4] = {side ? e0 : o0, side ? e1 : o1, side ? o0 : b0, side ? o1 : b1};
    const int k = side ? f_hi - 1 : f_lo - 1;
    const int key[2] = {k << key_shift | (side ? eoff : off), (k + 1) << key_shift | (side ? off : boff)};
#pragma unroll
    for (int q = 0; q < 2; ++q) {
      const A s = S[1 + q];
      if (!args.peak_raw && !(s > S[q] && s >= S[2 + q])) continue;
      const A thr = topI[kk - 1] >= 0 ? (A)topS[kk - 1] : (A)-INFINITY;
      if (!(s > thr || (s == thr && key[q] < topI[kk - 1]))) continue;
      list_insert(topS, topI, kk, (double)s, key[q], lane);
      changed = true;
    }
  }
  return changed;
}

// Step 4: peaks among the frequencies whose right neighbour is known by now
// (the tile's own except its last, and the previous tile's last), or every
// owned one in raw mode, ranked into the list: those in [f_lo, f_hi). c1, c2: S of the two
// frequencies before the tile. The ranking key of frequency k is (k <<
// key_shift) | extra; ce: the extra of the frequency before the tile.
// floor: no S below it can be among the curve's k best. Returns whether the list
// changed.
template <int R, class P>
__device__ __forceinline__ bool tile_peaks(const TileArgs& args, const Warp<P>& w, const typename P::S (&S)[R],
                                           const int (&extra)[R], int key_shift, int64_t s, int64_t f_lo, int64_t f_hi,
                                           double* topS, int* topI, typename P::S floor,
                                           typename P::S& c1, typename P::S& c2, int& ce) {
  using A = typename P::S;
  const int lane = w.lane, kk = w.kk;
  // values one and two frequencies left of the lane's first
  A l1 = __shfl_up_sync(0xffffffffu, S[R - 1], 1);
  A l2 = R > 1 ? __shfl_up_sync(0xffffffffu, S[R > 1 ? R - 2 : 0], 1) : __shfl_up_sync(0xffffffffu, S[0], 2);
  int e1 = key_shift ? __shfl_up_sync(0xffffffffu, extra[R - 1], 1) : 0;
  if (lane == 0) {
    l1 = c1;
    l2 = c2;
    e1 = ce;
  }
  if (R == 1 && lane == 1) l2 = c1;
  c2 = R > 1 ? __shfl_sync(0xffffffffu, S[R > 1 ? R - 2 : 0], 31) : __shfl_sync(0xffffffffu, S[0], 30);
  c1 = __shfl_sync(0xffffffffu, S[R - 1], 31);
  if (key_shift) ce = __shfl_sync(0xffffffffu, extra[R - 1], 31);
  // peaks that beat the k-th best so far, of this item or (floor) of any of the
  // curve's; the best of them is inserted, round by round, so a tile takes at
  // most k rounds whatever its peaks' order
  unsigned todo = 0u;  // bit r: the frequency before position r is a peak to look at
  A v[R];
#pragma unroll
  for (int r = 0; r < R; ++r) {
    const int64_t k = s + (int64_t)(lane * R + r) - 1;
    v[r] = r > 0 ? S[r > 0 ? r - 1 : 0] : l1;
    const A left = r > 1 ? S[r > 1 ? r - 2 : 0] : (r == 1 ? l1 : l2);
    if (k >= f_lo && k < f_hi && (args.peak_raw || (v[r] > left && v[r] >= S[r])) && v[r] >= floor) todo |= 1u << r;
  }
  bool changed = false;
  A bs = (A)-INFINITY;  // the lane's best candidate (lowest key first where equal)
  int bk = -1, br = 0;
  for (bool fresh = true;; fresh = false) {
    const A thr = topI[kk - 1] >= 0 ? (A)topS[kk - 1] : (A)-INFINITY;
    const int thrk = topI[kk - 1];
    if (fresh || bk < 0) {
      if (todo != 0u) {
        bs = (A)-INFINITY;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int key = (int)(((s + (int64_t)(lane * R + r) - 1) << key_shift) | (r > 0 ? extra[r > 0 ? r - 1 : 0] : e1));
          const bool beats = v[r] > thr || (v[r] == thr && thrk >= 0 && key < thrk);
          if ((todo >> r & 1u) && beats && (bk < 0 || v[r] > bs)) {
            bs = v[r];
            bk = key;
            br = r;
          }
        }
        if (bk < 0) todo = 0u;
      }
    } else if (!(bs > thr || (bs == thr && thrk >= 0 && bk < thrk))) {
      bk = -1;
      todo = 0u;
    }
    if (!__any_sync(0xffffffffu, bk >= 0)) break;
    A ws;
    const bool mine = warp_best(bs, bk, ws);
    const unsigned wk = __reduce_min_sync(0xffffffffu, mine ? (unsigned)bk : 0xffffffffu);
    list_insert(topS, topI, kk, (double)ws, (int)wk, lane);
    changed = true;
    if (mine && (unsigned)bk == wk) {
      todo &= ~(1u << br);
      bk = -1;
    }
  }
  return changed;
}

// Step 3: S of the lane's R frequencies, bins cleared for the next tile. The R
// sums advance together, two bins at a time: a loop short enough to stay in the
// instruction cache next to the hot loop (a warp reaches it at its own time; with
// eight bins per frequency unrolled, fetching the code cost short curves a
// quarter of their time).
template <int R, class P, bool PLAIN>
__device__ __forceinline__ void reduce_bins(const Warp<P>& w, typename P::S cal, typename P::S (&S)[R]) {
  using Bin = typename P::Bin;
  constexpr unsigned kStride = Warp<P>::kBinStride;
  const unsigned rstride = (unsigned)w.M * kStride;
  unsigned a = smem_u32(w.bins);
  Bin z;
  bin_zero(z);
#pragma unroll
  for (int r = 0; r < R; ++r) S[r] = (typename P::S)0;
  int m = 0;
#pragma unroll 1
  for (; m + 2 <= w.M; m += 2, a += 2 * kStride) {
    Bin v[R][2];
#pragma unroll
    for (int r = 0; r < R; ++r) {
      lds(a + (unsigned)r * rstride, v[r][0]);
      lds(a + (unsigned)r * rstride + kStride, v[r][1]);
    }
#pragma unroll
    for (int r = 0; r < R; ++r) {
      sts(a + (unsigned)r * rstride, z);
      sts(a + (unsigned)r * rstride + kStride, z);
#pragma unroll
      for (int u = 0; u < 2; ++u) S[r] += PLAIN ? bin_term_plain(v[r][u], cal) : bin_term(v[r][u], cal);
    }
  }
  if (m < w.M) {
#pragma unroll
    for (int r = 0; r < R; ++r) {
      Bin v;
      lds(a + (unsigned)r * rstride, v);
      sts(a + (unsigned)r * rstride, z);
      S[r] += bin_term(v, cal);
    }
  }
}

// Item prologue shared by both kernels: invalid curves produce NaN / empty
// candidates (returns false); otherwise the largest |t| of the curve (sets the
// grid-linearity tolerance; 0 where the whole grid is linear for every curve)
// and cleared top lists.
template <class P>
__device__ __forceinline__ bool item_begin(const TileArgs& args, const Warp<P>& w, const WorkItem& wi, int64_t base,
                                           int64_t n, bool grid_bad, bool all_lin, int groups, double& tm) {
  const int lane = w.lane, kk = w.kk;
  const int64_t c = wi.curve;
  if (grid_bad || (args.curve_bad[c] & kCurveBad)) {
    if (args.S_out)
      for (int g = 0; g < groups; ++g)
        for (int64_t q = wi.f_lo + lane; q < wi.f_hi; q += 32)
          args.S_out[(c * groups + g) * w.F + q] = __longlong_as_double(0x7ff8000000000000ll);
    for (int g = 0; g < groups; ++g)
      for (int q = lane; q < kk; q += 32) {
        args.cand_S[(g * args.group_rows + wi.slot) * kk + q] = -INFINITY;
        args.cand_idx[(g * args.group_rows + wi.slot) * kk + q] = -1;
      }
    return false;
  }
  tm = 0.0;
  if (!all_lin) {
    double m = 0.0;
    for (int64_t i = lane; i < n; i += 32) m = fmax(m, fabs(args.t[base + i]));
    tm = warp_max(m);
  }
  __syncwarp();
  for (int q = lane; q < kk * groups; q += 32) {
    w.topS[q] = -INFINITY;
    w.topI[q] = -1;
  }
  __syncwarp();
  return true;
}

template <class P>
__device__ __forceinline__ void item_end(const TileArgs& args, const Warp<P>& w, const WorkItem& wi, int groups) {
  const int kk = w.kk;
  __syncwarp();
  for (int q = w.lane; q < kk * groups; q += 32) {
    const int g = q / kk, j = q % kk;
    args.cand_S[(g * args.group_rows + wi.slot) * kk + j] = w.topS[q];
    args.cand_idx[(g * args.group_rows + wi.slot) * kk + j] = w.topI[q];
  }
}

// The warp's next item (>= nitems: none): the first by index, warp by warp
// over the blocks, so that few items spread over all SMs; then from the queue.
__device__ __forceinline__ int next_item(const TileArgs& args, bool first, int lane) {
  if (first) return (int)((threadIdx.x >> 5) * gridDim.x + blockIdx.x);
  unsigned q = 0;
  if (lane == 0) q = atomicAdd(args.counter, 1u);
  return (int)(gridDim.x * (blockDim.x >> 5) + __shfl_sync(0xffffffffu, q, 0));
}

// Do all blocks lie on lines for every curve's times, and are all anchors in reach
// of the fixed-point times (the usual case: a curve's own times and the anchors
// are then not looked at)?
__device__ __forceinline__ bool grid_is_linear(const TileArgs& args) {
  if (!args.rec || args.grid_dev[2] != 0u) return false;
  return (double)__uint_as_float(args.grid_dev[0]) * (double)__uint_as_float(args.grid_dev[1]) <= kGridTolCycles;
}

// The item's frequencies in the tile's block: [wi.f_lo, f_hi); whether they begin
// or end inside the block, where another item goes on, and whether the tile is
// their last.
struct Part {
  int f_hi;
  bool open, cut, last;
};
template <int W>
__device__ __forceinline__ Part part_of(const TileArgs& args, const WorkItem& wi, int64_t s, int q, int halo) {
  const int64_t lo = q * args.anchor_span, hi = lo + args.anchor_span;
  Part p;
  p.f_hi = (int)min((int64_t)wi.f_hi, hi);
  p.open = halo && wi.f_lo != lo;
  p.cut = halo && p.f_hi < args.nfreq && p.f_hi != hi;
  p.last = s + W >= (int64_t)p.f_hi + (p.cut ? 0 : halo);
  return p;
}

// At most kTileMaxThreads threads a block (wider shapes are launched as more
// blocks): 168 registers, where 128 made the R = 8 loop spill (N = 85, M = 10:
// 1.81 -> 1.85e12 evaluations/s).
template <int R, int PHASE, class P, bool DUMP>
__global__ void __launch_bounds__(kTileMaxThreads, 1) tile_kernel(const __grid_constant__ TileArgs args) {
  using Bin = typename P::Bin;
  using A = typename P::S;
  constexpr int W = 32 * R;
  extern __shared__ __align__(16) unsigned char smem[];
  const Warp<P> w = make_warp<R, P>(smem, args);
  const int64_t F = w.F;
  const bool grid_bad = (*(volatile unsigned*)args.status & kStatusGrid) != 0u;
  const A cal = (A)args.inv_alpha2;
  const bool every_lin = grid_is_linear(args);
  const bool plain_prior = args.inv_alpha2 == 0.0 || (args.inv_alpha2 > 0x1p-90 && args.inv_alpha2 < 0x1p+90);
  const int halo = w.kk > 0 ? 1 : 0;  // peaks need both neighbours of every owned frequency
  const int M = w.M, j0 = w.lane * R;

  for (int it = next_item(args, true, w.lane); it < args.nitems; it = next_item(args, false, w.lane)) {
    WorkItem wi = args.items[it];
    const int c = wi.curve;
    int64_t base = 0, n = args.n_single;
    if (args.offsets) {
      base = args.offsets[c];
      n = args.offsets[c + 1] - base;
    }
    double tm;
    if (!item_begin(args, w, wi, base, n, grid_bad, every_lin, 1, tm)) continue;
    const bool plain = !(args.curve_bad[c] & kCurveWide) && plain_prior;
    A c1 = (A)-INFINITY, c2 = (A)-INFINITY;
    int ce = 0;
    int q = (int)((unsigned)wi.f_lo / (unsigned)args.anchor_span);  // the anchor block of wi.f_lo and the tile
    int64_t s = (int64_t)wi.f_lo - (wi.f_lo == q * args.anchor_span ? halo : 0);
    while (wi.f_lo < wi.f_hi) {
      NlTile<R> nl;
      const Tile g = make_tile<R, P>(args, w, s, q, tm, every_lin, args.curve_bad[c] & kCurveUnfit, nl);
      const unsigned long long floor = w.kk > 0 ? curve_floor(args, c) : 0ull;
      accumulate_tile<R, PHASE, P, DUMP>(args, w, g, nl, base, n, wi);

      // S and the peak test stay in the policy's reduce type
      const Part part = part_of<W>(args, wi, s, q, halo);
      A S[R];
      if (plain)
        reduce_bins<R, P, true>(w, cal, S);
      else
        reduce_bins<R, P, false>(w, cal, S);
#pragma unroll
      for (int r = 0; r < R; ++r) {
        const int64_t k = s + (int64_t)(j0 + r);
        if (args.S_out && k >= wi.f_lo && k < part.f_hi) args.S_out[(int64_t)c * F + k] = (double)S[r];
        if (k < 0 || k >= F) S[r] = (A)-INFINITY;
      }
      if (w.kk > 0) {
        int zero[R];
#pragma unroll
        for (int r = 0; r < R; ++r) zero[r] = 0;
        bool changed = tile_peaks<R, P>(args, w, S, zero, 0, s, wi.f_lo + (part.open ? 1 : 0), part.f_hi, w.topS,
                                        w.topI, floor_value<A>(floor), c1, c2, ce);
        const bool left = part.open && s == wi.f_lo, right = part.last && part.cut;
        if (left || right)
          changed |= meet<A>(args, wi.slot, left, right, wi.f_lo, part.f_hi, __shfl_sync(0xffffffffu, S[0], 0),
                             __shfl_sync(0xffffffffu, S[R > 1 ? 1 : 0], R > 1 ? 0 : 1), 0, c2, c1, 0, 0, w.topS, w.topI,
                             w.kk, w.lane);
        if (changed) raise_floor(args, c, w.topS, w.topI, w.kk, w.lane);
      }
      s += W;
      if (part.last) {
        c1 = c2 = (A)-INFINITY;
        wi.f_lo = part.f_hi;
        s = part.f_hi - halo;
        ++q;
      }
    }
    item_end(args, w, wi, 1);
  }
}

// Several M from one M_max pass (Section 3.4): the kernel accumulates M_max
// bins; for each requested group g (M = M_max / g) it reports, per frequency,
// the largest S over the g bin offsets and that offset (ranking key
// (k << 6) | offset). FP32 sums. At most 256 threads per block (the host
// rejects more): that bound leaves the combination the registers it needs.
// Several-M combinations compiled for one M_max and three groups: the ones
// Section 3.4 suggests (M_max = 60 or 40, giving M = 20, 10 and 4) and the
// M = 20, 10, 5 split of M_max = 20. SPEC 0 is the generic combination.
template <int SPEC>
struct MultiSpec;
template <>
struct MultiSpec<1> {
  static constexpr int MX = 60, G0 = 3, G1 = 6, G2 = 15;
};
template <>
struct MultiSpec<2> {
  static constexpr int MX = 40, G0 = 2, G1 = 4, G2 = 10;
};
template <>
struct MultiSpec<3> {
  static constexpr int MX = 20, G0 = 1, G1 = 2, G2 = 4;
};

// One group's windows at bin m of the fixed combination: the window that ends
// at m, [m - g + 1, m], belongs to offset (m + 1) mod g; its sum is Q_m minus
// the prefix before its start (zero for the first window of offset 0).
template <int G, int M, int MX>
__device__ __forceinline__ void fixed_window(const float2 (&Q)[MX], float (&acc)[G], float cal) {
  if constexpr (M >= G) {
    acc[(M + 1) % G] += bin_term_plain(f2sub(Q[M], Q[M - G]), cal);
  } else if constexpr (M == G - 1) {
    acc[0] += bin_term_plain(f2sub(Q[M], make_float2(0.f, 0.f)), cal);
  }
}

// The wrapping window of each offset o >= 1, [M_max - g + o, M_max - 1] and
// [0, o - 1], added after the others; then the best offset (ties to the lower).
template <int G, int MX>
__device__ __forceinline__ void fixed_finish(const float2 (&Q)[MX], float (&acc)[G], float cal, float& best,
                                             int& bo) {
  const float2 total = Q[MX - 1];
#pragma unroll
  for (int o = 1; o < G; ++o) acc[o] += bin_term_plain(bin_add(f2sub(total, Q[MX - G + o - 1]), Q[o - 1]), cal);
  best = -INFINITY;
  bo = 0;
#pragma unroll
  for (int o = 0; o < G; ++o)
    if (acc[o] > best) {
      best = acc[o];
      bo = o;
    }
}

template <int MX, int G0, int G1, int G2, int M>
__device__ __forceinline__ void fixed_step(float2 (&Q)[MX], float2 v, float2& run, float (&a0)[G0], float (&a1)[G1],
                                           float (&a2)[G2], float cal) {
  run = bin_add(run, v);
  Q[M] = run;
  fixed_window<G0, M, MX>(Q, a0, cal);
  fixed_window<G1, M, MX>(Q, a1, cal);
  fixed_window<G2, M, MX>(Q, a2, cal);
}

template <int MX, int G0, int G1, int G2, int C, int U>
__device__ __forceinline__ void fixed_chunk(float2 (&Q)[MX], const float2 (&v)[4], float2& run, float (&a0)[G0],
                                            float (&a1)[G1], float (&a2)[G2], float cal) {
  if constexpr (U < 4) {
    fixed_step<MX, G0, G1, G2, C * 4 + U>(Q, v[U], run, a0, a1, a2, cal);
    fixed_chunk<MX, G0, G1, G2, C, U + 1>(Q, v, run, a0, a1, a2, cal);
  }
}

// Chunk C of four bins: the next chunk's bins are loaded before this chunk's
// bins are cleared, so the loads of two chunks are in flight together.
template <int MX, int G0, int G1, int G2, int C>
__device__ __forceinline__ void fixed_chunks(float2* col, int st, float2 (&Q)[MX], float2 (&v)[4], float2& run,
                                             float (&a0)[G0], float (&a1)[G1], float (&a2)[G2], float cal) {
  if constexpr (C < MX / 4) {
    float2 vn[4];
    if constexpr (C + 1 < MX / 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) vn[u] = col[((C + 1) * 4 + u) * st];
    }
#pragma unroll
    for (int u = 0; u < 4; ++u) col[(C * 4 + u) * st] = make_float2(0.f, 0.f);
    fixed_chunk<MX, G0, G1, G2, C, 0>(Q, v, run, a0, a1, a2, cal);
    if constexpr (C + 1 < MX / 4) {
#pragma unroll
      for (int u = 0; u < 4; ++u) v[u] = vn[u];
    }
    fixed_chunks<MX, G0, G1, G2, C + 1>(col, st, Q, v, run, a0, a1, a2, cal);
  }
}

// Several-M combination of one slot's M_max bins for a compiled (M_max, groups):
// one pass reads each bin once, clears it, forms the inclusive prefix sums Q_m
// in registers and adds every window that ends at bin m to its offset's sum;
// the windows that wrap past bin M_max - 1 are added last. The windows, terms
// and order of additions are those of the generic combination (in-place prefix
// sums, then per group and offset the windows in order, the wrapping one last),
// so S is the same bit for bit, while each bin costs one shared-memory read and
// one store instead of a read-modify-write for the prefix sums, a read per
// group and a clearing store. Curves whose weights allow bin_term_plain only.
template <int SPEC>
__device__ __forceinline__ void combine_fixed(float2* col, int st, float cal, float (&best)[3], int (&bo)[3]) {
  using SP = MultiSpec<SPEC>;
  constexpr int MX = SP::MX, G0 = SP::G0, G1 = SP::G1, G2 = SP::G2;
  static_assert(MX % 4 == 0 && MX % G0 == 0 && MX % G1 == 0 && MX % G2 == 0, "groups must divide M_max");
  float2 Q[MX];
  float a0[G0], a1[G1], a2[G2];
#pragma unroll
  for (int o = 0; o < G0; ++o) a0[o] = 0.f;
#pragma unroll
  for (int o = 0; o < G1; ++o) a1[o] = 0.f;
#pragma unroll
  for (int o = 0; o < G2; ++o) a2[o] = 0.f;
  float2 v[4];
#pragma unroll
  for (int u = 0; u < 4; ++u) v[u] = col[u * st];
  float2 run = make_float2(0.f, 0.f);
  fixed_chunks<MX, G0, G1, G2, 0>(col, st, Q, v, run, a0, a1, a2, cal);
  fixed_finish<G0, MX>(Q, a0, cal, best[0], bo[0]);
  fixed_finish<G1, MX>(Q, a1, cal, best[1], bo[1]);
  fixed_finish<G2, MX>(Q, a2, cal, best[2], bo[2]);
}

// The combination of one tile's M_max bins for any groups: in-place prefix sums first, then per
// group and offset the windows in order (window j of offset o spans bins [j g +
// o, j g + o + g - 1]; its sum is Q[end] - Q[start - 1], and its end is the next
// window's start - 1), the one that wraps past bin M_max - 1 last. The lane's R
// frequencies advance together. Short loops, as in reduce_bins.
template <int R>
__device__ __forceinline__ void prefix_bins(const Warp<AccF32>& w, float2 (&total)[R]) {
  constexpr unsigned kStride = Warp<AccF32>::kBinStride;
  const unsigned rstride = (unsigned)w.M * kStride;
  unsigned a = smem_u32(w.bins);
#pragma unroll
  for (int r = 0; r < R; ++r) total[r] = make_float2(0.f, 0.f);
  int m = 0;
#pragma unroll 1
  for (; m + 4 <= w.M; m += 4, a += 4 * kStride) {  // four bins loaded before any is stored back
    float2 v[R][4];
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int u = 0; u < 4; ++u) lds(a + (unsigned)r * rstride + u * kStride, v[r][u]);
#pragma unroll
    for (int r = 0; r < R; ++r)
#pragma unroll
      for (int u = 0; u < 4; ++u) {
        total[r] = bin_add(total[r], v[r][u]);
        sts(a + (unsigned)r * rstride + u * kStride, total[r]);
      }
  }
#pragma unroll 1
  for (; m < w.M; ++m, a += kStride)
#pragma unroll
    for (int r = 0; r < R; ++r) {
      float2 v;
      lds(a + (unsigned)r * rstride, v);
      total[r] = bin_add(total[r], v);
      sts(a + (unsigned)r * rstride, total[r]);
    }
}

// S_g of the lane's R frequencies: the largest S over the gs offsets (ties to
// the lower). OB offsets advance together (R OB independent sums: a window's
// load, reciprocal and addition take ~110 clk one after the other); offsets past
// gs - 1 repeat the last one, which changes nothing.
template <int R, int OB, bool PLAIN>
__device__ __forceinline__ void best_offset(const Warp<AccF32>& w, const float2 (&total)[R], int gs, float cal,
                                            float (&S)[R], int (&off)[R]) {
  constexpr unsigned kStride = Warp<AccF32>::kBinStride;
  const unsigned rstride = (unsigned)w.M * kStride, col = smem_u32(w.bins), step = (unsigned)gs * kStride;
  const int Mg = w.M / gs;
#pragma unroll
  for (int r = 0; r < R; ++r) {
    S[r] = -INFINITY;
    off[r] = 0;
  }
#pragma unroll 1
  for (int o0 = 0; o0 < gs; o0 += OB) {
    float2 prev[OB][R], q[OB][R];
    float acc[OB][R];
    unsigned e[OB];
#pragma unroll
    for (int b = 0; b < OB; ++b) {
      const int o = o0 + b < gs ? o0 + b : gs - 1;
      e[b] = col + (unsigned)(o + gs - 1) * kStride;
#pragma unroll
      for (int r = 0; r < R; ++r) {
        prev[b][r] = make_float2(0.f, 0.f);
        if (o > 0) lds(col + (unsigned)r * rstride + (unsigned)(o - 1) * kStride, prev[b][r]);
        q[b][r] = make_float2(0.f, 0.f);
        if (Mg > 1) lds(e[b] + (unsigned)r * rstride, q[b][r]);
        acc[b][r] = 0.f;
      }
    }
    const auto add = [&](float& a, float2 d) { a += PLAIN ? bin_term_plain(d, cal) : bin_term(d, cal); };
    float2 q0[OB][R];
#pragma unroll
    for (int b = 0; b < OB; ++b)
#pragma unroll
      for (int r = 0; r < R; ++r) q0[b][r] = prev[b][r];
#pragma unroll 1
    for (int j = 1; j < Mg; ++j) {  // the windows before the last; the next one's end is loaded ahead
#pragma unroll
      for (int b = 0; b < OB; ++b) {
        e[b] += step;
#pragma unroll
        for (int r = 0; r < R; ++r) {
          float2 n = make_float2(0.f, 0.f);
          if (j + 1 < Mg) lds(e[b] + (unsigned)r * rstride, n);
          add(acc[b][r], f2sub(q[b][r], prev[b][r]));
          prev[b][r] = q[b][r];
          q[b][r] = n;
        }
      }
    }
#pragma unroll
    for (int b = 0; b < OB; ++b)
#pragma unroll
      for (int r = 0; r < R; ++r) {
        // the last window: up to bin M_max - 1, and for o > 0 on to bin o - 1
        add(acc[b][r], bin_add(f2sub(total[r], prev[b][r]), q0[b][r]));
        if (acc[b][r] > S[r]) {
          S[r] = acc[b][r];
          off[r] = o0 + b;
        }
      }
  }
}

template <int R, int PHASE, int SPEC>
__global__ void __launch_bounds__(kMultiMaxThreads, 1) tile_kernel_multi(const __grid_constant__ TileArgs args) {
  using P = AccF32;
  using A = float;
  constexpr int W = 32 * R;
  extern __shared__ __align__(16) unsigned char smem[];
  const Warp<P> w = make_warp<R, P>(smem, args);
  const int64_t F = w.F;
  const int Mx = w.M, ng = args.ngroups, kk = w.kk;
  const bool grid_bad = (*(volatile unsigned*)args.status & kStatusGrid) != 0u;
  const A cal = (A)args.inv_alpha2;
  const bool every_lin = grid_is_linear(args);
  const bool plain_prior = args.inv_alpha2 == 0.0 || (args.inv_alpha2 > 0x1p-90 && args.inv_alpha2 < 0x1p+90);
  const int halo = kk > 0 ? 1 : 0;
  const int j0 = w.lane * R;

  for (int it = next_item(args, true, w.lane); it < args.nitems; it = next_item(args, false, w.lane)) {
    WorkItem wi = args.items[it];
    const int c = wi.curve;
    int64_t base = 0, n = args.n_single;
    if (args.offsets) {
      base = args.offsets[c];
      n = args.offsets[c + 1] - base;
    }
    double tm;
    if (!item_begin(args, w, wi, base, n, grid_bad, every_lin, ng, tm)) continue;
    const bool plain = !(args.curve_bad[c] & kCurveWide) && plain_prior;
    // S and offset of the two frequencies before the tile, per group (lane g holds group g's)
    A carry1 = -INFINITY, carry2 = -INFINITY;
    int carrye = 0;
    int q = (int)((unsigned)wi.f_lo / (unsigned)args.anchor_span);  // the anchor block of wi.f_lo and the tile
    int64_t s = (int64_t)wi.f_lo - (wi.f_lo == q * args.anchor_span ? halo : 0);
    while (wi.f_lo < wi.f_hi) {
      NlTile<R> nl;
      const Tile g0 = make_tile<R, P>(args, w, s, q, tm, every_lin, args.curve_bad[c] & kCurveUnfit, nl);
      accumulate_tile<R, PHASE, P, false>(args, w, g0, nl, base, n, wi);

      // the reported S of group g per owned frequency, and the peaks
      auto emit = [&](int g, const A (&S)[R], const int (&off)[R]) {
        const Part part = part_of<W>(args, wi, s, q, halo);
        if (args.S_out) {
#pragma unroll
          for (int r = 0; r < R; ++r) {
            const int64_t k = s + (int64_t)(j0 + r);
            if (k >= wi.f_lo && k < part.f_hi) args.S_out[((int64_t)c * ng + g) * F + k] = (double)S[r];
          }
        }
        if (kk > 0) {
          A c1 = __shfl_sync(0xffffffffu, carry1, g), c2 = __shfl_sync(0xffffffffu, carry2, g);
          int ce = __shfl_sync(0xffffffffu, carrye, g);
          const int64_t row = (int64_t)c * ng + g;
          double* const topS = w.topS + g * kk;
          int* const topI = w.topI + g * kk;
          bool changed = tile_peaks<R, P>(args, w, S, off, 6, s, wi.f_lo + (part.open ? 1 : 0), part.f_hi, topS, topI,
                                          floor_value<A>(curve_floor(args, row)), c1, c2, ce);
          const bool left = part.open && s == wi.f_lo, right = part.last && part.cut;
          if (left || right)
            changed |= meet<A>(args, g * args.group_rows + wi.slot, left, right, wi.f_lo, part.f_hi,
                               __shfl_sync(0xffffffffu, S[0], 0), __shfl_sync(0xffffffffu, S[R > 1 ? 1 : 0], R > 1 ? 0 : 1),
                               __shfl_sync(0xffffffffu, off[0], 0), c2, c1, ce, 6, topS, topI, kk, w.lane);
          if (changed) raise_floor(args, row, topS, topI, kk, w.lane);
          if (w.lane == g) {
            carry1 = c1;
            carry2 = c2;
            carrye = ce;
          }
        }
      };
      if constexpr (SPEC != 0) {
        if (plain) {
          A Sg[3][R];
          int offg[3][R];
#pragma unroll 1
          for (int r = 0; r < R; ++r) {  // one frequency at a time: the pass holds its prefix sums in registers
            float best[3];
            int bo[3];
            combine_fixed<SPEC>(reinterpret_cast<float2*>(w.bins) + r * Mx * 32, 32, cal, best, bo);
            const int64_t k = s + (int64_t)(j0 + r);
#pragma unroll
            for (int q = 0; q < 3; ++q) {
              Sg[q][r] = (k >= 0 && k < F) ? best[q] : (A)-INFINITY;
              offg[q][r] = bo[q];
            }
          }
#pragma unroll 1
          for (int g = 0; g < 3; ++g) {
            A S[R];
            int off[R];
#pragma unroll
            for (int r = 0; r < R; ++r) {
              S[r] = Sg[g][r];
              off[r] = offg[g][r];
            }
            emit(g, S, off);
          }
        }
      }
      float2 total[R];
      if (SPEC == 0 || !plain) prefix_bins<R>(w, total);
#pragma unroll 1
      for (int g = 0; g < ng && (SPEC == 0 || !plain); ++g) {
        A S[R];
        int off[R];
        const int gs = args.group_g[g];
        // as many offsets together as leave the registers for R frequencies each
        constexpr int kOb = R <= 3 ? 3 : (R <= 5 ? 2 : 1);
        if (!plain)
          best_offset<R, 1, false>(w, total, gs, cal, S, off);
        else if (gs == 1)
          best_offset<R, 1, true>(w, total, gs, cal, S, off);
        else if (R <= 2 && gs % 5 == 0)
          best_offset<R, R <= 2 ? 5 : 1, true>(w, total, gs, cal, S, off);
        else if (R <= 3 && gs % 3 != 0 && gs % 2 == 0)
          best_offset<R, 2, true>(w, total, gs, cal, S, off);
        else
          best_offset<R, kOb, true>(w, total, gs, cal, S, off);
#pragma unroll
        for (int r = 0; r < R; ++r) {
          const int64_t k = s + (int64_t)(j0 + r);
          if (k < 0 || k >= F) S[r] = (A)-INFINITY;
        }
        emit(g, S, off);
      }
      // clear the bins for the next tile
      for (int q = 0; q < R * Mx && (SPEC == 0 || !plain); ++q) reinterpret_cast<float2*>(w.bins)[q * 32] = make_float2(0.f, 0.f);
      const Part part = part_of<W>(args, wi, s, q, halo);
      s += W;
      if (part.last) {
        carry1 = carry2 = -INFINITY;
        wi.f_lo = part.f_hi;
        s = part.f_hi - halo;
        ++q;
      }
    }
    item_end(args, w, wi, ng);
  }
}

}  // namespace
#endif  // __CUDACC__

}  // namespace fpw
