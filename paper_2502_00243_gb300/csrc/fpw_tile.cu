// Host side of the persistent FPW tile kernels (device templates in
// fpw_tile.cuh): shared-memory sizes, kernel selection and launches.
#include <math.h>

#include "fpw_tile.cuh"

namespace fpw {
namespace {

const void* pick(int R, int phase_mode, int accum, bool multi, bool dump, int spec = 0) {
  if (multi) return dump ? nullptr : tile_fn_multi(R, phase_mode, spec);
  switch (accum) {
    case FPW_ACCUM_FP32: {
      const void* fn = tile_fn_f32(R, phase_mode, dump);
      return fn ? fn : tile_fn_f32_odd(R, phase_mode, dump);
    }
    case FPW_ACCUM_FP64: return tile_fn_f64(R, phase_mode, dump);
    case FPW_ACCUM_FP32_COMP: return tile_fn_comp(R, phase_mode, dump);
    default: return nullptr;
  }
}

}  // namespace

size_t tile_smem_bytes(int T, int R, int M, int k, int accum, int ngroups) {
  return (size_t)(T / 32) * warp_layout(R, M, accum_bin_bytes(accum), k, ngroups).total;
}

size_t tile_shape_bytes(int T, int R, int M, int NC, int accum, int ngroups) {
  const size_t bin = accum_bin_bytes(accum), tops = (size_t)(ngroups > 1 ? ngroups : 1) * FPW_MAX_TOPK;
  const size_t part[] = {(size_t)R * M * T * bin, (size_t)(NC + 2) * 16, (size_t)(NC + 2) * bin, (size_t)T * R * 8,
                         (size_t)T * R * 4, tops * 8, tops * 4, (size_t)(T / 32) * 16, 32 * 8, 64};
  size_t o = 0;
  for (size_t p : part) o = align16(o + p);
  return o;
}

int tile_max_warps(bool multi) { return (multi ? kMultiMaxThreads : kTileMaxThreads) / 32; }

bool tile_supported_R(int R) { return R >= 1 && R <= 8 && R != 7; }

bool tile_has_R(int R, int accum, bool multi) {
  if (R == 1 || R == 2 || R == 4 || R == 8) return true;
  return (R == 3 || R == 5 || R == 6) && accum == FPW_ACCUM_FP32 && !multi;
}

int tile_max_blocks_per_sm(int R, int phase_mode, int accum, int T, size_t smem, bool multi, bool dump, int spec) {
  const void* fn = pick(R, phase_mode, accum, multi, dump, spec);
  // (here, where it is known which one runs: the others need not be loaded)
  if (!fn || allow_shared_memory(fn, 0) != cudaSuccess) return 0;
  int nb = 0;
  if (cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, fn, T, smem) != cudaSuccess) return 0;
  return nb;
}

cudaError_t launch_tile(const TileArgs& a, const TileShape& s, int phase_mode, int accum, int grid, cudaStream_t st) {
  const void* fn = pick(s.lane_R, phase_mode, accum, a.ngroups > 0, a.bins_out != nullptr,
                        multi_spec_of(a.M, a.ngroups, a.group_g));
  if (!fn) return cudaErrorInvalidDeviceFunction;
  void* params[] = {const_cast<TileArgs*>(&a)};
  return cudaLaunchKernel(fn, dim3(grid), dim3(32 * s.warps), params, s.smem, st);
}

}  // namespace fpw
