// Instantiations of the tile kernel with compensated FP32 bin sums (fpw_tile.cuh).
#include "fpw_tile.cuh"

namespace fpw {

const void* tile_fn_comp(int R, int phase_mode, bool dump) {
  const bool fp32p = phase_mode == FPW_PHASE_FP32;
#define FPW_INST(RR)                                                                                         \
  if (R == RR) {                                                                                             \
    if (dump)                                                                                                \
      return fp32p ? (const void*)&tile_kernel<RR, FPW_PHASE_FP32, AccComp, true>                                 \
                   : (const void*)&tile_kernel<RR, FPW_PHASE_FIXED64, AccComp, true>;                             \
    return fp32p ? (const void*)&tile_kernel<RR, FPW_PHASE_FP32, AccComp, false>                                  \
                 : (const void*)&tile_kernel<RR, FPW_PHASE_FIXED64, AccComp, false>;                              \
  }
  FPW_INST(1)
  FPW_INST(2)
  FPW_INST(4)
  FPW_INST(8)
#undef FPW_INST
  return nullptr;
}

}  // namespace fpw
