// step_f32.cu -- instantiations of the fused step for ST_F32 storage.
#include "launch.h"
#include "pair_tile.cuh"

namespace cgevap {

// Every FP32 variant issues its own cells' pulls one plane ahead (PF): 16.2 -> 18.7 GLUPS on the
// 192^3 drop at the same 128 registers.
template <int Q, int TX, int TY, int MINB, int S = ST_F32>
static KernelRef reg_ref() {
  return pair_ref<Q, S, TX, TY, MINB, true>();
}

KernelRef step_kernel_f32(int q, int variant) {
  if (q == 19) {
    switch (variant) {
      case 0: return reg_ref<19, 32, 4, 4>();  // 128 threads, four CTAs per SM
      case 1: return reg_ref<19, 16, 8, 4>();
      case 2: return reg_ref<19, 16, 16, 2>();
      case 3: return reg_ref<19, 16, 4, 8>();  // 64 threads, eight CTAs per SM
      case 4: return reg_ref<19, 32, 8, 2>();
    }
  } else if (q == 9) {
    switch (variant) {
      case 0: return reg_ref<9, 128, 1, 4>();
      case 1: return reg_ref<9, 64, 1, 8>();
    }
  }
  return {nullptr, 0};
}

// FP32 pairs with exact colour masses (ST_F32X): the same tiles.
KernelRef step_kernel_f32x(int q, int variant) {
  if (q == 19) {
    switch (variant) {
      case 0: return reg_ref<19, 32, 4, 4, ST_F32X>();
      case 1: return reg_ref<19, 16, 8, 4, ST_F32X>();
      case 2: return reg_ref<19, 16, 16, 2, ST_F32X>();
      case 3: return reg_ref<19, 16, 4, 8, ST_F32X>();
      case 4: return reg_ref<19, 32, 8, 2, ST_F32X>();
    }
  } else if (q == 9) {
    switch (variant) {
      case 0: return reg_ref<9, 128, 1, 4, ST_F32X>();
      case 1: return reg_ref<9, 64, 1, 8, ST_F32X>();
    }
  }
  return {nullptr, 0};
}

KernelRef patch_kernel_f32(int storage, long long cells) {
  return storage == ST_F32X ? patch_pick<ST_F32X>(cells) : patch_pick<ST_F32>(cells);
}

}  // namespace cgevap
