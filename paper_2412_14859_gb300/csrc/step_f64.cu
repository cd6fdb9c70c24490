// step_f64.cu -- instantiations of the fused step for ST_F64 storage.
#include "launch.h"
#include "pair_tile.cuh"

namespace cgevap {

template <int Q, int TX, int TY, int MINB>
static KernelRef reg_ref() {
  return pair_ref<Q, ST_F64, TX, TY, MINB, false>();
}

KernelRef step_kernel_f64(int q, int variant) {
  if (q == 19) {
    switch (variant) {
      case 0: return reg_ref<19, 16, 8, 2>();
      case 1: return reg_ref<19, 32, 8, 1>();  // 240 registers a thread; variant 3: 128, two CTAs per SM
      case 2: return reg_ref<19, 16, 16, 1>();
      case 3: return reg_ref<19, 32, 8, 2>();
      case 4: return reg_ref<19, 32, 4, 2>();
    }
  } else if (q == 9) {
    switch (variant) {
      case 0: return reg_ref<9, 128, 1, 1>();
      case 1: return reg_ref<9, 64, 1, 2>();
    }
  }
  return {nullptr, 0};
}

KernelRef patch_kernel_f64(long long cells) { return patch_pick<ST_F64>(cells); }

}  // namespace cgevap
