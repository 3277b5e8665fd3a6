// Alternative k_ntt_batch shapes per degree (see NttCfg in ntt_info.cuh): the
// swizzled two-operand kernel at 128 registers.
#pragma once
#include "ntt_info.cuh"

namespace pm {

template <int MODE>
bool ntt_alt_u32(int logn, KernelInfo* ki) {
  switch (logn) {
#define PM_OLD(L)                                        \
  case L:                                                \
    *ki = ntt_info_rb<uint32_t, L, MODE, false, 4>();    \
    return true;
    PM_OLD(5) PM_OLD(6) PM_OLD(7) PM_OLD(8) PM_OLD(9) PM_OLD(10) PM_OLD(11) PM_OLD(12) PM_OLD(13)
#undef PM_OLD
    default:
      return false;
  }
}

}  // namespace pm
