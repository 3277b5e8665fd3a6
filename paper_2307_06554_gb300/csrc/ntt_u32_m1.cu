// k_ntt_batch instantiations: 32-bit words, reduction mode 1, n = 2^4 .. 2^14.
#include "ntt_info.cuh"

namespace pm {
bool lookup_ntt_u32_m1(int logn, KernelInfo* ki) {
  switch (logn) {
#define PM_CASE(L)                         \
  case L:                                  \
    *ki = ntt_info<uint32_t, L, 1>();      \
    return true;
    PM_CASE(4) PM_CASE(5) PM_CASE(6) PM_CASE(7) PM_CASE(8) PM_CASE(9) PM_CASE(10)
    PM_CASE(11) PM_CASE(12) PM_CASE(13) PM_CASE(14)
#undef PM_CASE
    default:
      return false;
  }
}

// One operand in registers at a time, for batches at 2^10, 2^11 that run ahead
// of their predecessor: the faster shape there (see NttCfg), as the other
// modes' default is.
bool lookup_ntt_u32_m1_seq(int logn, KernelInfo* ki) {
  if (logn == 10) *ki = ntt_info_x<uint32_t, 10, 1, false, 4, 96, 4, true>();
  if (logn == 11) *ki = ntt_info_x<uint32_t, 11, 1, false, 4, 96, 4, true>();
  return logn == 10 || logn == 11;
}
}  // namespace pm
