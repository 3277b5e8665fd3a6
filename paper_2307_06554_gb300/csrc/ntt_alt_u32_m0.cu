// k_ntt_batch alternative shapes, 32-bit words, reduction mode 0: the
// swizzled two-operand kernel at 128 registers for 2^12, 2^13, with the
// conditional subtractions unfused as in the other kernels of this mode that
// run 16 warps per SM (see kApart).
#include "ntt_alt.cuh"

namespace pm {
bool lookup_ntt_alt_u32_m0(int logn, KernelInfo* ki) {
  if (logn == 12) *ki = ntt_info_rb<uint32_t, 12, kApart, false, 4>();
  if (logn == 13) *ki = ntt_info_rb<uint32_t, 13, kApart, false, 4>();
  return logn == 12 || logn == 13;
}
}  // namespace pm
