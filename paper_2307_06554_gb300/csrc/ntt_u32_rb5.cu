// Radix-32 register passes (32 coefficients per operand per thread):
// candidates the autotuner weighs against the default radix-16 kernels
// (n <= 2^13) and against the thread-block-cluster kernel (n = 2^14, where
// a 512-thread CTA holds the whole product).
// 32-bit words, reduction modes 1 and 2, n = 2^9 .. 2^13; modes 0..2 at 2^14.
#include "ntt_info.cuh"

namespace pm {
bool lookup_ntt_u32_rb5(int logn, int mode, KernelInfo* ki) {
#define PM_V(L, M)                                  \
  if (logn == L && mode == M) {                     \
    *ki = ntt_info_rb<uint32_t, L, M, false, 5>();     \
    return true;                                    \
  }
  // 2^14: the padded layout, whose addresses are a base and constant offsets,
  // fits 128 registers where the swizzled one spilled 320 bytes a thread
  // (1000 rows, q < 2^31: 157.6 against 171.8 us; radix 16 with 1024 threads
  // of 64 registers 172.5)
#define PM_P(L, M)                                              \
  if (logn == L && mode == M) {                                 \
    *ki = ntt_info_x<uint32_t, L, M, false, 5, 128, 5, false>(); \
    return true;                                                \
  }
  PM_V(9, 1) PM_V(10, 1) PM_V(11, 1) PM_V(12, 1) PM_V(13, 1)
  PM_V(9, 2) PM_V(10, 2) PM_V(11, 2) PM_V(12, 2) PM_V(13, 2)
  PM_P(14, 0) PM_P(14, 1) PM_P(14, 2)
#undef PM_P
#undef PM_V
  return false;
}
}  // namespace pm
