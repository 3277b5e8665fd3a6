// k_ntt_batch with the unit for the smallest moduli (ntt_tiny.cuh), n = 2^8 .. 2^10.
//
// CTAs of eight warps at 96 registers or a little more, two per SM: the
// unit's straight-line body is long, and warps of one CTA, started together,
// share its instruction fetch.  n = 1024, q = 12289, overlapped batches of
// 4096 / 32768 products: 15.2 / 104 us, against 16.9 / 112 with five
// four-warp CTAs and 20.9 / 175 for the radix-16 kernel of the unreduced
// mode.
#include "ntt_info.cuh"

namespace pm {

constexpr int kTinyWarps = 8;

template <int LOGN>
static KernelInfo tiny_info() {
  // the padded layout of ntt_tiny.cuh takes n + n / 8 words per operand: PAD = 3
  using S = Shape<uint32_t, LOGN, 5, 3>;
  KernelInfo ki;
  ki.fn = (const void*)k_ntt_batch<S, kTiny, kTinyWarps, 96, false, true>;
  ki.rb = 5;
  ki.mode = kSmall;  // reported as the unreduced mode: no conditional subtraction either
  ki.regs = 96;
  ki.pad = 3;
  ki.seq = 1;
  ki.tiny = 1;
  ki.team = S::T;
  ki.block = 32 * kTinyWarps;
  ki.units_per_cta = kTinyWarps * (32 / S::T);
  ki.smem = ki.units_per_cta * S::SMEM_WORDS * 4;
  return ki;
}

bool lookup_ntt_tiny(int logn, KernelInfo* ki) {
  switch (logn) {
    case 8: *ki = tiny_info<8>(); return true;
    case 9: *ki = tiny_info<9>(); return true;
    case 10: *ki = tiny_info<10>(); return true;
    default: return false;
  }
}
}  // namespace pm
