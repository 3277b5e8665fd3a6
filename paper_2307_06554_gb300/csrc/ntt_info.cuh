// Launch description of one k_ntt_batch instantiation.
#pragma once
#include "kernels.h"
#include "ntt.cuh"

namespace pm {

constexpr int kNttWarps = 4;  // warps per CTA when a team fits in a warp

// Default shape of the batch kernel per word size and degree: stage bits per
// register pass (RB), exchange layout (PAD: 0 the XOR swizzle, else the
// padded layout with one word after every 2^PAD), register budget per thread
// and whether one operand at a time is held in registers (SEQ).  Measured on
// GB300 with 2^22 coefficients per batch (2^21 for 64-bit words), launches
// back to back:
//   32-bit words, n <= 2^9:      radix 16, padded, 96 registers, both operands;
//   32-bit words, 2^10, 2^11:    radix 16, padded, 96 registers, one operand
//                                 (n = 1024, q = 12289: 27.0 -> 25.7 us; 31-bit
//                                 primes, 3 M coefficients: 22.5 us at 2^10,
//                                 both operands 23.6; 24.0 / 25.1 at 2^11),
//                                 except
//   ... Harvey's bounds:         both operands, except in batches that run ahead
//                                 of their predecessor (q < 2^30, 3.2 M
//                                 coefficients, one operand / both: 23.6 / 22.7
//                                 us at 2^10, 24.4 / 24.3 at 2^11; overlapped
//                                 19.3 / 19.9 and 20.2 / 21.3: see
//                                 polymul_create);
//   32-bit words, n >= 2^12:     radix 16, padded, 64 registers, both operands:
//                                 32 warps per SM hold the multiply pipe at
//                                 74 % of its cycles.  16 M coefficients,
//                                 q < 2^31: 112.4 us at 2^12 (swizzled, 128
//                                 registers: 123.0), 141.3 at 2^13 (164.6);
//                                 8 M, q < 2^30, 2^12: 57.2 (62.0).  Few
//                                 products and batches that run ahead of their
//                                 predecessor take the 128-register kernel for
//                                 some sizes (see polymul_create).  2^14 takes a
//                                 512-thread CTA of its own (ntt_u32_rb5.cu);
//   64-bit words, 2^6 .. 2^11:   radix 8, padded, 96 registers, one operand
//                                 (radix 16 spills: 1.35-1.47x faster);
//   64-bit words, 2^12:          radix 8, padded, 64 registers, both operands:
//                                 twice the threads per unit and half the
//                                 straight-line code of radix 16, whose fetch
//                                 stalled it (n = 4096: 152 units 26.9 -> 20.3
//                                 us, 608 units 82.1 -> 67.2, 2048 units 233 ->
//                                 227; at 2^11 and 2^10 the spills of its 64
//                                 registers outweigh that).  The
//                                 multiply pipe then bounds it (65 % of its
//                                 cycles; loops over the passes in place of the
//                                 straight line cut the fetch stalls to nothing
//                                 and gained nothing more);
//   64-bit words, 2^13:          radix 16, padded, 128 registers (radix 8 with
//                                 1024 threads: the same time).
template <typename W, int LOGN, int MODE = 1>
struct NttCfg {
  static constexpr bool u32 = sizeof(W) == 4;
  static constexpr int RB = u32 ? 4 : (LOGN >= 6 && LOGN <= 12 ? 3 : 4);
  static constexpr bool SEQ = u32 ? MODE != kL4 && (LOGN == 10 || LOGN == 11) : (LOGN >= 6 && LOGN <= 11);
  static constexpr int PAD = u32 ? (LOGN >= 5 ? 4 : 0) : (LOGN >= 6 ? RB : 0);
  static constexpr int REGS = u32 ? (LOGN < 5 ? 128 : LOGN < 12 ? 96 : 64) : (LOGN >= 6 && LOGN <= 11 ? 96 : LOGN == 12 ? 64 : 128);
};

// Shape of the direct kernels (operands in host memory): one per word size and
// degree, both operands in registers.  The link bounds them, and what counts is
// loads in flight, so they did not follow the batch kernels to 64 registers
// (64-bit words, n = 1024, two primes, 89 products through polymul_batch_host:
// 38.2 us, radix 8 at 64 registers 40.0).
template <typename W, int LOGN>
struct DirectCfg {
  static constexpr bool u32 = sizeof(W) == 4;
  static constexpr bool mid = LOGN >= (u32 ? 5 : 6) && LOGN <= 11;
  static constexpr int RB = !u32 && mid ? 3 : 4;
  static constexpr int REGS = mid ? 96 : 128;
  static constexpr int PAD = mid ? RB : !u32 && LOGN > 11 ? RB : 0;
};

// every parameter explicit
template <typename W, int LOGN, int MODE, bool AUX, int RB, int REGS, int PAD, bool SEQ, bool DIRECT = false>
KernelInfo ntt_info_x() {
  using S = Shape<W, LOGN, RB, PAD>;
  KernelInfo ki;
  ki.fn = (const void*)k_ntt_batch<S, MODE, kNttWarps, REGS, AUX, SEQ, DIRECT>;
  ki.rb = RB;
  ki.mode = base_mode(MODE);
  ki.regs = REGS;
  ki.pad = PAD;
  ki.seq = SEQ ? 1 : 0;
  ki.team = S::T;
  if (S::T <= 32) {
    ki.block = 32 * kNttWarps;
    ki.units_per_cta = kNttWarps * (32 / S::T);
  } else {
    ki.block = S::T;
    ki.units_per_cta = 1;
  }
  ki.smem = ki.units_per_cta * S::SMEM_WORDS * (int)sizeof(W);
  return ki;
}

// the default shape for (W, LOGN)
template <typename W, int LOGN, int MODE, bool AUX = false>
KernelInfo ntt_info() {
  using C = NttCfg<W, LOGN, MODE>;
  return ntt_info_x<W, LOGN, MODE, AUX, C::RB, C::REGS, C::PAD, C::SEQ>();
}

// another register radix, swizzled layout, 128 registers, both operands
template <typename W, int LOGN, int MODE, bool AUX, int RB>
KernelInfo ntt_info_rb() {
  return ntt_info_x<W, LOGN, MODE, AUX, RB, 128, 0, false>();
}

}  // namespace pm
