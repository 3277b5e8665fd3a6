// One (product, prime) unit for the smallest moduli (q < 18500: the rings of
// lattice schemes, 12289 above all), n = 2^8 .. 2^10.
//
// Two things set it apart from polymul_unit (ntt.cuh):
//
//  * Plantard's multiplication by a constant (ntt_tiny_arith.h): one
//    precomputed word per root, two low products, two shifts (the second
//    fused with the butterfly's addition): 23.5 butterflies per SM per clock
//    measured, against 13 for the Shoup form of ntt.cuh (whose high product
//    takes two issue slots of the multiply pipe).  No reduction is needed on
//    the way forward.
//  * The transform stops at polynomials of 8 coefficients: the ring splits
//    into n / 8 rings x^8 - z, and the products there are 64 multiply-adds
//    of centred residues whose sums of eight fit 32 bits, reduced once per
//    output.  Eight coefficients cost 15.75 multiplies and 7.75 shifts each;
//    the three stages they replace, with the pointwise product, cost 14 and
//    about 20, and would bring a third exchange and the loads of 7/8 of the
//    twiddles.
//
// Layout: a thread holds 32 coefficients, n / 32 threads per unit.  The top
// layout (slot e is coefficient t + e n / 32) runs the first five stages
// with twiddles that all threads share; one exchange brings the low layout
// (coefficients 32 t .. 32 t + 31), where the remaining stages and the
// products run.  Coefficient j sits at word j + 4 (j >> 5): scalar accesses
// of the top layout and 16-byte accesses of the low one are both free of
// bank conflicts.
//
// Bounds, in units of (q - 1) / 2: inputs 2, one more per forward stage (at
// most 9); b is brought back to 1 before the products, a when it is parked.
// The inverse doubles per stage without a multiplication; tiny_bounds tracks
// it slot by slot at compile time and reduces a slot where a sum could pass
// kTinyLim, the largest factor the multiplication takes.
#pragma once
#include <cstdint>

#include "arith.cuh"
#include "ntt_tiny_arith.h"

namespace pm {

// Compile-time bounds of the inverse stages on 32 slots.
struct TinyBounds {
  int b[32] = {};
  bool reduce[5][32] = {};  // before stage bit i: slots to bring back to 1
  int out = 0;              // largest bound after the last stage run
};
// stages on slot bits lo .. hi - 1 from the uniform bound `in`; `last`: the
// final stage multiplies both outputs
constexpr TinyBounds tiny_bounds(int in, int lo, int hi, bool last) {
  TinyBounds t;
  for (int e = 0; e < 32; ++e) t.b[e] = in;
  for (int i = lo; i < hi; ++i) {
    for (int e = 0; e < 32; ++e) {
      if (e & (1 << i)) continue;
      const int f = e | (1 << i);
      if (t.b[e] + t.b[f] > kTinyLim) {
        const int big = t.b[e] >= t.b[f] ? e : f;
        t.reduce[i][big] = true;
        t.b[big] = 1;
      }
      if (t.b[e] + t.b[f] > kTinyLim) {
        const int big = t.b[e] >= t.b[f] ? e : f;
        t.reduce[i][big] = true;
        t.b[big] = 1;
      }
      const int s = t.b[e] + t.b[f];
      t.b[f] = 1;
      t.b[e] = (last && i == hi - 1) ? 1 : s;
    }
  }
  for (int e = 0; e < 32; ++e) t.out = t.out > t.b[e] ? t.out : t.b[e];
  return t;
}

template <int IN, int LO, int HI, bool LAST>
struct TinyStages {
  static constexpr TinyBounds v = tiny_bounds(IN, LO, HI, LAST);
};

template <class S>
struct TinyShape {
  static constexpr int T = S::N / 32;
  static constexpr int LOWLOG = S::LOGN - 5;            // lowest coefficient bit of the top layout
  static constexpr int LOW_HI = LOWLOG;                 // stages run in the low layout: bits LOW_HI - 1 .. kTinyLogM
  static constexpr int TOP_LO = LOWLOG < kTinyLogM ? kTinyLogM - LOWLOG : 0;  // first slot bit with a stage on top
  __host__ __device__ static constexpr int top_pos(int e) { return T * e + 4 * ((T * e) >> 5); }
};

// four words of a root table
__device__ __forceinline__ int4 tiny_ld4(const int* p) { return __ldg(reinterpret_cast<const int4*>(p)); }

// forward stages of the top layout: the roots are the same for every thread
template <class S>
__device__ __forceinline__ void tiny_fwd_top(int (&x)[32], const int* __restrict__ tw, const TinyMod& m) {
  using TS = TinyShape<S>;
  sfor<4, TS::TOP_LO - 1, -1>([&](auto hc) {
    constexpr int hb = decltype(hc)::value;       // slot bit; coefficient bit LOWLOG + hb
    constexpr int first = 1 << (4 - hb);          // root index of group 0
    auto apply = [&](auto gc, int w) {
      constexpr int g = decltype(gc)::value;
      sfor<0, (1 << hb)>([&](auto lc) {
        constexpr int u = (g << (hb + 1)) | decltype(lc)::value;
        tiny_ct(x[u], x[u | (1 << hb)], w, m);
      });
    };
    if constexpr (first < 4) {
      sfor<0, first>([&](auto gc) { apply(gc, __ldg(tw + first + decltype(gc)::value)); });
    } else {
      sfor<0, first, 4>([&](auto gc) {
        constexpr int g = decltype(gc)::value;
        const int4 w = tiny_ld4(tw + first + g);
        apply(std::integral_constant<int, g>{}, w.x);
        apply(std::integral_constant<int, g + 1>{}, w.y);
        apply(std::integral_constant<int, g + 2>{}, w.z);
        apply(std::integral_constant<int, g + 3>{}, w.w);
      });
    }
  });
}

// the roots of this thread's low-layout stage on coefficient bit h: 2^(4-h) words
template <class S, int H>
__device__ __forceinline__ void tiny_low_roots(int (&w)[1 << (4 - H)], const int* __restrict__ tw, uint32_t t) {
  constexpr int C = 1 << (4 - H);
  const int* p = tw + (1u << (S::LOGN - 1 - H)) + t * C;
  if constexpr (C == 1) {
    w[0] = __ldg(p);
  } else {
    const int2 v = __ldg(reinterpret_cast<const int2*>(p));
    w[0] = v.x;
    w[1] = v.y;
  }
}

template <class S>
__device__ __forceinline__ void tiny_fwd_low(int (&x)[32], const int* __restrict__ tw, const TinyMod& m, uint32_t t) {
  using TS = TinyShape<S>;
  if constexpr (TS::LOW_HI > kTinyLogM) {
    sfor<TS::LOW_HI - 1, kTinyLogM - 1, -1>([&](auto hc) {
      constexpr int h = decltype(hc)::value;
      int w[1 << (4 - h)];
      tiny_low_roots<S, h>(w, tw, t);
      sfor<0, (1 << (4 - h))>([&](auto gc) {
        constexpr int g = decltype(gc)::value;
        sfor<0, (1 << h)>([&](auto lc) {
          constexpr int u = (g << (h + 1)) | decltype(lc)::value;
          tiny_ct(x[u], x[u | (1 << h)], w[g], m);
        });
      });
    });
  }
}

__device__ __forceinline__ void tiny_st16(int* s, const int (&x)[32]) {
  sfor<0, 32, 4>([&](auto ec) {
    constexpr int e = decltype(ec)::value;
    *reinterpret_cast<int4*>(s + e) = make_int4(x[e], x[e + 1], x[e + 2], x[e + 3]);
  });
}
__device__ __forceinline__ void tiny_ld16(int (&x)[32], const int* s) {
  sfor<0, 32, 4>([&](auto ec) {
    constexpr int e = decltype(ec)::value;
    const int4 v = *reinterpret_cast<const int4*>(s + e);
    x[e] = v.x, x[e + 1] = v.y, x[e + 2] = v.z, x[e + 3] = v.w;
  });
}

// One operand through the forward transform; the result is in the low layout.
template <class S, class Sync>
__device__ __forceinline__ void tiny_forward(int (&x)[32], const uint32_t* in, int* s, const int* __restrict__ tw,
                                             const TinyMod& m, uint32_t t, Sync sync) {
  using TS = TinyShape<S>;
  sfor<0, 32>([&](auto ec) {
    constexpr int e = decltype(ec)::value;
    x[e] = (int)in[t + TS::T * e];
  });
  tiny_fwd_top<S>(x, tw, m);
  sync();  // every thread has its staged words
  sfor<0, 32>([&](auto ec) {
    constexpr int e = decltype(ec)::value;
    s[t + TS::top_pos(e)] = x[e];
  });
  sync();
  tiny_ld16(x, s + 36 * t);
  tiny_fwd_low<S>(x, tw, m, t);
}

// c = a b in the ring x^8 - z: a, b within (q - 1) / 2, wz the root's word
__device__ __forceinline__ void tiny_ring(int* b, const int (&a)[8], int wz, const TinyMod& m) {
  int az[8];
  sfor<1, 8>([&](auto ic) {
    constexpr int i = decltype(ic)::value;
    az[i] = tiny_mul(a[i], wz, m);
  });
  int acc[8];
  sfor<0, 8>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    acc[k] = a[0] * b[k];
    sfor<1, 8>([&](auto ic) {
      constexpr int i = decltype(ic)::value;
      acc[k] += (i <= k ? a[i] : az[i]) * b[(k - i) & 7];
    });
  });
  sfor<0, 8>([&](auto kc) {
    constexpr int k = decltype(kc)::value;
    b[k] = tiny_mul(acc[k], m.qinv, m);
  });
}

// One operand through the forward transform and back to centred residues (the
// low layout).
template <class S, class Sync>
__device__ __forceinline__ void tiny_transform(int (&x)[32], const uint32_t* in, int* s, const int* __restrict__ tw,
                                               const PrimeConst<uint32_t>& pc, uint32_t t, Sync sync) {
  const TinyMod m{(int)pc.q, (int)pc.qinv};
  tiny_forward<S>(x, in, s, tw, m, t, sync);
  sfor<0, 32>([&](auto ec) {
    constexpr int e = decltype(ec)::value;
    x[e] = tiny_mul(x[e], (int)pc.scale_p, m);
  });
}

// From b's transform in x and a's at sa (low layout): products, inverse
// through the exchange buffer sb, results to c.  `hook` as for polymul_unit.
template <class S, class Sync, class Hook>
__device__ __forceinline__ void tiny_finish(uint32_t* __restrict__ c, int (&x)[32], const int* sa, int* sb,
                                            const int* __restrict__ twf, const int* __restrict__ twi,
                                            const PrimeConst<uint32_t>& pc, uint32_t t, bool act, Sync sync,
                                            Hook&& hook) {
  using TS = TinyShape<S>;
  const TinyMod m{(int)pc.q, (int)pc.qinv};
  const int one = (int)pc.scale_p;
  // products: rings 2 i and 2 i + 1 of this thread are x^8 - z and x^8 + z
  // for the root z of the stage above
  int wz[2];
  tiny_low_roots<S, kTinyLogM>(wz, twf, t);
  sfor<0, 4>([&](auto rc) {
    constexpr int r = decltype(rc)::value;
    int a[8];
    const int4 a0 = *reinterpret_cast<const int4*>(sa + 36 * t + 8 * r);
    const int4 a1 = *reinterpret_cast<const int4*>(sa + 36 * t + 8 * r + 4);
    a[0] = a0.x, a[1] = a0.y, a[2] = a0.z, a[3] = a0.w, a[4] = a1.x, a[5] = a1.y, a[6] = a1.z, a[7] = a1.w;
    tiny_ring(x + 8 * r, a, (r & 1) ? -wz[r >> 1] : wz[r >> 1], m);
  });
  // inverse stages of the low layout
  using Low = TinyStages<1, kTinyLogM, (TS::LOW_HI > kTinyLogM ? TS::LOW_HI : kTinyLogM), false>;
  if constexpr (TS::LOW_HI > kTinyLogM) {
    sfor<kTinyLogM, TS::LOW_HI>([&](auto hc) {
      constexpr int h = decltype(hc)::value;
      int w[1 << (4 - h)];
      tiny_low_roots<S, h>(w, twi, t);
      sfor<0, (1 << (4 - h))>([&](auto gc) {
        constexpr int g = decltype(gc)::value;
        sfor<0, (1 << h)>([&](auto lc) {
          constexpr int u = (g << (h + 1)) | decltype(lc)::value;
          const int d = x[u] - x[u | (1 << h)];
          x[u] += x[u | (1 << h)];
          x[u | (1 << h)] = tiny_mul(d, w[g], m);
        });
      });
    });
  }
  tiny_st16(sb + 36 * t, x);
  sync();
  sfor<0, 32>([&](auto ec) {
    constexpr int e = decltype(ec)::value;
    x[e] = sb[t + TS::top_pos(e)];
  });
  sync();
  hook();
  using Top = TinyStages<Low::v.out, TS::TOP_LO, 5, true>;
  sfor<TS::TOP_LO, 5>([&](auto hc) {
    constexpr int hb = decltype(hc)::value;
    constexpr int first = 1 << (4 - hb);
    sfor<0, 32>([&](auto ec) {
      constexpr int e = decltype(ec)::value;
      if constexpr (Top::v.reduce[hb][e]) x[e] = tiny_mul(x[e], one, m);
    });
    auto apply = [&](auto gc, int w) {
      constexpr int g = decltype(gc)::value;
      sfor<0, (1 << hb)>([&](auto lc) {
        constexpr int u = (g << (hb + 1)) | decltype(lc)::value;
        constexpr int v = u | (1 << hb);
        const int d = x[u] - x[v];
        x[u] += x[v];
        x[v] = tiny_mul(d, w, m);
      });
    };
    if constexpr (hb == 4) {
      sfor<0, 16>([&](auto lc) {
        constexpr int u = decltype(lc)::value;
        const int s = x[u] + x[u + 16], d = x[u] - x[u + 16];
        x[u] = tiny_mul(s, (int)pc.scale, m);
        x[u + 16] = tiny_mul(d, (int)pc.scale_w, m);
      });
    } else if constexpr (first < 4) {
      sfor<0, first>([&](auto gc) { apply(gc, __ldg(twi + first + decltype(gc)::value)); });
    } else {
      sfor<0, first, 4>([&](auto gc) {
        constexpr int g = decltype(gc)::value;
        const int4 w = tiny_ld4(twi + first + g);
        apply(std::integral_constant<int, g>{}, w.x);
        apply(std::integral_constant<int, g + 1>{}, w.y);
        apply(std::integral_constant<int, g + 2>{}, w.z);
        apply(std::integral_constant<int, g + 3>{}, w.w);
      });
    }
  });
  if (act) {
    sfor<0, 32>([&](auto ec) {
      constexpr int e = decltype(ec)::value;
      // [-(q-1)/2, (q-1)/2] -> [0, q): as unsigned words the negative ones are the larger
      c[t + TS::T * e] = __viaddmin_u32((uint32_t)x[e], pc.q, (uint32_t)x[e]);
    });
  }
}

// One unit: c = a b mod (x^n +- 1, q).  Interface as polymul_unit; twf and
// twi are tables of n / 8 words (see build_tiny_tables), pc.scale_p the word
// of 1, pc.scale and pc.scale_w those of the last inverse stage.
template <class S, class Sync, class Hook>
__device__ __forceinline__ void polymul_unit_tiny(uint32_t* __restrict__ c, const int* __restrict__ twf,
                                                  const int* __restrict__ twi, const PrimeConst<uint32_t>& pc,
                                                  uint32_t* sa_, uint32_t* sb_, const uint32_t* ia, const uint32_t* ib,
                                                  uint32_t t, bool act, Sync sync, Hook&& hook) {
  int* sa = reinterpret_cast<int*>(sa_);
  int* sb = reinterpret_cast<int*>(sb_);
  int x[32];
  // a, then b, through the same instructions (a body of its own for each
  // would be fetched twice: the warps of an SM run through it at different
  // places, and instruction fetch was the first of its stalls)
#pragma unroll 1
  for (int op = 0; op < 2; ++op) {
    int* s = op ? sb : sa;
    tiny_transform<S>(x, op ? ib : ia, s, twf, pc, t, sync);
    if (op == 0) tiny_st16(s + 36 * t, x);  // a parked where this thread alone loaded it
  }
  tiny_finish<S>(c, x, sa, sb, twf, twi, pc, t, act, sync, hook);
}

}  // namespace pm
