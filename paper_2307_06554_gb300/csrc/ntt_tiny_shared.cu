// Shared-operand products c_i = a b_i for the smallest moduli (q < 18500,
// n = 2^10), one launch: the unit of ntt_tiny.cuh with a's transform done
// once per CTA and prime.
//
// The general form (ntt_shared.cu) transforms a in a launch of its own and
// every product waits for it.  Here each CTA serves one prime at a time: its
// first warp transforms a into shared memory while the others already load
// and transform their first products, and one barrier later all multiply by
// it.  That repeats a's transform in every CTA (304 of them against 4096
// products: 4 % of the forward work) and saves a launch, its scratch and the
// trip of a^ through memory.  A warp owns two row buffers: the next product's
// row arrives in one while the other serves this one's exchanges.
// n = 1024, q = 12289, 4096 products: 15.0 us, 25.4 in two launches of the
// general form; bound by issue slots and instruction fetch like the batch
// kernel, with a fill and a drain per call.
#include <cuda_runtime.h>

#include "kernels.h"
#include "ntt.cuh"
#include "polymul_types.h"

namespace pm {

constexpr int kTinySharedWarps = 8;

// barrier between a's transform and its use, reached by every warp of the CTA
// once per prime, from either of two places
__device__ __forceinline__ void ahat_barrier() { asm volatile("bar.sync 1, %0;" ::"n"(32 * kTinySharedWarps) : "memory"); }

template <class S>
__global__ void __launch_bounds__(32 * kTinySharedWarps, 2) k_ntt_tiny_shared(TinySharedArgs args) {
  static_assert(S::T == 32, "one warp per product");
  extern __shared__ __align__(16) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t mbar[kTinySharedWarps][2];
  constexpr uint32_t ROW = S::N * 4u;
  const uint32_t warp = threadIdx.x >> 5, t = threadIdx.x & 31;
  uint32_t* ahat = reinterpret_cast<uint32_t*>(smem_raw);
  uint32_t* buf = ahat + S::SLICE + (size_t)warp * 2 * S::SLICE;
  uint64_t* bar = mbar[warp];
  if (t == 0) {
    mbar_init(bar, 1);
    mbar_init(bar + 1, 1);
  }
  fence_mbar_init();
  __syncwarp();
  griddep_wait();               // everything before this launch is complete
  griddep_launch_dependents();  // only now: when the next one starts, so is everything before this one
  uint32_t parity = 0;  // bit i: phase of buffer i's barrier
  uint32_t cur_buf = 0;
  bool failed = false;
  const uint64_t step = (uint64_t)args.ctas_per_prime * kTinySharedWarps;
  for (uint64_t v = blockIdx.x; v < (uint64_t)args.k * args.ctas_per_prime; v += gridDim.x) {
    const uint32_t j = (uint32_t)(v / args.ctas_per_prime);
    const PrimeConst<uint32_t> pc = args.pc[j];
    const int* twf = args.tw_fwd + (size_t)j * (S::N / 8);
    const int* twi = args.tw_inv + (size_t)j * (S::N / 8);
    auto row = [&](uint64_t p) { return ((size_t)p * args.k + j) * S::N; };
    auto issue = [&](uint64_t p, uint32_t b) {  // lane 0 only
      fence_proxy_async();
      mbar_arrive_expect_tx(bar + b, ROW);
      bulk_g2s(buf + b * S::SLICE, args.b + row(p), ROW, bar + b);
    };
    uint64_t p = (v % args.ctas_per_prime) * kTinySharedWarps + warp;
    if (failed) p = args.batch;  // keeps its place at the barriers
    if (t == 0 && p < args.batch) issue(p, cur_buf);
    __syncthreads();  // every warp has finished with the previous prime's a^
    int x[32];
    if (warp == 0) {
      // this warp's other buffer serves the exchange: nothing is in flight into it
      tiny_transform<S>(x, args.a + (size_t)j * S::N, reinterpret_cast<int*>(buf + (cur_buf ^ 1u) * S::SLICE), twf, pc, t,
                        WarpSync{});
      tiny_st16(reinterpret_cast<int*>(ahat) + 36 * t, x);
      __syncwarp();
    }
    bool first = true;
    while (p < args.batch) {
      const bool ok = mbar_wait(bar + cur_buf, (parity >> cur_buf) & 1u);
      if (__any_sync(0xffffffffu, !ok)) {
        if (t == 0) atomicExch_system(args.err, 1);
        mbar_wait(bar + cur_buf, (parity >> cur_buf) & 1u);  // let the copy in flight land
        failed = true;
        break;
      }
      parity ^= 1u << cur_buf;
      const uint64_t nxt = p + step;
      if (t == 0 && nxt < args.batch) issue(nxt, cur_buf ^ 1u);
      int* s = reinterpret_cast<int*>(buf + cur_buf * S::SLICE);
      tiny_transform<S>(x, reinterpret_cast<const uint32_t*>(s), s, twf, pc, t, WarpSync{});
      if (first) ahat_barrier();
      first = false;
      tiny_finish<S>(args.c + row(p), x, reinterpret_cast<const int*>(ahat), s, twf, twi, pc, t, true, WarpSync{},
                     [] {});
      cur_buf ^= 1u;
      p = nxt;
    }
    if (first) ahat_barrier();
  }
}

bool lookup_ntt_tiny_shared(int logn, KernelInfo* ki) {
  if (logn != 10) return false;
  using S = Shape<uint32_t, 10, 5, 3>;
  ki->fn = (const void*)k_ntt_tiny_shared<S>;
  ki->block = 32 * kTinySharedWarps;
  ki->smem = (1 + 2 * kTinySharedWarps) * S::SLICE * 4;
  ki->team = S::T;
  ki->units_per_cta = kTinySharedWarps;
  ki->rb = 5;
  ki->tiny = 1;
  return true;
}

}  // namespace pm
