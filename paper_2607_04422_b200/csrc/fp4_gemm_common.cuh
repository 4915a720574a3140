// Device helpers shared by the kernels that run the products.
#pragma once

#include "fp4_kernels.h"

namespace fp4 {

__device__ __forceinline__ uint64_t globaltimer_ns() {
  uint64_t t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}

constexpr uint64_t kWaitLimitNs = 2000000000ull;  // two seconds

// Bounded wait on an mbarrier phase.  When a wait gives up (its own
// time-out, or another thread of the CTA gave up before) the abort flag is set and every later
// wait of the CTA falls through at once, so the kernel runs to its end on whatever data it has
// and the host reads FP4_ERR_DEVICE_TIMEOUT from the status word.  The polls carry a suspend-time
// hint: the thread sleeps in hardware until the phase completes instead of spinning.
__device__ __forceinline__ bool mbar_try_wait_hint(uint32_t bar_addr, uint32_t parity, uint32_t hint_ns) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2, %3;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar_addr), "r"(parity), "r"(hint_ns)
      : "memory");
  return ok != 0;
}
static __device__ __noinline__ void wait_limited_abort(uint32_t bar_addr, uint32_t parity, volatile uint32_t* abort_flag,
                                                       uint64_t limit_ns) {
  const uint64_t t0 = globaltimer_ns();
  for (;;) {
    if (*abort_flag) return;
    for (int i = 0; i < 64; ++i)
      if (mbar_try_wait_hint(bar_addr, parity, 4000u)) return;
    if (globaltimer_ns() - t0 > limit_ns) {
      *abort_flag = 1;
      return;
    }
  }
}
__device__ __forceinline__ void wait_or_abort(uint32_t bar_addr, uint32_t parity, volatile uint32_t* abort_flag) {
  uint32_t ok;
  asm volatile(
      "{\n\t.reg .pred p;\n\tmbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n\t"
      "selp.u32 %0, 1, 0, p;\n\t}"
      : "=r"(ok)
      : "r"(bar_addr), "r"(parity)
      : "memory");
  if (!ok) wait_limited_abort(bar_addr, parity, abort_flag, kWaitLimitNs);
}
__device__ __forceinline__ void wait_or_abort(uint64_t* bar, uint32_t parity, volatile uint32_t* abort_flag) {
  wait_or_abort(smem_u32(bar), parity, abort_flag);
}

// Barrier over all blocks of a cooperative launch: this block increments `counter` (zero before the launch) and waits until
// it is at least `want`, the number of blocks times that of the barrier.  Bounded like the other waits.
__device__ __forceinline__ void grid_barrier(uint32_t* counter, uint32_t want, volatile uint32_t* abort_flag,
                                             uint64_t limit_ns = kWaitLimitNs) {
  __syncthreads();
  if (threadIdx.x == 0) {
    asm volatile("red.release.gpu.global.add.u32 [%0], 1;" ::"l"(counter) : "memory");
    const uint64_t t0 = globaltimer_ns();
    for (;;) {
      uint32_t v;
      asm volatile("ld.acquire.gpu.global.u32 %0, [%1];" : "=r"(v) : "l"(counter) : "memory");
      if (v >= want) break;
      if (*abort_flag || globaltimer_ns() - t0 > limit_ns) { *abort_flag = 1; break; }
    }
  }
  __syncthreads();
}

// tile index of a launch -> (problem, tile row, tile column): bands of `band` tile rows, each walked column by column
// (only the tiles on and above the diagonal of a symmetric product); a band of one row is plain row order.  p comes in as a
// problem at or before the tile's (a thread's tiles are in ascending order).
__device__ __forceinline__ void decode_tile(int t, const GemmProblem* probs, int num_problems, int& p, int& ti, int& tj, bool sym) {
  while (p + 1 < num_problems && t >= probs[p + 1].first_tile) ++p;
  t -= probs[p].first_tile;
  const int tiles_n = (probs[p].blocks_n + 1) >> 1, band = probs[p].band;
  if (!sym) {
    const int b = t / (band * tiles_n);
    t -= b * band * tiles_n;
    const int h = min(band, ((probs[p].blocks_m + 1) >> 1) - b * band);   // the last band may be lower
    tj = t / h;
    ti = b * band + (t - tj * h);
  } else {
    int row = 0, h = min(band, tiles_n);
    for (;;) {
      // h rows from `row` on: a triangle of h columns, then whole columns
      const int in_band = h * (h + 1) / 2 + (tiles_n - row - h) * h;
      if (t < in_band) break;
      t -= in_band;
      row += h;
      h = min(band, tiles_n - row);
    }
    int col = 0;
    while (col < h && t > col) { t -= col + 1; ++col; }
    if (col == h) {
      const int c = t / h;
      col += c;
      t -= c * h;
    }
    ti = row + t;
    tj = row + col;
  }
}

// Per-call scalars of an epilogue: the factor that turns the accumulator into the
// product (tensor scales of the two operands) and the tensor scale of the quantised
// output, predicted from the running maxima (power of two); the bound is widened by
// args.q.widen when the output is rotated before quantisation (|x H| <= 4 amax(x)).
template <int MODE>
__device__ __forceinline__ void epilogue_scalars(const GemmProblem& pr, const GemmLaunch& args, float& scale,
                                                 float& sg_out, bool publish) {
  float* sc = pr.scalars;
  sg_out = 1.0f;
  if (MODE == kPlain) {
    scale = __fmul_rn(pr.sg_a, pr.sg_b);
  } else if (MODE == kG1) {
    const float sgx = sc[args.ix.sg_X0 + args.iter];
    const float ax = sc[args.ix.amax_X0 + args.iter];
    scale = __fmul_rn(sgx, sgx);
    float bound = __fmul_rn(__fmul_rn(__fmul_rn(2.0f, pr.l_cols), ax), ax);
    sg_out = scale_predicted(__fmul_rn(args.q.widen, fminf(bound, 4.0f)));
    if (publish) sc[args.ix.sg_A0 + args.iter] = sg_out;
  } else if (MODE == kG2) {
    const float sga = sc[args.ix.sg_A0 + args.iter];
    const float aa = sc[args.ix.amax_A0 + args.iter];
    scale = __fmul_rn(sga, sga);
    float bound = __fmul_rn(__fadd_rn(fabsf(pr.cb), __fmul_rn(4.0f, fabsf(pr.cc))), aa);
    sg_out = scale_predicted(__fmul_rn(args.q.widen, bound));
    if (publish) sc[args.ix.sg_B0 + args.iter] = sg_out;
  } else {
    const float sgb = sc[args.ix.sg_B0 + args.iter];
    const float sgx = sc[args.ix.sg_X0 + args.iter];
    const float ax = sc[args.ix.amax_X0 + args.iter];
    scale = __fmul_rn(sgb, sgx);
    float bound = __fmul_rn(__fmul_rn(4.0f, fabsf(pr.ca)), ax);
    sg_out = scale_predicted(__fmul_rn(args.q.widen, bound));
    if (publish) sc[args.ix.sg_X0 + args.iter + 1] = sg_out;
  }
}

}  // namespace fp4
