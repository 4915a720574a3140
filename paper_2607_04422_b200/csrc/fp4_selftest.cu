// fp4_selftest_rounding: the square roots, reciprocals and quotients that the kernels write out without the range tests of the
// general operations, against those operations - for every argument where that can be done, else for every argument that
// could round differently.
#include "fp4_kernels.h"
#include "fp4_state.cuh"

namespace fp4 {
namespace {

__device__ __forceinline__ void tally(uint32_t* count, uint32_t bad) {
  bad = __reduce_add_sync(0xffffffffu, bad);
  if ((threadIdx.x & 31) == 0 && bad) atomicAdd(count, bad);
}
__device__ __forceinline__ uint32_t differ(float a, float b) { return __float_as_uint(a) != __float_as_uint(b); }

// All floats of [2^lo, 2^hi), one per thread and step; whole warps.
template <typename F>
__device__ __forceinline__ uint32_t every_float(int lo, int hi, F&& f) {
  uint32_t bad = 0;
  const uint32_t first = (uint32_t)(lo + 127) << 23, last = (uint32_t)(hi + 127) << 23;
  for (uint32_t u = first + blockIdx.x * blockDim.x + threadIdx.x; u < last; u += gridDim.x * blockDim.x) bad += f(__uint_as_float(u));
  return bad;
}

__global__ void __launch_bounds__(256) k_selftest_unary(uint32_t* counts) {
  tally(counts + 0, every_float(-80, 30, [](float x) {
    float a, b;
    unpack2(neg_sqrt2<false>(pack2(-x, -x)), a, b);
    float c, d;
    unpack2(neg_sqrt2<true>(pack2(-x, -0.0f)), c, d);
    const float want = -__fsqrt_rn(x);
    return differ(a, want) + differ(b, want) + differ(c, want) + (d != 0.0f ? 1u : 0u);
  }));
  tally(counts + 1, every_float(-41, 36, [](float x) {
    const uint64_t den = pack2(x, x), ny = rcp_neg2(den);
    float a, b;
    unpack2(fma2(fma2(den, ny, pack2(1.0f, 1.0f)), ny, ny), a, b);
    const float want = -__frcp_rn(x);
    return differ(a, want) + differ(b, want);
  }));
  tally(counts + 2, every_float(-80, 80, [](float x) { return differ(rcp_newton(x), __frcp_rn(x)); }));
  tally(counts + 3, every_float(-100, 100, [](float x) { return differ(sixth_of(x), __fdiv_rn(x, 6.0f)); }));
  uint32_t bad = 0;
  for (uint32_t u = blockIdx.x * blockDim.x + threadIdx.x; u < 1u << 16; u += gridDim.x * blockDim.x) {
    const float d = __uint_as_float(u << 16);
    if (d >= 0x1p-110f && d <= 0x1p110f) bad += differ(rcp_bf16(d), __frcp_rn(d));
    if (u >= 1 && u <= 126) {   // every E4M3 scale
      uint16_t neg_s;
      float rcp;
      const float s = ue4m3_to_float(u);
      bad += (ue4m3_scale(s, neg_s, rcp) != u) + differ(rcp, __frcp_rn(s));
    }
  }
  tally(counts + 4, bad);
}

// Quotients a / b of 24-bit integers (significands) that lie within 3 b 2^-24 < 3 units of 2^-e / b of the midpoint M 2^-e of
// two floats, M odd in [2^24, 2^25): a 2^e - M b = r, |r| = 1 or 2; e = 24 for a >= b, 25 for a < b.  M is odd, so b has the
// factor 2 exactly as often as r, and M = -r / b modulo what remains of 2^e.
__global__ void __launch_bounds__(256) k_selftest_quotient(uint32_t* counts) {
  uint32_t bad = 0, bad_general = 0, seen = 0;
  for (uint32_t b = (1u << 23) + blockIdx.x * blockDim.x + threadIdx.x; b < 1u << 24; b += gridDim.x * blockDim.x) {
    const int j = (b & 1) ? 0 : (b & 2) ? 1 : -1;
    if (j < 0) continue;
    const uint32_t odd = b >> j;
    uint32_t inv = odd;   // modulo 2^3, then 6, 12, 24, 48 bits
    for (int i = 0; i < 4; ++i) inv *= 2 - odd * inv;
    for (int sign = -1; sign <= 1; sign += 2) {
      const int64_t r = sign * (1 << j);
      for (int e = 24; e <= 25; ++e) {
        const uint32_t mod = 1u << (e - j), m0 = ((uint32_t)(-sign) * inv) & (mod - 1);
        for (uint64_t M = m0; M < 1u << 25; M += mod) {
          if (M < 1u << 24) continue;
          const int64_t n = (int64_t)(M * b) + r;
          const uint32_t a = (uint32_t)(n >> e);
          if (a < 1u << 23 || a >= 1u << 24 || (a >= b) != (e == 24)) continue;
          ++seen;
          const float fa = (float)a, fb = (float)b, want = __fdiv_rn(fa, fb);
          float x, y;
          unpack2(neg_quotient2(pack2(fa, -fa), pack2(fb, fb)), x, y);
          bad += differ(x, -want) + differ(y, want) + (((int64_t)a << e) != n ? 1u : 0u);
          bad_general += differ(quotient(fa, fb, __frcp_rn(fb)), want);
        }
      }
    }
  }
  tally(counts + 5, bad);
  tally(counts + 6, bad_general);
  tally(counts + 7, seen);
}

}  // namespace

cudaError_t launch_selftest_rounding(uint32_t* counts, int sms, cudaStream_t st) {
  cudaError_t e = cudaMemsetAsync(counts, 0, 8 * sizeof(uint32_t), st);
  if (e != cudaSuccess) return e;
  count_launches(2);
  k_selftest_unary<<<8 * sms, 256, 0, st>>>(counts);
  k_selftest_quotient<<<8 * sms, 256, 0, st>>>(counts);
  return cudaGetLastError();
}

}  // namespace fp4
