// Device helpers shared by the kernels that keep optimiser moments in NVFP4 states (Section 3.3):
// the fixed 16-point Hadamard transform on register pairs, the two-candidate (4/6) block
// encoding with BF16 scales, hardware stochastic rounding, and 256-bit global accesses.
#pragma once

#include "fp4_common.cuh"

namespace fp4 {

__device__ __forceinline__ uint64_t splitmix64_at(uint64_t seed, uint64_t idx) {
  uint64_t z = seed + 0x9E3779B97F4A7C15ull * (idx + 1);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

// v <- v H_16 / 4 (QUARTER; else without the factor), the natural-order butterfly of hadamard16 with no signs: the stride-1 stage on
// scalars, the strides 2, 4, 8 and the factor 1/4 on packed pairs (v[2k], v[2k+1]); every lane
// is the same single rounded operation as in the scalar form.
template <bool QUARTER = true>
__device__ __forceinline__ void hadamard16_pairs(float (&v)[16]) {
  uint64_t p[8];
#pragma unroll
  for (int k = 0; k < 8; ++k) {
    const float a = v[2 * k], b = v[2 * k + 1];
    p[k] = pack2(__fadd_rn(a, b), __fsub_rn(a, b));
  }
#pragma unroll
  for (int h = 1; h < 8; h *= 2) {
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      if ((k & h) == 0) {
        const uint64_t a = p[k], b = p[k + h];
        p[k] = add2(a, b);
        p[k + h] = sub2(a, b);
      }
    }
  }
  const uint64_t q = pack2(0.25f, 0.25f);
#pragma unroll
  for (int k = 0; k < 8; ++k) unpack2(QUARTER ? mul2(p[k], q) : p[k], v[2 * k], v[2 * k + 1]);
}

// Nearest-rounding codes of one transformed block for the block scale d; returns the sum of the
// squared FP32 errors in element order.  Products are taken two at a time; every subtraction
// and every addition of the error sum stays a scalar operation, so none can fuse with a product.
__device__ __forceinline__ float mom_encode_rtn(const float (&h)[16], float d, uint32_t& lo, uint32_t& hi) {
  lo = 0; hi = 0;
  float err = 0.0f;
  if (d == 0.0f) {
#pragma unroll
    for (int i = 0; i < 16; ++i) err = __fadd_rn(err, __fmul_rn(h[i], h[i]));
    return err;
  }
  const float rcp = __frcp_rn(d);
  const uint64_t rcp2 = pack2(rcp, rcp), d2 = pack2(d, d);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    float y0, y1, p0, p1, s0, s1;
    unpack2(mul2(pack2(h[2 * i], h[2 * i + 1]), rcp2), y0, y1);
    const uint32_t byte = cvt_e2m1x2(y0, y1);
    const float2 q = e2m1x2_to_float2(byte);
    unpack2(mul2(pack2(q.x, q.y), d2), p0, p1);
    const float d0 = __fsub_rn(h[2 * i], p0), d1 = __fsub_rn(h[2 * i + 1], p1);
    const uint64_t dd = pack2(d0, d1);
    unpack2(mul2(dd, dd), s0, s1);
    err = __fadd_rn(err, s0);
    err = __fadd_rn(err, s1);
    if (i < 4) lo |= byte << (8 * i); else hi |= byte << (8 * (i - 4));
  }
  return err;
}

// Stochastic rounding of four values onto the E2M1 grid with the conversion instruction of
// sm_100a; the result holds v0 in bits 3:0 ... v3 in bits 15:12.  Measured behaviour of the
// instruction: with lo <= |v| < hi the neighbouring grid values and f = floor(65536 (|v| - lo) /
// (hi - lo)), v goes to hi when f + r >= 65536, where the 16 random bits r of the four values
// come from the bytes b3 b2 b1 b0 of the random word as
//   v0: b2 b0     v1: the same 16 bits in reverse order     v2: b3 b1     v3: those reversed.
// `w` is the word in the plain form (v0: low half, v2: high half), permuted here.
__device__ __forceinline__ uint32_t cvt_rs_e2m1x4(float v0, float v1, float v2, float v3, uint32_t w) {
  const uint32_t rbits = __byte_perm(w, 0u, 0x3120);  // b0, b2 <- low half; b1, b3 <- high half
  uint32_t r;
  asm("{\n\t.reg .b16 t;\n\tcvt.rs.satfinite.e2m1x4.f32 t, {%1, %2, %3, %4}, %5;\n\tcvt.u32.u16 %0, t;\n\t}"
      : "=r"(r)
      : "f"(v3), "f"(v2), "f"(v1), "f"(v0), "r"(rbits));
  return r;
}

__device__ __forceinline__ uint32_t hadd2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("add.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
__device__ __forceinline__ uint32_t hsub2(uint32_t a, uint32_t b) {
  uint32_t r;
  asm("sub.rn.f16x2 %0, %1, %2;" : "=r"(r) : "r"(a), "r"(b));
  return r;
}
// v = scale * (codes H_16 / 4).  The butterfly of the codes alone stays on multiples of 1/2 up to 96, exact in FP16, so it
// runs on half-precision pairs and the block scale is one product at the end: sum * d has at most 8 + 8 significant
// bits, as has every partial sum of the products code * d, so both are exact and equal.  Scales outside
// [2^-100, 2^100] (zero, negative, gradual underflow, overflow) take the butterfly of the FP32 products.
// HALF off takes the FP32 butterfly always.  AdamW of 2^26 parameters: 175 us against 181 without; momentum with the histogram
// of 8192 x 4096, where the counters and not the arithmetic bind: 58 us with, 56 without.
// ADD: plus `add`, a fused operation with that product, and so rounded once like the sum (`one`: 1, unknown to the compiler, which
// could fuse a plain sum with a product before it).
template <bool HALF, bool ADD = false>
__device__ __forceinline__ void mom_decode(uint2 c, uint32_t scale_bits, float (&v)[16], float add = 0.0f, float one = 1.0f) {
  const float d = __uint_as_float(scale_bits << 16);
  if (HALF && d >= 0x1p-100f && d <= 0x1p100f) {
    uint32_t p[8];
#pragma unroll
    for (int w = 0; w < 2; ++w) {
      asm("{\n\t.reg .b8 t0, t1, t2, t3;\n\t"
          "mov.b32 {t0, t1, t2, t3}, %4;\n\t"
          "cvt.rn.f16x2.e2m1x2 %0, t0;\n\t"
          "cvt.rn.f16x2.e2m1x2 %1, t1;\n\t"
          "cvt.rn.f16x2.e2m1x2 %2, t2;\n\t"
          "cvt.rn.f16x2.e2m1x2 %3, t3;\n\t}"
          : "=r"(p[4 * w]), "=r"(p[4 * w + 1]), "=r"(p[4 * w + 2]), "=r"(p[4 * w + 3])
          : "r"(w ? c.y : c.x));
    }
#pragma unroll
    for (int k = 0; k < 8; ++k)  // (a, b) -> (a + b, a - b) within a pair
      asm("{\n\t.reg .b16 a, b;\n\t.reg .b32 aa, bb;\n\t"
          "mov.b32 {a, b}, %0;\n\t"
          "mov.b32 aa, {a, a};\n\t"
          "mov.b32 bb, {b, b};\n\t"
          "fma.rn.f16x2 %0, bb, %1, aa;\n\t}"
          : "+r"(p[k]) : "r"(0xBC003C00u));
#pragma unroll
    for (int h = 1; h < 8; h *= 2) {
#pragma unroll
      for (int k = 0; k < 8; ++k) {
        if ((k & h) == 0) {
          const uint32_t a = p[k], b = p[k + h];
          p[k] = hadd2(a, b);
          p[k + h] = hsub2(a, b);
        }
      }
    }
    const float dq = __fmul_rn(d, 0.25f);
    const uint64_t d2 = pack2(dq, dq), add2s = pack2(add, add);
#pragma unroll
    for (int k = 0; k < 8; ++k) {
      float a, b;
      half2_to_float2(p[k], a, b);
      unpack2(ADD ? fma2(pack2(a, b), d2, add2s) : mul2(pack2(a, b), d2), v[2 * k], v[2 * k + 1]);
    }
    return;
  }
  const uint64_t d2 = pack2(d, d);
#pragma unroll
  for (int i = 0; i < 8; ++i) {
    const uint32_t byte = ((i < 4 ? c.x : c.y) >> (8 * (i & 3))) & 0xFFu;
    const float2 q = e2m1x2_to_float2(byte);
    unpack2(mul2(pack2(q.x, q.y), d2), v[2 * i], v[2 * i + 1]);
  }
  hadamard16_pairs(v);
  if (ADD) {
#pragma unroll
    for (int i = 0; i < 16; ++i) v[i] = __fmaf_rn(v[i], one, add);
  }
}

// Nearest-rounding codes of one transformed block for a BF16 block scale d in the normal range, with rcp = RN(1 / d);
// returns the sum of the squared FP32 errors in element order.  code * d has at most 2 + 8 significant bits, so one
// fused operation gives the rounded difference that a product and a subtraction would.
__device__ __forceinline__ float mom_encode_fast(const float (&h)[16], float d, float rcp, uint32_t& lo, uint32_t& hi) {
  const uint64_t rcp2 = pack2(rcp, rcp), nd2 = pack2(-d, -d);
  float err = 0.0f;
#pragma unroll
  for (int b = 0; b < 2; ++b) {
    float y[8];
    uint32_t codes, q[4];
#pragma unroll
    for (int i = 0; i < 4; ++i) unpack2(mul2(pack2(h[8 * b + 2 * i], h[8 * b + 2 * i + 1]), rcp2), y[2 * i], y[2 * i + 1]);
    cvt_e2m1x8_f16(y, codes, q);
#pragma unroll
    for (int i = 0; i < 4; ++i) {
      float q0, q1, s0, s1;
      half2_to_float2(q[i], q0, q1);
      const uint64_t dd = fma2(pack2(q0, q1), nd2, pack2(h[8 * b + 2 * i], h[8 * b + 2 * i + 1]));
      unpack2(mul2(dd, dd), s0, s1);
      err = __fadd_rn(err, s0);
      err = __fadd_rn(err, s1);
    }
    if (b == 0) lo = codes; else hi = codes;
  }
  return err;
}

// RN(1 / d) of a BF16 value in [2^-110, 2^110]: one Newton step on the approximation leaves a relative error near
// 2^-46, and the reciprocals of 8-bit significands lie at least 2^-33 from the midpoint of two floats.
__device__ __forceinline__ float rcp_bf16(float d) {
  float r;
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(r) : "f"(d));
  return __fmaf_rn(r, __fmaf_rn(-d, r, 1.0f), r);
}

// Two-candidate encoding of a transformed block with the errors of the definition: fused operations on pairs in a normal
// range, else its plain operations.
static __device__ __noinline__ uint3 encode_pair_exact(float h0, float h1, float h2, float h3, float h4, float h5, float h6,
                                                       float h7, float h8, float h9, float h10, float h11, float h12,
                                                       float h13, float h14, float h15, float amax) {
  const float h[16] = {h0, h1, h2, h3, h4, h5, h6, h7, h8, h9, h10, h11, h12, h13, h14, h15};
  uint32_t w, lo, hi, lo4, hi4;
  float err6, err4;
  if (amax >= 0x1p-100f && amax <= 0x1p100f) {
    w = cvt_bf16x2(sixth_of(amax), __fmul_rn(amax, 0.25f));
    err6 = mom_encode_fast(h, bf16_lo(w), rcp_bf16(bf16_lo(w)), lo, hi);
    err4 = mom_encode_fast(h, bf16_hi(w), rcp_bf16(bf16_hi(w)), lo4, hi4);
  } else {
    w = cvt_bf16x2(__fdiv_rn(amax, 6.0f), __fdiv_rn(amax, 4.0f));
    err6 = mom_encode_rtn(h, bf16_lo(w), lo, hi);
    err4 = mom_encode_rtn(h, bf16_hi(w), lo4, hi4);
  }
  uint32_t scale_bits = w & 0xFFFFu;
  if (err4 < err6) { scale_bits = w >> 16; lo = lo4; hi = hi4; }
  return make_uint3(lo, hi, scale_bits);
}

// Does every element have the same error with both scales, so that the definition's sums are equal?  What makes blocks tie:
// equal values (d4 = 1.5 d6, see codes_match), or a single magnitude amax beside zeros, midway between 6 d6 and 4 d4.
__device__ __forceinline__ bool same_errors(const float (&h4)[16], float amax4, float d6, float d4, uint32_t lo, uint32_t hi, uint32_t lo4,
                                            uint32_t hi4) {
  if (d4 == 1.5f * d6) return codes_match(lo, lo4) && codes_match(hi, hi4);
  bool one = __fmaf_rn(6.0f, d6, 4.0f * d4) == 0.5f * amax4;   // exact: sums of 10-bit numbers
#pragma unroll
  for (int i = 0; i < 16; ++i) one = one && (h4[i] == 0.0f || fabsf(h4[i]) == amax4);
  return one;
}

// Encodes a transformed block h = h4 / 4 (the quarter is taken by the reciprocals: a power of two changes no rounding in the
// normal range): candidate scales BF16(amax / 6) and BF16(amax / 4), nearest rounding with each, the
// smaller squared error (a tie keeps 6); SR: once more by stochastic rounding with the chosen scale, `first` =
// the matrix index of the block's first element.  The kernels that call this are bound by the instructions they issue, so the
// candidates are compared by the errors s6 and s4 of the scaled values, in units of the first scale d.  A scaled value is
// at most 6.05 and off by 2^-23 of itself, which moves a sum S of sixteen squares by less than 2 sqrt(S) 4 2^-20.4 + 2^-36;
// rounding the sums moves either form by less than 2^-19 of it, and the definition's loses another 32 2^-150 / d^2 < 2^-29
// to underflow while amax >= 2^-55.  With S the larger sum the order is certain when the difference exceeds
// sqrt(S) 2^-16.4 + S 2^-17 + 2^-28.9, whose square is below S (2^-32 + S 2^-32) + 2^-53.  Closer ones, 10^-4 of the blocks,
// and blocks out of range take the errors of the definition; blocks of few different magnitudes, of which a third can
// tie exactly because both scales give the same values, keep 6 at once; a block of zeros is all zeros.
// AdamW of 2^26 parameters, errors of the definition for all blocks / as here: 174.3 / 161.9 us; the same gradient every step with one
// non-zero per block 180 / 180 (without the look at ties 202, with a margin of 2^-14 of max(S, 1/16) 227), constant
// blocks 174 / 169 (195, 219), new constants every step 174 / 177 (184, 219); blocks out of range 252 / 246.
template <bool SR>
__device__ __forceinline__ void state_encode(const float (&h4)[16], uint64_t seed, uint64_t first, uint2& c, uint32_t& scale_bits) {
  const float amax4 = amax16(h4), amax = __fmul_rn(amax4, 0.25f);
  uint32_t lo = 0, hi = 0;
  float rcp = 0.0f;
  scale_bits = 0;
  bool certain = amax == 0.0f;
  if (amax >= 0x1p-55f && amax <= 0x1p55f) {
    const uint32_t w = cvt_bf16x2(sixth_of(amax), __fmul_rn(amax, 0.25f));
    const float d6 = bf16_lo(w), d4 = bf16_hi(w);
    const float r6 = rcp_bf16(d6), r4 = rcp_bf16(d4);
    uint32_t lo4, hi4;
    const float s6 = encode_block16_scaled(h4, 0.25f * r6, lo, hi);
    const float ratio = d4 * r6;
    const float s4 = encode_block16_scaled(h4, 0.25f * r4, lo4, hi4) * (ratio * ratio);
    const float diff = s4 - s6, S = fmaxf(s4, s6);
    certain = diff * diff > fmaf(S, fmaf(S, 0x1p-32f, 0x1p-32f), 0x1p-53f);
    bool four = diff < 0.0f;
    if (!certain && same_errors(h4, amax4, d6, d4, lo, hi, lo4, hi4)) {
      certain = true;
      four = false;
    }
    rcp = r6;
    scale_bits = w & 0xFFFFu;
    if (four) { rcp = r4; scale_bits = w >> 16; lo = lo4; hi = hi4; }
  }
  // one generator output per 8 elements of the matrix: its low word for the first four
  auto stochastic = [&](auto&& y) {
    const uint64_t z0 = splitmix64_at(seed, first >> 3), z1 = splitmix64_at(seed, (first >> 3) + 1);
    const uint32_t c0 = cvt_rs_e2m1x4(y(0), y(1), y(2), y(3), (uint32_t)z0), c1 = cvt_rs_e2m1x4(y(4), y(5), y(6), y(7), (uint32_t)(z0 >> 32));
    const uint32_t c2 = cvt_rs_e2m1x4(y(8), y(9), y(10), y(11), (uint32_t)z1);
    const uint32_t c3 = cvt_rs_e2m1x4(y(12), y(13), y(14), y(15), (uint32_t)(z1 >> 32));
    lo = c0 | (c1 << 16);
    hi = c2 | (c3 << 16);
  };
  if (certain) {
    if (SR && scale_bits != 0) {
      const float r = 0.25f * rcp;
      stochastic([&](int i) { return __fmul_rn(h4[i], r); });
    }
  } else {
    float h[16];
#pragma unroll
    for (int i = 0; i < 16; ++i) h[i] = __fmul_rn(h4[i], 0.25f);
    const uint3 e = encode_pair_exact(h[0], h[1], h[2], h[3], h[4], h[5], h[6], h[7], h[8], h[9], h[10], h[11], h[12], h[13],
                                      h[14], h[15], amax);
    lo = e.x; hi = e.y; scale_bits = e.z;
    const float d = __uint_as_float(scale_bits << 16);
    if (SR && d != 0.0f) {
      rcp = __frcp_rn(d);
      stochastic([&](int i) { return __fmul_rn(h[i], rcp); });
    }
  }
  c = make_uint2(lo, hi);
}

// Square root and quotient of register pairs for values in the normal range: an approximation, one Newton step and one residual (P.
// Markstein, IBM J. Res. Dev. 34, 1990).  They round correctly while no intermediate leaves that range: the square root
// agrees with __fsqrt_rn for every float in [2^-80, 2^30], the reciprocal with __frcp_rn for every float in [2^-41, 2^36];
// before its last rounding the quotient is off by less than 3 2^-25 units in the last place, and every pair of significands
// whose quotient lies that close to a midpoint of two floats agrees with __fdiv_rn (fp4_selftest_rounding repeats all three).
__device__ __forceinline__ uint64_t rsqrt_neg2(uint64_t v) {
  float a, b;
  unpack2(v, a, b);
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(-a));
  asm("rsqrt.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"(-b));
  return pack2(a, b);
}
__device__ __forceinline__ uint64_t rcp_neg2(uint64_t v) {
  float a, b;
  unpack2(v, a, b);
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(a) : "f"(-a));
  asm("rcp.approx.ftz.f32 %0, %1;" : "=f"(b) : "f"(-b));
  return pack2(a, b);
}

// -RN(sqrt(v)) from nv = -v.  ZEROS: nv may be -0 (any in-range reciprocal root will do; the result is a zero).
template <bool ZEROS>
__device__ __forceinline__ uint64_t neg_sqrt2(uint64_t nv) {
  uint64_t at = nv;
  if (ZEROS) {
    float a, b;
    unpack2(nv, a, b);
    at = pack2(fminf(a, -0x1p-80f), fminf(b, -0x1p-80f));
  }
  const uint64_t r = rsqrt_neg2(at);
  const uint64_t nt = mul2(nv, r);
  return fma2(fma2(nt, nt, nv), mul2(r, pack2(0.5f, 0.5f)), nt);
}
// -RN(m / den)
__device__ __forceinline__ uint64_t neg_quotient2(uint64_t m, uint64_t den) {
  const uint64_t ny = rcp_neg2(den);
  const uint64_t ny1 = fma2(fma2(den, ny, pack2(1.0f, 1.0f)), ny, ny);
  const uint64_t nq = mul2(m, ny1);
  return fma2(fma2(den, nq, m), ny1, nq);
}
// 256-bit global accesses (32-byte aligned): a thread moves its block of 16 floats as two full
// 32-byte sectors, so no sector is touched by two instructions -- with 128-bit pieces at a
// 64-byte lane stride every sector is looked up twice on loads and written as two partial
// sectors on stores.
__device__ __forceinline__ void ld_f32x8(const float* p, float* v) {
  asm volatile("ld.global.v8.f32 {%0,%1,%2,%3,%4,%5,%6,%7}, [%8];"
               : "=f"(v[0]), "=f"(v[1]), "=f"(v[2]), "=f"(v[3]), "=f"(v[4]), "=f"(v[5]), "=f"(v[6]), "=f"(v[7])
               : "l"(p));
}
__device__ __forceinline__ void stg_f32x8(float* p, const float* v) {
  asm volatile("st.global.v8.f32 [%0], {%1,%2,%3,%4,%5,%6,%7,%8};" ::"l"(p), "f"(v[0]), "f"(v[1]), "f"(v[2]),
               "f"(v[3]), "f"(v[4]), "f"(v[5]), "f"(v[6]), "f"(v[7])
               : "memory");
}


}  // namespace fp4
