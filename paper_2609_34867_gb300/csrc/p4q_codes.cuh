// Codes of a row's values from its scale (the rounding that the quantizers
// share): eight at a time, without a division per value.
#pragma once

#include <cstdint>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace p4q {

// Codes of eight values of a row (one 16-byte chunk of fp16 values).
//
// code = round_half_even(fl(x / s)). With inv = fl(1 / s) correctly rounded,
// fl(x / s) lies within 2^-23 (relative) of x * inv, so ip = fl(inv (1 +
// 2^-21)) and im = fl(inv (1 - 2^-21)) give products x * ip and x * im that
// enclose fl(x / s) (each is at least 2^-21 - 2^-23 away from x * inv). One
// fused multiply-add with the magic constant 1.5 * 2^23 rounds each exact
// product to the nearest integer (ties to even: the constant is even) and
// leaves its two's complement in the low mantissa bits. Rounding is
// monotone, so where the two agree their integer is the code of fl(x / s);
// a chunk where they differ for some value (a quotient within about 2^-21 of
// a .5 boundary) is recomputed with exact quotients fl(x / s). |x| <= max|x|
// bounds the codes to [-7, 7], so the clamp to [-8, 7] cannot bind. With
// NORM, squares of the codes are added to n2 (exact: sums below 2^24).
struct QRow {
  float s, ip, im;  // scale a / 7 and the two bracketing reciprocals (0 when a == 0)
};

__device__ __forceinline__ QRow quant_row(float a) {
  QRow r;
  r.s = __fdiv_rn(a, 7.0f);
  const float inv = (a != 0.0f) ? __frcp_rn(r.s) : 0.0f;
  r.ip = __fmul_rn(inv, 1.0f + 0x1p-21f);
  r.im = __fmul_rn(inv, 1.0f - 0x1p-21f);
  return r;
}

// Byte k of e holds the code of element 2k, byte k of o the code of element
// 2k + 1 (two's complement; the low nibble is the 4-bit code).
struct Codes8 {
  uint32_t e, o;
};

// packed: even-index codes in the low nibbles, odd-index codes in the high nibbles
__device__ __forceinline__ uint32_t packed4(Codes8 c) { return (c.e & 0x0F0F0F0Fu) | ((c.o << 4) & 0xF0F0F0F0u); }
// expanded, one byte per code u = v + 8: the four even-index codes, then the four odd-index codes
__device__ __forceinline__ uint32_t expanded_even(Codes8 c) { return (c.e & 0x0F0F0F0Fu) ^ 0x08080808u; }
__device__ __forceinline__ uint32_t expanded_odd(Codes8 c) { return (c.o & 0x0F0F0F0Fu) ^ 0x08080808u; }

// The magic-biased codes tb of eight fp32 values f (pairs in order).
__device__ __forceinline__ void quant_values(const float2 (&f)[4], const QRow& q, uint32_t (&tb)[8]) {
  const float2 ip2 = make_float2(q.ip, q.ip), im2 = make_float2(q.im, q.im);
  const float2 mg = make_float2(12582912.0f, 12582912.0f);
  uint32_t diff = 0;
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 tp = __ffma2_rn(f[k], ip2, mg);
    const float2 tm = __ffma2_rn(f[k], im2, mg);
    tb[2 * k] = __float_as_uint(tp.x);
    tb[2 * k + 1] = __float_as_uint(tp.y);
    diff |= (tb[2 * k] ^ __float_as_uint(tm.x)) | (tb[2 * k + 1] ^ __float_as_uint(tm.y));
  }
  if (diff != 0) {
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      tb[2 * k] = __float_as_uint(rintf(__fdiv_rn(f[k].x, q.s)) + 12582912.0f);
      tb[2 * k + 1] = __float_as_uint(rintf(__fdiv_rn(f[k].y, q.s)) + 12582912.0f);
    }
  }
}

__device__ __forceinline__ Codes8 gather_codes(const uint32_t (&tb)[8]) {
  Codes8 r;
  r.e = __byte_perm(__byte_perm(tb[0], tb[2], 0x0040), __byte_perm(tb[4], tb[6], 0x0040), 0x5410);
  r.o = __byte_perm(__byte_perm(tb[1], tb[3], 0x0040), __byte_perm(tb[5], tb[7], 0x0040), 0x5410);
  return r;
}

template <bool NORM>
__device__ __forceinline__ Codes8 quant_chunk(const uint4 v, const QRow& q, float2& n2) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  float2 f[4];
#pragma unroll
  for (int k = 0; k < 4; ++k) f[k] = __half22float2(*reinterpret_cast<const __half2*>(&w[k]));
  uint32_t tb[8];
  quant_values(f, q, tb);
  if (NORM) {
    const float2 nmg = make_float2(-12582912.0f, -12582912.0f);
#pragma unroll
    for (int k = 0; k < 4; ++k) {
      const float2 c = __fadd2_rn(make_float2(__uint_as_float(tb[2 * k]), __uint_as_float(tb[2 * k + 1])), nmg);
      n2 = __ffma2_rn(c, c, n2);
    }
  }
  return gather_codes(tb);
}

}  // namespace p4q
