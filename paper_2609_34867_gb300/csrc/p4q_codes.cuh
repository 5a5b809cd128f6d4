// Codes of a row's values from its scale (the rounding that the quantizers
// share): eight at a time, without a division per value.
#pragma once

#include <cstdint>
#include <type_traits>
#include <cuda_fp16.h>
#include <cuda_runtime.h>

namespace p4q {

// code = round_half_even(fl(x / s)), s = fl(a / 7), a = max|x| of the row. One
// fused multiply-add with the magic constant 1.5 * 2^23 rounds an exact product
// x * m to the nearest integer (ties to even: the constant is even) and leaves
// its two's complement in the low mantissa bits. |x| <= a bounds the codes to
// [-7, 7], so the clamp to [-8, 7] cannot bind.

// Rows of fp16 values. A quotient x / a of two fp16 values that is not exactly
// (2k + 1) / 14 lies at least 2^-15 (relative) from it: 14 |x| and (2k + 1) a
// are different multiples of a unit of at least 2^-11 of either. So any m
// within 2^-16 of 1 / s gives the code of every x off the ties, and only the
// ties 14 |x| = (2k + 1) a are left to the rounding of s and of the quotient:
//   k = 3, x = a / 2, is possible in every row; its code, 3 or 4, decides
//   whether m lies 2^-20 above or below 1 / s;
//   the others need 7 to divide a's significand: then s = a / 7 is exact, a
//   tie's quotient is exactly k + 1/2, and its code is the even one.
// (Compared with round_half_even(fl(x / s)) for all 503 856 639 pairs |x| <= a
// of finite fp16 values: equal.) Before, every chunk was rounded with two
// bracketing products and, where they differed for some value, recomputed by
// eight divisions: a / 2 is a common value (18 % of a warp's chunks of 256
// values), and that was a quarter of the instructions of a token pass.
struct QRow {
  float s, m;  // scale a / 7; the multiplier (0 when a == 0)
  bool tie;    // s is exactly a / 7: m = fl(1 / s), ties to even
};

__device__ __forceinline__ QRow quant_row(float a) {
  QRow r;
  r.s = __fdiv_rn(a, 7.0f);
  const float inv = (a != 0.0f) ? __frcp_rn(r.s) : 0.0f;
  r.tie = a != 0.0f && __fmaf_rn(r.s, 7.0f, -a) == 0.0f;
  const bool up = __fdiv_rn(0.5f * a, r.s) >= 3.5f;  // (3.5 itself goes to 4, the even one)
  r.m = r.tie ? inv : __fmul_rn(inv, up ? 1.0f + 0x1p-20f : 1.0f - 0x1p-20f);
  return r;
}

// Rows of fp32 values. With inv = fl(1 / s) correctly rounded, fl(x / s) lies
// within 2^-23 (relative) of x * inv, so ip = fl(inv (1 + 2^-21)) and im =
// fl(inv (1 - 2^-21)) give products x * ip and x * im that enclose fl(x / s)
// (each is at least 2^-21 - 2^-23 away from x * inv). Rounding is monotone, so
// where the two agree their integer is the code of fl(x / s); a chunk where
// they differ for some value (a quotient within about 2^-21 of a .5 boundary)
// is recomputed with exact quotients fl(x / s).
struct QRowF {
  float s, ip, im;  // scale a / 7 and the two bracketing reciprocals (0 when a == 0)
};

__device__ __forceinline__ QRowF quant_row_f(float a) {
  QRowF r;
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
__device__ __forceinline__ void quant_values(const float2 (&f)[4], const QRowF& q, uint32_t (&tb)[8]) {
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

// Codes of eight fp16 values of a row (a 16-byte chunk); TIE: the row's q.tie,
// where 1 / s is bracketed and, of two different neighbours (a tie), the even
// one is the code. With NORM, squares of the codes are added to n2 (exact: sums
// below 2^24).
template <bool NORM, bool TIE>
__device__ __forceinline__ Codes8 quant_chunk(const uint4 v, const QRow& q, float2& n2) {
  const uint32_t w[4] = {v.x, v.y, v.z, v.w};
  const float m = TIE ? q.m * (1.0f + 0x1p-21f) : q.m, mm = q.m * (1.0f - 0x1p-21f);
  const float2 m2 = make_float2(m, m), mm2 = make_float2(mm, mm);
  const float2 mg = make_float2(12582912.0f, 12582912.0f), nmg = make_float2(-12582912.0f, -12582912.0f);
  uint32_t tb[8];
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[k]));
    float2 t = __ffma2_rn(f, m2, mg);
    if (TIE) {
      const float2 t2 = __ffma2_rn(f, mm2, mg);
      t.x = (__float_as_uint(t.x) & 1u) ? t2.x : t.x;
      t.y = (__float_as_uint(t.y) & 1u) ? t2.y : t.y;
    }
    tb[2 * k] = __float_as_uint(t.x);
    tb[2 * k + 1] = __float_as_uint(t.y);
    if (NORM) {
      const float2 c = __fadd2_rn(t, nmg);
      n2 = __ffma2_rn(c, c, n2);
    }
  }
  return gather_codes(tb);
}

// f(std::integral_constant<bool, q.tie>): a row's loop over its chunks, once
// for each of the two roundings.
template <class F>
__device__ __forceinline__ void by_rounding(const QRow& q, F f) {
  if (q.tie) f(std::true_type());
  else f(std::false_type());
}

}  // namespace p4q
