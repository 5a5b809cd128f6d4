// SwiGLU before down_proj, fused with the per-token 4-bit quantizer of
// down_proj's input (App. A: every linear's input is quantized per token):
//   h = silu(gate) * up, silu(g) = g * (1 / (1 + exp32(-g))) (each
//   operation one rounded fp32 step, the reciprocal correctly rounded),
//   then a = max|h|, s = a / 7, code = clamp(round_half_even(h / s), -8, 7).
// exp32 is an own fp32 exponential (Cody-Waite reduction with ln 2 split as
// 355/512 + a low part, degree-7 Taylor polynomial by Horner's rule with fused
// multiply-adds, two exact power-of-two scalings; within 0.9 ulp of e^x; 0
// below -87, inf above 88.72284). The fp32 h is within 2.9 ulp (3.5e-7
// relative: 0.9 ulp from exp32 and four roundings of 2^-24) of the real
// silu(g) * up, the row's abs-max likewise, the scale a / 7 adds one
// rounding and the quotient h / s one more, so h / s is within 8.1e-7
// relative, 5.7e-6 absolute (|h / s| <= 7), of the exact quotient: the codes
// are those of the exact SwiGLU except where that quotient falls within
// 5.7e-6 of a .5 boundary.
//
// Kernel: one CTA per row (256, 384 or 512 threads); each thread holds its
// chunks of 8 values of h in registers (computed once), the row's abs-max comes
// from a block reduction, then the codes are written packed and, optionally, expanded one byte per code (u =
// code + 8, the GEMM's order) with their row sum.
//
// Bound: instruction issue, then HBM. Gates within [-87, 87] (nearly all
// chunks; the others take the scalar form below) are evaluated two at a time
// (fma.rn.f32x2), the power of two enters the exponent by an integer addition,
// the reciprocal is the hardware approximation with one Newton step (Markstein's
// correction: residual by a fused multiply-add; compared with the correctly
// rounded reciprocal for every significand at the exponents 0 .. 125, which hold
// 1 + e^87: equal, so that both forms give the same h), and the codes come from
// the bracketing products of p4q_codes.cuh: about 20 instructions per value
// where one at a time with a library reciprocal took about 45. Measured (us,
// inputs past L2; before): 6144 x 11008 84 (140) = 4.4 TB/s, 6144 x 13824 104
// (180), 600 x 13824 13.9 (21.8), 1 x 13824 4.0 (6.8).
#include <cuda_fp16.h>

#include "p4q.h"
#include "p4q_codes.cuh"
#include "p4q_device.cuh"
#include "p4q_internal.h"

namespace p4q {
namespace {

__device__ __forceinline__ float pow2f(int k) { return __int_as_float((k + 127) << 23); }

__device__ __forceinline__ float exp32(float x) {
  if (x > 0x1.62e430p+6f) return __int_as_float(0x7f800000);
  if (x < -87.0f) return 0.0f;
  // n = round_half_even(x * log2 e) by adding 1.5 * 2^23 (|n| <= 128); its
  // bits hold n in the low mantissa bits
  const float nm = __fadd_rn(__fmul_rn(x, 0x1.715476p+0f), 12582912.0f);
  const float n = __fsub_rn(nm, 12582912.0f);
  const int k = __float_as_int(nm) - 0x4B400000;
  float r = __fmaf_rn(-n, 0x1.630000p-1f, x);
  r = __fmaf_rn(-n, -0x1.bd0106p-13f, r);
  float p = 0x1.a01a02p-13f;
  p = __fmaf_rn(p, r, 0x1.6c16c2p-10f);
  p = __fmaf_rn(p, r, 0x1.111112p-7f);
  p = __fmaf_rn(p, r, 0x1.555556p-5f);
  p = __fmaf_rn(p, r, 0x1.555556p-3f);
  p = __fmaf_rn(p, r, 0.5f);
  p = __fmaf_rn(p, r, 1.0f);
  p = __fmaf_rn(p, r, 1.0f);
  // p * 2^n is exact (a normal result): one multiplication, two when 2^n
  // itself overflows (n = 128)
  if (k <= 127) return __fmul_rn(p, pow2f(k));
  return __fmul_rn(__fmul_rn(p, pow2f(64)), pow2f(k - 64));
}

// silu(g) * u = (g * (1 / (1 + exp32(-g)))) * u, four rounded fp32 steps
__device__ __forceinline__ float swiglu(float g, float u) {
  const float sig = __frcp_rn(__fadd_rn(1.0f, exp32(-g)));
  return __fmul_rn(__fmul_rn(g, sig), u);
}

__device__ __forceinline__ float max3_abs(float m, float a, float b) {
  float d;
  asm("{\n\t.reg .f32 x, y;\n\tabs.f32 x, %2;\n\tabs.f32 y, %3;\n\tmax.f32 %0, %1, x, y;\n\t}\n"
      : "=f"(d)
      : "f"(m), "f"(a), "f"(b));
  return d;
}

__device__ __forceinline__ float rcp_approx(float x) {
  float y;
  asm("rcp.approx.f32 %0, %1;" : "=f"(y) : "f"(x));
  return y;
}

// -h of eight values, gates ng = -g given (their sign bits flipped), all
// |g| <= 87: swiglu's steps two values at a time. The polynomial is negated
// (np = -p) so that nd = -(1 + e) is at hand for the Newton step.
__device__ __forceinline__ void swiglu8(const uint32_t (&ng)[4], const uint32_t (&uw)[4], float2 (&nh)[4]) {
  auto two = [](float c) { return make_float2(c, c); };
#pragma unroll
  for (int k = 0; k < 4; ++k) {
    const float2 x = __half22float2(*reinterpret_cast<const __half2*>(&ng[k]));
    const float2 u = __half22float2(*reinterpret_cast<const __half2*>(&uw[k]));
    const float2 nm = __ffma2_rn(x, two(0x1.715476p+0f), two(12582912.0f));
    const float2 n = __fadd2_rn(nm, two(-12582912.0f));
    float2 r = __ffma2_rn(n, two(-0x1.630000p-1f), x);
    r = __ffma2_rn(n, two(0x1.bd0106p-13f), r);
    float2 np = two(-0x1.a01a02p-13f);
    np = __ffma2_rn(np, r, two(-0x1.6c16c2p-10f));
    np = __ffma2_rn(np, r, two(-0x1.111112p-7f));
    np = __ffma2_rn(np, r, two(-0x1.555556p-5f));
    np = __ffma2_rn(np, r, two(-0x1.555556p-3f));
    np = __ffma2_rn(np, r, two(-0.5f));
    np = __ffma2_rn(np, r, two(-1.0f));
    np = __ffma2_rn(np, r, two(-1.0f));
    // -p * 2^n: n, in the low bits of nm, into the exponent field (|n| <= 126, p in [0.7, 1.42])
    const float2 ne = make_float2(__uint_as_float(__float_as_uint(np.x) + (__float_as_uint(nm.x) << 23)),
                                  __uint_as_float(__float_as_uint(np.y) + (__float_as_uint(nm.y) << 23)));
    const float2 nd = __fadd2_rn(ne, two(-1.0f));
    const float2 y = make_float2(rcp_approx(-nd.x), rcp_approx(-nd.y));
    const float2 sig = __ffma2_rn(y, __ffma2_rn(nd, y, two(1.0f)), y);
    nh[k] = __fmul2_rn(__fmul2_rn(x, sig), u);
  }
}

template <int THREADS, int MAXC, bool EXPANDED>
__global__ void __launch_bounds__(THREADS, THREADS == 256 ? (MAXC <= 3 ? 4 : 2) : THREADS == 384 ? 3 : 2)
    swiglu_quant_kernel(const __half* gate, long long ldg, const __half* up, long long ldu, int K, uint8_t* Xq,
                        float* s_a, uint8_t* Xu, int32_t* sum_xu) {
  pdl_launch_dependents();  // before the wait: see p4q_device.cuh
  pdl_wait();
  __shared__ float wmax[THREADS / 32];
  __shared__ int wsum[THREADS / 32];
  const int row = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int nch = K >> 3;
  const uint4* g4 = reinterpret_cast<const uint4*>(gate + static_cast<size_t>(row) * ldg);
  const uint4* u4 = reinterpret_cast<const uint4*>(up + static_cast<size_t>(row) * ldu);
  float2 nh[MAXC][4];  // -h
  float m = 0.0f;
  constexpr int kBatch = 3;  // chunks on their way together
#pragma unroll
  for (int j0 = 0; j0 < MAXC; j0 += kBatch) {
    uint4 gv[kBatch], uv[kBatch];
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      const int c = t + (j0 + j) * THREADS;
      const bool in = j0 + j < MAXC && c < nch;
      gv[j] = in ? ldg_stream16(g4 + c) : make_uint4(0u, 0u, 0u, 0u);
      uv[j] = in ? ldg_stream16(u4 + c) : make_uint4(0u, 0u, 0u, 0u);
    }
#pragma unroll
    for (int j = 0; j < kBatch; ++j) {
      if (j0 + j >= MAXC) break;
      float2(&h)[4] = nh[j0 + j < MAXC ? j0 + j : 0];
      const uint32_t ng[4] = {gv[j].x ^ 0x80008000u, gv[j].y ^ 0x80008000u, gv[j].z ^ 0x80008000u,
                              gv[j].w ^ 0x80008000u};
      const uint32_t uw[4] = {uv[j].x, uv[j].y, uv[j].z, uv[j].w};
      auto abs2 = [](uint32_t w) { return __habs2(*reinterpret_cast<const __half2*>(&w)); };
      const __half2 gm = __hmax2(__hmax2(abs2(ng[0]), abs2(ng[1])), __hmax2(abs2(ng[2]), abs2(ng[3])));
      if (__hble2(gm, __float2half2_rn(87.0f))) {
        swiglu8(ng, uw, h);
      } else {
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 gf = __half22float2(*reinterpret_cast<const __half2*>(&ng[e]));
          const float2 uf = __half22float2(*reinterpret_cast<const __half2*>(&uw[e]));
          h[e] = make_float2(-swiglu(-gf.x, uf.x), -swiglu(-gf.y, uf.y));
        }
      }
#pragma unroll
      for (int e = 0; e < 4; ++e) m = max3_abs(m, h[e].x, h[e].y);
    }
  }
  // non-negative floats order as their bits
  const uint32_t wm = __reduce_max_sync(0xFFFFFFFFu, __float_as_uint(m));
  if (lane == 0) wmax[warp] = __uint_as_float(wm);
  __syncthreads();
  float a = 0.0f;
#pragma unroll
  for (int w = 0; w < THREADS / 32; ++w) a = fmaxf(a, wmax[w]);
  QRowF q = quant_row_f(a);
  const float s = q.s;
  q.s = -q.s;  // the values are held negated
  q.ip = -q.ip;
  q.im = -q.im;
  uint32_t* q4 = reinterpret_cast<uint32_t*>(Xq + static_cast<size_t>(row) * (K >> 1));
  uint2* up2 = EXPANDED ? reinterpret_cast<uint2*>(Xu + static_cast<size_t>(row) * K) : nullptr;
  uint32_t su = 0;
#pragma unroll
  for (int j = 0; j < MAXC; ++j) {
    const int c = t + j * THREADS;
    if (c < nch) {
      Codes8 cd{0u, 0u};
      if (a != 0.0f) {
        uint32_t tb[8];
        quant_values(nh[j], q, tb);
        cd = gather_codes(tb);
      }
      q4[c] = packed4(cd);
      if (EXPANDED) {
        // the even values, then the odd ones, offset by 8 (the GEMM's order)
        const uint32_t eu = expanded_even(cd), ou = expanded_odd(cd);
        up2[c] = make_uint2(eu, ou);
        su = __dp4a(eu + ou, 0x01010101u, su);
      }
    }
  }
  if (t == 0) s_a[row] = (a != 0.0f) ? s : 0.0f;
  if (EXPANDED) {
    const int ws = static_cast<int>(__reduce_add_sync(0xFFFFFFFFu, su));
    if (lane == 0) wsum[warp] = ws;
    __syncthreads();
    if (t == 0) {
      int tot = 0;
#pragma unroll
      for (int w = 0; w < THREADS / 32; ++w) tot += wsum[w];
      sum_xu[row] = tot;
    }
  }
}

template <int THREADS, int MAXC>
cudaError_t launch_c(const __half* g, long long ldg, const __half* u, long long ldu, int M, int K, uint8_t* Xq,
                     float* s_a, uint8_t* Xu, int32_t* sum_xu, cudaStream_t stream) {
  if (Xu)
    return launch_pdl(swiglu_quant_kernel<THREADS, MAXC, true>, dim3(M), dim3(THREADS), 0, stream, g, ldg, u, ldu, K,
                      Xq, s_a, Xu, sum_xu);
  return launch_pdl(swiglu_quant_kernel<THREADS, MAXC, false>, dim3(M), dim3(THREADS), 0, stream, g, ldg, u, ldu, K,
                    Xq, s_a, Xu, sum_xu);
}

}  // namespace

cudaError_t launch_swiglu_quant(const uint16_t* gate, long long ldg, const uint16_t* up, long long ldu, int M, int K,
                                uint8_t* Xq, float* s_a, uint8_t* Xu, int32_t* sum_xu, cudaStream_t stream) {
  if (M <= 0) return cudaSuccess;
  const __half* g = reinterpret_cast<const __half*>(gate);
  const __half* u = reinterpret_cast<const __half*>(up);
  const int chunks = K / 8;
  // Few rows: as many threads per row as they fill. Otherwise CTAs of 384
  // threads, three per SM (6144 x 11008 and x 13824, us: 384 threads 84 and 104,
  // 256 threads 87 and 132, 512 threads 88 and 116); shorter rows 256, longer
  // ones 256 with 8 chunks.
  if (M <= 4 * num_sms()) {
    if (chunks <= 512) return launch_c<512, 1>(g, ldg, u, ldu, M, K, Xq, s_a, Xu, sum_xu, stream);
    if (chunks <= 3 * 512) return launch_c<512, 3>(g, ldg, u, ldu, M, K, Xq, s_a, Xu, sum_xu, stream);
    return launch_c<512, 4>(g, ldg, u, ldu, M, K, Xq, s_a, Xu, sum_xu, stream);
  }
  if (chunks <= 3 * 256) return launch_c<256, 3>(g, ldg, u, ldu, M, K, Xq, s_a, Xu, sum_xu, stream);
  if (chunks <= 4 * 384) return launch_c<384, 4>(g, ldg, u, ldu, M, K, Xq, s_a, Xu, sum_xu, stream);
  if (chunks <= 5 * 384) return launch_c<384, 5>(g, ldg, u, ldu, M, K, Xq, s_a, Xu, sum_xu, stream);
  return launch_c<256, 8>(g, ldg, u, ldu, M, K, Xq, s_a, Xu, sum_xu, stream);
}

}  // namespace p4q
