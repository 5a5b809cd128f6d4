// RMSNorm before the quantized linears, fused with the per-token 4-bit
// quantizer of their input (App. A: every linear's input is quantized per
// token; the decoder's input norms feed q/k/v/gate/up):
//   S = sum_k x_k^2 exactly, rounded once to fp32; ms = S / d;
//   r = 1 / sqrt(ms + eps) (0 when ms + eps == 0); t_k = fp16(x_k * r);
//   y_k = fp16(t_k * w_k); then a = max|y|, s = a / 7,
//   code = clamp(round_half_even(y / s), -8, 7).
// Every fp16 value is an integer multiple of 2^-24, so its square is an
// integer count of 2^-48 below 2^80 and the row's sum fits 128 bits: the sum
// is exact whatever the order of the additions, and its one rounding to fp32
// (to nearest, ties to even) is the same on every evaluation. The remaining
// steps are single correctly rounded operations.
//
// The exact sum on the fp32 pipes: a square q = x^2 is exact in fp32 (at most
// 22 significant bits, at least 2^-48). Adding M = 1.5 * 2^(t + 23) to a value
// below 2^(t + 22) rounds it to a multiple of 2^t, and the bits of the sum
// minus those of M are that multiple as an integer; the residual is exact.
// Four such splits (t = 10, -12, -34, -48) write q as
// H1 2^10 + H2 2^-12 + H3 2^-34 + H4 2^-48 with integers |H| <= 2^22; each
// thread adds the bit patterns in four 32-bit words and turns them into one
// 128-bit integer count of 2^-48 at the end.
//
// Kernel: one CTA per row, 128, 160, 256 or 512 threads (so that a thread has
// at most 4 chunks of 8 values, kept in registers as fp16); a warp's four words
// are added by integer reductions of their halfwords, every thread adds the
// warps' sums into the 128-bit count and forms r, then y, the row's abs-max (a
// second block reduction) and the codes, written packed and, optionally,
// expanded one byte per code (u = code + 8, the GEMM's order) with their row
// sum.
//
// Bound: instruction issue. The splits run two values at a time
// (add/fma.rn.f32x2), t w is one fp16 multiplication (its exact product
// rounded once, as the fp32 product rounded to fp16 is), the maxima are taken
// on fp16 pairs and the codes take one product per value (p4q_codes.cuh).
// Measured (us; one value at a time before): 2048 x 4096 8.5 (14.2) = 3.4 TB/s;
// with two products per value 2048 x 5120 13.0 (21.3), 16000 x 5120 79 (149).
#include <cuda_fp16.h>

#include "p4q.h"
#include "p4q_codes.cuh"
#include "p4q_device.cuh"
#include "p4q_internal.h"

namespace p4q {
namespace {

constexpr int kRnMaxChunks = 4;  // chunks of 8 values per thread, at most

__device__ __forceinline__ float pow2f(int k) { return __int_as_float((k + 127) << 23); }

constexpr float kM1 = 0x1.8p+33f, kM2 = 0x1.8p+11f, kM3 = 0x1.8p-11f, kM4 = 0x1.8p-25f;

// acc[i] += bits of (residual + M_i) for the four splits of the two squares q = x^2
__device__ __forceinline__ void add_squares(float2 x, uint32_t (&acc)[4]) {
  auto two = [](float c) { return make_float2(c, c); };
  const float2 q = __fmul2_rn(x, x);
  const float2 a1 = __fadd2_rn(q, two(kM1));
  const float2 r1 = __ffma2_rn(__fadd2_rn(a1, two(-kM1)), two(-1.0f), q);  // q - (a1 - M1), exact
  const float2 a2 = __fadd2_rn(r1, two(kM2));
  const float2 r2 = __ffma2_rn(__fadd2_rn(a2, two(-kM2)), two(-1.0f), r1);
  const float2 a3 = __fadd2_rn(r2, two(kM3));
  const float2 r3 = __ffma2_rn(__fadd2_rn(a3, two(-kM3)), two(-1.0f), r2);
  const float2 a4 = __fadd2_rn(r3, two(kM4));
  acc[0] += __float_as_uint(a1.x) + __float_as_uint(a1.y);
  acc[1] += __float_as_uint(a2.x) + __float_as_uint(a2.y);
  acc[2] += __float_as_uint(a3.x) + __float_as_uint(a3.y);
  acc[3] += __float_as_uint(a4.x) + __float_as_uint(a4.y);
}

// The warp's sum of the integers h (|h| < 2^31), by halfwords.
__device__ __forceinline__ long long warp_sum(int h) {
  const int lo = __reduce_add_sync(0xFFFFFFFFu, h & 0xFFFF), hi = __reduce_add_sync(0xFFFFFFFFu, h >> 16);
  return static_cast<long long>(hi) * 65536 + lo;
}

__device__ __forceinline__ void add128(uint64_t& lo, uint64_t& hi, uint64_t lo2, uint64_t hi2) {
  lo += lo2;
  hi += hi2 + (lo < lo2 ? 1ull : 0ull);
}

// H1 2^58 + H2 2^36 + H3 2^14 + H4 (the count of 2^-48) as a 128-bit integer.
__device__ __forceinline__ void splits_to_u128(const long long (&h)[4], uint64_t& lo, uint64_t& hi) {
  lo = static_cast<uint64_t>(h[0]) << 58;  // h[0] >= 0
  hi = static_cast<uint64_t>(h[0]) >> 6;
  add128(lo, hi, static_cast<uint64_t>(h[1]) << 36, static_cast<uint64_t>(h[1] >> 28));
  add128(lo, hi, static_cast<uint64_t>(h[2]) << 14, static_cast<uint64_t>(h[2] >> 50));
  add128(lo, hi, static_cast<uint64_t>(h[3]), static_cast<uint64_t>(h[3] >> 63));
}

// fl32(S * 2^-48) for S = hi * 2^64 + lo, hi < 2^30: the top 64 bits of S with
// every lower bit folded into a sticky bit 0 round to 24 bits exactly as S
// does; the power-of-two scaling is exact (the result is a normal number).
__device__ __forceinline__ float sum_to_f32(uint64_t lo, uint64_t hi) {
  if (hi == 0) return __fmul_rn(__ull2float_rn(lo), 0x1p-48f);
  const int lz = __clzll(static_cast<long long>(hi));  // 34 .. 63
  const uint64_t top = (hi << lz) | (lo >> (64 - lz));
  const uint64_t sticky = (lo << lz) != 0ull ? 1ull : 0ull;
  return __fmul_rn(__ull2float_rn(top | sticky), pow2f(16 - lz));
}

template <int THREADS, int MAXC, bool EXPANDED>
__global__ void __launch_bounds__(THREADS)
    rmsnorm_quant_kernel(const __half* X, long long ldx, const __half* w, float eps, int K, uint8_t* Xq, float* s_a,
                         uint8_t* Xu, int32_t* sum_xu) {
  pdl_launch_dependents();  // before the wait: see p4q_device.cuh
  pdl_wait();
  constexpr int kWarps = THREADS / 32;
  __shared__ long long sh[kWarps][4];
  __shared__ uint32_t wmax[kWarps];
  __shared__ int wsum[kWarps];
  const int row = blockIdx.x, t = threadIdx.x, lane = t & 31, warp = t >> 5;
  const int nch = K >> 3;
  const uint4* x4 = reinterpret_cast<const uint4*>(X + static_cast<size_t>(row) * ldx);
  const uint4* w4 = reinterpret_cast<const uint4*>(w);
  uint4 xv[MAXC];
#pragma unroll
  for (int j = 0; j < MAXC; ++j) {
    const int c = t + j * THREADS;
    xv[j] = c < nch ? x4[c] : make_uint4(0u, 0u, 0u, 0u);
  }
  // exact sum of squares
  uint32_t acc[4] = {0u, 0u, 0u, 0u};
#pragma unroll
  for (int j = 0; j < MAXC; ++j) {
    const uint32_t xw[4] = {xv[j].x, xv[j].y, xv[j].z, xv[j].w};
#pragma unroll
    for (int e = 0; e < 4; ++e) add_squares(__half22float2(*reinterpret_cast<const __half2*>(&xw[e])), acc);
  }
  // each word holds 8 MAXC values' bits: as many times the bits of M_i plus the sum of the H_i
  const float kM[4] = {kM1, kM2, kM3, kM4};
  long long h[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) h[i] = warp_sum(static_cast<int>(acc[i] - 8u * MAXC * __float_as_uint(kM[i])));
  if (lane == 0) {
#pragma unroll
    for (int i = 0; i < 4; ++i) sh[warp][i] = h[i];
  }
  __syncthreads();
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    h[i] = sh[0][i];
#pragma unroll
    for (int v = 1; v < kWarps; ++v) h[i] += sh[v][i];
  }
  uint64_t lo, hi;
  splits_to_u128(h, lo, hi);
  const float ms = __fdiv_rn(sum_to_f32(lo, hi), static_cast<float>(K));
  const float den = __fadd_rn(ms, eps);
  const float r = den == 0.0f ? 0.0f : __frcp_rn(__fsqrt_rn(den));
  // y = fp16(fp16(x * r) * w), in place of x
  const float2 r2 = make_float2(r, r);
  uint32_t m = 0;  // per-halfword max of |y| bit patterns
#pragma unroll
  for (int j = 0; j < MAXC; ++j) {
    const int c = t + j * THREADS;
    const uint4 wv = c < nch ? w4[c] : make_uint4(0u, 0u, 0u, 0u);
    uint32_t xw[4] = {xv[j].x, xv[j].y, xv[j].z, xv[j].w};
    const uint32_t ww[4] = {wv.x, wv.y, wv.z, wv.w};
#pragma unroll
    for (int e = 0; e < 4; ++e) {
      const float2 tf = __fmul2_rn(__half22float2(*reinterpret_cast<const __half2*>(&xw[e])), r2);
      const __half2 y = __hmul2_rn(__floats2half2_rn(tf.x, tf.y), *reinterpret_cast<const __half2*>(&ww[e]));
      xw[e] = *reinterpret_cast<const uint32_t*>(&y);
      m = __vmaxu2(m, xw[e] & 0x7FFF7FFFu);
    }
    xv[j] = make_uint4(xw[0], xw[1], xw[2], xw[3]);
  }
  const uint32_t wm = __reduce_max_sync(0xFFFFFFFFu, max(m & 0xFFFFu, m >> 16));
  if (lane == 0) wmax[warp] = wm;
  __syncthreads();
  uint32_t am = wmax[0];
#pragma unroll
  for (int v = 1; v < kWarps; ++v) am = max(am, wmax[v]);
  const float a = __half2float(__ushort_as_half(static_cast<unsigned short>(am)));
  const QRow q = quant_row(a);
  const float s = q.s;
  uint32_t* q4 = reinterpret_cast<uint32_t*>(Xq + static_cast<size_t>(row) * (K >> 1));
  uint2* up2 = EXPANDED ? reinterpret_cast<uint2*>(Xu + static_cast<size_t>(row) * K) : nullptr;
  uint32_t su = 0;
  float2 n2 = make_float2(0.0f, 0.0f);  // unused
  by_rounding(q, [&](auto tie) {
#pragma unroll
    for (int j = 0; j < MAXC; ++j) {
      const int c = t + j * THREADS;
      if (c < nch) {
        const Codes8 cd = quant_chunk<false, decltype(tie)::value>(xv[j], q, n2);
        q4[c] = packed4(cd);
        if (EXPANDED) {
          // the even values, then the odd ones, offset by 8 (the GEMM's order)
          const uint32_t eu = expanded_even(cd), ou = expanded_odd(cd);
          up2[c] = make_uint2(eu, ou);
          su = __dp4a(eu + ou, 0x01010101u, su);
        }
      }
    }
  });
  if (t == 0) s_a[row] = (a != 0.0f) ? s : 0.0f;
  if (EXPANDED) {
    const int ws = static_cast<int>(__reduce_add_sync(0xFFFFFFFFu, su));
    if (lane == 0) wsum[warp] = ws;
    __syncthreads();
    if (t == 0) {
      int tot = 0;
#pragma unroll
      for (int v = 0; v < kWarps; ++v) tot += wsum[v];
      sum_xu[row] = tot;
    }
  }
}

template <int THREADS, int MAXC>
cudaError_t launch_c(const __half* X, long long ldx, const __half* w, float eps, int M, int K, uint8_t* Xq, float* s_a,
                     uint8_t* Xu, int32_t* sum_xu, cudaStream_t stream) {
  if (Xu)
    return launch_pdl(rmsnorm_quant_kernel<THREADS, MAXC, true>, dim3(M), dim3(THREADS), 0, stream, X, ldx, w, eps,
                      K, Xq, s_a, Xu, sum_xu);
  return launch_pdl(rmsnorm_quant_kernel<THREADS, MAXC, false>, dim3(M), dim3(THREADS), 0, stream, X, ldx, w, eps, K,
                    Xq, s_a, Xu, sum_xu);
}

template <int THREADS>
cudaError_t launch_t(const __half* X, long long ldx, const __half* w, float eps, int M, int K, uint8_t* Xq, float* s_a,
                     uint8_t* Xu, int32_t* sum_xu, cudaStream_t stream) {
  const int per = (K / 8 + THREADS - 1) / THREADS;  // chunks per thread, at most kRnMaxChunks
  if (per <= 1) return launch_c<THREADS, 1>(X, ldx, w, eps, M, K, Xq, s_a, Xu, sum_xu, stream);
  if (per <= 2) return launch_c<THREADS, 2>(X, ldx, w, eps, M, K, Xq, s_a, Xu, sum_xu, stream);
  if (per <= 3) return launch_c<THREADS, 3>(X, ldx, w, eps, M, K, Xq, s_a, Xu, sum_xu, stream);
  return launch_c<THREADS, kRnMaxChunks>(X, ldx, w, eps, M, K, Xq, s_a, Xu, sum_xu, stream);
}

}  // namespace

cudaError_t launch_rmsnorm_quant(const uint16_t* X16, long long ldx, const uint16_t* w16, float eps, int M, int K,
                                 uint8_t* Xq, float* s_a, uint8_t* Xu, int32_t* sum_xu, cudaStream_t stream) {
  if (M <= 0) return cudaSuccess;
  const __half* X = reinterpret_cast<const __half*>(X16);
  const __half* w = reinterpret_cast<const __half*>(w16);
  static_assert(P4Q_MAX_ROW <= 8 * 512 * kRnMaxChunks, "rows longer than 512 threads x 4 chunks");
  if (K <= 8 * 128 * kRnMaxChunks) return launch_t<128>(X, ldx, w, eps, M, K, Xq, s_a, Xu, sum_xu, stream);
  if (K <= 8 * 160 * kRnMaxChunks) return launch_t<160>(X, ldx, w, eps, M, K, Xq, s_a, Xu, sum_xu, stream);
  if (K <= 8 * 256 * kRnMaxChunks) return launch_t<256>(X, ldx, w, eps, M, K, Xq, s_a, Xu, sum_xu, stream);
  return launch_t<512>(X, ldx, w, eps, M, K, Xq, s_a, Xu, sum_xu, stream);
}

}  // namespace p4q
