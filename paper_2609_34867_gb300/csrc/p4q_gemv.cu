// W4A4 linear for a few token rows (decode steps, small batches): the same
// exact integer products and dequantization as the GEMMs (App. A / App. B.3
// of the paper: per-token INT4 activations, per-output-channel INT4 weights,
// acc = sum_k a_k w_k exact, y = fp16_rne((float(acc) * s_a) * s_w)), for
// M <= 2 rows, where the cost is streaming the packed weights from HBM.
//
// Kernel: the M activation rows are sign-extended once into shared memory,
// one byte per code (for each packed 32-bit word: its four low-nibble codes,
// then its four high-nibble codes; the weights use the same order, so every
// dot product is unchanged). Each warp streams pairs of whole weight rows,
// every lane a 16-byte chunk (32 codes) of each at a time, four chunks of both
// in flight (the next pair's first ones while the current pair is summed), and
// dp4a's them against the activation rows (read from shared memory once for
// the two weight rows). The weight codes enter as unsigned bytes w + 8 (low
// nibbles) and 16 (w + 8) (high nibbles, left in place: one logic operation
// per four codes each) in two accumulators: acc = lo + hi / 16 - 8 sum x,
// exact. A warp sum per row gives the int32 accumulators, and lane m writes row
// m's outputs.
//
// Bound: instruction issue (half of it dp4a), then HBM. Measured (us, the four
// linears and quantizers of a decode step as one graph; before, with
// sign-extended weights, one row at a time, about 50 instructions per chunk):
// 1 row 7B 38.2 (43.3) = 2.7 TB/s, 1 row 13B 51.5 (61.1), 2 rows 13B 63.3
// (78.7).
#include <cuda_fp16.h>

#include "p4q.h"
#include "p4q_device.cuh"
#include "p4q_internal.h"

namespace p4q {
namespace {

constexpr int kGemvWarps = 8;
constexpr int kGemvCtas = 3;  // per SM, one wave (4 at 64 registers, us: 40.0 / 57.4 for the steps above, 6: 48 / 60)
constexpr int kGemvMaxRows = 2;  // above, the tensor-core kernel (p4q_fewrows.cu) is faster: 4 x 11008 x 4096 16.6 us here, 10.4 there
constexpr int kGemvUnroll = 4;                  // weight chunks in flight per lane
constexpr size_t kGemvSmemMax = 200u * 1024u;   // sign-extended activation rows

__device__ __forceinline__ int sext4(uint32_t n) {
  return static_cast<int>((n & 0x0F0F0F0Fu) | ((n & 0x08080808u) * 0x1Eu));
}

// c + the dot product of four unsigned bytes a with four signed bytes b.
__device__ __forceinline__ int dp4a_us(uint32_t a, int b, int c) {
  int d;
  asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

template <int MR, bool S32>
__global__ void __launch_bounds__(kGemvWarps * 32, kGemvCtas)
    gemv_w4a4_kernel(const uint8_t* Xq, const float* s_a, int M, int K, const uint8_t* Wq, const float* s_w, int N,
                     void* out) {
  extern __shared__ __align__(16) int8_t xs[];  // [M][K] sign-extended activation codes
  __shared__ int xsum[MR];                       // their row sums
  const int kb = K >> 1;                         // packed bytes per row
  const int nch = kb >> 4;                       // 16-byte packed chunks per row
  const int lane = threadIdx.x & 31;
  const int stride = 2 * gridDim.x * kGemvWarps;  // N is even
  // This warp's weight rows into L2 while the previous kernel (the quantizer
  // of the activations) still runs: a prefetch changes no memory, so it may run
  // ahead of a kernel that still writes the weights.
  int n = 2 * (blockIdx.x * kGemvWarps + (threadIdx.x >> 5));
  for (int r = n + (lane >> 1) * stride + (lane & 1); r < N; r += 16 * stride)
    prefetch_l2_bulk(Wq + static_cast<size_t>(r) * kb, static_cast<uint32_t>(kb));
  if (threadIdx.x < MR) xsum[threadIdx.x] = 0;
  pdl_launch_dependents();
  pdl_wait();
  // the first weight chunks of this warp's first rows are on their way while
  // the activations are staged
  uint4 wv[2][kGemvUnroll];
  auto load = [&](int row, int c0) {
#pragma unroll
    for (int i = 0; i < 2; ++i) {
      const uint4* wrow = reinterpret_cast<const uint4*>(Wq + static_cast<size_t>(row + i) * kb);
#pragma unroll
      for (int u = 0; u < kGemvUnroll; ++u) {
        const int c = c0 + 32 * u;
        if (row < N && c < nch) wv[i][u] = ldg_stream16(wrow + c);
      }
    }
  };
  load(n, lane);
  __syncthreads();
  // stage the activations: 16 packed bytes -> 32 signed bytes
#pragma unroll
  for (int m = 0; m < MR; ++m) {
    if (m >= M) break;
    int sum = 0;
    for (int c = threadIdx.x; c < nch; c += blockDim.x) {
      const uint4 p = *reinterpret_cast<const uint4*>(Xq + static_cast<size_t>(m) * kb + 16 * c);
      const uint32_t w[4] = {p.x, p.y, p.z, p.w};
      int4* dst = reinterpret_cast<int4*>(xs + static_cast<size_t>(m) * K + 32 * c);
      int e[8];
#pragma unroll
      for (int k = 0; k < 4; ++k) {
        e[2 * k] = sext4(w[k]);
        e[2 * k + 1] = sext4(w[k] >> 4);
        sum = __dp4a(e[2 * k], 0x01010101, __dp4a(e[2 * k + 1], 0x01010101, sum));
      }
      dst[0] = make_int4(e[0], e[1], e[2], e[3]);
      dst[1] = make_int4(e[4], e[5], e[6], e[7]);
    }
    sum = __reduce_add_sync(0xFFFFFFFFu, sum);
    if (lane == 0) atomicAdd(&xsum[m], sum);
  }
  __syncthreads();
  for (; n < N; n += stride) {
    int lo[2][MR], hi[2][MR];
#pragma unroll
    for (int m = 0; m < MR; ++m) lo[0][m] = lo[1][m] = hi[0][m] = hi[1][m] = 0;
    for (int c0 = lane; c0 < nch; c0 += 32 * kGemvUnroll) {
      if (c0 != lane) load(n, c0);  // the rows' first chunks were loaded ahead
#pragma unroll
      for (int u = 0; u < kGemvUnroll; ++u) {
        const int c = c0 + 32 * u;
        if (c >= nch) break;
        uint32_t l[2][4], h[2][4];
#pragma unroll
        for (int i = 0; i < 2; ++i) {
          const uint32_t w[4] = {wv[i][u].x, wv[i][u].y, wv[i][u].z, wv[i][u].w};
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            l[i][k] = (w[k] ^ 0x88888888u) & 0x0F0F0F0Fu;
            h[i][k] = (w[k] ^ 0x88888888u) & 0xF0F0F0F0u;
          }
        }
#pragma unroll
        for (int m = 0; m < MR; ++m) {
          if (m < M) {
            const int4* xr = reinterpret_cast<const int4*>(xs + static_cast<size_t>(m) * K + 32 * c);
            const int4 x0 = xr[0], x1 = xr[1];
#pragma unroll
            for (int i = 0; i < 2; ++i) {
              int a = lo[i][m], b = hi[i][m];
              a = dp4a_us(l[i][0], x0.x, a); b = dp4a_us(h[i][0], x0.y, b);
              a = dp4a_us(l[i][1], x0.z, a); b = dp4a_us(h[i][1], x0.w, b);
              a = dp4a_us(l[i][2], x1.x, a); b = dp4a_us(h[i][2], x1.y, b);
              a = dp4a_us(l[i][3], x1.z, a); b = dp4a_us(h[i][3], x1.w, b);
              lo[i][m] = a;
              hi[i][m] = b;
            }
          }
        }
      }
    }
    // the next rows' first chunks go out before this pair's sums
    load(n + stride, lane);
#pragma unroll
    for (int m = 0; m < MR; ++m) {
      if (m < M) {
        int tot[2];
#pragma unroll
        for (int i = 0; i < 2; ++i)  // hi is a sum of multiples of 16
          tot[i] = __reduce_add_sync(0xFFFFFFFFu, lo[i][m] + (hi[i][m] >> 4)) - 8 * xsum[m];
        if (lane == m) {
          const size_t at = static_cast<size_t>(m) * N + n;
          if (S32) {
            *reinterpret_cast<int2*>(static_cast<int32_t*>(out) + at) = make_int2(tot[0], tot[1]);
          } else {
            const float y0 = __fmul_rn(__fmul_rn(static_cast<float>(tot[0]), s_a[m]), s_w[n]);
            const float y1 = __fmul_rn(__fmul_rn(static_cast<float>(tot[1]), s_a[m]), s_w[n + 1]);
            *reinterpret_cast<__half2*>(static_cast<__half*>(out) + at) = __floats2half2_rn(y0, y1);
          }
        }
      }
    }
  }
}

template <int MR, bool S32>
cudaError_t launch_mr(const GemmArgs& g, cudaStream_t stream) {
  const size_t smem = static_cast<size_t>(g.M) * g.K;
  static SmemLimit limit;
  const cudaError_t le = limit.allow(gemv_w4a4_kernel<MR, S32>, kGemvSmemMax);
  if (le != cudaSuccess) return le;
  // enough warps for every pair of weight rows, at most the CTAs that fit on the SMs
  const int per_sm = smem <= 64u * 1024u ? kGemvCtas : smem <= 100u * 1024u ? 2 : 1;
  const int want = (g.N / 2 + kGemvWarps - 1) / kGemvWarps;
  const int blocks = want < per_sm * num_sms() ? want : per_sm * num_sms();
  return launch_pdl(gemv_w4a4_kernel<MR, S32>, dim3(blocks), dim3(kGemvWarps * 32), smem, stream, g.A, g.s_a, g.M,
                    g.K, g.B, g.s_b, g.N, g.D);
}

}  // namespace

bool gemv_applies(const GemmArgs& g) {
  return (g.out == GemmOut::kHalf || g.out == GemmOut::kS32) && g.batch == 1 && g.M >= 1 && g.M <= kGemvMaxRows &&
         g.N % 2 == 0 && g.K % 32 == 0 && (g.d_pitch == 0 || g.d_pitch == g.N) && static_cast<size_t>(g.M) * g.K <= kGemvSmemMax;
}

cudaError_t launch_gemv(const GemmArgs& g, cudaStream_t stream) {
  return g.out == GemmOut::kS32 ? launch_mr<kGemvMaxRows, true>(g, stream) : launch_mr<kGemvMaxRows, false>(g, stream);
}

}  // namespace p4q
