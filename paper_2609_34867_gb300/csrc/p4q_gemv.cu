// W4A4 linear for a few token rows (decode steps, small batches): the same
// exact integer products and dequantization as the GEMMs (App. A / App. B.3
// of the paper: per-token INT4 activations, per-output-channel INT4 weights,
// acc = sum_k a_k w_k exact, y = fp16_rne((float(acc) * s_a) * s_w)), for
// M <= 2 rows, where the cost is streaming the packed weights from HBM, and for
// up to 8 rows on small weights, where it is the launch's start.
//
// Kernel: the M activation rows are sign-extended once into shared memory,
// one byte per code (for each packed 32-bit word: its four low-nibble codes,
// then its four high-nibble codes; the weights use the same order, so every
// dot product is unchanged). Each warp streams pairs of whole weight rows (one
// row where there are few), every lane a 16-byte chunk (32 codes) of each at a
// time, four chunks of both in flight (the next pair's first ones while the
// current pair is summed), and dp4a's them against the activation rows (read
// from shared memory once for the two weight rows). The weight codes enter as unsigned bytes w + 8 (low
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
constexpr int kGemvMaxRows = 8;  // rows of activations, up to 2 whatever the weights' size
constexpr int kGemvUnroll = 4;                  // weight chunks in flight per lane
constexpr size_t kGemvSmemMax = 56u * 1024u;    // sign-extended activation rows (gemv_applies' M (K + N))

__device__ __forceinline__ int sext4(uint32_t n) {
  return static_cast<int>((n & 0x0F0F0F0Fu) | ((n & 0x08080808u) * 0x1Eu));
}

// c + the dot product of four unsigned bytes a with four signed bytes b.
__device__ __forceinline__ int dp4a_us(uint32_t a, int b, int c) {
  int d;
  asm("dp4a.u32.s32 %0, %1, %2, %3;" : "=r"(d) : "r"(a), "r"(b), "r"(c));
  return d;
}

// RW weight rows per warp and step: two share each read of the activations.
template <int MR, int RW, bool S32>
__global__ void __launch_bounds__(kGemvWarps * 32, MR * RW > 8 ? 2 : kGemvCtas)
    gemv_w4a4_kernel(const uint8_t* Xq, const float* s_a, int M, int K, const uint8_t* Wq, const float* s_w, int N,
                     void* out, bool early) {
  extern __shared__ __align__(16) int8_t xs[];  // [M][K] sign-extended activation codes
  __shared__ int xsum[MR];                       // their row sums
  const int kb = K >> 1;                         // packed bytes per row
  const int nch = kb >> 4;                       // 16-byte packed chunks per row
  const int lane = threadIdx.x & 31;
  const int stride = RW * gridDim.x * kGemvWarps;  // N is even
  // This warp's weight rows into L2 while the previous kernel (the quantizer
  // of the activations) still runs: a prefetch changes no memory, so it may run
  // ahead of a kernel that still writes the weights.
  int n = RW * (blockIdx.x * kGemvWarps + (threadIdx.x >> 5));
  for (int r = n + lane / RW * stride + lane % RW; r < N; r += 32 / RW * stride)
    prefetch_l2_bulk(Wq + static_cast<size_t>(r) * kb, static_cast<uint32_t>(kb));
  if (threadIdx.x < MR) xsum[threadIdx.x] = 0;
  if (early) pdl_launch_dependents();
  pdl_wait();
  if (!early) pdl_launch_dependents();
  // the first weight chunks of this warp's first rows are on their way while
  // the activations are staged
  uint4 wv[RW][kGemvUnroll];
  auto load = [&](int row, int c0) {
#pragma unroll
    for (int i = 0; i < RW; ++i) {
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
  // stage the activations, 16 packed bytes -> 32 signed bytes: the rows side by
  // side, each by its share of the warps
  {
    constexpr int kLog = MR == 2 ? 2 : MR == 4 ? 1 : 0;
    static_assert(MR << kLog == kGemvWarps, "warps per row");
    const int log = M == 1 ? 3 : kLog, t = threadIdx.x, m = t >> (5 + log), step = 32 << log;  // step threads per row
    if (m < M) {
      const uint4* x = reinterpret_cast<const uint4*>(Xq + static_cast<size_t>(m) * kb);
      int4* dst = reinterpret_cast<int4*>(xs + static_cast<size_t>(m) * K);
      int sum = 0;
      for (int c = t & (step - 1); c < nch; c += step) {
        const uint4 p = x[c];
        const uint32_t w[4] = {p.x, p.y, p.z, p.w};
        int e[8];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          e[2 * k] = sext4(w[k]);
          e[2 * k + 1] = sext4(w[k] >> 4);
          sum = __dp4a(e[2 * k], 0x01010101, __dp4a(e[2 * k + 1], 0x01010101, sum));
        }
        dst[2 * c] = make_int4(e[0], e[1], e[2], e[3]);
        dst[2 * c + 1] = make_int4(e[4], e[5], e[6], e[7]);
      }
      sum = __reduce_add_sync(0xFFFFFFFFu, sum);
      if (lane == 0) atomicAdd(&xsum[m], sum);
    }
  }
  __syncthreads();
  for (; n < N; n += stride) {
    int lo[RW][MR], hi[RW][MR];
#pragma unroll
    for (int i = 0; i < RW; ++i)
#pragma unroll
      for (int m = 0; m < MR; ++m) lo[i][m] = hi[i][m] = 0;
    for (int c0 = lane; c0 < nch; c0 += 32 * kGemvUnroll) {
      if (c0 != lane) load(n, c0);  // the rows' first chunks were loaded ahead
#pragma unroll
      for (int u = 0; u < kGemvUnroll; ++u) {
        const int c = c0 + 32 * u;
        if (c >= nch) break;
        uint32_t l[RW][4], h[RW][4];
#pragma unroll
        for (int i = 0; i < RW; ++i) {
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
            for (int i = 0; i < RW; ++i) {
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
    // the next rows' first chunks go out before these rows' sums
    load(n + stride, lane);
#pragma unroll
    for (int m = 0; m < MR; ++m) {
      if (m < M) {
        int tot[RW];
#pragma unroll
        for (int i = 0; i < RW; ++i)  // hi is a sum of multiples of 16
          tot[i] = __reduce_add_sync(0xFFFFFFFFu, lo[i][m] + (hi[i][m] >> 4)) - 8 * xsum[m];
        if (lane == m) {
          const size_t at = static_cast<size_t>(m) * N + n;
          if constexpr (S32 && RW == 2) {
            *reinterpret_cast<int2*>(static_cast<int32_t*>(out) + at) = make_int2(tot[0], tot[RW - 1]);
          } else if constexpr (S32) {
            static_cast<int32_t*>(out)[at] = tot[0];
          } else {
            float y[RW];
#pragma unroll
            for (int i = 0; i < RW; ++i) y[i] = __fmul_rn(__fmul_rn(static_cast<float>(tot[i]), s_a[m]), s_w[n + i]);
            if constexpr (RW == 2)
              *reinterpret_cast<__half2*>(static_cast<__half*>(out) + at) = __floats2half2_rn(y[0], y[RW - 1]);
            else
              static_cast<__half*>(out)[at] = __float2half_rn(y[0]);
          }
        }
      }
    }
  }
}

template <int MR, int RW, bool S32>
cudaError_t launch_mr(const GemmArgs& g, cudaStream_t stream) {
  const size_t smem = static_cast<size_t>(g.M) * g.K;
  static SmemLimit limit;
  const cudaError_t le = limit.allow(gemv_w4a4_kernel<MR, RW, S32>, kGemvSmemMax);
  if (le != cudaSuccess) return le;
  // enough warps for every RW weight rows, at most the CTAs that fit on the SMs
  const int per_sm = MR * RW > 8 ? 2 : kGemvCtas;
  const int want = (g.N / RW + kGemvWarps - 1) / kGemvWarps;
  const int blocks = want < per_sm * num_sms() ? want : per_sm * num_sms();
  // A grid that leaves SMs free lets the next kernel launch only after its own
  // wait: its CTAs would take those SMs and, where it is another linear, run
  // beside this one on some and alone on others (2 x 2048 x 4096 after another,
  // us: 3.8 early, 2.7 so; between quantizers no difference).
  return launch_pdl(gemv_w4a4_kernel<MR, RW, S32>, dim3(blocks), dim3(kGemvWarps * 32), smem, stream, g.A, g.s_a, g.M,
                    g.K, g.B, g.s_b, g.N, g.D, blocks > num_sms());
}

}  // namespace

// One or two rows always. Three to eight while the weights are small: above,
// the tensor-core kernel (p4q_fewrows.cu) is faster, which starts slower (3.7 -
// 8 us for weights of any size up to 4 MB) and hardly depends on the rows. The
// time here grows with the rows' staging and outputs and with the products; the
// line's two terms are fitted to 858 sizes (on average 0.8 % above the faster
// kernel), us here / there: 3 x 1024 x 1024 (N x K) 2.2 / 4.8, 8 x 1024 x 4096 5.0 /
// 5.3, 8 x 4096 x 1024 4.0 / 6.2, 4 x 4096 x 4096 6.7 / 6.8, 8 x 4096 x 4096 7.8 / 6.9, 3 x
// 2048 x 8192 4.8 / 7.5, 8 x 512 x 11008 9.6 / 7.0, 8 x 8192 x 512 5.8 / 6.1.
bool gemv_applies(const GemmArgs& g) {
  const long long m = g.M, mnk = m * g.N * g.K;
  if (g.M > 2 && (m * (g.K + g.N) > static_cast<long long>(kGemvSmemMax) || mnk > 5ll << 24)) return false;
  return (g.out == GemmOut::kHalf || g.out == GemmOut::kS32) && g.batch == 1 && g.M >= 1 && g.M <= kGemvMaxRows &&
         g.N % 2 == 0 && g.K % 32 == 0 && (g.d_pitch == 0 || g.d_pitch == g.N) &&
         static_cast<size_t>(g.M) * g.K <= kGemvSmemMax;
}

namespace {

template <int RW, bool S32>
cudaError_t launch_rows(const GemmArgs& g, cudaStream_t stream) {
  if (g.M <= 2) return launch_mr<2, RW, S32>(g, stream);
  if (g.M <= 4) return launch_mr<4, RW, S32>(g, stream);
  return launch_mr<8, RW, S32>(g, stream);
}

}  // namespace

// A weight row per warp while that leaves no SM two CTAs (us, one / two: 2 x 1024 x
// 4096 2.5 / 2.7, 2 x 2048 x 4096 3.1 / 2.7).
cudaError_t launch_gemv(const GemmArgs& g, cudaStream_t stream) {
  if (g.N <= kGemvWarps * num_sms())
    return g.out == GemmOut::kS32 ? launch_rows<1, true>(g, stream) : launch_rows<1, false>(g, stream);
  return g.out == GemmOut::kS32 ? launch_rows<2, true>(g, stream) : launch_rows<2, false>(g, stream);
}

}  // namespace p4q
