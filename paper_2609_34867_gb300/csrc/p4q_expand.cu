// Expansion of packed INT4 codes to one byte per code (u = v + 8, the E4M3
// byte the FP8 MMAs read exactly as u * 2^-9) with the per-row sums of u:
// the operands of the expanded-operand GEMM (p4q_gemm8.cu), both of them in
// one launch. HBM-bound streaming kernel: bytes per row K/2 in, K + 4 out.
// 11008 + 2048 rows of 4096 codes (80 MB): two launches with 16-byte stores and
// no prefetch 19 us; one launch 12.5, part of it beside the quantizer whose time
// the prefetch fills (quantizer + linear together 89.2 -> 75.2 us).
#include "p4q_device.cuh"
#include "p4q_internal.h"

namespace p4q {
namespace {

struct ExpandOperand {
  const uint8_t* src;
  uint8_t* dst;
  int32_t* sums;
  int rows;
};

__device__ __forceinline__ void st_global32(void* p, const uint4& a, const uint4& b) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};" ::"l"(p), "r"(a.x), "r"(a.y), "r"(a.z),
               "r"(a.w), "r"(b.x), "r"(b.y), "r"(b.z), "r"(b.w)
               : "memory");
}

// One warp per row, the rows of first, then of second: packed codes [rows,
// K/2] -> one byte per code u = v + 8 [rows, K] (per packed 32-bit word: its
// four low-nibble codes, then its four high-nibble codes) and sum_u[row]. All
// of a lane's 16-byte loads of the row are issued before the first store (MAXC
// chunks per lane). WIDE (32-byte aligned outputs): a chunk's 32 bytes in one
// store, so that no sector is written in halves. Before it waits for the
// previous kernel of the stream, a warp prefetches a row of first (the GEMM's
// weights) into L2: a prefetch changes no memory, so it may run ahead of a
// kernel that still writes them.
template <int MAXC, bool WIDE>
__global__ void __launch_bounds__(256) expand_codes_kernel(const ExpandOperand first, const ExpandOperand second,
                                                           int K) {
  int row = blockIdx.x * 8 + (threadIdx.x >> 5);
  const int lane = threadIdx.x & 31;
  const bool is1 = row < first.rows;
  if (!is1) row -= first.rows;
  const uint8_t* src = (is1 ? first.src : second.src) + static_cast<size_t>(row) * (K >> 1);
  if (is1 && lane == 0) prefetch_l2_bulk(src, static_cast<uint32_t>(K) >> 1);
  pdl_wait();
  pdl_launch_dependents();
  if (row >= (is1 ? first.rows : second.rows)) return;
  const uint4* s4 = reinterpret_cast<const uint4*>(src);
  uint4* d4 = reinterpret_cast<uint4*>((is1 ? first.dst : second.dst) + static_cast<size_t>(row) * K);
  const int nch = K >> 5;  // 16-byte packed chunks per row
  uint4 w[MAXC];
#pragma unroll
  for (int i = 0; i < MAXC; ++i) {
    const int c = lane + 32 * i;
    if (c < nch) w[i] = ldg_stream16(s4 + c);
  }
  constexpr uint32_t ones = 0x01010101u;
  uint32_t acc = 0;
#pragma unroll
  for (int i = 0; i < MAXC; ++i) {
    const int c = lane + 32 * i;
    if (c < nch) {
      const uint32_t l0 = (w[i].x & 0x0F0F0F0Fu) ^ 0x08080808u, h0 = ((w[i].x >> 4) & 0x0F0F0F0Fu) ^ 0x08080808u;
      const uint32_t l1 = (w[i].y & 0x0F0F0F0Fu) ^ 0x08080808u, h1 = ((w[i].y >> 4) & 0x0F0F0F0Fu) ^ 0x08080808u;
      const uint32_t l2 = (w[i].z & 0x0F0F0F0Fu) ^ 0x08080808u, h2 = ((w[i].z >> 4) & 0x0F0F0F0Fu) ^ 0x08080808u;
      const uint32_t l3 = (w[i].w & 0x0F0F0F0Fu) ^ 0x08080808u, h3 = ((w[i].w >> 4) & 0x0F0F0F0Fu) ^ 0x08080808u;
      if (WIDE) {
        st_global32(d4 + 2 * c, make_uint4(l0, h0, l1, h1), make_uint4(l2, h2, l3, h3));
      } else {
        d4[2 * c] = make_uint4(l0, h0, l1, h1);
        d4[2 * c + 1] = make_uint4(l2, h2, l3, h3);
      }
      // byte-wise sum of the eight words first (each byte <= 8 x 15 < 256), then one dp4a
      acc = __dp4a(l0 + h0 + l1 + h1 + l2 + h2 + l3 + h3, ones, acc);
    }
  }
  acc = __reduce_add_sync(0xFFFFFFFFu, acc);
  if (lane == 0) (is1 ? first.sums : second.sums)[row] = static_cast<int32_t>(acc);
}

template <bool WIDE>
cudaError_t launch_expand(const ExpandOperand& a, const ExpandOperand& b, int K, cudaStream_t stream) {
  const dim3 grid((static_cast<long long>(a.rows) + b.rows + 7) / 8), block(256);
  const int nch = K >> 5;
  if (nch <= 32 * 4) return launch_pdl_l1(expand_codes_kernel<4, WIDE>, grid, block, 0, 0, stream, a, b, K);
  if (nch <= 32 * 8) return launch_pdl_l1(expand_codes_kernel<8, WIDE>, grid, block, 0, 0, stream, a, b, K);
  return launch_pdl_l1(expand_codes_kernel<16, WIDE>, grid, block, 0, 0, stream, a, b, K);
}

}  // namespace

cudaError_t launch_expand_codes(const uint8_t* q, int rows, int K, uint8_t* u, int32_t* sum_u, const uint8_t* q2,
                                int rows2, uint8_t* u2, int32_t* sum_u2, cudaStream_t stream) {
  if (rows <= 0 && rows2 <= 0) return cudaSuccess;
  const ExpandOperand a{q, u, sum_u, rows}, b{q2, u2, sum_u2, rows2};
  const uintptr_t at = reinterpret_cast<uintptr_t>(u) | reinterpret_cast<uintptr_t>(u2);  // K is a multiple of 32
  return at % 32 == 0 ? launch_expand<true>(a, b, K, stream) : launch_expand<false>(a, b, K, stream);
}

}  // namespace p4q
