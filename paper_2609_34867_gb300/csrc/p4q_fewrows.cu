// W4A4 linear for few token rows (decode batches, the prefill of one pruned
// image): the exact integer products and the dequantization of the GEMMs
// (App. A / App. B.3: acc = sum_k a_k w_k over INT4 codes, y =
// fp16_rne((float(acc) * s_a) * s_w)) where the packed weights, read once,
// are most of the bytes.
//
// The weights are the M = 128 side of the MMAs and the activation rows the N
// side, so a few rows fill the tensor instruction, and the reduction over k
// is split over a cluster of up to 8 CTAs, so that a 4096-row weight matrix
// (32 row tiles) still occupies the whole GPU. Per CTA: 128 weight rows x its
// share of the 128-deep k-blocks,
//   all warps   first unpack the CTA's activation codes x to E4M3 bytes x + 8
//               (exactly (x + 8) * 2^-9) in shared memory, in the 128-byte-
//               swizzled layout the MMAs read, with their row sums, and one
//               more row of ones;
//   warp 0      loads the packed weights by TMA, 128 rows x 128 bytes (a pair
//               of k-blocks), into a ring of stages;
//   warps 2-9   unpack them: four lanes per weight row turn its 16-byte chunks
//               into E4M3 bytes u = w + 8 (exactly u * 2^-9) and store them to
//               TMEM;
//   warp 1      MMAs (tcgen05 kind::f8f6f4): A (weights) from TMEM, B
//               (activations) from shared memory, fp32 accumulator in TMEM.
// P = sum (x + 8) (w + 8) is exact in fp32 (at most 225 * 16384 < 2^22), the
// row of ones gives sum (w + 8) of each weight row in a column of its own, and
// acc = P - 8 sum (x + 8) - 8 sum (w + 8) + 64 K. The unpacked weights pass no
// shared memory. The partial sums of a cluster meet in shared memory: CTA r
// adds the cluster's partials (exact integers) of the activation rows r, r +
// S, ... and writes the outputs.
// Order of the codes of a k-block: the 16x256b TMEM store puts word w of
// lane c's 16-byte chunk (8 codes) into columns 8 w + 2 c (its low nibbles)
// and 8 w + 2 c + 1, so MMA step w (8 columns = 32 codes) takes word w of the
// four chunks; the activations are laid out in the same order.
// Bound: a CTA takes a pair of k-blocks in about 900 cycles (the chain
// barrier -> shared loads -> unpack -> TMEM store -> MMA, two CTAs per SM side
// by side) and 4 - 8 k cycles around them. Measured (CUDA graph of calls over
// distinct weights, us; before: the 256-column tiles of p4q_gemm.cu or, up to
// 8 rows, the dp4a stream): 96 x 4096 x 4096 29.6 -> 12.2, 24 x 5120 x 13824
// (N x K) 79 -> 20, 24 x 15360 x 5120 42 -> 21, 8 x 4096 x 11008 29.9 -> 10.7.
// Before it waits for the previous kernel of the stream, a CTA prefetches its
// weights into L2 (a prefetch changes no memory, so it may run ahead of a
// kernel that still writes them): the weight stream then runs beside the
// quantizer of the linear's input.
#include <cuda_fp16.h>

#include <algorithm>

#include "p4q_device.cuh"
#include "p4q_internal.h"

namespace p4q {

__device__ unsigned int g_fewrows_err;

namespace {

constexpr int kTileN = 128;     // weight rows per CTA (TMEM lanes)
constexpr int kBK = 128;        // codes per k-block
constexpr int kBKP = kBK / 2;   // packed bytes per row and k-block
constexpr int kUnpackWarps = 8;  // 16 weight rows each
constexpr int kThreads = 64 + kUnpackWarps * 32;
constexpr int kPairBytes = kTileN * 2 * kBKP;  // packed weights of a pair of k-blocks
constexpr int kMaxStages = 6;
constexpr int kMaxCluster = 8;
constexpr int kSmemMax = 231424;  // dynamic, beside 1 KB of barriers and sums
constexpr int kSmemTwo = 113664;  // dynamic (without the alignment slack) with two CTAs per SM

constexpr int kMaxRowTile = 127;   // activation rows of a tile: with the row of ones at most 128 columns of D
constexpr uint32_t kTmem = 256;    // TMEM columns: D (fp32) from 0, then the A stages; two CTAs per SM
constexpr uint32_t kStageCols = 64;  // an A stage: a pair of k-blocks, 4 codes per column
constexpr int kMaxConv = 3;

struct FewParams {
  const uint8_t* X;  // [M, K/2] packed
  const uint8_t* W;  // [N, K/2] packed
  const float* s_a;
  const float* s_w;
  void* out;
  int M, N, K, split;
  int mt;      // activation rows per tile
  int ncol;    // columns of D: mt + 1 rounded up to 16
  int xrows;   // rows per k-block of the unpacked activations: mt + 1 rounded up to 8
  int stages;  // of packed weights
  int col_a;   // first column of the A stages, and their number
  int conv;
};

// Shared memory: the ring of packed weights, then the unpacked activations
// [nkb][xrows][128] with slack for an MMA's rows past them (the partial sums
// float [mt][128] take their place afterwards).
constexpr int few_x_bytes(int mt, int ncol, int xrows, int nkb) {
  return std::max(kBK * (nkb * xrows + ncol - xrows), mt * kTileN * 4);
}

// 16 lanes (TMEM rows) x 64 columns: register 4 j + i of thread t is row
// t / 4 (+ 8 for i >= 2), column 8 j + 2 (t % 4) + (i & 1).
__device__ __forceinline__ void tmem_st_16x256b_x8(uint32_t taddr, const uint32_t (&r)[32]) {
  asm volatile(
      "tcgen05.st.sync.aligned.16x256b.x8.b32 [%0], "
      "{%1, %2, %3, %4, %5, %6, %7, %8, %9, %10, %11, %12, %13, %14, %15, %16, "
      "%17, %18, %19, %20, %21, %22, %23, %24, %25, %26, %27, %28, %29, %30, %31, %32};" ::"r"(taddr),
      "r"(r[0]), "r"(r[1]), "r"(r[2]), "r"(r[3]), "r"(r[4]), "r"(r[5]), "r"(r[6]), "r"(r[7]), "r"(r[8]),
      "r"(r[9]), "r"(r[10]), "r"(r[11]), "r"(r[12]), "r"(r[13]), "r"(r[14]), "r"(r[15]), "r"(r[16]), "r"(r[17]),
      "r"(r[18]), "r"(r[19]), "r"(r[20]), "r"(r[21]), "r"(r[22]), "r"(r[23]), "r"(r[24]), "r"(r[25]), "r"(r[26]),
      "r"(r[27]), "r"(r[28]), "r"(r[29]), "r"(r[30]), "r"(r[31])
      : "memory");
}

__device__ __forceinline__ void tmem_ld_32x32b_x1(uint32_t taddr, uint32_t& r) {
  asm volatile("tcgen05.ld.sync.aligned.32x32b.x1.b32 {%0}, [%1];" : "=r"(r) : "r"(taddr) : "memory");
}

__device__ __forceinline__ void tmem_st_wait() { asm volatile("tcgen05.wait::st.sync.aligned;" ::: "memory"); }

// A from TMEM (lanes = rows, four 8-bit values of K per column), B from shared memory.
__device__ __forceinline__ void mma_f8f6f4_ts(uint32_t d_tmem, uint32_t a_tmem, uint64_t b_desc, uint32_t idesc,
                                              uint32_t accumulate) {
  asm volatile(
      "{\n\t.reg .pred p;\n\t"
      "setp.ne.b32 p, %4, 0;\n\t"
      "tcgen05.mma.cta_group::1.kind::f8f6f4 [%0], [%1], %2, %3, p;\n\t}\n" ::"r"(d_tmem),
      "r"(a_tmem), "l"(b_desc), "r"(idesc), "r"(accumulate)
      : "memory");
}

__device__ __forceinline__ float2 ld_shared_cluster_f32x2(uint32_t cluster_saddr) {
  float2 v;
  asm volatile("ld.shared::cluster.v2.f32 {%0, %1}, [%2];" : "=f"(v.x), "=f"(v.y) : "r"(cluster_saddr) : "memory");
  return v;
}

// Offset codes u = v + 8 of the low / high nibbles of a packed word, one per byte.
__device__ __forceinline__ uint32_t u_lo(uint32_t w) { return (w ^ 0x88888888u) & 0x0F0F0F0Fu; }
__device__ __forceinline__ uint32_t u_hi(uint32_t w) { return ((w >> 4) ^ 0x08080808u) & 0x0F0F0F0Fu; }

template <bool S32>
__global__ void __launch_bounds__(kThreads, 2)
    w4a4_fewrows_kernel(const __grid_constant__ CUtensorMap tmW, const FewParams p) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  __shared__ __align__(8) uint64_t full[kMaxStages];  // TMA -> unpack
  __shared__ __align__(8) uint64_t empty[kMaxStages]; // unpack -> TMA
  __shared__ __align__(8) uint64_t conv_full[kMaxConv];   // unpack -> MMA
  __shared__ __align__(8) uint64_t conv_empty[kMaxConv];  // MMA -> unpack
  __shared__ __align__(8) uint64_t acc_full;          // MMA -> epilogue
  __shared__ uint32_t tmem_slot;
  __shared__ int abort_word;
  __shared__ int loads;                                // issued, for the give-up path
  __shared__ int sums[kMaxRowTile + 1];                // of x + 8, per activation row
  volatile int* abort_flag = &abort_word;

  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int rank = static_cast<int>(cluster_ctarank());
  const int n0 = static_cast<int>(blockIdx.x) / p.split * kTileN;
  const int m0 = static_cast<int>(blockIdx.y) * p.mt;
  const int KB = p.K / kBK;
  const int kb0 = KB * rank / p.split;             // this CTA's k-blocks
  const int nkb = KB * (rank + 1) / p.split - kb0;
  const int np = (nkb + 1) >> 1;                   // pairs of them
  const size_t pitch = static_cast<size_t>(p.K) >> 1;
  uint8_t* xs = smem + p.stages * kPairBytes;

  if (threadIdx.x == 0) {
    for (int i = 0; i < p.stages; ++i) {
      mbar_init(&full[i], 1);
      mbar_init(&empty[i], kUnpackWarps);
    }
    for (int i = 0; i < p.conv; ++i) {
      mbar_init(&conv_full[i], kUnpackWarps);
      mbar_init(&conv_empty[i], 1);
    }
    mbar_init(&acc_full, 1);
    abort_word = 0;
    fence_barrier_init();
    tma_prefetch_desc(&tmW);
  }
  if (warp == 1) {
    tmem_alloc(&tmem_slot, kTmem);
    tmem_relinquish();
  }
  if (threadIdx.x >= kThreads - kTileN) {  // one thread per weight row: its bytes of this CTA's k-blocks
    const int n = n0 + static_cast<int>(threadIdx.x) - (kThreads - kTileN);
    if (n < p.N)
      prefetch_l2_bulk(p.W + static_cast<size_t>(n) * pitch + static_cast<size_t>(kb0) * kBKP,
                       static_cast<uint32_t>(nkb) * kBKP);
  }
  if (threadIdx.x <= kMaxRowTile) sums[threadIdx.x] = 0;
  // This CTA holds its TMEM before the next kernel's CTAs may come to the SM
  // (they would wait for this grid while holding TMEM it still needs).
  __syncthreads();
  pdl_launch_dependents();
  pdl_wait();

  int issued = 0;  // warp 0, lane 0: loads in flight or done
  if (threadIdx.x == 0) {
    for (; issued < min(np, p.stages); ++issued) {
      mbar_arrive_expect_tx(&full[issued], kPairBytes);
      tma_load_3d(&tmW, &full[issued], smem + issued * kPairBytes, (kb0 + 2 * issued) * kBKP, n0, 0);
    }
  }
  // Activations: task i = 16-byte chunk (32 codes) c of row m of k-block kb, c
  // fastest, then m (so that a warp's stores fall into different banks). Rows
  // past M are left as they are: they reach only accumulator columns that
  // nobody reads.
  const int rows = min(p.mt, p.M - m0);
  {
    const uint32_t inv = 0xFFFFFFFFu / static_cast<uint32_t>(rows) + 1u;  // a / rows = umulhi(a, inv), a < 2^16
    const uint8_t* xp = p.X + static_cast<size_t>(m0) * pitch + static_cast<size_t>(kb0) * kBKP;
    const int tasks = rows * nkb * 4, c = lane & 3;
    constexpr int kXU = 4;  // chunks per thread in flight
    for (int i0 = threadIdx.x; i0 - lane < tasks; i0 += kXU * kThreads) {
      uint4 x[kXU];
      int kb[kXU], m[kXU];
#pragma unroll
      for (int j = 0; j < kXU; ++j) {
        const int i = i0 + j * kThreads;
        kb[j] = rows == 1 ? i >> 2 : static_cast<int>(__umulhi(static_cast<uint32_t>(i >> 2), inv));
        m[j] = (i >> 2) - kb[j] * rows;
        if (i < tasks)
          x[j] = *reinterpret_cast<const uint4*>(xp + static_cast<size_t>(m[j]) * pitch + kBKP * kb[j] + 16 * c);
      }
#pragma unroll
      for (int j = 0; j < kXU; ++j) {
        const int i = i0 + j * kThreads;
        if (i - lane >= tasks) break;
        const bool in = i < tasks;
        uint32_t t = 0;
        if (in) {
          const uint32_t pw[4] = {x[j].x, x[j].y, x[j].z, x[j].w};
          uint8_t* row = xs + (kb[j] * p.xrows + m[j]) * kBK + 8 * (c & 1);
#pragma unroll
          for (int w = 0; w < 4; ++w) {
            const uint32_t lo = u_lo(pw[w]), hi = u_hi(pw[w]);
            t += lo + hi;  // byte-wise, at most 8 x 15
            // logical byte 32 w + 8 c of the 128-byte row: 16-byte chunk 2 w + (c >> 1)
            *reinterpret_cast<uint2*>(row + (((2 * w + (c >> 1)) ^ (m[j] & 7)) << 4)) = make_uint2(lo, hi);
          }
        }
        t = __dp4a(t, 0x01010101u, 0u);
        t += __shfl_xor_sync(0xFFFFFFFFu, t, 1);  // the four chunks of a k-block's row
        t += __shfl_xor_sync(0xFFFFFFFFu, t, 2);
        if (in && c == 0) atomicAdd(&sums[m[j]], static_cast<int>(t));
      }
    }
  }
  for (int i = threadIdx.x; i < nkb * 8; i += kThreads)  // the row of ones (the E4M3 byte 1 = 2^-9)
    *reinterpret_cast<uint4*>(xs + ((i >> 3) * p.xrows + rows) * kBK + 16 * (i & 7)) =
        make_uint4(0x01010101u, 0x01010101u, 0x01010101u, 0x01010101u);
  fence_proxy_async_smem();
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = tmem_slot;

  if (warp == 0) {
    // ------------------------------------------------------------ packed weights by TMA
    if (lane == 0) {
      int s = 0, ph = 0;
      for (; issued < np; ++issued) {
        if (!mbar_wait_spin(&empty[s], ph, abort_flag, &g_fewrows_err)) break;
        mbar_arrive_expect_tx(&full[s], kPairBytes);
        tma_load_3d(&tmW, &full[s], smem + s * kPairBytes, (kb0 + 2 * issued) * kBKP, n0, 0);
        if (++s == p.stages) {
          s = 0;
          ph ^= 1;
        }
      }
      loads = issued;
    }
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMAs
    // The whole warp runs the loop (its operands stay in uniform registers),
    // one elected thread issues.
    const uint32_t idesc = idesc_e4m3_f32(kTileN, p.ncol);
    const uint32_t kbu = static_cast<uint32_t>(p.xrows) * (kBK / 16);  // a k-block's activations, in 16-byte units
    const bool leader = elect_one();
    bool ok = true;
    uint64_t bd = sw128_kmajor_desc(smem_u32(xs));  // this pair's activations (16-byte units in the low bits)
    for (int g = 0, c = 0, ph = 0; g < np; ++g, bd += 2 * kbu) {
      if (!(ok = mbar_wait_all(&conv_full[c], ph, abort_flag, &g_fewrows_err))) break;
      tc_fence_after();
      const uint32_t a0 = tmem + p.col_a + kStageCols * static_cast<uint32_t>(c);
      const bool both = 2 * g + 1 < nkb;
      if (leader) {
#pragma unroll
        for (int k = 0; k < kBK / 32; ++k)
          mma_f8f6f4_ts(tmem, a0 + 8u * k, bd + 2 * k, idesc, (g | k) != 0 ? 1u : 0u);
        if (both) {
#pragma unroll
          for (int k = 0; k < kBK / 32; ++k)
            mma_f8f6f4_ts(tmem, a0 + 32u + 8u * k, bd + kbu + 2 * k, idesc, 1u);
        }
        mma_commit(&conv_empty[c]);
      }
      if (++c == p.conv) {
        c = 0;
        ph ^= 1;
      }
    }
    // every MMA of this CTA completes before the accumulator is read (or TMEM released)
    if (leader) mma_commit(&acc_full);
    if (!ok && leader) {
      volatile int never = 0;
      mbar_wait(&acc_full, 0, &never, &g_fewrows_err, 100000000ull);
    }
  } else {
    // ------------------------------------------------------------ unpack
    const int quad = warp & 3, sub = (warp - 2) >> 2;  // TMEM lanes 32 quad + 16 sub .. + 15 of this warp
    const int r = 32 * quad + 16 * sub + (lane >> 2);  // weight rows r and r + 8 of the tile
    const uint32_t ta = tmem + (static_cast<uint32_t>(32 * quad + 16 * sub) << 16) + p.col_a;
    bool ok = true;
    uint4 v[4];  // chunks (lane & 3) of row r, row r + 8 (first k-block), then of the second k-block
    auto load = [&](int s, int ph) -> bool {
      if (!mbar_wait_all(&full[s], ph, abort_flag, &g_fewrows_err)) return false;
      const uint8_t* w = smem + s * kPairBytes + r * (2 * kBKP);  // 128-byte rows, 128-byte swizzle
#pragma unroll
      for (int i = 0; i < 4; ++i)
        v[i] = *reinterpret_cast<const uint4*>(w + (i & 1) * (16 * kBKP) +
                                               (((static_cast<uint32_t>(lane) & 3u) + 4 * (i >> 1)) ^ (r & 7)) * 16);
      return true;
    };
    int s = 0, ph = 0, st = 0, use = 0;
    ok = load(s, ph);
    for (int g = 0; g < np && ok; ++g) {
      uint32_t u[32];
#pragma unroll
      for (int h = 0; h < 2; ++h) {
        const uint32_t a[4] = {v[2 * h].x, v[2 * h].y, v[2 * h].z, v[2 * h].w};
        const uint32_t b[4] = {v[2 * h + 1].x, v[2 * h + 1].y, v[2 * h + 1].z, v[2 * h + 1].w};
#pragma unroll
        for (int w = 0; w < 4; ++w) {
          u[16 * h + 4 * w] = u_lo(a[w]);
          u[16 * h + 4 * w + 1] = u_hi(a[w]);
          u[16 * h + 4 * w + 2] = u_lo(b[w]);
          u[16 * h + 4 * w + 3] = u_hi(b[w]);
        }
      }
      __syncwarp();
      if (lane == 0) mbar_arrive(&empty[s]);
      if (++s == p.stages) {
        s = 0;
        ph ^= 1;
      }
      if (use > 0) {
        if (!(ok = mbar_wait_all(&conv_empty[st], (use - 1) & 1, abort_flag, &g_fewrows_err))) break;
        tc_fence_after();
      }
      tmem_st_16x256b_x8(ta + kStageCols * static_cast<uint32_t>(st), u);
      if (g + 1 < np && !(ok = load(s, ph))) break;  // the next pair on its way under the store
      tmem_st_wait();
      tc_fence_before();
      __syncwarp();
      if (lane == 0) mbar_arrive(&conv_full[st]);
      if (++st == p.conv) {
        st = 0;
        ++use;
      }
    }
    if (ok) ok = mbar_wait_all(&acc_full, 0, abort_flag, &g_fewrows_err);
    else tmem_st_wait();  // given up: no store in flight when TMEM is released
    tc_fence_after();
    // this CTA's partial accumulators (exact integers) as [MP][128] floats in
    // place of the activations (every MMA that read them is complete)
    float* part = reinterpret_cast<float*>(xs);
    const uint32_t td = tmem + (static_cast<uint32_t>(quad * 32) << 16);
    if (ok) {
      // P - 8 sum (x + 8) - 8 sum (w + 8) + 64 K': integers below 2^24, exact
      uint32_t ones;
      tmem_ld_32x32b_x1(td + rows, ones);
      tmem_ld_wait();
      const float corr_w = __fmaf_rn(__uint_as_float(ones), -8.0f * 262144.0f, static_cast<float>(64 * nkb * kBK));
#pragma unroll 1
      for (int c0 = sub * 16; c0 < rows; c0 += 32) {
        uint32_t d[16];
        tmem_ld_32x32b_x16(td + c0, d);
        tmem_ld_wait();
#pragma unroll
        for (int i = 0; i < 16; ++i) {
          if (c0 + i < rows) {
            const float corr = corr_w - static_cast<float>(8 * sums[c0 + i]);
            part[(c0 + i) * kTileN + quad * 32 + lane] = __fmaf_rn(__uint_as_float(d[i]), 262144.0f, corr);
          }
        }
      }
    }
  }
  __syncwarp();
  tc_fence_before();
  if (p.split > 1) cluster_sync();
  else __syncthreads();
  if (warp > 1) {
    // ------------------------------------------------------------ sums over the cluster, dequantization
    const int t = static_cast<int>(threadIdx.x) - 64;
    const int n = n0 + 2 * (t & 63);
    const bool in = n < p.N;  // N is even
    float2 sw = make_float2(0.0f, 0.0f);
    if (!S32 && in) sw = make_float2(p.s_w[n], p.s_w[n + 1]);
    const uint32_t part = smem_u32(xs) + 8u * static_cast<uint32_t>(t & 63);
    for (int m = rank + p.split * (t >> 6); m < rows; m += 4 * p.split) {
      const float sa = S32 ? 0.0f : p.s_a[m0 + m];
      float2 v[kMaxCluster];
#pragma unroll
      for (int q = 0; q < kMaxCluster; ++q)
        v[q] = q < p.split ? ld_shared_cluster_f32x2(mapa_shared(part + static_cast<uint32_t>(m) * (kTileN * 4), q))
                           : make_float2(0.0f, 0.0f);
      float2 a = v[0];
#pragma unroll
      for (int q = 1; q < kMaxCluster; ++q) {
        a.x += v[q].x;
        a.y += v[q].y;
      }
      if (in && !*abort_flag) {
        const size_t at = static_cast<size_t>(m0 + m) * p.N + n;
        if (S32)
          *reinterpret_cast<int2*>(static_cast<int32_t*>(p.out) + at) =
              make_int2(__float2int_rn(a.x), __float2int_rn(a.y));
        else
          *reinterpret_cast<__half2*>(static_cast<__half*>(p.out) + at) =
              __floats2half2_rn(__fmul_rn(__fmul_rn(a.x, sa), sw.x), __fmul_rn(__fmul_rn(a.y, sa), sw.y));
      }
    }
  }
  if (p.split > 1) cluster_sync();  // no CTA leaves while its partials are read
  else __syncthreads();
  if (threadIdx.x == 0 && *abort_flag) {
    // given up (whichever warp did): leave no TMA load in flight into this CTA's shared memory
    int fresh = 0;
    for (int j = (loads > p.stages ? loads - p.stages : 0); j < loads; ++j)
      mbar_wait(&full[j % p.stages], (j / p.stages) & 1, reinterpret_cast<volatile int*>(&fresh), &g_fewrows_err,
                100000000ull);
  }
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmem);
  }
}

// 3-D map over packed rows: dims (K/2 bytes, rows), boxes of a pair of
// k-blocks (128 bytes) x 128 rows, 128-byte swizzle.
bool make_packed_map(CUtensorMap* map, const uint8_t* base, int K, int rows) {
  auto enc = get_encode_fn();
  if (!enc) return false;
  const cuuint64_t kb = static_cast<cuuint64_t>(K / 2);
  cuuint64_t dims[3] = {kb, static_cast<cuuint64_t>(rows), 1};
  cuuint64_t strides[2] = {kb, kb * static_cast<cuuint64_t>(rows)};
  cuuint32_t box[3] = {2 * kBKP, kTileN, 1};
  cuuint32_t estr[3] = {1, 1, 1};
  return enc(map, CU_TENSOR_MAP_DATA_TYPE_UINT8, 3, const_cast<uint8_t*>(base), dims, strides, box, estr,
             CU_TENSOR_MAP_INTERLEAVE_NONE, CU_TENSOR_MAP_SWIZZLE_128B, CU_TENSOR_MAP_L2_PROMOTION_L2_256B,
             CU_TENSOR_MAP_FLOAT_OOB_FILL_NONE) == CUDA_SUCCESS;
}

template <bool S32>
cudaError_t launch_out(const GemmArgs& g, cudaStream_t stream) {
  static SmemLimit limit;
  const cudaError_t le = limit.allow(w4a4_fewrows_kernel<S32>, kSmemMax);
  if (le != cudaSuccess) return le;
  const int KB = g.K / kBK;
  FewParams p;
  p.X = g.A;
  p.W = g.B;
  p.s_a = g.s_a;
  p.s_w = g.s_b;
  p.out = g.D;
  p.M = g.M;
  p.N = g.N;
  p.K = g.K;
  int mtiles = (g.M + kMaxRowTile - 1) / kMaxRowTile;
  const int ntiles = (g.N + kTileN - 1) / kTileN;
  // Split of k: as many CTAs as SMs (3 .. 16 x 4096 x 4096: 10.7 us at 1, 7.0
  // at 4, 6.6 at 8), no further, as the start and the sums over the cluster
  // cost a CTA about as much as six pairs of k-blocks (22016 x 4096: 17 us at
  // 1 and 2, 21 at 4) ...
  int split = 1;
  while (split < kMaxCluster && 2 * split <= KB && ntiles * mtiles * split < num_sms()) split *= 2;
  // ... and, where its activations and two stages leave no room for a second
  // CTA on the SM, more (24 x 5120 x 13824: 28.4 -> 20.0 us at 8 instead of 4).
  int nkb, xb;
  while (true) {
    p.mt = (g.M + mtiles - 1) / mtiles;
    p.ncol = (p.mt + 16) / 16 * 16;
    p.xrows = (p.mt + 8) / 8 * 8;
    nkb = (KB + split - 1) / split;
    xb = few_x_bytes(p.mt, p.ncol, p.xrows, nkb);
    const bool grow = split < kMaxCluster && 2 * split <= KB;
    if (xb + 2 * kPairBytes <= kSmemTwo || (!grow && 1024 + xb + 2 * kPairBytes <= kSmemMax)) break;
    if (grow) split *= 2;
    else ++mtiles;
  }
  p.split = split;
  // ring: every pair of the CTA if two CTAs still fit an SM, at least two pairs
  p.stages = std::max(2, std::min(std::min(kMaxStages, (nkb + 1) / 2), (kSmemTwo - xb) / kPairBytes));
  p.col_a = p.ncol <= 64 ? 64 : 128;
  p.conv = (static_cast<int>(kTmem) - p.col_a) / static_cast<int>(kStageCols);
  CUtensorMap mw;
  if (!make_packed_map(&mw, g.B, g.K, g.N)) return cudaErrorInvalidValue;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(ntiles * split), static_cast<unsigned>((g.M + p.mt - 1) / p.mt));
  cfg.blockDim = dim3(kThreads);
  cfg.dynamicSmemBytes = static_cast<size_t>(1024 + xb + p.stages * kPairBytes);
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = static_cast<unsigned>(split);
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = 2;
  return cudaLaunchKernelEx(&cfg, w4a4_fewrows_kernel<S32>, mw, p);
}

}  // namespace

// Up to 128 rows, and fewer for more weight rows: every CTA unpacks its share
// of the activations, and with M * ceil(N / 128) past 8192 that costs more
// than the in-kernel unpack of p4q_gemm.cu on 256-row weight tiles (measured,
// us, this kernel / that one: 64 x 12288 x 4096 21.7 / 26.0, 64 x 22016 x 4096
// 34.2 / 29.6, 96 x 12288 x 4096 35.0 / 25.9, 128 x 4096 x 4096 13.3 / 25.4).
// Past K = 8192 only where the activations are one row tile of the CTA's shared
// memory: a second tile reads the weights again, against that file's CTA pairs
// (128 x 5120 x 5120 27.9 / 29.3, 96 x 5120 x 13824 45.3 / 62.2, 128 x 4096 x
// 11008 56.2 / 51.5, 128 x 5120 x 13824 74.6 / 62.2).
// Its int32 outputs have no pairs there: a second tile while the CTAs are at most
// three rounds (128 x 2048 x 11008 32.3 / 50.9, 128 x 5120 x 8320 59.1 / 40.0).
// Short rows: the unpacking, sums and outputs of a row tile cost this kernel more
// per row than that file's, whose time is that of its k loop (64 x 256 x 128 8.1 /
// 5.4, 32 x 256 x 256 5.6 / 6.0, 48 x 256 x 256 6.7 / 6.0, 64 x 256 x 512 6.3 / 7.0, 96 x
// 256 x 512 7.8 / 7.0; fp16 outputs from N = 1024, where that file takes wider tiles:
// 48 x 1024 x 128 7.2 / 7.4, 64 x 1024 x 256 7.6 / 8.3, 80 x 1024 x 256 8.9 / 8.4, 96 x 1024 x
// 512 8.0 / 9.7).
bool fewrows_applies(const GemmArgs& g) {
  const int nkb = (g.K / kBK + kMaxCluster - 1) / kMaxCluster;
  const bool one_tile = g.M <= kMaxRowTile && 1024 + few_x_bytes(g.M, (g.M + 16) / 16 * 16, (g.M + 8) / 8 * 8, nkb) +
                                                      2 * kPairBytes <= kSmemMax;
  const bool pairs_serve = g.out == GemmOut::kHalf && g.N >= 1024 && (g.N + 255) / 256 <= num_sms() / 2;
  const long long ntiles = (g.N + kTileN - 1) / kTileN;
  const bool second_tile = g.out == GemmOut::kHalf ? !pairs_serve : 2 * kMaxCluster * ntiles <= 3 * num_sms();
  const int mt = g.M <= kMaxRowTile ? g.M : (g.M + 1) / 2;
  const int rows = std::max(24, g.K / 8) + (g.out == GemmOut::kHalf && g.N >= 1024 ? 32 : 0);
  return (g.out == GemmOut::kHalf || g.out == GemmOut::kS32) && g.batch == 1 && g.M >= 1 && g.M <= 128 &&
         g.M * ntiles <= (g.K >= 512 ? 8192 : 6144) && (g.K >= 1024 || mt <= rows) && g.N % 2 == 0 && g.K % kBK == 0 &&
         (g.d_pitch == 0 || g.d_pitch == g.N) && (g.K <= 8192 || one_tile || second_tile);
}

cudaError_t launch_fewrows(const GemmArgs& g, cudaStream_t stream) {
  return g.out == GemmOut::kS32 ? launch_out<true>(g, stream) : launch_out<false>(g, stream);
}

unsigned int fewrows_read_and_clear_error() {
  unsigned int v = 0, z = 0;
  cudaMemcpyFromSymbol(&v, g_fewrows_err, sizeof(v));
  cudaMemcpyToSymbol(g_fewrows_err, &z, sizeof(z));
  return v;
}

}  // namespace p4q
