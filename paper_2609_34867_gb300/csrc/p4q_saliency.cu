// CLS-to-patch saliency A_cls (Sec. 3.2 of the paper, Visual Saliency): in
// the vision tower's final self-attention layer each crop's [CLS] token is
// the query; its attention row is the softmax, over the CLS key and the
// crop's patch keys, of q . k / sqrt(d_h), and the saliency of a patch is its
// weight averaged over the heads.
//
// Kernel: one CTA per (image, crop) or, where that leaves SMs idle, a cluster of
// up to 8, its heads dealt out to the CTAs and each head's tokens to the CTA's
// warps. A token's key row for the head (dh fp16 values, rows of consecutive
// tokens H x dh apart) is read by dh / 8 lanes with one 16-byte load each, so
// that a warp load covers whole rows; the lanes' partial dot products (fp16
// products accumulated in fp32) are summed by shuffles. The head's max and sum
// (over its warps, in warp order) give its softmax; the per-head weights stay in
// the CTA's shared memory, and each CTA sums its share of the tokens over the
// heads in head order, reading the other CTAs' weights through distributed
// shared memory (deterministic for a given shape).
//
// Bound: load latency for few crops, HBM for many. Measured (16 heads x 64, us;
// one CTA per crop and one warp per head before): 8 crops of 576 tokens 8.2
// (24.3), 32 crops 13.7 (31.9), 80 crops 29.1 (29.9), 160 crops 44.3 (47.4) =
// 4.2 TB/s, 4 crops of 3600 at 128 wide 66 (390).
#include <cuda_fp16.h>

#include "p4q.h"
#include "p4q_device.cuh"
#include "p4q_internal.h"

namespace p4q {
namespace {

constexpr int kWarps = 16;
constexpr int kMaxHeads = 32;
constexpr int kMaxCluster = 8;
constexpr size_t kSmemMax = 227u * 1024u - 256u;  // dynamic, beside the reductions

// Lanes that share one token's key row: the row's dh / 8 16-byte chunks, one
// per lane, rounded up to a power of two (idle lanes past the row).
template <int DH>
constexpr int lanes_per_token() {
  return DH / 8 <= 4 ? 4 : DH / 8 <= 8 ? 8 : DH / 8 <= 16 ? 16 : 32;
}

// Heads of CTA `rank` of a cluster of cs: h = rank + cs * i, i = 0 .. heads - 1.
__device__ __forceinline__ int heads_of(int H, int cs, int rank) { return (H - rank + cs - 1) / cs; }

__device__ __forceinline__ float ld_shared_cluster_f32(uint32_t cluster_saddr) {
  float v;
  asm volatile("ld.shared::cluster.f32 %0, [%1];" : "=f"(v) : "r"(cluster_saddr) : "memory");
  return v;
}

// wph warps per head (a power of two); the CTA's heads in rounds of its warps / wph.
template <int DH, bool ONE>
__global__ void __launch_bounds__(32 * kWarps, 2)
    cls_saliency_kernel(const __half* q_cls, const __half* k_cls, const __half* k, int N, int C, int H, int cs_,
                        int wph_, float* A) {
  // ONE: one CTA per crop, one warp per head
  const int cs = ONE ? 1 : cs_, wph = ONE ? 1 : wph_;
  pdl_wait();
  pdl_launch_dependents();
  constexpr int R = DH / 8;                  // 16-byte chunks per key row
  constexpr int LPT = lanes_per_token<DH>();  // lanes per token
  constexpr int CPL = (R + LPT - 1) / LPT;    // chunks per lane
  constexpr int TPI = 32 / LPT;               // tokens per warp iteration
  extern __shared__ float p[];  // [heads of this CTA][n] softmax weights of the crop's patches
  __shared__ float red[2][kWarps];  // per warp: max, then sum
  const int c = blockIdx.x / cs, rank = blockIdx.x - c * cs;
  const int b = blockIdx.y, n = N / C;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int sub = lane % LPT, tok = lane / LPT;
  const int mine = heads_of(H, cs, rank);
  const int hpr = static_cast<int>(blockDim.x >> 5) / wph;  // heads per round
  const int part = warp % wph;               // this warp's part of the head's tokens
  const int per = (n + wph - 1) / wph, t0 = part * per, t1 = min(n, t0 + per);
  const float scale = 1.0f / sqrtf(static_cast<float>(DH));
  for (int i0h = 0; i0h < mine; i0h += hpr) {
    const int ih = i0h + warp / wph;         // the CTA's head index
    const bool live = ih < mine;
    const int h = rank + cs * (live ? ih : 0);
    const size_t head = (static_cast<size_t>(b) * C + c) * H + h;
    // this lane's chunks of the query, as fp32
    float qf[CPL][8];
    const uint4* q4 = reinterpret_cast<const uint4*>(q_cls + head * DH);
#pragma unroll
    for (int u = 0; u < CPL; ++u) {
      const int ch = sub + u * LPT;
      const uint4 v = ch < R ? q4[ch] : make_uint4(0u, 0u, 0u, 0u);
      const uint32_t w[4] = {v.x, v.y, v.z, v.w};
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[e]));
        qf[u][2 * e] = f.x;
        qf[u][2 * e + 1] = f.y;
      }
    }
    // this lane's chunks of a key row (zeros past the row or for no token)
    auto load = [&](const uint4* row, bool in, uint4 (&v)[CPL]) {
#pragma unroll
      for (int u = 0; u < CPL; ++u) {
        const int ch = sub + u * LPT;
        v[u] = (in && ch < R) ? ldg_stream16(row + ch) : make_uint4(0u, 0u, 0u, 0u);
      }
    };
    // partial dot of the loaded chunks, then the sum over the token's lanes
    auto dot = [&](const uint4 (&v)[CPL]) {
      float acc = 0.0f;
#pragma unroll
      for (int u = 0; u < CPL; ++u) {
        const uint32_t w[4] = {v[u].x, v[u].y, v[u].z, v[u].w};
#pragma unroll
        for (int e = 0; e < 4; ++e) {
          const float2 f = __half22float2(*reinterpret_cast<const __half2*>(&w[e]));
          acc = fmaf(qf[u][2 * e], f.x, acc);
          acc = fmaf(qf[u][2 * e + 1], f.y, acc);
        }
      }
#pragma unroll
      for (int o = LPT / 2; o > 0; o >>= 1) acc += __shfl_xor_sync(0xFFFFFFFFu, acc, o);
      return acc;
    };
    uint4 v0[CPL];
    load(reinterpret_cast<const uint4*>(k_cls + head * DH), true, v0);
    const float l0 = dot(v0) * scale;
    float mx = l0;
    float* ph = p + static_cast<size_t>(live ? ih : 0) * n;
    constexpr int U = ONE ? 8 : 4;  // token rows in flight per lane (several warps per head: 4 keeps 64 registers)
    for (int i0 = t0; i0 < t1; i0 += TPI * U) {
      uint4 v[U][CPL];
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * TPI + tok;
        const bool in = live && i < t1;
        const size_t row = (static_cast<size_t>(b) * N + static_cast<size_t>(c) * n + (in ? i : 0)) * H + h;
        load(reinterpret_cast<const uint4*>(k + row * DH), in, v[u]);
      }
#pragma unroll
      for (int u = 0; u < U; ++u) {
        const int i = i0 + u * TPI + tok;
        const float l = dot(v[u]) * scale;
        if (live && i < t1) {
          if (sub == 0) ph[i] = l;
          mx = fmaxf(mx, l);
        }
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) mx = fmaxf(mx, __shfl_xor_sync(0xFFFFFFFFu, mx, o));
    if (wph > 1) {
      if (lane == 0) red[0][warp] = mx;
      __syncthreads();
      for (int w = warp - part; w < warp - part + wph; ++w) mx = fmaxf(mx, red[0][w]);
    } else {
      __syncwarp();
    }
    float z = (lane == 0 && part == 0) ? expf(l0 - mx) : 0.0f;
    if (live) {
      for (int i = t0 + lane; i < t1; i += 32) {
        const float e = expf(ph[i] - mx);
        ph[i] = e;
        z += e;
      }
    }
#pragma unroll
    for (int o = 16; o > 0; o >>= 1) z += __shfl_xor_sync(0xFFFFFFFFu, z, o);
    if (wph > 1) {
      if (lane == 0) red[1][warp] = z;
      __syncthreads();
      z = 0.0f;
      for (int w = warp - part; w < warp - part + wph; ++w) z += red[1][w];
    }
    const float inv = 1.0f / z;
    if (live)
      for (int i = t0 + lane; i < t1; i += 32) ph[i] *= inv;
  }
  if (cs > 1) cluster_sync();
  else __syncthreads();
  const float invh = 1.0f / static_cast<float>(H);
  const uint32_t pb = smem_u32(p);
  for (int i = rank * blockDim.x + threadIdx.x; i < n; i += cs * blockDim.x) {
    float s = 0.0f;
    if (cs > 1) {
#pragma unroll 8
      for (int hh = 0; hh < H; ++hh)
        s += ld_shared_cluster_f32(mapa_shared(pb + 4u * static_cast<uint32_t>((hh / cs) * n + i), hh % cs));
    } else {
      for (int hh = 0; hh < H; ++hh) s += p[static_cast<size_t>(hh) * n + i];
    }
    A[static_cast<size_t>(b) * N + static_cast<size_t>(c) * n + i] = s * invh;
  }
  if (cs > 1) cluster_sync();  // no CTA leaves while its weights are read
}

template <int DH>
cudaError_t launch_dh(const __half* q_cls, const __half* k_cls, const __half* k, int B, int N, int C, int H,
                      float* A, cudaStream_t stream) {
  // CTAs per crop. A cluster pays where a crop's keys are some work for a CTA and
  // SMs are free: from 80 KB of keys (twice that when every SM has a crop), as many
  // CTAs as one per SM, or two per SM from 1 MB. Elsewhere one CTA, a warp per
  // head, is faster: 16 heads x 64, us, clusters of up to two CTAs per SM always /
  // this: 8 crops of 49 tokens 4.8 / 4.4, 75 of 49 9.0 / 4.6, 75 of 196 14.4 / 9.5, 100
  // of 400 22.1 / 16.7, 40 of 576 16.8 / 16.6. More CTAs where one's weights exceed
  // its shared memory.
  const long long crops = static_cast<long long>(B) * C, sms = num_sms();
  const long long keys = 2ll * H * (N / C) * DH;  // bytes
  int cs = 1;
  auto weights = [&](int x) { return static_cast<size_t>((H + x - 1) / x) * (N / C) * sizeof(float); };
  auto split = [&](int x) {
    return weights(x) > kSmemMax || (keys * sms >= 80 * 1024 * (sms + crops) &&
                                     crops * 2 * x <= (keys >= 1 << 20 ? 2 * sms : sms));
  };
  while (cs < kMaxCluster && 2 * cs <= H && split(cs)) cs *= 2;
  // Warps per head. In a cluster, all of the block's; one CTA's, several where the
  // head's tokens are many rounds of loads and the SMs have room (16 warps each,
  // 32 for long crops): 400 crops of 49 tokens, 4 heads x 64, two / one 7.2 / 4.3.
  const int heads = (H + cs - 1) / cs, n = N / C;
  constexpr int kTokens = 32 / lanes_per_token<DH>();  // per warp and load
  int wph = 1;
  auto share = [&](int x) {
    const long long warps = crops * heads * x * 2;
    return cs > 1 || (warps <= 16 * sms && n > 12 * x * kTokens) || (warps <= 32 * sms && n > 64 * x * kTokens);
  };
  while (2 * wph * heads <= kWarps && share(wph)) wph *= 2;
  const int warps = heads * wph < kWarps ? heads * wph : kWarps;
  const size_t smem = weights(cs);
  static SmemLimit limit_one, limit_more;
  const cudaError_t le = cs == 1 && wph == 1 ? limit_one.allow(cls_saliency_kernel<DH, true>, kSmemMax)
                                             : limit_more.allow(cls_saliency_kernel<DH, false>, kSmemMax);
  if (le != cudaSuccess) return le;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(static_cast<unsigned>(C) * cs, B);
  cfg.blockDim = dim3(32 * warps);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = stream;
  cudaLaunchAttribute attr[2];
  attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  attr[0].val.programmaticStreamSerializationAllowed = 1;
  attr[1].id = cudaLaunchAttributeClusterDimension;
  attr[1].val.clusterDim.x = static_cast<unsigned>(cs);
  attr[1].val.clusterDim.y = 1;
  attr[1].val.clusterDim.z = 1;
  cfg.attrs = attr;
  cfg.numAttrs = cs > 1 ? 2 : 1;
  if (cs == 1 && wph == 1)
    return cudaLaunchKernelEx(&cfg, cls_saliency_kernel<DH, true>, q_cls, k_cls, k, N, C, H, cs, wph, A);
  return cudaLaunchKernelEx(&cfg, cls_saliency_kernel<DH, false>, q_cls, k_cls, k, N, C, H, cs, wph, A);
}

}  // namespace

size_t cls_saliency_smem_bytes(int N, int C, int H) { return static_cast<size_t>(H) * (N / C) * sizeof(float); }

int cls_saliency_max_heads(int) { return kMaxHeads; }

cudaError_t launch_cls_saliency(const uint16_t* q_cls16, const uint16_t* k_cls16, const uint16_t* k16, int B, int N,
                                int C, int H, int dh, float* A, cudaStream_t stream) {
  const __half* q_cls = reinterpret_cast<const __half*>(q_cls16);
  const __half* k_cls = reinterpret_cast<const __half*>(k_cls16);
  const __half* k = reinterpret_cast<const __half*>(k16);
  switch (dh) {
    case 32: return launch_dh<32>(q_cls, k_cls, k, B, N, C, H, A, stream);
    case 64: return launch_dh<64>(q_cls, k_cls, k, B, N, C, H, A, stream);
    case 80: return launch_dh<80>(q_cls, k_cls, k, B, N, C, H, A, stream);
    case 128: return launch_dh<128>(q_cls, k_cls, k, B, N, C, H, A, stream);
    default: return cudaErrorInvalidValue;
  }
}

}  // namespace p4q
