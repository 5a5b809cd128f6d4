// Block-level ranking helpers of the selector kernels (Sec. 3.2, Eq. 4:
// every stage keeps the best-ranked tokens, ties to the lower token index).
// Token i of an image is held by thread i / PER of the block's first nt
// threads (element i % PER); the other threads of the block do not take part.
#pragma once

#include <cstdint>

#include "p4q_device.cuh"

namespace p4q {

constexpr int kPer = 4;  // tokens per ranking thread where the block has other work: token i = kPer * threadIdx.x + e

// Shared memory of the rankings.
struct RankScratch {
  __align__(16) unsigned int hist[256];
  unsigned int wsum[32];
  float wlo[32], whi[32];           // per warp: smallest and largest free value
  unsigned long long list[32];      // the boundary bin's (key, ~token) pairs
  unsigned long long threshold;     // the last pair taken
  int count;                        // of the list
  int digit, above, inbin;
};

// Barrier of the first nt threads of the block (group 0, the token owners);
// the other row groups do not take part in the rankings.
__device__ __forceinline__ void group_sync(int nt) { named_bar_sync(1, static_cast<uint32_t>(nt)); }

// Exclusive prefix sum of per-thread counts over the first nt threads (thread order).
template <class Scratch>
__device__ int block_exclusive_scan(int v, int* total, int nt, Scratch& s) {
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  int x = v;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const int y = __shfl_up_sync(0xFFFFFFFFu, x, o);
    if (lane >= o) x += y;
  }
  if (lane == 31) s.wsum[warp] = x;
  group_sync(nt);
  if (warp == 0) {
    int w = lane < (nt >> 5) ? s.wsum[lane] : 0;
#pragma unroll
    for (int o = 1; o < 32; o <<= 1) {
      const int y = __shfl_up_sync(0xFFFFFFFFu, w, o);
      if (lane >= o) w += y;
    }
    s.wsum[lane] = w;  // inclusive
  }
  group_sync(nt);
  const int before = (warp ? s.wsum[warp - 1] : 0) + x - v;
  *total = s.wsum[(nt >> 5) - 1];
  group_sync(nt);
  return before;
}

// The float whose order-preserving key is k (float_order_key's inverse).
__device__ __forceinline__ float order_key_float(uint32_t k) {
  return __uint_as_float((k & 0x80000000u) ? (k & 0x7FFFFFFFu) : ~k);
}

// Warp 0: the digit at which the count from the top of s.hist reaches need,
// the count above it and its own; clears the histogram.
template <class Scratch>
__device__ __forceinline__ void find_digit(int need, Scratch& s) {
  const int lane = threadIdx.x & 31;
  // lane l owns digits [8l, 8l+8)
  const uint4 c0 = *reinterpret_cast<const uint4*>(&s.hist[8 * lane]);
  const uint4 c1 = *reinterpret_cast<const uint4*>(&s.hist[8 * lane + 4]);
  *reinterpret_cast<uint4*>(&s.hist[8 * lane]) = make_uint4(0u, 0u, 0u, 0u);
  *reinterpret_cast<uint4*>(&s.hist[8 * lane + 4]) = make_uint4(0u, 0u, 0u, 0u);
  const unsigned int c[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
  unsigned int own = 0;
#pragma unroll
  for (int k = 0; k < 8; ++k) own += c[k];
  unsigned int x = own;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned int y = __shfl_down_sync(0xFFFFFFFFu, x, o);
    if (lane + o < 32) x += y;
  }
  const unsigned int above = x - own;  // sum over lanes > lane
  if (above < static_cast<unsigned>(need) && above + own >= static_cast<unsigned>(need)) {
    unsigned int acc = above;
    bool found = false;
#pragma unroll
    for (int k = 7; k >= 0; --k) {
      if (!found && acc + c[k] >= static_cast<unsigned>(need)) {
        s.digit = 8 * lane + k;
        s.above = static_cast<int>(acc);
        s.inbin = static_cast<int>(c[k]);
        found = true;
      }
      acc += c[k];
    }
  }
}

// Marks as kept the q free tokens with the largest keys (keys are the
// order-preserving images of fp32 scores, or with INV their complements: the
// smallest scores; ties go to the lower token index); q is at most the number
// of free tokens.
//
// A histogram of 256 bins, linear between the smallest and the largest free
// value (the bin is monotone in the key), finds the bin that the q-th token
// lies in, a second one splits that bin; when the bin holds at most 32 tokens
// (it nearly always does after one or two: scores spread over the range), one
// warp ranks those and publishes the last pair taken: five or seven barriers.
// The counts are plain shared atomics: combining a warp's equal bins by
// match_any first costs more than the collisions that it saves (whole selector
// call, 8 images of 2880 heavy-tailed tokens: 229 us with it, 214 without).
// Otherwise (many equal scores, non-finite values) the bin's tokens go through
// a radix select of their keys, 8 bits per pass, as every ranking did before
// (about 20 barriers).
template <bool INV, int PER>
__device__ void block_take_top(const uint32_t (&key)[PER], bool (&kept)[PER], int base, int N, int q, int nt,
                               RankScratch& s) {
  if (q <= 0) return;
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5, nw = nt >> 5;
  float v[PER];
  bool live[PER];
  float lo = INFINITY, hi = -INFINITY;
#pragma unroll
  for (int e = 0; e < PER; ++e) {
    live[e] = base + e < N && !kept[e];
    v[e] = INV ? -order_key_float(~key[e]) : order_key_float(key[e]);
    if (live[e]) {
      lo = fminf(lo, v[e]);
      hi = fmaxf(hi, v[e]);
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xFFFFFFFFu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xFFFFFFFFu, hi, o));
  }
  if (lane == 0) {
    s.wlo[warp] = lo;
    s.whi[warp] = hi;
  }
  for (int h = threadIdx.x; h < 256; h += nt) s.hist[h] = 0;
  if (threadIdx.x == 0) s.count = 0;
  group_sync(nt);
  lo = lane < nw ? s.wlo[lane] : INFINITY;
  hi = lane < nw ? s.whi[lane] : -INFINITY;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    lo = fminf(lo, __shfl_xor_sync(0xFFFFFFFFu, lo, o));
    hi = fmaxf(hi, __shfl_xor_sync(0xFFFFFFFFu, hi, o));
  }
  int need = q;
  // 255.99 / (hi - lo), or 0 (every token in bin 0) where that is not a finite positive number
  const float width = hi - lo;
  const float scale = (width > 0.0f && width < INFINITY) ? fminf(__fdividef(255.99f, width), 3.0e38f) : 0.0f;
  float x[PER];  // position in the current bin's range, [0, 256)
#pragma unroll
  for (int e = 0; e < PER; ++e) x[e] = scale > 0.0f ? fminf((v[e] - lo) * scale, 255.99f) : 0.0f;
  for (int level = 0; level < 2; ++level) {
    int bin[PER];
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      bin[e] = static_cast<int>(x[e]);
      if (live[e]) atomicAdd(&s.hist[bin[e]], 1u);
    }
    group_sync(nt);
    if (warp == 0) find_digit(need, s);
    group_sync(nt);
    need -= s.above;
    const int digit = s.digit, inbin = s.inbin;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      if (live[e] && bin[e] > digit) kept[e] = true;
      live[e] = live[e] && bin[e] == digit;
      x[e] = fminf((x[e] - static_cast<float>(digit)) * 256.0f, 255.99f);
    }
    if (inbin > 32) continue;
    if (inbin > need) {
#pragma unroll
      for (int e = 0; e < PER; ++e)
        if (live[e])
          s.list[atomicAdd(&s.count, 1)] =
              (static_cast<unsigned long long>(key[e]) << 32) | (0xFFFFFFFFu - static_cast<uint32_t>(base + e));
      group_sync(nt);
      if (warp == 0) {
        const unsigned long long mine = lane < inbin ? s.list[lane] : 0ull;
        int rank = 0;
        for (int k = 0; k < inbin; ++k) rank += s.list[k] > mine ? 1 : 0;
        if (lane < inbin && rank == need - 1) s.threshold = mine;
      }
      group_sync(nt);
    }
    const unsigned long long last = inbin > need ? s.threshold : 0ull;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const unsigned long long pair =
          (static_cast<unsigned long long>(key[e]) << 32) | (0xFFFFFFFFu - static_cast<uint32_t>(base + e));
      if (live[e] && pair >= last) kept[e] = true;
    }
    return;
  }
  // the bin's tokens by radix select
  uint32_t prefix = 0, mask = 0;
  for (int pass = 0; pass < 4; ++pass) {
    const int shift = 24 - 8 * pass;
#pragma unroll
    for (int e = 0; e < PER; ++e) {
      const bool in = live[e] && (key[e] & mask) == prefix;
      const uint32_t dig = in ? ((key[e] >> shift) & 255u) : 256u;  // 256: not counted
      const unsigned peers = __match_any_sync(0xFFFFFFFFu, dig);
      if (in && (__ffs(peers) - 1) == lane) atomicAdd(&s.hist[dig], static_cast<unsigned>(__popc(peers)));
    }
    group_sync(nt);
    if (warp == 0) find_digit(need, s);
    group_sync(nt);
    need -= s.above;
    prefix |= static_cast<uint32_t>(s.digit) << shift;
    mask |= 255u << shift;
    group_sync(nt);
  }
  // keys > prefix are taken; among keys == prefix the first `need` in index order
  int eq = 0;
#pragma unroll
  for (int e = 0; e < PER; ++e)
    if (live[e] && key[e] == prefix) ++eq;
  int total;
  int rank = block_exclusive_scan(eq, &total, nt, s);
#pragma unroll
  for (int e = 0; e < PER; ++e) {
    if (live[e]) {
      if (key[e] > prefix) {
        kept[e] = true;
      } else if (key[e] == prefix) {
        if (rank < need) kept[e] = true;
        ++rank;
      }
    }
  }
  group_sync(nt);
}

}  // namespace p4q
