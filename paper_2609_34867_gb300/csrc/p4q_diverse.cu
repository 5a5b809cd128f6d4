// Stage 3 of the selector (Sec. 3.2, Eq. 4, visual diversity): greedy
// max-min selection on the cosines of fake-quantized tokens. With R the kept
// set (R0 after stages 1-2), m_i = max over r in R of cos(i, r) (-inf while R
// is empty); each of the K_d rounds keeps the free token with the smallest
// m (lower index on ties) and m absorbs its cosines.
//
// One CTA per image (and, while that leaves SMs free, one or three helpers that
// share phase 2's cosines). The largest cosine of every token to R0 comes from the
// tensor-core GEMM before this kernel (its cosine-max epilogue, or a row pass
// over its int32 tiles; in Gram mode a row pass over the token-pair GEMM)
// as m. After that no cosine row of the whole image is ever formed. The kernel holds, for every free token, a
// lower bound of m (exact up to the first ex picks) and runs in phases:
//   1. pool: the 128 smallest free (bound, token) pairs (block_take_top);
//      tau = the largest of them. Every token outside the pool has a pair
//      above tau, and its true pair is at least its bound's.
//   2. the pool's exact cosines: code dot products of the pool rows with the
//      pool rows and with every pick the pool's bounds have not seen yet, on
//      the tensor cores (tcgen05 kind::f8f6f4, M = 128 pool rows, N <= 256
//      columns per chunk, operand rows gathered from the expanded codes into
//      a 4-deep ring of shared-memory stages by cp.async in the
//      128-byte-swizzled K-major layout),
//      turned into Eq. 4 cosines in the epilogue: the pool block and, per
//      pool row, the largest cosine to those picks (the bound becomes m).
//   3. greedy rounds on the pool by the block (pool_rounds): a pool entry
//      whose pair is at most tau is below every token outside, so the
//      smallest such entry is the next pick, and runs of the next smallest
//      are picked together while no earlier pick raises them; their cosines
//      to the pool come from the block.
//   4. the pool's m go back to their tokens (exact up to the picks so far).
// A phase that picks nothing still makes its pool exact, so phases end.
#include <cuda_fp16.h>

#include "p4q.h"
#include "p4q_device.cuh"
#include "p4q_internal.h"
#include "p4q_rank.cuh"

namespace p4q {

__device__ unsigned int g_diverse_err;

namespace {

constexpr int kPool = 128;
constexpr int kPickMax = 64;  // picks confirmed per pool iteration at most
constexpr int kPoolPer = kPool / 32;
static_assert(kPoolPer == 4, "pool warp layout: four slots per lane");
constexpr int kArows = 128;   // pool rows per MMA (M = 128: the TMEM lanes)
constexpr int kBrows = 128;   // extra column rows per stage
constexpr int kBK = 128;      // bytes of K per stage (one 128-byte swizzle row)
constexpr int kStages = 4;    // k-blocks in flight: the gathered rows come at L2 latency
constexpr int kLag = 2;       // k-blocks a producer keeps loading before it hands one over
constexpr int kAbytes = kArows * kBK;
constexpr int kStageBytes = (kArows + kBrows) * kBK;
constexpr uint32_t kTmemCols = 256;

struct DivScratch {
  RankScratch rank;
  int t, npool, tmin;
  unsigned long long tau;
  __align__(16) uint32_t skey[kPool];   // pool rounds: order keys of the certain entries' m
  int prank[kPool];                     // pool rounds: their ranks
  int sorted[kPool];                    // pool rounds: slots of the certain entries in key order
  int L;                                // pool rounds: length of the confirmed prefix
  int ptok[kPool];                      // pool slot -> token (ascending)
  float pm[kPool];                      // m of the pool tokens (bound, then exact)
  unsigned int pmx[kPool];              // order key of the largest cosine to the pick columns; pool rounds: of m
  int psum[kPool], pnorm[kPool];        // pool rows: sum of u, squared code norm
  float prs[kPool];                     // pool rows: rsqrtf of the squared code norm (0 for a zero row)
  int csum[kBrows], cnorm[kBrows];      // extra columns of the current chunk
  unsigned int keptbits[P4Q_MAX_TOKENS / 32];
  int16_t list[P4Q_MAX_TOKENS];         // the greedy picks, in order
  signed char slotof[P4Q_MAX_TOKENS];   // token -> pool slot, -1 outside the pool
  int16_t candof[P4Q_MAX_TOKENS];       // token -> candidate index, -1 for the others
  int pci[kPool];                       // pool slot -> candidate index (-1: not a candidate)
  uint64_t bar_full[kStages];           // producer warps -> the stage is in shared memory
  uint64_t bar_empty[kStages];          // MMA commit -> the stage may be overwritten
  uint64_t bar_acc;                     // MMA commit -> the chunk's accumulator is complete
  uint64_t bar_done;                    // MMA commit at teardown -> nothing in flight
  uint32_t tmem_slot;
  volatile int abort_flag;
  int go, ncp;                          // to the helper CTAs: another phase's cosines, and its unseen picks
  __align__(16) float cp[kPool][kPool + 1]; // cos(ptok[i], ptok[j]), i <= j (Eq. 4, exact; padded: column reads)
};

__device__ __forceinline__ float pool_cos(const DivScratch& s, int i, int j) { return s.cp[min(i, j)][max(i, j)]; }

// Greedy rounds on the pool, by the whole block, with exact m of the pool
// entries in s.pm. The next pick is the smallest free
// (m, token) pair. A pool entry is certain to be in order while its pair is at
// most tau (every token outside the pool is above tau and m only grows). Per
// iteration the certain entries are ranked by their pairs (four warps per
// 32 slots count the smaller keys, every load a broadcast), giving c_0 < c_1 < ...; c_0 is the next pick, and
// c_a the pick after c_0 .. c_{a-1} whenever none of their cosines exceeds
// m(c_a) (nothing else can pass it: every other pair only grows). The pairs
// (b < a) are checked in parallel; the longest such prefix (at most kPickMax)
// is picked at once, the pool's m absorbs the picks' cosines, and the picks
// are appended to s.list. Ends when Kd picks are made or no entry is certain;
// s.t and s.pm hold the results.
// Two to five iterations make the picks of a 576-token image (about 30 each),
// of about 3250 cycles (640 threads; 4000 with 768): half of it the 16 K key
// comparisons of the ranks, bound by the integer pipe. With a thread per slot
// in all but the pair check an iteration took 4300 (4700).
template <int kThreads>
__device__ void pool_rounds(int npool, int Kd, DivScratch& s) {
  constexpr uint32_t kNone = 0xFFFFFFFFu;
  constexpr int kParts = 4;                    // warps per 32 slots
  constexpr int kCheck = kThreads / kPickMax;  // threads per candidate of the pair check
  static_assert(kPool == 128 && kPickMax == 64 && kThreads % 64 == 0 && kThreads >= kParts * kPool, "thread layout");
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const int slot = tid & (kPool - 1), part = warp >> 2;  // (slot of the warp's lanes: 32 (warp % 4) + lane)
  const unsigned long long tau = s.tau;
  if (tid < kPool) s.pmx[tid] = tid < npool ? float_order_key(s.pm[tid]) : kNone;
  bool alive = tid < npool;  // of thread tid's slot, tid < kPool
  while (true) {
    const int t = s.t;  // every thread has passed the barrier that published it
    if (t >= Kd) break;
    bool certain = false;
    if (tid < kPool) {
      const uint32_t k = s.pmx[tid];
      certain = alive && ((static_cast<unsigned long long>(k) << 32) | tid) <= tau;
      s.skey[tid] = certain ? k : kNone;
      s.prank[tid] = 0;
    }
    if (tid == 0) s.L = kPickMax;
    const int nc = __syncthreads_count(certain);
    const int r = min(min(nc, Kd - t), kPickMax);
    if (r == 0) break;
    // rank of each certain entry among them: the smaller keys, and the equal
    // ones of lower slots (keys below kNone: no cosine's key is that large)
    if (part < kParts) {
      const uint32_t key = s.skey[slot];
      int cnt = 0;
      if (part != (warp & 3)) {
        const uint32_t lim = key + (part < (warp & 3) ? 1u : 0u);
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint4 k = *reinterpret_cast<const uint4*>(&s.skey[32 * part + 4 * i]);
          cnt += (k.x < lim ? 1 : 0) + (k.y < lim ? 1 : 0) + (k.z < lim ? 1 : 0) + (k.w < lim ? 1 : 0);
        }
      } else {
#pragma unroll
        for (int i = 0; i < 8; ++i) {
          const uint4 k = *reinterpret_cast<const uint4*>(&s.skey[32 * part + 4 * i]);
          cnt += (k.x < key + (4 * i < lane ? 1u : 0u) ? 1 : 0) + (k.y < key + (4 * i + 1 < lane ? 1u : 0u) ? 1 : 0) +
                 (k.z < key + (4 * i + 2 < lane ? 1u : 0u) ? 1 : 0) + (k.w < key + (4 * i + 3 < lane ? 1u : 0u) ? 1 : 0);
        }
      }
      if (key != kNone) atomicAdd(&s.prank[slot], cnt);
    }
    __syncthreads();
    const int rank = certain ? s.prank[tid] : kPool;
    if (rank < r) s.sorted[rank] = tid;
    __syncthreads();
    // pairs b < a < r: a violation (an earlier candidate raises c_a) ends the prefix at a
    {
      const int a2 = tid & (kPickMax - 1);
      bool bad = false;
      if (a2 < r) {
        const int ca = s.sorted[a2];
        const float mc = s.pm[ca];
#pragma unroll 4
        for (int b2 = tid / kPickMax; b2 < a2; b2 += kCheck) bad |= pool_cos(s, s.sorted[b2], ca) > mc;
      }
      const unsigned int v = __ballot_sync(0xFFFFFFFFu, bad);
      if (v != 0 && lane == __ffs(v) - 1) atomicMin(&s.L, a2);
    }
    __syncthreads();
    const int L = min(s.L, r);  // >= 1: c_0 never fails
    if (rank < L) {
      alive = false;
      const int tok = s.ptok[tid];
      s.list[t + rank] = static_cast<int16_t>(tok);
      atomicOr(&s.keptbits[tok >> 5], 1u << (tok & 31));
    }
    if (part < kParts) {
      float mx = -INFINITY;
#pragma unroll 4
      for (int b2 = part; b2 < L; b2 += kParts) mx = fmaxf(mx, pool_cos(s, s.sorted[b2], slot));
      atomicMax(&s.pmx[slot], float_order_key(mx));
    }
    if (tid == 0) s.t = t + L;
    __syncthreads();
    if (tid < kPool) s.pm[tid] = order_key_float(s.pmx[tid]);
  }
}

// Arguments of one launch.
struct DivArgs {
  const uint32_t* kept12;  // [B, words] R0 as bits
  const float* m;          // [B, N] largest cosine to R0 (R0 > 0)
  const int32_t* cand;     // [B, C] candidates, ascending (nullptr: every token, C = N)
  const int32_t* candnorm; // [B, C]
  const float* cdots;      // [B, C, cpitch] their pairwise code dot products
  int C, cpitch;
  const uint8_t* vu;       // [B*N, d] expanded codes
  const int32_t* vsum;     // [B*N]
  const int32_t* vnorm;    // [B*N]
  int N, d, R0, K, Kd;
  int32_t* idx;            // [B, K]
};

struct PickCols {
  int* c;     // candidate index
  int* n;     // squared code norm
  float* rs;  // its rsqrtf (0 for a zero row)
};

__device__ __forceinline__ PickCols pick_cols(uint8_t* stages) {
  static_assert(P4Q_MAX_TOKENS * 12 <= kStages * kStageBytes, "pick columns");
  int* c = reinterpret_cast<int*>(stages);
  return PickCols{c, c + P4Q_MAX_TOKENS, reinterpret_cast<float*>(c + 2 * P4Q_MAX_TOKENS)};
}

// The same variable of CTA rank of the cluster (a generic address).
template <class T>
__device__ __forceinline__ T* cluster_ptr(T* p, uint32_t rank) {
  uint64_t r;
  asm volatile("mapa.u64 %0, %1, %2;" : "=l"(r) : "l"(reinterpret_cast<uint64_t>(p)), "r"(rank));
  return reinterpret_cast<T*>(r);
}

// Pool rows rank, rank + cs, ... of a phase whose tokens are all candidates:
// their exact cosines to the pool (into out.cp) and the largest to the ncp
// unseen picks pk (into out.pmx), from the candidates' dot products; the
// pool's data from s.
template <int kThreads>
__device__ __forceinline__ void cand_cosines(const DivArgs& a, int b, int npool, int ncp, int rank, int cs,
                                             const DivScratch& s, const PickCols& pk, DivScratch& out) {
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int step = cs * (kThreads / 32);
  const float* cd = a.cdots + static_cast<size_t>(b) * a.C * a.cpitch;
  // the pool block, a warp per row, two rows of four columns per lane in
  // flight; it is symmetric: each pair once (f >= e)
  constexpr int kR = 2;
  int fc[kPoolPer], fn[kPoolPer];
#pragma unroll
  for (int k = 0; k < kPoolPer; ++k) {
    const int f = lane + 32 * k;
    fc[k] = f < npool ? s.pci[f] : 0;
    fn[k] = f < npool ? s.pnorm[f] : 0;
  }
  for (int e0 = rank + cs * warp; e0 < npool; e0 += kR * step) {
    float v[kR][kPoolPer];
#pragma unroll
    for (int j = 0; j < kR; ++j) {
      const int e = e0 + j * step;
      const float* row = cd + static_cast<size_t>(e < npool ? s.pci[e] : 0) * a.cpitch;
#pragma unroll
      for (int k = 0; k < kPoolPer; ++k) {
        const int f = lane + 32 * k;
        v[j][k] = f < npool && f >= e ? row[fc[k]] : 0.0f;
      }
    }
#pragma unroll
    for (int j = 0; j < kR; ++j) {
      const int e = e0 + j * step;
#pragma unroll
      for (int k = 0; k < kPoolPer; ++k) {
        const int f = lane + 32 * k;
        if (f < npool && f >= e) {
          const float c = code_cosine(static_cast<int>(v[j][k]), s.pnorm[e], fn[k]);
          out.cp[e][f] = c;
        }
      }
    }
  }
  // per pool row: the largest cosine to the unseen picks, 128 columns of
  // two rows at a time: approximate, then exact for the columns near the
  // largest so far (from the row's bound on: less does not raise it)
  if (ncp > 0) {
    for (int e0 = rank + cs * warp; e0 < npool; e0 += kR * step) {
      float amax[kR], emax[kR], rs[kR];
      const float* row[kR];
#pragma unroll
      for (int j = 0; j < kR; ++j) {
        const int e = min(e0 + j * step, npool - 1);
        amax[j] = s.pm[e];
        emax[j] = -INFINITY;
        rs[j] = s.prs[e];
        row[j] = cd + static_cast<size_t>(s.pci[e]) * a.cpitch;
      }
      for (int c0 = 0; c0 < ncp; c0 += 128) {
        float v[kR][4];
#pragma unroll
        for (int k = 0; k < 4; ++k) {
          const int cj = pk.c[min(c0 + lane + 32 * k, ncp - 1)];
#pragma unroll
          for (int j = 0; j < kR; ++j)
            if (e0 + j * step < npool) v[j][k] = row[j][cj];
        }
#pragma unroll
        for (int j = 0; j < kR; ++j) {
          if (e0 + j * step >= npool) break;
          float ap[4], am = amax[j];
#pragma unroll
          for (int k = 0; k < 4; ++k) {
            ap[k] = v[j][k] * rs[j] * pk.rs[min(c0 + lane + 32 * k, ncp - 1)];
            am = fmaxf(am, ap[k]);
          }
          amax[j] = order_key_float(__reduce_max_sync(0xFFFFFFFFu, float_order_key(am)));
#pragma unroll
          for (int k = 0; k < 4; ++k)
            if (ap[k] >= amax[j] - kCosMargin)
              emax[j] = fmaxf(emax[j], code_cosine(static_cast<int>(v[j][k]),
                                                   s.pnorm[min(e0 + j * step, npool - 1)],
                                                   pk.n[min(c0 + lane + 32 * k, ncp - 1)]));
        }
      }
#pragma unroll
      for (int j = 0; j < kR; ++j) {
        const uint32_t mx = __reduce_max_sync(0xFFFFFFFFu, float_order_key(emax[j]));
        if (lane == 0 && e0 + j * step < npool) out.pmx[e0 + j * step] = mx;
      }
    }
  }
}

// A helper CTA: its share of the cosines of each phase that takes them from
// the candidates' dot products, written into the first CTA's shared memory.
template <int kThreads>
__device__ void diverse_helper(const DivArgs& a, int b, int rank, int cs, DivScratch& s, uint8_t* stages) {
  DivScratch& s0 = *cluster_ptr(&s, 0);
  const PickCols pk = pick_cols(stages), pk0 = pick_cols(cluster_ptr(stages, 0));
  while (true) {
    cluster_sync();  // the phase's pool and picks are in place, or the picks are complete
    if (!s0.go) break;
    const int npool = s0.npool, ncp = s0.ncp;
    for (int r = threadIdx.x; r < npool; r += kThreads) {
      s.pci[r] = s0.pci[r];
      s.pnorm[r] = s0.pnorm[r];
      s.prs[r] = s0.prs[r];
      s.pm[r] = s0.pm[r];
    }
    for (int c = threadIdx.x; c < ncp; c += kThreads) {
      pk.c[c] = pk0.c[c];
      pk.n[c] = pk0.n[c];
      pk.rs[c] = pk0.rs[c];
    }
    __syncthreads();
    cand_cosines<kThreads>(a, b, npool, ncp, rank, cs, s, pk, s0);
    cluster_sync();
  }
  cluster_sync();  // the first CTA stays until every helper has read its word
}

// Token i of the image is held by thread i / PER (element i % PER).
template <int kThreads, int PER>
__global__ void __launch_bounds__(kThreads, 1) select_diverse_kernel(const DivArgs a) {
  extern __shared__ uint8_t smem_raw[];
  uint8_t* stages = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) & ~uintptr_t(1023));
  DivScratch& s = *reinterpret_cast<DivScratch*>(stages + kStages * kStageBytes);
  constexpr int kWarps = kThreads / 32;
  const int cs = static_cast<int>(cluster_nctarank()), rank = static_cast<int>(cluster_ctarank());
  const int b = blockIdx.x / cs, N = a.N, d = a.d;
  const int warp = threadIdx.x >> 5, lane = threadIdx.x & 31;
  const int tpg = ((N + PER - 1) / PER + 31) / 32 * 32;  // token owners (group 0)
  const bool g0 = threadIdx.x < tpg;
  const int base = PER * threadIdx.x;
  const int words = (N + 31) / 32;
  const size_t row0 = static_cast<size_t>(b) * N;

  if (rank > 0) {
    pdl_wait();
    pdl_launch_dependents();
    diverse_helper<kThreads>(a, b, rank, cs, s, stages);
    return;
  }
  if (threadIdx.x == 0) {
    for (int i = 0; i < kStages; ++i) {
      mbar_init(&s.bar_full[i], kThreads / 32 - 1);
      mbar_init(&s.bar_empty[i], 1);
    }
    mbar_init(&s.bar_acc, 1);
    mbar_init(&s.bar_done, 1);
    s.abort_flag = 0;
    s.t = 0;
    fence_barrier_init();
  }
  if (warp == 0) {
    tmem_alloc(&s.tmem_slot, kTmemCols);
    tmem_relinquish();
  }
  for (int i = threadIdx.x; i < N; i += kThreads) {
    s.slotof[i] = -1;
    s.candof[i] = a.cand ? -1 : static_cast<int16_t>(i);  // (without candidates, C = N: the token itself)
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = s.tmem_slot;
  volatile int* abort_flag = &s.abort_flag;
  pdl_wait();  // R0 bits and maxima come from the kernels before
  pdl_launch_dependents();
  for (int w = threadIdx.x; w < words; w += kThreads) s.keptbits[w] = a.kept12[static_cast<size_t>(b) * words + w];
  if (a.cand)
    for (int c = threadIdx.x; c < a.C; c += kThreads)
      s.candof[a.cand[static_cast<size_t>(b) * a.C + c]] = static_cast<int16_t>(c);

  bool kept[PER];
  float m[PER];
  int ex[PER];  // m of the token is exact up to the first ex picks
#pragma unroll
  for (int e = 0; e < PER; ++e) {
    const int i = base + e;
    kept[e] = false;  // (set from the bits at the top of each phase)
    m[e] = g0 && i < N && a.R0 > 0 ? a.m[row0 + i] : -INFINITY;
    ex[e] = 0;
  }
  const int KB = d / kBK;
  const int phase_limit = a.Kd * (N / kPool + 2) + 8;
  int g = 0;       // k-blocks staged so far (mbarrier phases of bar_full / bar_empty)
  int chunks = 0;  // accumulators completed so far (phases of bar_acc)
  uint32_t key[PER];

  // Every thread leaves the loop at the same phase: what it decides on changes
  // only behind a later barrier of the block (s.t; the abort flag of the bounded
  // waits), or is its own count of the phases.
  for (int phase = 0;; ++phase) {
    __syncthreads();
    const int t = s.t;
    if (t >= a.Kd || s.abort_flag) break;
    if (phase >= phase_limit) {
      if (threadIdx.x == 0) atomicOr(&g_diverse_err, kErrTimeout);
      break;
    }
#pragma unroll
    for (int e = 0; e < PER; ++e)
      if (g0 && base + e < N && ((s.keptbits[(base + e) >> 5] >> ((base + e) & 31)) & 1u)) kept[e] = true;
    // ---- 1. pool: the q smallest free (bound, token) pairs, in token order
    const int nfree = N - a.R0 - t;
    const int q = min(kPool, nfree);
    if (threadIdx.x == 0) s.tmin = t;
    int npool = 0;
    if (g0) {
      bool member[PER];
#pragma unroll
      for (int e = 0; e < PER; ++e) {
        member[e] = kept[e];
        key[e] = (base + e < N) ? ~float_order_key(m[e]) : 0u;
      }
      block_take_top<true>(key, member, base, N, q, tpg, s.rank);
      int cnt = 0, emin = t;
#pragma unroll
      for (int e = 0; e < PER; ++e) {
        const bool in = base + e < N && member[e] && !kept[e];
        cnt += in ? 1 : 0;
        emin = in ? min(emin, ex[e]) : emin;
      }
      group_sync(tpg);
      int pos = block_exclusive_scan(cnt, &npool, tpg, s.rank);
#pragma unroll
      for (int e = 0; e < PER; ++e) {
        if (base + e < N && member[e] && !kept[e]) {
          const int i = base + e;
          s.ptok[pos] = i;
          s.pm[pos] = m[e];
          s.pmx[pos] = 0u;  // below the key of every float
          s.slotof[i] = static_cast<signed char>(pos);
          ++pos;
        }
      }
      if (emin < t) atomicMin(&s.tmin, emin);
      if (threadIdx.x == 0) s.npool = npool;
    }
    __syncthreads();
    npool = s.npool;
    const int tmin = s.tmin;
    const int ncp = t - tmin;  // picks whose cosines some pool bound has not seen
    // tau: the largest pool pair (everything certain when the pool holds every free token)
    if (warp == kWarps - 1) {
      unsigned long long mx = 0;
#pragma unroll
      for (int k = 0; k < kPoolPer; ++k) {
        const int slot = kPoolPer * lane + k;
        if (slot < npool) {
          const unsigned long long pr = (static_cast<unsigned long long>(float_order_key(s.pm[slot])) << 32) | slot;
          mx = pr > mx ? pr : mx;
        }
      }
      const uint32_t thi = __reduce_max_sync(0xFFFFFFFFu, static_cast<uint32_t>(mx >> 32));
      const uint32_t tlo =
          __reduce_max_sync(0xFFFFFFFFu, static_cast<uint32_t>(mx >> 32) == thi ? static_cast<uint32_t>(mx) : 0u);
      if (lane == 0) s.tau = (q >= nfree) ? ~0ull : ((static_cast<unsigned long long>(thi) << 32) | tlo);
    }
    // ---- 2. the pool's exact dot products with the pool and with the picks
    // its bounds have not seen: from the candidates' dot products when every
    // one of those tokens is a candidate, else on the tensor cores here
    bool mine_ok = true;
    for (int r = threadIdx.x; r < npool + ncp; r += kThreads) {
      const int tok = r < npool ? s.ptok[r] : s.list[tmin + r - npool];
      const int ci = s.candof[tok];
      mine_ok = mine_ok && ci >= 0;
      if (r < npool) {  // its row's data (a thread per slot: one global latency)
        const int ns = a.vnorm[row0 + tok];
        s.psum[r] = a.vsum[row0 + tok];
        s.pnorm[r] = ns;
        s.prs[r] = ns > 0 ? rsqrtf(static_cast<float>(ns)) : 0.0f;
        s.pci[r] = ci;
      }
    }
    const bool from_cand = __syncthreads_and(mine_ok) != 0;
    if (from_cand) {
      // the unseen picks' columns (in the stage ring, which nothing uses here)
      const PickCols pk = pick_cols(stages);
      const int32_t* cn = a.candnorm + static_cast<size_t>(b) * a.C;
      for (int c = threadIdx.x; c < ncp; c += kThreads) {
        const int cj = s.candof[s.list[tmin + c]];
        const int nj = cn[cj];
        pk.c[c] = cj;
        pk.n[c] = nj;
        pk.rs[c] = nj > 0 ? rsqrtf(static_cast<float>(nj)) : 0.0f;
      }
      if (threadIdx.x == 0) {
        s.go = 1;
        s.ncp = ncp;
      }
      if (cs > 1) cluster_sync();
      else __syncthreads();
      cand_cosines<kThreads>(a, b, npool, ncp, 0, cs, s, pk, s);
      if (cs > 1) cluster_sync();
      else __syncthreads();
    } else {
    // the rows this phase reads, toward L2 ahead of the staged loads
    for (int r = threadIdx.x; r < npool + ncp; r += kThreads) {
      const int tok = r < npool ? s.ptok[r] : s.list[tmin + r - npool];
      prefetch_l2_bulk(a.vu + (row0 + tok) * d, static_cast<uint32_t>(d));
    }
    // chunk 0: columns = the 128 pool rows (the A stage itself) + up to 128 picks;
    // chunk c >= 1: up to 128 further picks.
    const int extra0 = min(ncp, kArows);
    const int nchunks = 1 + (ncp - extra0 + kBrows - 1) / kBrows;
    for (int ch = 0; ch < nchunks; ++ch) {
      const int pick0 = (ch == 0) ? tmin : tmin + extra0 + (ch - 1) * kBrows;  // first pick column of the chunk
      const int nextra = (ch == 0) ? extra0 : min(kBrows, ncp - extra0 - (ch - 1) * kBrows);
      const int ncol = (ch == 0) ? (extra0 > 0 ? kArows + ((nextra + 15) & ~15) : ((npool + 15) & ~15))
                                 : ((nextra + 15) & ~15);
      for (int c = threadIdx.x; c < nextra; c += kThreads) {
        const int tok = s.list[pick0 + c];
        s.csum[c] = a.vsum[row0 + tok];
        s.cnorm[c] = a.vnorm[row0 + tok];
      }
      const int items = (npool + nextra) * (kBK / 16);
      if (warp == 0) {
        // MMA issuer: each stage once its producers have arrived on full[st]
        if (lane == 0) {
          const uint32_t idesc = idesc_e4m3_f32(kArows, ncol);
          for (int kb = 0; kb < KB; ++kb, ++g) {
            const int st = g % kStages;
            if (!mbar_wait_spin(&s.bar_full[st], (g / kStages) & 1, abort_flag, &g_diverse_err)) continue;
            tc_fence_after();
            const uint32_t a0 = smem_u32(stages + st * kStageBytes);
            const uint32_t b0 = (ch == 0) ? a0 : a0 + kAbytes;
#pragma unroll
            for (int k = 0; k < kBK / 32; ++k)
              mma_f8f6f4(tmem, sw128_kmajor_desc(a0 + 32 * k), sw128_kmajor_desc(b0 + 32 * k), idesc,
                         (kb > 0 || k > 0) ? 1u : 0u);
            mma_commit(&s.bar_empty[st]);
          }
          mma_commit(&s.bar_acc);
        } else {
          g += KB;
        }
        __syncwarp();
      } else {
        // producers: warps 1.. gather the k-block's 16-byte row chunks by
        // cp.async; k-block kb is handed over (wait, proxy fence, arrive) kLag
        // k-blocks later, so kLag loads per thread stay in flight
        const int pt = threadIdx.x - 32, np = kThreads - 32;
        for (int kb = 0; kb < KB + kLag; ++kb) {
          if (kb < KB) {
            const int st = (g + kb) % kStages;
            if (g + kb >= kStages) {
              if (lane == 0)
                mbar_wait_spin(&s.bar_empty[st], (((g + kb) / kStages) - 1) & 1, abort_flag, &g_diverse_err);
              __syncwarp();
            }
            const uint32_t sbase = smem_u32(stages + st * kStageBytes);
            for (int it = pt; it < items; it += np) {
              // pool rows at stage rows 0.., extra columns at stage rows 128.. (the B region)
              const int r = it >> 3, c16 = it & 7;
              const bool pool_row = r < npool;
              const int tok = pool_row ? s.ptok[r] : s.list[pick0 + r - npool];
              const int srow = pool_row ? r : kArows + (r - npool);
              const uint8_t* src = a.vu + (row0 + tok) * d + kb * kBK + c16 * 16;
              cp_async16(sbase + srow * kBK + ((c16 ^ (srow & 7)) << 4), src);
            }
          }
          cp_async_commit();  // empty groups past KB keep the accounting uniform
          const int kc = kb - kLag;
          if (kc >= 0) {
            cp_async_wait<kLag>();
            fence_proxy_async_smem();
            __syncwarp();
            if (lane == 0) mbar_arrive(&s.bar_full[(g + kc) % kStages]);
          }
        }
        g += KB;
      }
      // epilogue: TMEM lanes = pool rows, 16-column groups spread over the warps
      if (lane == 0 && !*abort_flag) mbar_wait(&s.bar_acc, chunks & 1, abort_flag, &g_diverse_err);
      __syncwarp();
      ++chunks;
      tc_fence_after();
      {
        const int qd = warp & 3;
        const int e = 32 * qd + lane;
        const bool erow = e < npool;
        const float corr = erow ? static_cast<float>(64 * d - 8 * s.psum[e]) : 0.0f;
        const int ne = erow ? s.pnorm[e] : 0;
        // pool columns: every cosine, exactly (the block); pick columns: the
        // largest approximate cosine, then the exact cosine of the columns
        // near it (two passes over TMEM)
        float amax = -INFINITY, emax = -INFINITY;
        const int g_first = (ch == 0) ? kArows / 16 : 0;  // first group of pick columns
#pragma unroll 1
        for (int pass = 0; pass < 2; ++pass) {
#pragma unroll 1
          for (int grp = warp >> 2; grp < ncol / 16; grp += kWarps / 4) {  // the same groups in both passes
            if (pass == 1 && grp < g_first) continue;
            uint32_t v[16];
            tmem_ld_32x32b_x16(tmem + (static_cast<uint32_t>(32 * qd) << 16) + 16 * grp, v);
            tmem_ld_wait();
            if (!erow) continue;
            if (grp < g_first) {  // pool columns (pass 0 only)
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const int slot = 16 * grp + i;
                if (slot < npool) {
                  const int dot = __float2int_rn(__fmaf_rn(__uint_as_float(v[i]), 262144.0f,
                                                           corr - 8.0f * static_cast<float>(s.psum[slot])));
                  s.cp[slot][e] = code_cosine(dot, ne, s.pnorm[slot]);  // the block is symmetric
                }
              }
            } else {
#pragma unroll
              for (int i = 0; i < 16; ++i) {
                const int ci = 16 * grp + i - (ch == 0 ? kArows : 0);
                if (ci < nextra) {
                  const int dot = __float2int_rn(__fmaf_rn(__uint_as_float(v[i]), 262144.0f,
                                                           corr - 8.0f * static_cast<float>(s.csum[ci])));
                  const float ap = cos_approx(dot, ne, s.cnorm[ci]);
                  if (pass == 0) {
                    amax = fmaxf(amax, ap);
                  } else if (ap >= amax - kCosMargin) {
                    emax = fmaxf(emax, code_cosine(dot, ne, s.cnorm[ci]));
                  }
                }
              }
            }
          }
        }
        if (erow && emax > -INFINITY) atomicMax(&s.pmx[e], float_order_key(emax));
      }
      tc_fence_before();
      __syncthreads();
    }
    }  // tensor-core path
    // the bounds of the pool become m
    if (threadIdx.x < npool && s.pmx[threadIdx.x] != 0u)
      s.pm[threadIdx.x] = fmaxf(s.pm[threadIdx.x], order_key_float(s.pmx[threadIdx.x]));
    __syncthreads();
    // ---- 3. greedy rounds on the pool
    if (!s.abort_flag) pool_rounds<kThreads>(npool, a.Kd, s);
    __syncthreads();
    // ---- 4. exact m back to the pool's tokens
    const int tn = s.t;
    if (g0) {
#pragma unroll
      for (int e = 0; e < PER; ++e) {
        const int i = base + e;
        if (i < N && s.slotof[i] >= 0) {
          const int slot = s.slotof[i];
          if ((s.keptbits[i >> 5] >> (i & 31)) & 1u) {
            kept[e] = true;
          } else {
            m[e] = s.pm[slot];
            ex[e] = tn;
          }
          s.slotof[i] = -1;
        }
      }
    }
  }
  if (cs > 1) {  // the helpers leave
    __syncthreads();
    if (threadIdx.x == 0) s.go = 0;
    cluster_sync();
  }
  // Output: the kept set in ascending index order.
  if (g0) {
    int cnt = 0;
#pragma unroll
    for (int e = 0; e < PER; ++e)
      cnt += (base + e < N && ((s.keptbits[(base + e) >> 5] >> ((base + e) & 31)) & 1u)) ? 1 : 0;
    int total;
    int pos = block_exclusive_scan(cnt, &total, tpg, s.rank);
#pragma unroll
    for (int e = 0; e < PER; ++e)
      if (base + e < N && ((s.keptbits[(base + e) >> 5] >> ((base + e) & 31)) & 1u) && pos < a.K)
        a.idx[static_cast<size_t>(b) * a.K + pos++] = base + e;
  }
  // Teardown: every MMA this CTA issued has completed (a commit after the last
  // one, waited for with a bound) before the accumulator is released.
  if (threadIdx.x == 0) {
    mma_commit(&s.bar_done);
    int fresh = 0;
    mbar_wait(&s.bar_done, 0, reinterpret_cast<volatile int*>(&fresh), &g_diverse_err, 100000000ull);
  }
  tc_fence_before();
  if (cs > 1) cluster_sync();
  else __syncthreads();
  if (warp == 0) {
    tc_fence_after();
    tmem_dealloc(tmem, kTmemCols);
  }
}

constexpr size_t kDivSmem = 1024 + kStages * kStageBytes + sizeof(DivScratch);
static_assert(kDivSmem <= 232448, "shared memory budget");

}  // namespace

cudaError_t launch_select_diverse(const SelectPlan& p, const SelectWorkspace& ws, int32_t* idx, cudaStream_t stream) {
  if (p.Kd <= 0) return cudaSuccess;
  DivArgs a;
  a.kept12 = ws.kept12;
  a.m = ws.m;
  a.cand = ws.gram ? nullptr : ws.cand;
  a.candnorm = ws.gram ? ws.vnorm : ws.candnorm;  // Gram mode: candidate c is token c
  a.cdots = ws.cdots;
  a.C = ws.C;
  a.cpitch = ws.cpitch;
  a.vu = ws.vu;
  a.vsum = ws.vsum;
  a.vnorm = ws.vnorm;
  a.N = p.N;
  a.d = p.d;
  a.R0 = p.Kq + p.Ks;
  a.K = p.K;
  a.Kd = p.Kd;
  a.idx = idx;
  // Each CTA takes an SM, most of whose time a helper waits: so as many per image
  // as leave room for another selection's on a second stream. Four while two
  // calls' take half the SMs (9 images of 152 SMs), two while they fit (38).
  // Whole selector call of 576 tokens (K = 192) / 2880 tokens (K = 640), us,
  // clusters of 1, 2, 4:
  //   one stream: 1 image 66.4 -> 63.4, 60.7 / 458 -> 454, 449; 8 images 89.0 ->
  //     86.7, 83.0 / 675 -> 671, 664; 32 images 162 -> 159, 156 / 1002 -> 994, 990;
  //   two streams, per call: 8 images 57.0 -> 55.6, 55.7 / 374 -> 371, 372; 12
  //     64.9 -> 62.5, 70.2 / 430 -> 427, 429; 16 86.0 -> 85.9, 89.6 / 489 -> 488,
  //     517; 32 141 -> 130, 137 / 705 -> 718, 833.
  const int sms = num_sms(), cs = 16 * p.B <= sms ? 4 : 4 * p.B <= sms ? 2 : 1;
  auto go = [&](auto kern, int threads) -> cudaError_t {
    cudaError_t e = cudaFuncSetAttribute(kern, cudaFuncAttributeMaxDynamicSharedMemorySize, static_cast<int>(kDivSmem));
    if (e != cudaSuccess) return e;
    cudaLaunchConfig_t cfg = {};
    cfg.gridDim = dim3(p.B * cs);
    cfg.blockDim = dim3(threads);
    cfg.dynamicSmemBytes = kDivSmem;
    cfg.stream = stream;
    cudaLaunchAttribute attr[2];
    attr[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
    attr[0].val.programmaticStreamSerializationAllowed = 1;
    attr[1].id = cudaLaunchAttributeClusterDimension;
    attr[1].val.clusterDim.x = static_cast<unsigned>(cs);
    attr[1].val.clusterDim.y = 1;
    attr[1].val.clusterDim.z = 1;
    cfg.attrs = attr;
    cfg.numAttrs = 2;
    return cudaLaunchKernelEx(&cfg, kern, a);
  };
  // a token per thread where a block allows (the ranking of the pool and the
  // scatter around it, cycles per phase: 576 tokens on 144 threads of four each
  // 10.0 k, one each 6.4 k), and the narrowest of these blocks: barriers cost
  // by the warp. Past 768 tokens two or four each (three: more registers than
  // 1024 threads leave).
  if (p.N <= 512) return go(select_diverse_kernel<512, 1>, 512);
  if (p.N <= 640) return go(select_diverse_kernel<640, 1>, 640);
  if (p.N <= 768) return go(select_diverse_kernel<768, 1>, 768);
  if (p.N <= 1536) return go(select_diverse_kernel<768, 2>, 768);
  if (p.N <= 3072) return go(select_diverse_kernel<768, 4>, 768);
  return go(select_diverse_kernel<1024, 4>, 1024);
}

unsigned int diverse_read_and_clear_error() {
  unsigned int v = 0, z = 0;
  cudaMemcpyFromSymbol(&v, g_diverse_err, sizeof(v));
  cudaMemcpyToSymbol(g_diverse_err, &z, sizeof(z));
  return v;
}

}  // namespace p4q
