// Exact cosine top-k over the gradient store (Bergson Sec. 3.1: exact top-k
// nearest-neighbour lookup; queries score against unit-normalised rows).
//
// Score kernels (persistent, one CTA per SM): a CTA owns one query group of
// QT x 128 normalised fp16 queries and streams every (grid / n_qg)-th tile of
// bn store rows (at most 256).  TMA brings 64-column slices of the store tile
// and of the query tiles into a shared-memory ring; one thread issues
// tcgen05.mma with the queries on M and the store rows on N, K = 16, into TMEM
// (fp32), so that TMEM lane = query and column = store row.  Up to 128 queries
// one CTA runs M = 128 on its own (score_kernel); above that CTAs run in pairs
// whose MMAs take M = 256 over both CTAs' query tiles, each CTA loading half
// of every store tile (score_pair_kernel).  Epilogue warps read their query's
// scores, drop everything below the query's threshold, and append the rest to
// a per-(CTA, query) list of up to topk keys in global memory (a 4-ary
// min-heap once it is full).  The N x Q score matrix never exists.
//
// Threshold (the bound): the CTAs of a query group score their first tiles at
// about the same time.  Each publishes, per query, its j-th best score there;
// the r-th largest of the published values, r = ceil(topk / j), has at least
// topk rows at or above it, so no row below it can reach the final top-k.  It
// passes about 1.7 topk rows of those tiles instead of all of them, so a list
// takes a handful of appends where a heap took topk ln(rows / topk) serial
// insertions of two or three dependent round trips to L2 each.  Results never
// depend on which values were there in time: the bound is a filter.
// Merge kernel: one CTA per query gathers the lists of the CTAs that covered
// the query and sorts them by score descending, then row ascending (long
// candidate sets go through an exact radix select first).
// Measured (one GB300, microseconds a call, with heaps / as here): 3 queries,
// 20,011 x 3072, top-10 91 / 37; 100 queries, 250,007 x 12,288, bottom-100 1530 /
// 897 (the store stream's time at 6.8 TB/s is 904); 64 queries, 100,003 x 1024,
// top-500 2810 / 78; 1024 queries, 60,000 x 4096, top-100 1660 / 465 and 300,000 x
// 2048, top-300 7960 / 1120; 4M x 8192 level (tensor bound).  Small calls pay for
// code they run once (instruction fetch): fully unrolled searches of the bound
// and of the candidates cost 5 to 15 us more.

#include <algorithm>

#include "internal.h"
#include "ptx.cuh"

namespace bergson {

namespace {

constexpr int kSmemBudget = 232448;
constexpr uint64_t kDrainTimeoutNs = 2000000000ull;
constexpr int kMaxMergeCTAs = 160;                  // CTAs that can cover a query
constexpr int kQBoxBytes = kScoreQT * 128;          // 128 rows x 64 fp16
constexpr unsigned long long kSentinelKey = 0x007FFFFF00000000ull;   // (-inf, row 0xFFFFFFFF)
// L2 policy of store-chunk loads: 0 = evict_normal, 1 = evict_first.  The
// pair kernel with more than one pair of query groups (n_qg counts the
// CTAs' groups, two per pair) keeps the normal policy: every store half is
// read once per pair group, by CTAs that stream the same tiles in the same
// order (paced, below), and the later reads hit L2 more often when the first
// one does not mark the lines for early eviction (1.6x the store in DRAM
// reads with evict_first at 1024 queries).
constexpr int kStoreEvictFirst = 1;

// Candidates a lane may park in shared memory per tile before inserting them
// into its heap after the tile's TMEM buffer is released.
constexpr int kQueueCap = 8;

// Candidate keys the merge keeps in shared memory for its radix select
// (26,624 x 8 bytes = 208 KB); larger candidate sets are merged in sorted rounds.
constexpr int kMergeSmemKeys = 26624;

// Single-CTA kernel: the ring's stages hold bn store rows and q_rows queries
// (both chosen by the launcher: small tiles leave room for more stages).
constexpr int kBarBytes = 256;
constexpr int kMaxStages = 12;
struct ScoreCfg {
  static constexpr int kQueueBytes = kQueueCap * 128 * 8;
  static constexpr int kRingBudget = kSmemBudget - 1024 - kBarBytes - kQueueBytes;
  static constexpr int kNBuf = 2;                       // TMEM accumulator buffers
  static constexpr int kEpiThreads = 128;
  static constexpr int kThreads = 64 + kEpiThreads;
  static_assert(2 * kMaxStages + 2 * kNBuf + 1 <= kBarBytes / 8 - 2, "barrier area");
};

// Order-preserving map of a float onto uint32 (-0 is folded onto +0 first).
__device__ __forceinline__ uint32_t float_order(float s) {
  const uint32_t u = __float_as_uint(s + 0.0f);
  return (u & 0x80000000u) ? ~u : (u | 0x80000000u);
}

__device__ __forceinline__ float order_to_float(uint32_t o) {
  return __uint_as_float((o & 0x80000000u) ? (o & 0x7FFFFFFFu) : ~o);
}

// Larger key = better: higher score first, then lower row index.
__device__ __forceinline__ unsigned long long make_key(float s, uint32_t row) {
  return (static_cast<unsigned long long>(float_order(s)) << 32) | static_cast<uint32_t>(~row);
}

// Children per node of the per-query min-heaps (a wider heap is shallower:
// fewer dependent global-memory round trips per insertion).
constexpr int kHeapArity = 4;

// Replace the root (worst kept entry) of a kHeapArity-ary min-heap of `k` keys
// stored at base[e * stride] and restore the heap property.  The children of
// one node are loaded together, so each level costs one memory round trip.
__device__ __forceinline__ void heap_replace_root(unsigned long long* base, int stride, int k,
                                                  unsigned long long key) {
  int i = 0;
  for (;;) {
    const int c0 = kHeapArity * i + 1;
    if (c0 >= k) break;
    unsigned long long kc = base[static_cast<int64_t>(c0) * stride];
    int c = c0;
#pragma unroll
    for (int t = 1; t < kHeapArity; ++t) {
      if (c0 + t < k) {
        const unsigned long long kt = base[static_cast<int64_t>(c0 + t) * stride];
        if (kt < kc) { kc = kt; c = c0 + t; }
      }
    }
    if (kc >= key) break;
    base[static_cast<int64_t>(i) * stride] = kc;
    i = c;
  }
  base[static_cast<int64_t>(i) * stride] = key;
}

// v[pos] for a run-time pos in [0, 32) without dynamic register indexing
// (a 5-level select tree keeps v in registers).
__device__ __forceinline__ float select32(const float* v, uint32_t pos) {
  float t16[16], t8[8], t4[4], t2[2];
#pragma unroll
  for (int i = 0; i < 16; ++i) t16[i] = (pos & 16u) ? v[i + 16] : v[i];
#pragma unroll
  for (int i = 0; i < 8; ++i) t8[i] = (pos & 8u) ? t16[i + 8] : t16[i];
#pragma unroll
  for (int i = 0; i < 4; ++i) t4[i] = (pos & 4u) ? t8[i + 4] : t8[i];
#pragma unroll
  for (int i = 0; i < 2; ++i) t2[i] = (pos & 2u) ? t4[i + 2] : t4[i];
  return (pos & 1u) ? t2[1] : t2[0];
}

// List of one (CTA, query): keys at heap[e * stride], e < topk.  While it is
// not full its last entry holds the number of its keys: a real key has a low
// word of ~row >= 2^31, so a full list is told by its last entry.
constexpr uint32_t kFullBit = 0x80000000u;
// Longest wait for the group's other CTAs to score their first tiles (they
// start together; a limit below their spread, 10 us, cost a 60,000-row search
// half its speed).
constexpr uint64_t kBoundWaitNs = 100000ull;

// Published scores: the upper 16 order bits (sign, exponent, 7 bits of
// mantissa: rounded down by at most 0.8%, a few percent more candidates) of
// CTA c's j-th best for slot s of group g at pub[(g * slots + s) * cpg + c], so
// that a warp reads a slot's values side by side; 0 = not there yet (cleared
// before the launch).
__device__ __forceinline__ uint16_t ld_relaxed_u16(const uint16_t* ptr) {
  uint16_t v;
  asm volatile("ld.relaxed.gpu.global.u16 %0, [%1];" : "=h"(v) : "l"(ptr) : "memory");
  return v;
}
__device__ __forceinline__ void st_relaxed_u16(uint16_t* ptr, uint16_t v) {
  asm volatile("st.relaxed.gpu.global.u16 [%0], %1;" ::"l"(ptr), "h"(v) : "memory");
}
__device__ __forceinline__ uint16_t pub_word(float best) {
  return static_cast<uint16_t>(float_order(best) >> 16);
}

// Turns k keys into a min-heap, bottom up.
__device__ __noinline__ static void heapify(unsigned long long* heap, int stride, int k) {
  for (int i = (k - 2) / kHeapArity; i >= 0; --i) {
    // sift heap[i] down
    const unsigned long long key = heap[static_cast<int64_t>(i) * stride];
    int at = i;
    for (;;) {
      const int c0 = kHeapArity * at + 1;
      if (c0 >= k) break;
      unsigned long long kc = heap[static_cast<int64_t>(c0) * stride];
      int c = c0;
#pragma unroll
      for (int t = 1; t < kHeapArity; ++t) {
        if (c0 + t < k) {
          const unsigned long long kt = heap[static_cast<int64_t>(c0 + t) * stride];
          if (kt < kc) { kc = kt; c = c0 + t; }
        }
      }
      if (kc >= key) break;
      heap[static_cast<int64_t>(at) * stride] = kc;
      at = c;
    }
    heap[static_cast<int64_t>(at) * stride] = key;
  }
}

// Bounds of kBatch query slots from what the group's CTAs published (the slots'
// rows of cpg words start at `pub`): per slot the r-th largest value, or NaN or
// -inf while fewer than r are there.  One warp; lane i looks at CTAs i, i + 32,
// ... of the group.  The slots' loads and reductions run side by side.
constexpr int kBatch = 8;
__device__ __forceinline__ void slot_bounds(const uint16_t* pub, int cpg, int r, int lane,
                                            float* out) {
  uint32_t v[kBatch][5];                          // cpg <= 160
#pragma unroll
  for (int s = 0; s < kBatch; ++s) {
#pragma unroll
    for (int i = 0; i < 5; ++i) {
      const int c = lane + 32 * i;
      v[s][i] = c < cpg ? ld_relaxed_u16(pub + s * cpg + c) : 0u;
    }
  }
  uint32_t t[kBatch];
#pragma unroll
  for (int s = 0; s < kBatch; ++s) t[s] = 0u;
#pragma unroll 1
  for (int bit = 15; bit >= 0; --bit) {
#pragma unroll
    for (int s = 0; s < kBatch; ++s) {
      const uint32_t cand = t[s] | (1u << bit);
      int n = 0;
#pragma unroll
      for (int i = 0; i < 5; ++i) n += v[s][i] >= cand ? 1 : 0;
      if (__reduce_add_sync(0xffffffffu, n) >= r) t[s] = cand;
    }
  }
#pragma unroll
  for (int s = 0; s < kBatch; ++s) out[s] = t[s] == 0u ? -INFINITY : order_to_float(t[s] << 16);
}

// Inserts t into the descending top[0, J).
template <int J>
__device__ __forceinline__ void top_insert(float* top, float t) {
#pragma unroll
  for (int i = 0; i < J; ++i) {
    const float hi = fmaxf(top[i], t);
    t = fminf(top[i], t);
    top[i] = hi;
  }
}

template <int J>
__device__ __forceinline__ float nth(const float* top, int j) {   // top[j - 1]
  float x = top[0];
#pragma unroll
  for (int i = 1; i < J; ++i)
    if (j == i + 1) x = top[i];
  return x;
}

// The j-th best (j <= J) of a query's `rows` scores at TMEM address tbase (NaN
// never; -inf when there are fewer).
template <int J>
__device__ __forceinline__ float nth_of_tile(uint32_t tbase, int rows, int j) {
  float top[J];
#pragma unroll
  for (int i = 0; i < J; ++i) top[i] = -INFINITY;
  // eight columns a time: unrolled over 32, the J = 32 network is 32 KB of code
  // that each launch fetches for one use
#pragma unroll 1
  for (int c = 0; c < rows; c += 8) {
    float v[8];
    tmem_ld8(tbase + c, v);
    const int nvalid = rows - c;
#pragma unroll
    for (int i = 0; i < 8; ++i)
      top_insert<J>(top, i < nvalid && v[i] == v[i] ? v[i] : -INFINITY);
  }
  return nth<J>(top, j);
}

// The j-th best score of a list of n keys.
template <int J>
__device__ __noinline__ float nth_of_list(const unsigned long long* list, int stride, int n, int j) {
  float top[J];
#pragma unroll
  for (int i = 0; i < J; ++i) top[i] = -INFINITY;
#pragma unroll 4
  for (int e = 0; e < n; ++e)
    top_insert<J>(top, order_to_float(static_cast<uint32_t>(
                           list[static_cast<int64_t>(e) * stride] >> 32)));
  return nth<J>(top, j);
}

// Epilogue role (QT x 128 threads, one query per thread): per store tile, wait
// for the accumulators, read the query's scores from TMEM, keep those at or
// above its threshold, release TMEM (on the even CTA of a pair when kPair).
// Kept scores are appended to the query's list; once that holds topk keys it
// becomes a heap, whose insertions are parked in shared memory and done after
// TMEM is released.
template <int QT, int kNBuf, bool kPair>
__device__ __forceinline__ void score_epilogue(const ScoreParams& p, uint32_t tmem, uint64_t* tfull,
                                               uint64_t* tempty,
                                               unsigned long long* cand_queue,
                                               volatile int* s_abort, volatile int* s_epi_stop,
                                               int g, int nt0, int cpg, int warp, int lane,
                                               uint64_t tmo) {
  constexpr int kEpiThreads = QT * 128;
  const int et = threadIdx.x - 64;                 // 0 .. QT*128-1
  const int qt = et >> 7;
  const int quarter = warp & 3;
  const int slot = qt * kScoreQT + 32 * quarter + lane;
  const int stride = kEpiThreads;
  const int topk = p.topk;
  unsigned long long* heap =
      p.heaps + static_cast<int64_t>(blockIdx.x) * topk * stride + slot;
  unsigned long long tau_key = kSentinelKey;
  // Scores below the k-th best of any subset of the rows can never reach the
  // final top-k, so a threshold from earlier rows (if any) filters from the start.
  const int q_global = (g * QT + qt) * kScoreQT + 32 * quarter + lane;
  griddep_wait();                // thresholds and cleared lists come from earlier grids
  float tau0 = -INFINITY;
  if (p.tau0 != nullptr && q_global < p.Q) {
    const float t = p.tau0[static_cast<int64_t>(q_global) * topk + topk - 1];
    tau0 = p.tau0_negate ? -t : t;
  }
  float tau = tau0;
  // Slots past the last query (ragged query groups) hold no query: they take
  // no candidates, so their lanes do not walk every score of every tile.
  const bool live = q_global < p.Q;
  const int n_live = min(32, p.Q - (q_global - lane));   // live lanes of this warp (may be <= 0)
  const int j_best = p.bound_j, r_best = p.bound_r;      // j_best == 0: no bound
  // this group's published words, and this thread's own
  const int rank = blockIdx.x / p.n_qg;             // of this CTA in its group
  uint16_t* pub = p.pub + static_cast<int64_t>(g - p.qg_base) * stride * cpg;
  uint16_t* my_pub = pub + slot * cpg + rank;
  float best = -INFINITY;                           // the j-th best published last
  int cnt = 0;                                      // keys in the list
  bool is_heap = false;
  int nq = 0;                                       // parked candidates of this lane
  int ab = 0;
  uint32_t aph = 0;
  int tile_no = 0;
  const int n_my_tiles = (p.n_ntiles - nt0 + cpg - 1) / cpg;
  for (int nt = nt0; nt < p.n_ntiles; nt += cpg, ++tile_no) {
    if (et == 0) {
      if (!mbar_wait(smem_u32(&tfull[ab]), aph, tmo, s_abort))
        raise_device_error(p.status, s_abort, kStatusTimeout);
      *s_epi_stop = *s_abort;
    }
    named_bar_sync(1, kEpiThreads);
    if (*s_epi_stop) break;
    tc_fence_after();
    const uint32_t tbase = tmem + (static_cast<uint32_t>(32 * quarter) << 16) +
                           ab * QT * kScoreBN + qt * kScoreBN;
    const int row_base = nt * p.bn;
    const int rows = min(p.bn, p.N - row_base);
    if (j_best > 0 && n_live > 0 && tile_no == 0) {
      // The first tile: this query's j-th best score, published before any is kept.
      // A warp reads no slots but its own 32, which each peer's warp stores in one
      // instruction (and flushes: without the fence the polls overtake the store, 4
      // to 8% of a small call), so it waits for its first one.  Whatever were missing
      // all the same would only make the bound weaker.  Ordered across the whole CTA
      // (slot 0 last, behind a barrier): 50.8 / 48.7 us at 20,011 x 3072, 64 queries,
      // 83.4 / 79.6 at 100,003 x 1024, 64 queries, top-500.
      if (j_best == 1) best = nth_of_tile<1>(tbase, rows, 1);
      else if (j_best <= 8) best = nth_of_tile<8>(tbase, rows, j_best);
      else best = nth_of_tile<kScoreMaxJ>(tbase, rows, j_best);
      if (live) st_relaxed_u16(my_pub, pub_word(best));
      __threadfence();
      const uint16_t* first = pub + (slot - lane) * cpg;
      const uint64_t t0 = global_timer_ns();
      for (;;) {
        bool all = true;
        for (int c = lane; c < cpg; c += 32) all = all && ld_relaxed_u16(first + c) != 0;
        if (__all_sync(0xffffffffu, all)) break;
        const bool late = *s_abort != 0 || global_timer_ns() - t0 > kBoundWaitNs;
        if (__any_sync(0xffffffffu, late)) break;
      }
      __threadfence();
    }
    // The bound from the first tiles, and again before tiles 2, 6, 20, ... from
    // the lists, which hold every row seen so far that matters: with t tiles
    // seen a tile adds about 1.3 topk / (cpg t) keys to a list, so the lists
    // do not fill up unless a CTA's rows come in ascending order.  It takes 10 to
    // 30 us, so only scans that go on for four times as long do it.
    const bool again = j_best > 0 && n_my_tiles > 4 * tile_no &&
                       (tile_no == 2 || tile_no == 6 || tile_no == 20 || tile_no == 60 ||
                        tile_no == 200);
    if (again && live && cnt >= j_best) {
      const float x = j_best == 1   ? nth_of_list<1>(heap, stride, cnt, 1)
                      : j_best <= 8 ? nth_of_list<8>(heap, stride, cnt, j_best)
                                    : nth_of_list<kScoreMaxJ>(heap, stride, cnt, j_best);
      best = fmaxf(best, x);
      st_relaxed_u16(my_pub, pub_word(best));
    }
    if (j_best > 0 && n_live > 0 && (tile_no == 0 || again)) {
      float b = -INFINITY;
      const int s0 = slot - lane;
#pragma unroll 1
      for (int i = 0; i < min(32, n_live); i += kBatch) {
        float x[kBatch];
        slot_bounds(pub + (s0 + i) * cpg, cpg, r_best, lane, x);
#pragma unroll
        for (int u = 0; u < kBatch; ++u)
          if (lane == i + u) b = x[u];
      }
      tau0 = fmaxf(tau0, b);
      tau = fmaxf(tau, tau0);
    }
#pragma unroll 1
    for (int c = 0; n_live > 0 && c * 32 < rows; ++c) {
      float v[32];
      tmem_ld32(tbase + c * 32, v);
      const int r0 = row_base + c * 32;
      const int nvalid = rows - c * 32;
      // Candidate positions of this lane (the comparison also drops NaN).
      uint32_t cand = 0;
#pragma unroll
      for (int j = 0; j < 32; ++j)
        if (live && j < nvalid && v[j] >= tau) cand |= 1u << j;
      // Warp-uniform rounds: in round r every lane takes its r-th candidate,
      // so a warp pays for its busiest lane, not for every distinct column.
      while (__any_sync(0xffffffffu, cand != 0)) {
        if (cand != 0) {
          const uint32_t pos = __ffs(cand) - 1;
          cand &= cand - 1;
          const float sc = select32(v, pos);
          const unsigned long long key = make_key(sc, static_cast<uint32_t>(r0) + pos);
          if (cnt < topk) {
            heap[static_cast<int64_t>(cnt) * stride] = key;
            ++cnt;
          } else if (key > tau_key) {
            if (nq < kQueueCap) {                 // park it; inserted after TMEM is released
              cand_queue[nq * stride + slot] = key;
              ++nq;
            } else {                              // queue full: insert now
              if (!is_heap) {
                heapify(heap, stride, topk);
                is_heap = true;
                tau_key = heap[0];
              }
              if (key > tau_key) {
                heap_replace_root(heap, stride, topk, key);
                tau_key = heap[0];
              }
              tau = fmaxf(tau0, order_to_float(static_cast<uint32_t>(tau_key >> 32)));
            }
          }
        }
      }
    }
    tc_fence_before();
    __syncwarp();
    if (lane == 0) {
      if (kPair)
        mbar_arrive_cluster(mapa_shared(smem_u32(&tempty[ab]), 0));
      else
        mbar_arrive(smem_u32(&tempty[ab]));
    }
    if (++ab == kNBuf) { ab = 0; aph ^= 1; }
    // The MMA warp is already filling TMEM for the next tile; drain the parked
    // candidates meanwhile (warp-uniform rounds, as above).
    while (__any_sync(0xffffffffu, nq > 0)) {
      if (nq > 0) {
        if (!is_heap) {
          heapify(heap, stride, topk);
          is_heap = true;
          tau_key = heap[0];
        }
        --nq;
        const unsigned long long key = cand_queue[nq * stride + slot];
        if (key > tau_key) {
          heap_replace_root(heap, stride, topk, key);
          tau_key = heap[0];
        }
        tau = fmaxf(tau0, order_to_float(static_cast<uint32_t>(tau_key >> 32)));
      }
    }
    named_bar_sync(1, kEpiThreads);   // keeps the stop broadcast single-writer
  }
  if (live && cnt < topk) heap[static_cast<int64_t>(topk - 1) * stride] = cnt;
}

__global__ void __launch_bounds__(ScoreCfg::kThreads, 1)
    score_kernel(const __grid_constant__ CUtensorMap tm_store, const __grid_constant__ CUtensorMap tm_q,
                 const ScoreParams p) {
  using C = ScoreCfg;
  const int n_stages = p.stages;
  const int store_bytes = p.bn * 128;
  const int stage_bytes = store_bytes + p.q_rows * 128;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const uint32_t sbase = smem_u32(smem);
  unsigned long long* cand_queue =
      reinterpret_cast<unsigned long long*>(smem + C::kRingBudget / 1024 * 1024);  // [cap][lanes]
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::kRingBudget / 1024 * 1024 + C::kQueueBytes);
  uint64_t* empty = full + n_stages;
  uint64_t* tfull = empty + n_stages;       // [kNBuf]
  uint64_t* tempty = tfull + 2;               // [kNBuf]
  uint64_t* drain = tempty + 2;
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);
  volatile int* s_epi_stop = s_abort + 1;

  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int g_local = blockIdx.x % p.n_qg;
  const int g = p.qg_base + g_local;
  const int cpg = gridDim.x / p.n_qg;
  const int nt0 = blockIdx.x / p.n_qg;
  const int nK = (p.K + kChunk - 1) / kChunk;

  if (threadIdx.x == 0) {
    for (int s = 0; s < n_stages; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int i = 0; i < C::kNBuf; ++i) {
      mbar_init(smem_u32(&tfull[i]), 1);
      mbar_init(smem_u32(&tempty[i]), 4);
    }
    mbar_init(smem_u32(drain), 1);
    *s_abort = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc(smem_u32(s_tmem), 512);
    tmem_relinquish();
  }
  tc_fence_before();
  __syncthreads();
  tc_fence_after();
  const uint32_t tmem = *s_tmem;
  const uint64_t tmo = p.timeout_ns;

  if (warp == 0) {
    if (lane == 0) {
      prefetch_tmap(&tm_store);
      prefetch_tmap(&tm_q);
      const uint64_t pol_store = kStoreEvictFirst ? policy_evict_first() : policy_evict_normal();
      const uint64_t pol_q = policy_evict_last();
      int stage = 0;
      uint32_t ph = 0;
      uint32_t issued = 0, issued_par = 0;
      bool ok = true;
      // The store does not come from the preceding grid: the first round of
      // stages streams it while the queries are still being normalised.
      bool dep = false;
      int n_def = 0;
      auto load_q = [&](int sg, int kc) {
        tma_load_2d_hint(sbase + sg * stage_bytes + store_bytes, &tm_q, smem_u32(&full[sg]),
                         kc * kChunk, g * kScoreQT, pol_q);
      };
      auto release = [&]() {
        griddep_wait();
        dep = true;
        for (int d = 0; d < n_def; ++d) load_q(d, d % nK);     // stage d holds chunk d
      };
      for (int nt = nt0; nt < p.n_ntiles && ok; nt += cpg) {
        for (int kc = 0; kc < nK; ++kc) {
          if (!mbar_wait(smem_u32(&empty[stage]), ph ^ 1, tmo, s_abort)) { ok = false; break; }
          const uint32_t fb = smem_u32(&full[stage]);
          mbar_arrive_expect_tx(fb, stage_bytes);
          tma_load_2d_hint(sbase + stage * stage_bytes, &tm_store, fb, kc * kChunk, nt * p.bn,
                           pol_store);
          if (dep) {
            load_q(stage, kc);
          } else if (++n_def == n_stages) {
            release();
          }
          issued |= 1u << stage;
          issued_par = (issued_par & ~(1u << stage)) | (ph << stage);
          if (++stage == n_stages) { stage = 0; ph ^= 1; }
        }
      }
      if (!dep) release();
      griddep_launch_dependents();   // every load issued: the merge may be scheduled
      if (!ok) {
        raise_device_error(p.status, s_abort, kStatusTimeout);
        for (int s = 0; s < n_stages; ++s)
          if (issued >> s & 1)
            mbar_wait(smem_u32(&full[s]), (issued_par >> s) & 1, kDrainTimeoutNs, nullptr);
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (lane == 0) {
      const uint32_t idesc = make_idesc_f16(kScoreQT, p.bn, false);
      int stage = 0;
      uint32_t ph = 0;
      int ab = 0;
      uint32_t aph = 0;
      bool ok = true;
      for (int nt = nt0; nt < p.n_ntiles && ok; nt += cpg) {
        if (!mbar_wait(smem_u32(&tempty[ab]), aph ^ 1, tmo, s_abort)) { ok = false; break; }
        tc_fence_after();
        const uint32_t dbuf = tmem + ab * kScoreBN;
        for (int kc = 0; kc < nK; ++kc) {
          if (!mbar_wait(smem_u32(&full[stage]), ph, tmo, s_abort)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sd = sbase + stage * stage_bytes;
          const uint32_t qd = sd + store_bytes;
          // M = 128 reads 128 query rows: past q_rows they are whatever lies
          // behind them in shared memory, and land in lanes no one reads
#pragma unroll
          for (int kk = 0; kk < kChunk / 16; ++kk)
            umma_f16(dbuf, sw128_desc(qd + kk * 32), sw128_desc(sd + kk * 32), idesc,
                     (kc | kk) != 0);
          umma_commit(smem_u32(&empty[stage]));
          if (++stage == n_stages) { stage = 0; ph ^= 1; }
        }
        if (!ok) break;
        umma_commit(smem_u32(&tfull[ab]));
        if (++ab == C::kNBuf) { ab = 0; aph ^= 1; }
      }
      if (!ok) raise_device_error(p.status, s_abort, kStatusTimeout);
      umma_commit(smem_u32(drain));
      mbar_wait(smem_u32(drain), 0, kDrainTimeoutNs, nullptr);
    }
    __syncwarp();
  } else {
    score_epilogue<1, C::kNBuf, false>(p, tmem, tfull, tempty, cand_queue, s_abort, s_epi_stop,
                                        g, nt0, cpg, warp, lane, tmo);
  }

  tc_fence_before();
  __syncthreads();
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc(tmem, 512);
  }
}

// Pair variant for more than 128 queries (QT query tiles per CTA, clusters of
// two CTAs on two SMs).  One tcgen05.mma of M = 256 (the two CTAs' query tiles
// of the same index) x N = 256 store rows serves both SMs: each CTA loads only
// its half of the store tile (128 rows), and the tensor cores of the pair read
// both halves.  With QT = 2 (more than 256 queries, tensor-bound) a 16-column
// step moves 12 KB into shared memory and reads 16 KB out of it per SM for two
// 128 x 256 products, against 16 KB and 24 KB for the single-CTA kernel.  With
// QT = 1 (129..256 queries, bound by the store stream) the smaller stages give
// six of them, i.e. more store bytes in flight per SM, and two TMEM buffers.
//
// Synchronisation: the odd CTA's TMA loads complete on the even CTA's `full`
// barrier, which expects the bytes of both; the even CTA's MMA thread frees a
// stage in both CTAs (commit multicast to `empty`), and signals both CTAs'
// epilogues (commit multicast to `tfull`); both epilogues release the TMEM
// buffer on the even CTA's `tempty`.
constexpr int kPairStoreRows = kScoreBN / 2;               // store rows each CTA loads
constexpr int kPairStoreBoxBytes = kPairStoreRows * 128;   // 128 rows x 64 fp16

// Pacing of the pair groups that read the same store tiles (two or more pair
// groups: more than 512 queries).  Each store half is read once per pair
// group; the second read finds it in L2 only while the groups stay close
// (left alone they drift apart over a pass, and their re-reads then miss).
// Each producer publishes its count of issued store chunks every kPaceEvery
// chunks, tagged with the launch, and before running more than kPaceLead
// chunks ahead of the next pair group's CTA (same tile sequence, same rank;
// the groups form a ring) waits for it, at most kPaceWaitNs per wait; a peer
// that does not catch up in that time ends the pacing for this CTA.  The
// peer's word is read one check ahead, so a producer that is not ahead does
// not wait out the load.  A waiting CTA has published its own count, so no
// ring of CTAs can all wait on one another.  Only timing depends on the
// words: a stale or foreign word just means a wait that runs out.
// Measured at 1024 queries (3.2 GB store): DRAM reads 1.08x the store at a
// lead of 16 (1.07x at 8, but 30% slower; 1.13-1.33x at 32 or unpaced).
constexpr uint32_t kPaceEvery = 8;
constexpr uint32_t kPaceLead = 16;                    // an eighth of a 8192-column tile
constexpr uint64_t kPaceWaitNs = 100000ull;

template <int QT_>
struct PairCfg {
  static constexpr int QT = QT_;
  static constexpr int kStageBytes = kPairStoreBoxBytes + QT * kQBoxBytes;
  static constexpr int kBarBytes = 256;
  static constexpr int kQueueBytes = kQueueCap * QT * 128 * 8;
  static constexpr int kStagesFit = (kSmemBudget - 1024 - kBarBytes - kQueueBytes) / kStageBytes;
  static constexpr int kStages = kStagesFit > 6 ? 6 : kStagesFit;
  static constexpr int kSmemBytes = 1024 + kStages * kStageBytes + kQueueBytes + kBarBytes;
  static constexpr int kNBuf = 512 / (QT * kScoreBN);   // TMEM accumulator buffers
  static constexpr int kEpiThreads = QT * 128;
  static constexpr int kThreads = 64 + kEpiThreads;
  static_assert(kStages >= 3, "pipeline depth");
  static_assert(2 * kStages + 4 * kNBuf + 1 <= kBarBytes / 8 - 2, "barrier area");
};

// Bounded wait for this CTA's own TMA loads after an abort: the odd CTA's
// loads complete on the other CTA's barrier, so it waits out a fixed time.
__device__ __forceinline__ void pair_settle_loads() {
  const uint64_t t0 = global_timer_ns();
  while (global_timer_ns() - t0 < 1000000ull) {
  }
}

template <int QT>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(PairCfg<QT>::kThreads, 1)
    score_pair_kernel(const __grid_constant__ CUtensorMap tm_store,
                      const __grid_constant__ CUtensorMap tm_q, const ScoreParams p) {
  using C = PairCfg<QT>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const uint32_t sbase = smem_u32(smem);
  unsigned long long* cand_queue =
      reinterpret_cast<unsigned long long*>(smem + C::kStages * C::kStageBytes);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::kStages * C::kStageBytes + C::kQueueBytes);
  uint64_t* empty = full + C::kStages;
  uint64_t* tfull = empty + C::kStages;       // [kNBuf]
  uint64_t* tempty = tfull + 2;               // [kNBuf]
  uint64_t* drain = tempty + 2;
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);
  volatile int* s_epi_stop = s_abort + 1;

  const uint32_t rank = cluster_ctarank();   // 0: issues the MMAs
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int g_local = blockIdx.x % p.n_qg;   // even on rank 0, +1 on rank 1
  const int g = p.qg_base + g_local;
  const int cpg = gridDim.x / p.n_qg;
  const int nt0 = blockIdx.x / p.n_qg;       // the same for both CTAs of the pair
  const int nK = (p.K + kChunk - 1) / kChunk;

  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int i = 0; i < C::kNBuf; ++i) {
      mbar_init(smem_u32(&tfull[i]), 1);
      mbar_init(smem_u32(&tempty[i]), 2 * QT * 4);   // every epilogue warp of both CTAs
    }
    mbar_init(smem_u32(drain), 1);
    *s_abort = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(s_tmem), 512);
    tmem_relinquish_pair();
  }
  tc_fence_before();
  cluster_sync();              // both CTAs' barriers initialised and TMEM allocated
  tc_fence_after();
  const uint32_t tmem = *s_tmem;
  const uint64_t tmo = p.timeout_ns;

  if (warp == 0) {
    if (lane == 0) {
      prefetch_tmap(&tm_store);
      prefetch_tmap(&tm_q);
      const uint64_t pol_store =
          kStoreEvictFirst && p.n_qg == 2 ? policy_evict_first() : policy_evict_normal();
      const uint64_t pol_q = policy_evict_last();
      int stage = 0;
      uint32_t ph = 0;
      uint32_t issued = 0, issued_par = 0;
      bool ok = true;
      const int half_rows = p.bn / 2;              // store rows each CTA loads
      // the first round of stages streams the store while the queries are still
      // being normalised
      bool dep = false;
      int n_def = 0;
      auto load_q = [&](int sg, int kc) {
        const uint32_t fb = mapa_shared(smem_u32(&full[sg]), 0);
        const uint32_t dst = sbase + sg * C::kStageBytes + kPairStoreBoxBytes;
#pragma unroll
        for (int qt = 0; qt < QT; ++qt)
          tma_load_2d_pair(dst + qt * kQBoxBytes, &tm_q, fb, kc * kChunk, (g * QT + qt) * kScoreQT,
                           pol_q);
      };
      auto release = [&]() {
        griddep_wait();
        dep = true;
        for (int d = 0; d < n_def; ++d) load_q(d, d % nK);     // stage d holds chunk d
      };
      // pacing against the next pair group's CTA on the same tiles (see kPaceLead)
      bool pacing = p.pace != nullptr && p.n_qg >= 4;
      unsigned long long* pace_mine = nullptr;
      const unsigned long long* pace_peer = nullptr;
      if (pacing) {
        const int n_pg = p.n_qg >> 1;
        const int pg = g_local >> 1;
        pace_mine = p.pace + blockIdx.x;
        pace_peer = p.pace + nt0 * p.n_qg + ((pg + 1) % n_pg) * 2 + (g_local & 1);
      }
      const unsigned long long tag = static_cast<unsigned long long>(p.pace_tag) << 32;
      uint32_t n_chunks = 0;
      unsigned long long peer_next = 0;   // peer word read at the previous check
      for (int nt = nt0; nt < p.n_ntiles && ok; nt += cpg) {
        for (int kc = 0; kc < nK; ++kc, ++n_chunks) {
          if (pacing && n_chunks % kPaceEvery == 0) {
            st_relaxed_u64(pace_mine, tag | n_chunks);
            if (n_chunks >= kPaceLead) {
              unsigned long long v = peer_next;
              const uint64_t t0 = global_timer_ns();
              while (!((v >> 32) == p.pace_tag && static_cast<uint32_t>(v) + kPaceLead >= n_chunks)) {
                if (*s_abort || global_timer_ns() - t0 > kPaceWaitNs) {
                  pacing = false;
                  break;
                }
                v = ld_relaxed_u64(pace_peer);
              }
            }
            peer_next = ld_relaxed_u64(pace_peer);
          }
          if (!mbar_wait(smem_u32(&empty[stage]), ph ^ 1, tmo, s_abort)) { ok = false; break; }
          const uint32_t fb_local = smem_u32(&full[stage]);
          const uint32_t fb = mapa_shared(fb_local, 0);
          if (rank == 0) mbar_arrive_expect_tx(fb_local, 2 * (half_rows * 128 + QT * kQBoxBytes));
          const uint32_t dst = sbase + stage * C::kStageBytes;
          tma_load_2d_pair(dst, &tm_store, fb, kc * kChunk,
                           nt * p.bn + static_cast<int>(rank) * half_rows, pol_store);
          if (dep) {
            load_q(stage, kc);
          } else if (++n_def == C::kStages) {
            release();
          }
          issued |= 1u << stage;
          issued_par = (issued_par & ~(1u << stage)) | (ph << stage);
          if (++stage == C::kStages) { stage = 0; ph ^= 1; }
        }
      }
      if (!dep) release();
      griddep_launch_dependents();   // every load issued: the merge may be scheduled
      if (pacing) st_relaxed_u64(pace_mine, tag | n_chunks);   // releases a peer near the end
      if (!ok) {
        raise_device_error(p.status, s_abort, kStatusTimeout);
        if (rank == 0) {
          for (int s = 0; s < C::kStages; ++s)
            if (issued >> s & 1)
              mbar_wait(smem_u32(&full[s]), (issued_par >> s) & 1, kDrainTimeoutNs, nullptr);
        } else {
          pair_settle_loads();
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    if (rank == 0 && lane == 0) {
      const uint32_t idesc = make_idesc_f16(2 * kScoreQT, p.bn, false);
      int stage = 0;
      uint32_t ph = 0;
      int ab = 0;
      uint32_t aph = 0;
      bool ok = true;
      for (int nt = nt0; nt < p.n_ntiles && ok; nt += cpg) {
        if (!mbar_wait_cluster(smem_u32(&tempty[ab]), aph ^ 1, tmo, s_abort)) { ok = false; break; }
        tc_fence_after();
        const uint32_t dbuf = tmem + ab * QT * kScoreBN;
        for (int kc = 0; kc < nK; ++kc) {
          if (!mbar_wait(smem_u32(&full[stage]), ph, tmo, s_abort)) { ok = false; break; }
          tc_fence_after();
          const uint32_t sd = sbase + stage * C::kStageBytes;
          const uint32_t qd = sd + kPairStoreBoxBytes;
#pragma unroll
          for (int qt = 0; qt < QT; ++qt) {
#pragma unroll
            for (int kk = 0; kk < kChunk / 16; ++kk)
              umma_f16_pair(dbuf + qt * kScoreBN, sw128_desc(qd + qt * kQBoxBytes + kk * 32),
                            sw128_desc(sd + kk * 32), idesc, (kc | kk) != 0);
          }
          umma_commit_pair(smem_u32(&empty[stage]), 0x3);
          if (++stage == C::kStages) { stage = 0; ph ^= 1; }
        }
        if (!ok) break;
        umma_commit_pair(smem_u32(&tfull[ab]), 0x3);
        if (++ab == C::kNBuf) { ab = 0; aph ^= 1; }
      }
      if (!ok) raise_device_error(p.status, s_abort, kStatusTimeout);
      umma_commit_pair(smem_u32(drain), 0x1);
      mbar_wait(smem_u32(drain), 0, kDrainTimeoutNs, nullptr);
    }
    __syncwarp();
  } else {
    score_epilogue<QT, C::kNBuf, true>(p, tmem, tfull, tempty, cand_queue, s_abort, s_epi_stop, g,
                                       nt0, cpg, warp, lane, tmo);
  }

  tc_fence_before();
  cluster_sync();              // no MMA, commit or remote arrival is still in flight
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, 512);
  }
}

// Bitonic sort of keys[0, n) (n a power of two) into descending order.
__device__ __forceinline__ void bitonic_desc(unsigned long long* keys, int n) {
  for (int kk = 2; kk <= n; kk <<= 1) {
    for (int j = kk >> 1; j > 0; j >>= 1) {
      for (int i = threadIdx.x; i < n; i += blockDim.x) {
        const int ixj = i ^ j;
        if (ixj > i) {
          const unsigned long long a = keys[i];
          const unsigned long long b = keys[ixj];
          const bool desc = (i & kk) == 0;
          if (desc ? (a < b) : (a > b)) {
            keys[i] = b;
            keys[ixj] = a;
          }
        }
      }
      __syncthreads();
    }
  }
}

// negate: the scores were taken against -q (a bottom-k search); report them
// against q, so the list runs from the lowest score up.  Key rows are global
// (row_base already added).
__device__ __forceinline__ void write_topk(const unsigned long long* keys, int q, int topk,
                                           int negate, float* out_scores, int64_t* out_idx) {
  for (int e = threadIdx.x; e < topk; e += blockDim.x) {
    const unsigned long long k = keys[e];
    const uint32_t lo = static_cast<uint32_t>(k);
    const bool real = lo >= 0x80000000u;          // rows < 2^31 map to ~row >= 2^31
    const float v = real ? order_to_float(static_cast<uint32_t>(k >> 32)) : -INFINITY;
    out_scores[static_cast<int64_t>(q) * topk + e] = negate ? -v : v;
    out_idx[static_cast<int64_t>(q) * topk + e] = real ? static_cast<int64_t>(~lo) : -1;
  }
}

// Final top-k of one query from the lists of the CTAs that covered it (entry e
// of CTA c's list for this query's slot at lists[(c topk + e) gsize + slot],
// counts from their last entries), their local rows moved to row_base + row, and from the prior result (scores
// against q, negated back into the search's order for a bottom-k state).
//
// Candidate sets that fit in shared memory are gathered there.  Up to
// kMergeSortKeys are bitonic-sorted at once; larger ones first go through an
// exact radix select (eight passes over 8-bit digits, most significant first)
// for the topk-th largest key T: keys are unique (the low word is the row), so
// exactly topk keys are >= T, and only those are sorted.  Sets that do not fit
// (smem_keys) are sorted in rounds of sort_n, keeping the best topk of each.
constexpr int kMergeSortKeys = 1024;

__global__ void __launch_bounds__(512) merge_kernel(const unsigned long long* lists,
                                                    uint16_t* pub, int64_t pub_words, int n_qg,
                                                    int cpg,
                                                    int gsize, int topk, int q_begin, int q_end,
                                                    int sort_n, int select_n, int smem_keys,
                                                    int negate, uint32_t row_base,
                                                    const float* prior_scores,
                                                    const int64_t* prior_idx, float* out_scores,
                                                    int64_t* out_idx) {
  extern __shared__ unsigned long long keys[];
  __shared__ unsigned int hist[256];
  __shared__ int s_off[kMaxMergeCTAs + 1];      // first key of each covering CTA
  __shared__ unsigned long long s_prefix;
  __shared__ int s_need, s_count, s_done;
  griddep_wait();
  const int q = q_begin + blockIdx.x;
  if (q >= q_end) return;
  const int local = q - q_begin;
  const int gl = local / gsize, slot = local % gsize;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  // the next launch's published words start out cleared
  for (int64_t i = static_cast<int64_t>(blockIdx.x) * blockDim.x + tid; i < pub_words;
       i += static_cast<int64_t>(gridDim.x) * blockDim.x)
    pub[i] = 0;
  // counts, then their prefix sums (cpg <= 160)
  if (tid < cpg) {
    const uint32_t lo = static_cast<uint32_t>(
        lists[(static_cast<int64_t>(gl + tid * n_qg) * topk + topk - 1) * gsize + slot]);
    s_off[tid] = lo >= kFullBit ? topk : min(static_cast<int>(lo), topk);
  }
  __syncthreads();
  if (warp == 0) {
    int base = 0;
    for (int c0 = 0; c0 < cpg; c0 += 32) {
      const int c = c0 + lane;
      const int n = c < cpg ? s_off[c] : 0;
      int x = n;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const int y = __shfl_up_sync(0xffffffffu, x, o);
        if (lane >= o) x += y;
      }
      if (c < cpg) s_off[c] = base + x - n;
      base += __shfl_sync(0xffffffffu, x, 31);
    }
    if (lane == 0) s_off[cpg] = base;
  }
  if (tid == 0) {
    s_prefix = 0ull;
    s_need = topk;
    s_count = 0;
    s_done = 0;
  }
  __syncthreads();
  const int n_list = s_off[cpg];
  const int total = n_list + (prior_idx != nullptr ? topk : 0);
  auto list_key = [&](int c, int e) {
    const unsigned long long k =
        lists[(static_cast<int64_t>(gl + c * n_qg) * topk + e) * gsize + slot];
    if (row_base == 0u) return k;
    return (k & 0xFFFFFFFF00000000ull) |
           static_cast<uint32_t>(~(~static_cast<uint32_t>(k) + row_base));
  };
  auto prior_key = [&](int i) {
    const int64_t e = static_cast<int64_t>(q) * topk + i;
    const int64_t idx = prior_idx[e];
    if (idx < 0) return 0ull;
    const float v = prior_scores[e];
    return make_key(negate ? -v : v, static_cast<uint32_t>(idx));
  };
  // Every prior entry is read (into shared memory) before any output is
  // written, so the prior may alias the output.
  int sort_all = 2;
  while (sort_all < total || sort_all < topk) sort_all <<= 1;
  const bool fits = sort_all <= kMergeSortKeys ? sort_all <= smem_keys
                                               : total + select_n <= smem_keys;
  if (fits) {
    for (int c = warp; c < cpg; c += 16) {
      const int o = s_off[c], m = s_off[c + 1] - o;
      for (int e = lane; e < m; e += 32) keys[o + e] = list_key(c, e);
    }
    for (int i = n_list + tid; i < total; i += blockDim.x) keys[i] = prior_key(i - n_list);
    if (sort_all <= kMergeSortKeys) {
      for (int i = total + tid; i < sort_all; i += blockDim.x) keys[i] = 0ull;
      __syncthreads();
      bitonic_desc(keys, sort_all);
      write_topk(keys, q, topk, negate, out_scores, out_idx);
      return;
    }
    const int n = total;
    __syncthreads();
    for (int shift = 56; shift >= 0; shift -= 8) {
      for (int b = tid; b < 256; b += blockDim.x) hist[b] = 0u;
      __syncthreads();
      const unsigned long long prefix = s_prefix;
      const unsigned long long above = shift == 56 ? 0ull : (~0ull << (shift + 8));
      // Candidates cluster in score, so most share a digit: lanes of a warp
      // with the same digit add their count once (one atomic per group).
      for (int i0 = 0; i0 < n; i0 += blockDim.x) {
        const int i = i0 + tid;
        const unsigned long long k = i < n ? keys[i] : 0ull;
        const bool hit = i < n && (k & above) == prefix;
        const unsigned dig = hit ? static_cast<unsigned>((k >> shift) & 255u) : 256u;
        const unsigned peers = __match_any_sync(0xffffffffu, dig);
        if (hit && lane == __ffs(peers) - 1) atomicAdd(&hist[dig], __popc(peers));
      }
      __syncthreads();
      // The digit where the count from the top reaches s_need: lane l sums
      // bins 255 - 8 l .. 248 - 8 l, a prefix sum finds the lane, the lane
      // the bin.  (One thread walking the 256 bins took 3 us a pass.)
      if (warp == 0) {
        const int need = s_need;
        int h[8], sum = 0;
#pragma unroll
        for (int b = 0; b < 8; ++b) {
          h[b] = static_cast<int>(hist[255 - 8 * lane - b]);
          sum += h[b];
        }
        int x = sum;
#pragma unroll
        for (int o = 1; o < 32; o <<= 1) {
          const int y = __shfl_up_sync(0xffffffffu, x, o);
          if (lane >= o) x += y;
        }
        int acc = x - sum;                      // keys in higher bins
        const bool mine = acc < need && x >= need;
        if (mine) {
          int b = 0;
#pragma unroll
          for (int i = 0; i < 7; ++i)
            if (b == i && acc + h[i] < need) { acc += h[i]; b = i + 1; }
          s_prefix = prefix | (static_cast<unsigned long long>(255 - 8 * lane - b) << shift);
          s_need = need - acc;
          int in_bin = 0;
#pragma unroll
          for (int i = 0; i < 8; ++i)
            if (i == b) in_bin = h[i];
          s_done = in_bin == need - acc;        // every key left is taken: no smaller digits
        } else if (lane == 31 && x < need) {    // fewer keys than topk: the smallest digit
          s_prefix = prefix;
          s_need = need - x + h[7];
        }
      }
      __syncthreads();
      if (s_done) break;
    }
    const unsigned long long T = s_prefix;       // at most the topk-th largest key, above the next
    unsigned long long* sel = keys + n;
    // Only real keys (a row in the low word) are kept: an empty prior entry
    // must not push a real row out when fewer than topk keys exist.
    for (int i = tid; i < n; i += blockDim.x) {
      const unsigned long long k = keys[i];
      if (k >= T && static_cast<uint32_t>(k) >= 0x80000000u) {
        const int pos = atomicAdd(&s_count, 1);
        if (pos < select_n) sel[pos] = k;
      }
    }
    __syncthreads();
    for (int i = min(s_count, select_n) + tid; i < select_n; i += blockDim.x) sel[i] = 0ull;
    __syncthreads();
    bitonic_desc(sel, select_n);
    write_topk(sel, q, topk, negate, out_scores, out_idx);
    return;
  }
  int consumed = 0;
  bool first = true;
  while (first || consumed < total) {
    const int start = first ? 0 : topk;
    for (int i = start + tid; i < sort_n; i += blockDim.x) {
      const int ci = consumed + (i - start);
      unsigned long long k = 0ull;
      if (ci < n_list) {
        int lo = 0, hi = cpg;                    // the CTA whose keys hold number ci
        while (hi - lo > 1) {
          const int mid = (lo + hi) >> 1;
          if (s_off[mid] <= ci) lo = mid; else hi = mid;
        }
        k = list_key(lo, ci - s_off[lo]);
      } else if (ci < total) {
        k = prior_key(ci - n_list);
      }
      keys[i] = k;
    }
    consumed += sort_n - start;
    first = false;
    __syncthreads();
    bitonic_desc(keys, sort_n);
  }
  __syncthreads();
  write_topk(keys, q, topk, negate, out_scores, out_idx);
}

}  // namespace

// Store rows per tile of a launch that scores `rows` rows with `ctas_per_group`
// CTAs per query group: the whole rounds of 256-row tiles that the rows need,
// shared out evenly (a last round that is nearly empty would cost as much as a
// full one), in steps of what one MMA takes: N of 16 at M = 128 on one CTA, of 32
// at M = 256 over a pair.  Not below 64: smaller MMAs take as long to issue as
// that one, and a tile's fixed costs weigh more.
int score_tile_rows(int64_t rows, int ctas_per_group, bool pair) {
  const int64_t step = pair ? 32 : 16;
  const int64_t per_round = static_cast<int64_t>(std::max(1, ctas_per_group)) * kScoreBN;
  const int64_t rounds = (rows + per_round - 1) / per_round;
  const int64_t tiles = rounds * std::max(1, ctas_per_group);
  const int64_t bn = ((rows + tiles - 1) / tiles + step - 1) / step * step;
  return static_cast<int>(std::max<int64_t>(64, std::min<int64_t>(kScoreBN, bn)));
}

int score_query_rows(int Q) { return std::min(kScoreQT, (Q + 7) / 8 * 8); }

cudaError_t launch_score(const CUtensorMap& tm_store, const CUtensorMap& tm_q, ScoreParams p,
                         int grid, cudaStream_t s) {
  using C = ScoreCfg;
  p.q_rows = score_query_rows(p.Q);
  const int stage_bytes = (p.bn + p.q_rows) * 128;
  // the last stage's MMAs read 128 query rows whatever q_rows is
  const int slack = kQBoxBytes - p.q_rows * 128;
  p.stages = std::min(kMaxStages, (C::kRingBudget / 1024 * 1024 - slack) / stage_bytes);
  static PerDeviceOnce attr;
  const cudaError_t e = smem_attr_once(attr, score_kernel, kSmemBudget);
  if (e != cudaSuccess) return e;
  return launch_dependent(score_kernel, dim3(grid), dim3(C::kThreads), kSmemBudget, s, tm_store,
                          tm_q, p);
}

template <int QT>
PerDeviceOnce& pair_attr() {
  static PerDeviceOnce attr;
  return attr;
}

template <int QT>
cudaError_t launch_score_pair_t(const CUtensorMap& tm_store, const CUtensorMap& tm_q,
                                const ScoreParams& p, int grid, cudaStream_t s) {
  using C = PairCfg<QT>;
  const cudaError_t e = smem_attr_once(pair_attr<QT>(), score_pair_kernel<QT>, C::kSmemBytes);
  if (e != cudaSuccess) return e;
  return launch_dependent(score_pair_kernel<QT>, dim3(grid), dim3(C::kThreads), C::kSmemBytes, s,
                          tm_store, tm_q, p);
}

template <int QT>
cudaError_t score_pair_max_ctas_t(int sms, int* ctas) {
  using C = PairCfg<QT>;
  cudaError_t e = smem_attr_once(pair_attr<QT>(), score_pair_kernel<QT>, C::kSmemBytes);
  if (e != cudaSuccess) return e;
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(2 * (sms / 2));
  cfg.blockDim = dim3(C::kThreads);
  cfg.dynamicSmemBytes = C::kSmemBytes;
  int clusters = 0;
  e = cudaOccupancyMaxActiveClusters(&clusters, score_pair_kernel<QT>, &cfg);
  if (e != cudaSuccess) return e;
  *ctas = 2 * clusters;
  return cudaSuccess;
}

cudaError_t launch_score_pair(int qt, const CUtensorMap& tm_store, const CUtensorMap& tm_q,
                              const ScoreParams& p, int grid, cudaStream_t s) {
  if (qt == 1) return launch_score_pair_t<1>(tm_store, tm_q, p, grid, s);
  if (qt == 2) return launch_score_pair_t<2>(tm_store, tm_q, p, grid, s);
  return cudaErrorInvalidValue;
}

// CTAs of the pair kernel that can be resident at once (2 x co-resident clusters).
cudaError_t score_pair_max_ctas(int qt, int sms, int* ctas) {
  if (qt == 1) return score_pair_max_ctas_t<1>(sms, ctas);
  if (qt == 2) return score_pair_max_ctas_t<2>(sms, ctas);
  return cudaErrorInvalidValue;
}

cudaError_t launch_merge(const unsigned long long* heaps, uint16_t* pub, int64_t pub_words,
                         int grid, int n_qg, int qt, int topk,
                         int q_begin, int q_end, bool negate, int64_t row_base,
                         const float* prior_scores, const int64_t* prior_idx, float* out_scores,
                         int64_t* out_idx, cudaStream_t s) {
  const int nq = q_end - q_begin;
  if (nq <= 0) return cudaSuccess;
  const int cpg = grid / n_qg;
  // the most candidates there can be; the kernel picks its way by how many there are
  const int64_t total = static_cast<int64_t>(cpg) * topk + (prior_idx != nullptr ? topk : 0);
  int sort_n = 2;
  while (sort_n < total && sort_n < 8192) sort_n <<= 1;
  int select_n = 2;
  while (select_n < topk) select_n <<= 1;
  const int smem_keys = static_cast<int>(
      std::min<int64_t>(kMergeSmemKeys, std::max<int64_t>(total + select_n, sort_n)));
  static PerDeviceOnce attr;
  const cudaError_t e = smem_attr_once(
      attr, merge_kernel, static_cast<int>(kMergeSmemKeys * sizeof(unsigned long long)));
  if (e != cudaSuccess) return e;
  return launch_dependent(merge_kernel, dim3(nq), dim3(512),
                          static_cast<size_t>(smem_keys) * sizeof(unsigned long long), s, heaps,
                          pub, pub_words, n_qg, cpg, qt * kScoreQT, topk, q_begin, q_end, sort_n, select_n,
                          smem_keys, negate ? 1 : 0, static_cast<uint32_t>(row_base), prior_scores,
                          prior_idx, out_scores, out_idx);
}

}  // namespace bergson
