// Square products of the Fisher preconditioner (C[b, q] = <x_b, y_q> for two
// operands of thousands of rows, fp32 accuracy) on the tensor cores.
//
// Operands are split once, by the pass that writes them, into three bf16 planes
//   x = x0 + x1 + x2,  x0 = bf16(x), x1 = bf16(x - x0), x2 = bf16(x - x0 - x1)
// (each rounded to nearest), which hold all 24 bits of every entry at any
// magnitude, and the product is taken as the six terms down to 2^-16,
//   <x, y> ~= <x0, y0> + <x0, y1> + <x1, y0> + <x1, y1> + <x0, y2> + <x2, y0>
// (Ootomo and Yokota 2022 with bf16 parts; what is left out is below 2^-25).
// Two fp16 planes with a scale per row take half the MMAs, but keep those bits
// only down to 2^-17 of a row's largest entry: entries of M = R^-1/2 that are
// small beside the diagonal (columns of R that differ by e^4: half of them) lost
// every digit.
//
// Bound: the tensor pipe.  CTA pairs take 256 x 256 output tiles (M = 256 rows
// of y over the pair, N = 256 rows of x, K = 16 per MMA): a 64-column stage is
// 96 KB per CTA for 24 MMAs of 128 cycles, 32 bytes of L2 reads per SM and cycle.
// A Newton-Schulz update (three products and their passes) at K = 256 / 1024 /
// 3072: 34 / 66 / 653 us; 35 / 52 / 408 with two fp16 planes.
//
// The tensor cores' fp32 accumulation rounds toward zero, so an accumulation
// chain is one stage or half of one, its smallest terms first: four MMAs (two)
// round a sum of full size.  The epilogue adds the chains in registers with IEEE
// adds, in order, while the next chain runs in the other half of TMEM.  No
// partial sums go to memory.

#include <algorithm>

#include "internal.h"
#include "ptx.cuh"

namespace bergson {

namespace {

constexpr int kSqM = 256;                 // rows of y per tile (128 per CTA)
constexpr int kSqK = 64;                  // bf16 columns per stage: one 128-byte row
constexpr int kPlanes = SplitOperand::kPlanes;
// Columns up to which a stage is two accumulation chains of 32 columns: there a
// chain is a larger part of the sum.  M = R^-1/2 of K columns of unequal scale
// (e^1), error against fp64 as a multiple of that with tf32 parts and chains of 32
// columns or more, one chain / two: K = 128 1.28 / 0.79, 384 1.64 / 0.91, 512 0.89 /
// 0.53, 1024 0.2.  Two cost 42 -> 48 us an update at K = 512, 66 -> 78 at K = 1024.
constexpr int kShortChainK = 512;
constexpr int kSqThreads = 64 + 256;      // producer, MMA, 8 epilogue warps
constexpr int kSqBarBytes = 256;
constexpr int kSqSmemBudget = 232448;
constexpr int kOutTile = 32 * 33;         // floats of an epilogue warp's output tile
constexpr int kOutBytes = 8 * kOutTile * 4;
constexpr uint64_t kSqDrainTimeoutNs = 2000000000ull;

template <int TN_>
struct SqCfg {
  static constexpr int TN = TN_;                           // rows of x per tile
  static constexpr int kABytes = kPlanes * 128 * 128;      // y: 128 rows of each plane
  static constexpr int kBBytes = kPlanes * (TN / 2) * 128; // x: this CTA's half of the N side
  static constexpr int kStageBytes = kABytes + kBBytes;
  static constexpr int kStages = (kSqSmemBudget - 1024 - kSqBarBytes - kOutBytes) / kStageBytes;
  static constexpr int kSmemBytes = 1024 + kStages * kStageBytes + kSqBarBytes + kOutBytes;
  static constexpr int kTmemCols = 2 * TN;                 // two accumulators
  static constexpr int kCols = TN / 2;                     // accumulator columns per epilogue warp
};

struct SqParams {
  float* c[2];               // [N, ldc] of each product; nullptr: the splits below instead
  int n_prob;                // products of the launch (one, or two of the same shape)
  int chains;                // accumulation chains per stage, 1 or 2
  int M, N, K;               // rows of y (q), rows of x (b), columns
  int n_mt, n_nt;            // tiles
  int n_tiles;               // of one product
  int symmetric;             // x == y: tiles with some b <= q, mirrored into C[q, b]
  int accumulate;            // the product is added to C
  float alpha;
  const float* alpha_s;      // or nullptr
  float gamma;               // added on the diagonal
  int64_t ldc;
  SplitOperand row, col;     // splits of C's rows and columns (c == nullptr)
  const int* stop;           // nonzero: nothing is computed or written (nullptr: never)
  float* part;               // [n_tiles, 16] sums of (C - I)^2 per tile and epilogue warp, or nullptr
  int* status;
  uint64_t timeout_ns;
};

// Tile i of the launch.  Symmetric products enumerate the tiles with some b <=
// q row by row (row mt has TN == 256 ? mt + 1 : 2 mt + 2 of them, the last row
// maybe one fewer); others go in groups of kGroup tile rows, so that the tiles
// in flight form a near-square block and share operand panels in L2.
constexpr int kGroup = 8;
template <int TN>
__device__ __forceinline__ void tile_of(const SqParams& p, int i, int* mt, int* nt) {
  if (p.symmetric) {
    constexpr int w = kSqM / TN;                     // row mt starts at w mt (mt + 1) / 2
    int m = static_cast<int>((sqrtf(8.0f * static_cast<float>(i / w) + 1.0f) - 1.0f) * 0.5f);
    while (w * (m + 1) * (m + 2) / 2 <= i) ++m;
    while (w * m * (m + 1) / 2 > i) --m;
    *mt = m;
    *nt = i - w * m * (m + 1) / 2;
    return;
  }
  const int per = kGroup * p.n_nt;
  const int g = i / per, r = i % per;
  const int m0 = g * kGroup;
  const int gm = min(kGroup, p.n_mt - m0);
  *mt = m0 + r % gm;
  *nt = r / gm;
}

// TMA load of a {64 columns, rows, planes} box for a CTA pair's barrier.
__device__ __forceinline__ void tma_load_3d_pair(uint32_t dst, const void* tmap, uint32_t bar,
                                                 int c0, int c1, uint64_t policy) {
  asm volatile(
      "cp.async.bulk.tensor.3d.cta_group::2.shared::cluster.global.mbarrier::complete_tx::bytes"
      ".L2::cache_hint [%0], [%1, {%3, %4, %5}], [%2], %6;" ::"r"(dst),
      "l"(tmap), "r"(bar), "r"(c0), "r"(c1), "r"(0), "l"(policy)
      : "memory");
}

// The planes of two values.
__device__ __forceinline__ void split_bf16x2(float a, float b, __nv_bfloat162* out) {
#pragma unroll
  for (int i = 0; i < kPlanes; ++i) {
    out[i] = __floats2bfloat162_rn(a, b);
    const float2 h = __bfloat1622float2(out[i]);
    a -= h.x;
    b -= h.y;
  }
}

// The split of v at columns col.. of a row (4 | col: 8-byte aligned).
__device__ __forceinline__ void put_four(const SplitOperand& o, int row, int col, float4 v) {
  __nv_bfloat162 lo[kPlanes], hi[kPlanes];
  split_bf16x2(v.x, v.y, lo);
  split_bf16x2(v.z, v.w, hi);
  __nv_bfloat16* d = o.planes + static_cast<int64_t>(row) * o.ld + col;
#pragma unroll
  for (int i = 0; i < kPlanes; ++i, d += static_cast<int64_t>(o.rows) * o.ld) {
    uint2 w;
    w.x = *reinterpret_cast<const uint32_t*>(&lo[i]);
    w.y = *reinterpret_cast<const uint32_t*>(&hi[i]);
    *reinterpret_cast<uint2*>(d) = w;
  }
}

// Writes a warp's 32 x 32 output tile (tile[j * 33 + i] = C[bc + j, q0 + i]) to
// the splits of C's rows and columns, four entries per lane and 64 bytes per
// row and plane (sizes are multiples of 4; lanes 8 r + l read banks r + 4 l).
__device__ __forceinline__ void put_splits(const SqParams& p, const float* tile, int lane, int bc,
                                           int nb, int q0) {
  const int l4 = 4 * (lane & 7);
  const int nq = min(32, p.M - q0);
#pragma unroll 2
  for (int j = lane >> 3; j < 32; j += 4) {
    if (j < nb && l4 < nq) {                       // row bc + j of C, columns q0 + l4, ..
      const float* v = tile + j * 33 + l4;
      put_four(p.row, bc + j, q0 + l4, make_float4(v[0], v[1], v[2], v[3]));
    }
    if (p.col.planes != nullptr && j < nq && l4 < nb) {   // column q0 + j of C, rows bc + l4, ..
      const float* v = tile + l4 * 33 + j;
      put_four(p.col, q0 + j, bc + l4, make_float4(v[0], v[33], v[66], v[99]));
    }
  }
}

__device__ __forceinline__ bool sq_warp_wait(uint32_t bar, uint32_t parity, uint64_t tmo,
                                             const volatile int* abort_flag) {
  bool ok = true;
  if ((threadIdx.x & 31) == 0) ok = mbar_wait_inline(bar, parity, tmo, abort_flag);
  return __shfl_sync(0xffffffffu, ok ? 1 : 0, 0) != 0;
}

// The MMAs of one chain of 16 kMmas columns, the terms y_i x_j smallest first
// (descriptors hold addresses in 16 bytes: 16 bf16 = 2).  Unrolled: in a loop an
// MMA of N = 128 is issued later than the pipe could take it (K = 1024: 64 -> 80 us
// an update).
template <int TN, int kMmas>
__device__ __forceinline__ void issue_chain(uint32_t d, uint64_t y, uint64_t x, uint32_t idesc) {
  using C = SqCfg<TN>;
  constexpr int kTerms = 6;
  constexpr uint8_t kI[kTerms] = {2, 0, 1, 1, 0, 0}, kJ[kTerms] = {0, 2, 1, 0, 1, 0};
#pragma unroll
  for (int t = 0; t < kTerms; ++t) {
    const uint64_t yi = y + kI[t] * (C::kABytes / kPlanes / 16);
    const uint64_t xj = x + kJ[t] * (C::kBBytes / kPlanes / 16);
#pragma unroll
    for (int kk = 0; kk < kMmas; ++kk)
      umma_f16_pair(d, yi + 2 * kk, xj + 2 * kk, idesc, t != 0 || kk != 0);
  }
}

// C[b, q] = alpha' <x_b, y_q> + gamma [b == q] over persistent CTA pairs.
// Synchronisation as in the pair scorer: the odd CTA's loads complete on the
// even CTA's `full`, the even CTA's MMA thread frees a stage in both CTAs and
// hands accumulators to both epilogues by multicast commits, and every
// epilogue warp of both CTAs releases an accumulator on the even CTA's
// `tempty`.  Every wait is bounded.
template <int TN>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kSqThreads, 1)
    square_kernel(const __grid_constant__ CUtensorMap tm_y0,
                  const __grid_constant__ CUtensorMap tm_x0,
                  const __grid_constant__ CUtensorMap tm_y1,
                  const __grid_constant__ CUtensorMap tm_x1, const __grid_constant__ SqParams p) {
  using C = SqCfg<TN>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = reinterpret_cast<uint8_t*>((reinterpret_cast<uintptr_t>(smem_raw) + 1023) &
                                             ~static_cast<uintptr_t>(1023));
  const uint32_t sbase = smem_u32(smem);
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + C::kStages * C::kStageBytes);
  uint64_t* empty = full + C::kStages;
  uint64_t* tfull = empty + C::kStages;
  uint64_t* tempty = tfull + 2;
  uint64_t* drain = tempty + 2;
  uint32_t* s_tmem = reinterpret_cast<uint32_t*>(drain + 1);
  volatile int* s_abort = reinterpret_cast<volatile int*>(s_tmem + 1);

  const uint32_t rank = cluster_ctarank();
  const int cid = blockIdx.x >> 1;
  const int n_cl = gridDim.x >> 1;
  const int warp = threadIdx.x >> 5;
  const int lane = threadIdx.x & 31;
  const int nK = (p.K + kSqK - 1) / kSqK;
  griddep_launch_dependents();   // the next grid sets itself up and waits for this one to end
  if (threadIdx.x == 0) {
    for (int s = 0; s < C::kStages; ++s) {
      mbar_init(smem_u32(&full[s]), 1);
      mbar_init(smem_u32(&empty[s]), 1);
    }
    for (int i = 0; i < 2; ++i) {
      mbar_init(smem_u32(&tfull[i]), 1);
      mbar_init(smem_u32(&tempty[i]), 16);           // 8 epilogue warps of each CTA
    }
    mbar_init(smem_u32(drain), 1);
    *s_abort = 0;
    fence_barrier_init();
  }
  if (warp == 1) {
    tmem_alloc_pair(smem_u32(s_tmem), C::kTmemCols);
    tmem_relinquish_pair();
  }
  griddep_wait();                // the operands come from earlier grids
  tc_fence_before();
  cluster_sync();
  tc_fence_after();
  const uint32_t tmem = *s_tmem;
  const uint64_t tmo = p.timeout_ns;
  const int n_all = p.stop != nullptr && *p.stop != 0 ? 0 : p.n_prob * p.n_tiles;

  if (warp == 0) {
    // ------------------------------------------------------------ producer
    if (lane == 0) {
      prefetch_tmap(&tm_y0);
      prefetch_tmap(&tm_x0);
      const uint64_t pol = policy_evict_normal();
      int stage = 0;
      uint32_t ph = 0;
      uint32_t issued = 0, issued_par = 0;
      bool ok = true;
      for (int t = cid; t < n_all && ok; t += n_cl) {
        const bool second = t >= p.n_tiles;
        const CUtensorMap* tm_y = second ? &tm_y1 : &tm_y0;
        const CUtensorMap* tm_x = second ? &tm_x1 : &tm_x0;
        int mt, nt;
        tile_of<TN>(p, second ? t - p.n_tiles : t, &mt, &nt);
        for (int kc = 0; kc < nK; ++kc) {
          if (!mbar_wait(smem_u32(&empty[stage]), ph ^ 1, tmo, s_abort)) { ok = false; break; }
          const uint32_t fb_local = smem_u32(&full[stage]);
          const uint32_t fb = mapa_shared(fb_local, 0);
          if (rank == 0) mbar_arrive_expect_tx(fb_local, 2 * C::kStageBytes);
          const uint32_t dst = sbase + stage * C::kStageBytes;
          tma_load_3d_pair(dst, tm_y, fb, kc * kSqK, mt * kSqM + static_cast<int>(rank) * 128,
                           pol);
          tma_load_3d_pair(dst + C::kABytes, tm_x, fb, kc * kSqK,
                           nt * TN + static_cast<int>(rank) * (TN / 2), pol);
          issued |= 1u << stage;
          issued_par = (issued_par & ~(1u << stage)) | (ph << stage);
          if (++stage == C::kStages) { stage = 0; ph ^= 1; }
        }
      }
      if (!ok) {
        raise_device_error(p.status, s_abort, kStatusTimeout);
        if (rank == 0) {
          for (int s = 0; s < C::kStages; ++s)
            if (issued >> s & 1)
              mbar_wait(smem_u32(&full[s]), (issued_par >> s) & 1, kSqDrainTimeoutNs, nullptr);
        } else {
          const uint64_t t0 = global_timer_ns();      // its loads complete on the other CTA's barrier
          while (global_timer_ns() - t0 < 1000000ull) {
          }
        }
      }
    }
    __syncwarp();
  } else if (warp == 1) {
    // ------------------------------------------------------------ MMA issuer (even CTA)
    if (rank == 0 && lane == 0) {
      const uint32_t idesc = make_idesc_f16(kSqM, TN, true);
      int stage = 0;
      uint32_t ph = 0;
      int ab = 0;
      uint32_t aph = 0;
      bool ok = true;
      for (int t = cid; t < n_all && ok; t += n_cl) {
        for (int kc = 0; kc < nK; ++kc) {
          if (!mbar_wait(smem_u32(&full[stage]), ph, tmo, s_abort)) { ok = false; break; }
          const uint32_t sa = sbase + stage * C::kStageBytes;
          const uint64_t y = sw128_desc(sa), x = sw128_desc(sa + C::kABytes);
          for (int ch = 0; ch < p.chains && ok; ++ch) {
            if (!mbar_wait(smem_u32(&tempty[ab]), aph ^ 1, tmo, s_abort)) { ok = false; break; }
            tc_fence_after();
            const uint32_t d = tmem + ab * TN;
            if (p.chains == 1) issue_chain<TN, kSqK / 16>(d, y, x, idesc);
            else issue_chain<TN, kSqK / 32>(d, y + kSqK / 16 * ch, x + kSqK / 16 * ch, idesc);
            if (ch == p.chains - 1) umma_commit_pair(smem_u32(&empty[stage]), 0x3);
            umma_commit_pair(smem_u32(&tfull[ab]), 0x3);
            if (++ab == 2) { ab = 0; aph ^= 1; }
          }
          if (++stage == C::kStages) { stage = 0; ph ^= 1; }
        }
      }
      if (!ok) raise_device_error(p.status, s_abort, kStatusTimeout);
      umma_commit_pair(smem_u32(drain), 0x1);
      mbar_wait(smem_u32(drain), 0, kSqDrainTimeoutNs, nullptr);
    }
    __syncwarp();
  } else {
    // ------------------------------------------------------------ epilogue
    // Thread = row q of this CTA's half (TMEM lane) and kCols columns b.
    const int ew = warp - 2;
    const int quarter = warp & 3;
    const int half = ew >> 2;
    float* tile = reinterpret_cast<float*>(smem + C::kStages * C::kStageBytes + kSqBarBytes) +
                  ew * kOutTile;
    const float al = p.alpha_s != nullptr ? p.alpha * *p.alpha_s : p.alpha;
    int ab = 0;
    uint32_t aph = 0;
    bool aborted = false;
    for (int t = cid; t < n_all && !aborted; t += n_cl) {
      float* out = p.c[t >= p.n_tiles ? 1 : 0];
      int mt, nt;
      tile_of<TN>(p, t >= p.n_tiles ? t - p.n_tiles : t, &mt, &nt);
      float acc[C::kCols];               // 0 + v = v: the first chain lands unchanged
#pragma unroll
      for (int j = 0; j < C::kCols; ++j) acc[j] = 0.0f;
      for (int ch = 0; ch < p.chains * nK; ++ch) {
        if (!sq_warp_wait(smem_u32(&tfull[ab]), aph, tmo, s_abort)) {
          raise_device_error(p.status, s_abort, kStatusTimeout);
          aborted = true;
          break;
        }
        tc_fence_after();
        const uint32_t tb = tmem + (static_cast<uint32_t>(32 * quarter) << 16) + ab * TN +
                            half * C::kCols;
#pragma unroll
        for (int c = 0; c < C::kCols; c += 16) {
          float v[16];
          tmem_ld16(tb + c, v);
#pragma unroll
          for (int j = 0; j < 16; ++j) acc[c + j] += v[j];
        }
        tc_fence_before();
        __syncwarp();
        if (lane == 0) mbar_arrive_remote(mapa_shared(smem_u32(&tempty[ab]), 0));
        if (++ab == 2) { ab = 0; aph ^= 1; }
      }
      if (aborted) break;
      // Out through a 32 x 32 tile of shared memory per warp, in rolled loops
      // (unrolled over the registers, the same code is 80 KB of instructions
      // fetched once per tile: 15 us of a 23 us launch at K = 256).
      const int q0 = mt * kSqM + static_cast<int>(rank) * 128 + 32 * quarter;
      const int q = q0 + lane;
      const bool qin = q < p.M;
      const int b0 = nt * TN + half * C::kCols;
      float ssq = 0.0f, comp = 0.0f;
#pragma unroll
      for (int c = 0; c < C::kCols; c += 32) {
        const int bc = b0 + c;
        const int nb = min(32, p.N - bc);
        __syncwarp();
#pragma unroll
        for (int j = 0; j < 32; ++j) tile[j * 33 + lane] = acc[c + j];
        __syncwarp();
        float* dst = out + static_cast<int64_t>(bc) * p.ldc + q;
#pragma unroll 4
        for (int j = 0; j < 32; ++j, dst += p.ldc) {
          const int b = bc + j;
          float v = al * tile[j * 33 + lane];
          if (b == q) v += p.gamma;
          const bool in = qin && j < nb;
          if (p.accumulate && in && (!p.symmetric || b <= q)) v += *dst;
          if (in && out != nullptr && (!p.symmetric || b <= q)) *dst = v;
          tile[j * 33 + lane] = in ? v : 0.0f;
          const float r = in ? v - (b == q ? 1.0f : 0.0f) : 0.0f;
          const float y = r * r - comp;
          const float u = ssq + y;
          comp = (u - ssq) - y;
          ssq = u;
        }
        __syncwarp();
        if (out == nullptr) put_splits(p, tile, lane, bc, nb, q0);
        if (p.symmetric && lane < nb) {                 // the mirror image C[q, b], b < q
          float* mir = out + static_cast<int64_t>(q0) * p.ldc + bc + lane;
          const int nq = min(32, p.M - q0);
#pragma unroll 4
          for (int i = 0; i < nq; ++i, mir += p.ldc)
            if (bc + lane < q0 + i) *mir = tile[lane * 33 + i];
        }
      }
      if (p.part != nullptr) {
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) ssq += __shfl_xor_sync(0xffffffffu, ssq, o);
        if (lane == 0) p.part[static_cast<int64_t>(t) * 16 + rank * 8 + ew] = ssq;
      }
    }
  }

  tc_fence_before();
  cluster_sync();              // no MMA, commit or remote arrival is still in flight
  if (warp == 1) {
    tc_fence_after();
    tmem_dealloc_pair(tmem, C::kTmemCols);
  }
}

// ------------------------------------------------------------ operand passes

constexpr int kPassTile = 64;

// Writes 64 values of one row of a split operand, two per lane.
__device__ __forceinline__ void put_row(const SplitOperand& o, int row, int col0, int lane, float a,
                                        float b) {
  const int c = col0 + 2 * lane;
  if (row >= o.rows || c >= o.K) return;
  __nv_bfloat162 v[kPlanes];
  split_bf16x2(a, b, v);
  __nv_bfloat16* d = o.planes + static_cast<int64_t>(row) * o.ld + c;
#pragma unroll
  for (int i = 0; i < kPlanes; ++i, d += static_cast<int64_t>(o.rows) * o.ld) {
    if (c + 1 < o.K) *reinterpret_cast<__nv_bfloat162*>(d) = v[i];
    else *d = v[i].x;
  }
}

// One pass over a K x K matrix c, or two of them (grid.y), that writes the split
// of its rows (o.row) and / or of the rows of its symmetric part (c + c^T) / 2
// (o.sym).  Memory bound: 4 bytes read and 6 written per entry and operand.  One
// CTA per pair of 64 x 64 tiles (ti <= tj); a thread takes a 4 x 4 block of the
// upper tile and the mirrored block of the lower one as eight 16-byte loads,
// adds them across the diagonal in registers and writes both 8 bytes a row and
// plane.  A warp's blocks are 4 x 8, so every access covers whole 32-byte
// sectors.
struct SquarePass {
  const float* c;
  int64_t ldc;
  int K;
  SplitOperand row, sym;         // planes == nullptr: not written
};

struct SquarePasses {
  SquarePass p[2];
  const int* stop;               // nonzero: nothing is written (nullptr: never)
};

__global__ void __launch_bounds__(256)
    square_pass_kernel(const __grid_constant__ SquarePasses pp) {
  const SquarePass& p = pp.p[blockIdx.y];
  const int pair = blockIdx.x;                 // tj (tj + 1) / 2 + ti
  int tj = static_cast<int>((sqrtf(8.0f * static_cast<float>(pair) + 1.0f) - 1.0f) * 0.5f);
  while ((tj + 1) * (tj + 2) / 2 <= pair) ++tj;
  while (tj * (tj + 1) / 2 > pair) --tj;
  const int ti = pair - tj * (tj + 1) / 2;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  const int i = ti * kPassTile + 16 * (w >> 1) + 4 * (lane >> 3);      // rows of the upper block
  const int j = tj * kPassTile + 32 * (w & 1) + 4 * (lane & 7);        // and its columns
  griddep_launch_dependents();
  griddep_wait();
  if (pp.stop != nullptr && *pp.stop != 0) return;
  if (i >= p.K || j >= p.K) return;            // 4 | K: a block lies inside or outside
  float4 a[4], b[4];
#pragma unroll
  for (int u = 0; u < 4; ++u)
    a[u] = *reinterpret_cast<const float4*>(p.c + static_cast<int64_t>(i + u) * p.ldc + j);
#pragma unroll
  for (int u = 0; u < 4; ++u)
    b[u] = *reinterpret_cast<const float4*>(p.c + static_cast<int64_t>(j + u) * p.ldc + i);
  const bool lower = ti != tj;                 // on the diagonal another thread holds the mirror
  if (p.row.planes != nullptr) {
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      put_four(p.row, i + u, j, a[u]);
      if (lower) put_four(p.row, j + u, i, b[u]);
    }
  }
  if (p.sym.planes != nullptr) {
    float s[4][4];                             // s[u][v]: entry (i + u, j + v), and (j + v, i + u)
    const float au[4][4] = {{a[0].x, a[0].y, a[0].z, a[0].w}, {a[1].x, a[1].y, a[1].z, a[1].w},
                            {a[2].x, a[2].y, a[2].z, a[2].w}, {a[3].x, a[3].y, a[3].z, a[3].w}};
    const float bu[4][4] = {{b[0].x, b[0].y, b[0].z, b[0].w}, {b[1].x, b[1].y, b[1].z, b[1].w},
                            {b[2].x, b[2].y, b[2].z, b[2].w}, {b[3].x, b[3].y, b[3].z, b[3].w}};
#pragma unroll
    for (int u = 0; u < 4; ++u)
#pragma unroll
      for (int v = 0; v < 4; ++v) s[u][v] = 0.5f * (au[u][v] + bu[v][u]);
#pragma unroll
    for (int u = 0; u < 4; ++u) {
      put_four(p.sym, i + u, j, make_float4(s[u][0], s[u][1], s[u][2], s[u][3]));
      if (lower) put_four(p.sym, j + u, i, make_float4(s[0][u], s[1][u], s[2][u], s[3][u]));
    }
  }
}

// to = the split of from's columns: its planes transposed (both K x K).  64 x 64
// tiles through shared memory, 16 bytes an access; columns past K lie within ld.
__global__ void __launch_bounds__(256) split_transpose_kernel(const SplitOperand from,
                                                              const SplitOperand to,
                                                              const int* stop) {
  __shared__ __align__(16) __nv_bfloat16 tile[kPassTile][kPassTile + 8];
  griddep_launch_dependents();
  griddep_wait();
  if (stop != nullptr && *stop != 0) return;
  const int64_t plane = static_cast<int64_t>(blockIdx.z) * from.rows * from.ld;
  const int i0 = blockIdx.y * kPassTile, j0 = blockIdx.x * kPassTile;
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int r = (threadIdx.x >> 3) + 32 * u, c = 8 * (threadIdx.x & 7);
    if (i0 + r < from.rows && j0 + c < from.K)
      *reinterpret_cast<uint4*>(&tile[r][c]) = *reinterpret_cast<const uint4*>(
          from.planes + plane + static_cast<int64_t>(i0 + r) * from.ld + j0 + c);
  }
  __syncthreads();
#pragma unroll
  for (int u = 0; u < 2; ++u) {
    const int r = (threadIdx.x >> 3) + 32 * u, c = 8 * (threadIdx.x & 7);
    if (j0 + r >= to.rows || i0 + c >= to.K) continue;
    __align__(16) __nv_bfloat16 v[8];
#pragma unroll
    for (int x = 0; x < 8; ++x) v[x] = tile[c + x][r];
    *reinterpret_cast<uint4*>(to.planes + plane + static_cast<int64_t>(j0 + r) * to.ld + i0 + c) =
        *reinterpret_cast<const uint4*>(v);
  }
}

// m = (c + c^T) / 2 * (*scale)
__global__ void __launch_bounds__(256) symmetric_scale_kernel(const float* c, int K, int64_t ldc,
                                                              const float* scale, float* m,
                                                              int64_t ldm) {
  __shared__ float sa[32][33], sb[32][33];
  const int ti = blockIdx.y, tj = blockIdx.x;
  if (ti > tj) return;
  griddep_wait();
  const int i0 = ti * 32, j0 = tj * 32, x = threadIdx.x;
  for (int r = threadIdx.y; r < 32; r += 8) {
    sa[r][x] = (i0 + r < K && j0 + x < K) ? c[static_cast<int64_t>(i0 + r) * ldc + j0 + x] : 0.0f;
    sb[r][x] = (j0 + r < K && i0 + x < K) ? c[static_cast<int64_t>(j0 + r) * ldc + i0 + x] : 0.0f;
  }
  __syncthreads();
  const float s = *scale;
  for (int r = threadIdx.y; r < 32; r += 8) {
    if (i0 + r < K && j0 + x < K)
      m[static_cast<int64_t>(i0 + r) * ldm + j0 + x] = 0.5f * (sa[r][x] + sb[x][r]) * s;
    if (ti != tj && j0 + r < K && i0 + x < K)
      m[static_cast<int64_t>(j0 + r) * ldm + i0 + x] = 0.5f * (sb[r][x] + sa[x][r]) * s;
  }
}

// The split of x^T (K rows of n entries) from x [n, ldx].
__global__ void __launch_bounds__(256) transpose_split_kernel(const float* __restrict__ x, int n,
                                                              int K, int64_t ldx,
                                                              const SplitOperand o) {
  __shared__ float s[kPassTile][kPassTile + 1];
  griddep_launch_dependents();
  const int i0 = blockIdx.x * kPassTile, k0 = blockIdx.y * kPassTile;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float v[16];
#pragma unroll
  for (int u = 0; u < 16; ++u) {
    const int r = w + 8 * (u >> 1), cc = lane + 32 * (u & 1);
    v[u] = (i0 + r < n && k0 + cc < K) ? x[static_cast<int64_t>(i0 + r) * ldx + k0 + cc] : 0.0f;
  }
#pragma unroll
  for (int u = 0; u < 16; ++u) s[w + 8 * (u >> 1)][lane + 32 * (u & 1)] = v[u];
  __syncthreads();
#pragma unroll 4
  for (int r = w; r < kPassTile; r += 8)
    put_row(o, k0 + r, i0, lane, s[2 * lane][r], s[2 * lane + 1][r]);
}

int64_t square_tiles(int M, int N, int tn, bool symmetric) {
  const int64_t mt = (M + kSqM - 1) / kSqM, nt = (N + tn - 1) / tn;
  // symmetric: rows of (mt + 1) 256 / tn tiles, the last clipped to nt
  return symmetric ? (kSqM / tn) * mt * (mt - 1) / 2 + nt : mt * nt;
}

// Tile width: the one whose rounds over the clusters cost least.  A 128-wide
// tile is half the products of a 256-wide one but reads more of shared memory
// per product and pays the same fill and epilogue, so it counts 0.7 (an update at
// K = 2052, three rounds of 128 / two of 256: 449 / 442 us, at K = 2560 520 / 507).
int square_tile_width(int M, int N, int n, int clusters, bool symmetric) {
  const int64_t r256 = (n * square_tiles(M, N, 256, symmetric) + clusters - 1) / clusters;
  const int64_t r128 = (n * square_tiles(M, N, 128, symmetric) + clusters - 1) / clusters;
  return static_cast<double>(r128) * 0.7 < static_cast<double>(r256) ? 128 : 256;
}

template <int TN>
cudaError_t launch_square_t(const SquareArgs* a, int n, SqParams p, int clusters, cudaStream_t s) {
  using C = SqCfg<TN>;
  CUtensorMap tm_y[2], tm_x[2];
  for (int i = 0; i < 2; ++i) {
    const SquareArgs& g = a[i < n ? i : 0];
    if (encode_tmap_planes(&tm_y[i], g.y.planes, g.y.K, g.y.rows, g.y.ld, kSqK, 128) !=
            CUDA_SUCCESS ||
        encode_tmap_planes(&tm_x[i], g.x.planes, g.x.K, g.x.rows, g.x.ld, kSqK, TN / 2) !=
            CUDA_SUCCESS)
      return cudaErrorInvalidValue;
  }
  static PerDeviceOnce attr;
  const cudaError_t e = smem_attr_once(attr, square_kernel<TN>, C::kSmemBytes);
  if (e != cudaSuccess) return e;
  p.n_mt = (p.M + kSqM - 1) / kSqM;
  p.n_nt = (p.N + TN - 1) / TN;
  p.n_tiles = static_cast<int>(square_tiles(p.M, p.N, TN, p.symmetric != 0));
  const int grid = 2 * std::max(1, std::min(clusters, n * p.n_tiles));
  return launch_dependent(square_kernel<TN>, dim3(grid), dim3(kSqThreads), C::kSmemBytes, s,
                          tm_y[0], tm_x[0], tm_y[1], tm_x[1], p);
}

}  // namespace

// Most sums a product writes to `part`, and how many it does.
int64_t square_part_floats(int M, int N) {
  return 16 * static_cast<int64_t>((M + kSqM - 1) / kSqM) * ((N + 127) / 128);
}

int square_part_count(int M, int N, int sms) {
  const int clusters = std::max(1, sms / 2);
  return static_cast<int>(
      16 * square_tiles(M, N, square_tile_width(M, N, 1, clusters, false), false));
}

cudaError_t launch_square(const SquareArgs* a, int n, int sms, cudaStream_t s) {
  SqParams p = {};
  p.n_prob = n;
  p.M = a->y.rows;
  p.N = a->x.rows;
  p.K = a->y.K;
  p.chains = p.K <= kShortChainK ? 2 : 1;
  p.symmetric = a->symmetric ? 1 : 0;
  p.accumulate = a->accumulate ? 1 : 0;
  for (int i = 0; i < n; ++i) p.c[i] = a[i].c;
  p.alpha = a->alpha;
  p.alpha_s = a->alpha_s;
  p.gamma = a->gamma;
  p.ldc = a->ldc;
  p.row = a->row_out;
  p.col = a->col_out;
  p.stop = a->stop;
  p.part = a->part;
  p.status = a->status;
  p.timeout_ns = kWaitTimeoutNs;
  const int clusters = std::max(1, sms / 2);
  return square_tile_width(p.M, p.N, n, clusters, a->symmetric) == 256
             ? launch_square_t<256>(a, n, p, clusters, s)
             : launch_square_t<128>(a, n, p, clusters, s);
}

cudaError_t launch_square_pass(const SquarePassArgs* a, int n, int K, const int* stop,
                               cudaStream_t s) {
  SquarePasses pp = {};
  pp.stop = stop;
  for (int i = 0; i < n; ++i) {
    pp.p[i].c = a[i].c;
    pp.p[i].ldc = K;
    pp.p[i].K = K;
    pp.p[i].row = a[i].row;
    pp.p[i].sym = a[i].sym;
  }
  const int t = (K + kPassTile - 1) / kPassTile;
  return launch_dependent(square_pass_kernel, dim3(t * (t + 1) / 2, n), dim3(256), 0, s, pp);
}

cudaError_t launch_split_transpose(const SplitOperand& from, const SplitOperand& to,
                                   const int* stop, cudaStream_t s) {
  const int t = (from.K + kPassTile - 1) / kPassTile;
  return launch_dependent(split_transpose_kernel, dim3(t, t, kPlanes), dim3(256), 0, s, from, to,
                          stop);
}

cudaError_t launch_symmetric_scale(const float* c, int K, int64_t ldc, const float* scale, float* m,
                                   int64_t ldm, cudaStream_t s) {
  const int t = (K + 31) / 32;
  return launch_dependent(symmetric_scale_kernel, dim3(t, t), dim3(32, 8), 0, s, c, K, ldc, scale,
                          m, ldm);
}

cudaError_t launch_transpose_split(const float* x, int n, int K, int64_t ldx,
                                   const SplitOperand& o, cudaStream_t s) {
  const dim3 grid((n + kPassTile - 1) / kPassTile, (K + kPassTile - 1) / kPassTile);
  transpose_split_kernel<<<grid, 256, 0, s>>>(x, n, K, ldx, o);
  return cudaGetLastError();
}

}  // namespace bergson
