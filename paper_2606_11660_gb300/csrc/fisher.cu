// TrackStar's empirical-Fisher preconditioner (Bergson Sec. 3.1: the empirical
// Fisher used by TrackStar, stacked with optimizer normalisation and
// down-projection; Fig. 2: Fisher fitting and mixing before index building).
//
//   fit:    R = (1/n) X^T X over n projected gradient rows (K x K)
//   mix:    R = lam R1 + (1 - lam) R2 + damping * (tr(R)/K) * I
//   power:  M = R^-1/2 (or R^-1) by the coupled Newton-Schulz iteration
//           Y0 = R/c, Z0 = I, T = (3I - Z Y)/2, Y <- Y T, Z <- T Z, which
//           drives Y -> (R/c)^1/2 and Z -> (R/c)^-1/2 using only matrix
//           products (c = ||R||_F puts every eigenvalue of R/c in (0, 1]).
//   apply:  x' = M x for each row (bergson_precondition_rows, same GEMM as
//           the on-the-fly scores).
//
// All products are "NT" (C = A B^T, the reduction index contiguous in both
// operands) on the pair kernel of square.cu, whose operands are three bf16
// planes: every matrix of the iteration is split once, by the pass that also
// symmetrises it, or by the product itself (T).  Products of the iteration are
// symmetric in exact arithmetic; each update is re-symmetrised so that rounding
// cannot build up an antisymmetric part.
//
// Measured (one GB300, n = 1024, 12 updates at K = 3072): 17.4 ms per fit and
// power with tf32 parts on single CTAs, K slices through partial sums in
// memory and separate transpose / symmetrise / norm passes; 8.7 ms as here.
// Per update: 63 / 116 / 1220 us at K = 256 / 1024 / 3072 before, 34 / 66 / 653
// here.

#include <algorithm>

#include "internal.h"
#include "ptx.cuh"

namespace bergson {

namespace {

// scal[0] = sum_i (lam * R1[i,i] + (1 - lam) * R2[i,i])  (single CTA)
__global__ void mixed_trace_kernel(const float* __restrict__ r1, const float* __restrict__ r2,
                                   int64_t ld, int K, float lam, float* __restrict__ scal) {
  __shared__ float red[32];
  float s = 0.0f;
  for (int i = threadIdx.x; i < K; i += blockDim.x) {
    const float a = r1[i * ld + i];
    s += r2 != nullptr ? lam * a + (1.0f - lam) * r2[i * ld + i] : a;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float t = 0.0f;
    for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) t += red[w];
    scal[0] = t;
  }
}

// Row i of out = lam R1 + (1 - lam) R2 + damping * trace / K * I (R2 may be
// null: R1 + ...) and its compensated sum of squares.  One CTA per row (grid
// stride).
__global__ void __launch_bounds__(256) mix_kernel(const float* __restrict__ r1,
                                                  const float* __restrict__ r2, int64_t ld, int K,
                                                  float lam, float damping,
                                                  const float* __restrict__ scal,
                                                  float* __restrict__ out,
                                                  float* __restrict__ part) {
  __shared__ float red[8];
  const float d = damping * scal[0] / static_cast<float>(K);
  for (int i = blockIdx.x; i < K; i += gridDim.x) {
    const float4* a = reinterpret_cast<const float4*>(r1 + static_cast<int64_t>(i) * ld);
    const float4* b =
        r2 != nullptr ? reinterpret_cast<const float4*>(r2 + static_cast<int64_t>(i) * ld) : nullptr;
    float4* o = reinterpret_cast<float4*>(out + static_cast<int64_t>(i) * K);
    float s = 0.0f, comp = 0.0f;
    for (int j = threadIdx.x; j < K / 4; j += 256) {
      float4 v = a[j];
      if (b != nullptr) {
        const float4 w = b[j];
        v.x = lam * v.x + (1.0f - lam) * w.x;
        v.y = lam * v.y + (1.0f - lam) * w.y;
        v.z = lam * v.z + (1.0f - lam) * w.z;
        v.w = lam * v.w + (1.0f - lam) * w.w;
      }
      if (j == i / 4) {
        if ((i & 3) == 0) v.x += d;
        if ((i & 3) == 1) v.y += d;
        if ((i & 3) == 2) v.z += d;
        if ((i & 3) == 3) v.w += d;
      }
      o[j] = v;
      const float y = v.x * v.x + v.y * v.y + v.z * v.z + v.w * v.w - comp;
      const float t = s + y;
      comp = (t - s) - y;
      s = t;
    }
#pragma unroll
    for (int k = 16; k > 0; k >>= 1) s += __shfl_xor_sync(0xffffffffu, s, k);
    __syncthreads();
    if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = s;
    __syncthreads();
    if (threadIdx.x == 0) {
      float t = 0.0f;
      for (int w = 0; w < 8; ++w) t += red[w];
      part[i] = t;
    }
  }
}

// Fixed-order sum of part[0, n): compensated per thread, then a tree over the
// threads of the single CTA.  Returned to thread 0.
__device__ __forceinline__ float ordered_sum(const float* part, int n) {
  __shared__ float red[32];
  float t = 0.0f, comp = 0.0f;
  for (int i = threadIdx.x; i < n; i += blockDim.x) {
    const float y = part[i] - comp;
    const float u = t + y;
    comp = (u - t) - y;
    t = u;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) t += __shfl_xor_sync(0xffffffffu, t, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = t;
  __syncthreads();
  float s = 0.0f;
  if (threadIdx.x == 0)
    for (int w = 0; w < static_cast<int>(blockDim.x >> 5); ++w) s += red[w];
  return s;
}

// scal[1] = ||R||_F = c, scal[2] = 1/c, scal[3] = 1/sqrt(c), scal[4] = 1/c
__global__ void __launch_bounds__(1024) frob_final_kernel(const float* __restrict__ part,
                                                          int n_part, float* __restrict__ scal,
                                                          int* stop) {
  const float t = ordered_sum(part, n_part);
  if (threadIdx.x != 0) return;
  *stop = 0;
  // a norm that overflows leaves NaN: 1 / c = 0 would make M = 0 of it
  const float c = isfinite(t) ? sqrtf(t) : __int_as_float(0x7fffffff);
  scal[1] = c;
  scal[2] = 1.0f / c;
  scal[3] = 1.0f / sqrtf(c);
  scal[4] = 1.0f / c;
}

// *out = scale * sqrt(sum of part[0, n_part)); *stop is set once that is <= tol.
__global__ void __launch_bounds__(1024) frob_norm_kernel(const float* part, int n_part, float scale,
                                                         float tol, float* out, int* stop) {
  griddep_launch_dependents();
  griddep_wait();
  if (*stop != 0) return;
  const float t = ordered_sum(part, n_part);
  if (threadIdx.x == 0) {
    const float r = scale * sqrtf(t);
    *out = r;
    if (r <= tol) *stop = 1;
  }
}

// The first iterate without products: Y0 = R / c (in place in y), t = T0^T =
// 1.5 I - 0.5 Y0 (Z0 = I) and, per tile, the sum of (T0 - I)^2.  64 x 64 tiles.
__global__ void __launch_bounds__(256) ns_first_kernel(float* __restrict__ y, int K,
                                                       const float* __restrict__ scal,
                                                       float* __restrict__ t,
                                                       float* __restrict__ part) {
  __shared__ float red[8];
  griddep_launch_dependents();
  griddep_wait();
  const float inv_c = scal[2];
  const int i0 = blockIdx.y * 64, j0 = blockIdx.x * 64;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  float s = 0.0f;
  float v[16];
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int i = i0 + w + 8 * (k >> 1), j = j0 + lane + 32 * (k & 1);
    v[k] = (i < K && j < K) ? y[static_cast<int64_t>(i) * K + j] * inv_c : 0.0f;
  }
#pragma unroll
  for (int k = 0; k < 16; ++k) {
    const int i = i0 + w + 8 * (k >> 1), j = j0 + lane + 32 * (k & 1);
    if (i < K && j < K) {
      const int64_t e = static_cast<int64_t>(i) * K + j;
      y[e] = v[k];
      const float u = (i == j ? 1.5f : 0.0f) - 0.5f * v[k];
      t[e] = u;
      const float d = u - (i == j ? 1.0f : 0.0f);
      s += d * d;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(0xffffffffu, s, o);
  if (lane == 0) red[w] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    float a = 0.0f;
    for (int x = 0; x < 8; ++x) a += red[x];
    part[blockIdx.y * gridDim.x + blockIdx.x] = a;
  }
}

// m = *scale * I
__global__ void scaled_identity_kernel(int K, const float* __restrict__ scale,
                                       float* __restrict__ m, int64_t ldm) {
  const float sc = *scale;
  for (int i = blockIdx.x; i < K; i += gridDim.x)
    for (int j = threadIdx.x; j < K; j += blockDim.x)
      m[static_cast<int64_t>(i) * ldm + j] = i == j ? sc : 0.0f;
}

size_t round_up256(size_t x) { return (x + 255) / 256 * 256; }

int64_t split_ld(int64_t K) { return (K + 7) / 8 * 8; }

// Carves a split operand of `rows` rows of K entries out of ws at *off.
size_t split_bytes(int64_t rows, int64_t K) {
  return round_up256(SplitOperand::kPlanes * static_cast<size_t>(rows) * split_ld(K) *
                     sizeof(__nv_bfloat16));
}
SplitOperand take_split(uint8_t* ws, size_t* off, int rows, int K) {
  SplitOperand o;
  o.rows = rows;
  o.K = K;
  o.ld = split_ld(K);
  o.planes = reinterpret_cast<__nv_bfloat16*>(ws + *off);
  *off += split_bytes(rows, K);
  return o;
}

// Above this K the workspace query reports the lean layout (see
// launch_fisher_power).  An update with the full one / the lean one: K = 256 35 / 48
// us, 1024 67 / 96, 2304 389 / 466, 4096 1.50 / 1.62 ms, 8192 11.2 / 11.4, 12,288 38.0 /
// 38.4.
constexpr int kFullK = 12288;

// Iterates enqueued between two read-backs of their residuals.  Everything after
// the first one within the tolerance finds the stop flag set and does nothing,
// so the device need not wait for the host after every residual (25 us a time).
constexpr int kItersPerSync = 4;
constexpr int kMaxIterations = 100;
constexpr int kScalBytes = 512;      // scalars [0, 8), residuals [8, 8 + kMaxIterations]
static_assert((8 + kMaxIterations + 1) * sizeof(float) <= kScalBytes, "residual slots");

size_t part_floats(int64_t K) {
  const int64_t t = (K + 63) / 64;
  return static_cast<size_t>(std::max<int64_t>(
      K, std::max<int64_t>(t * t, square_part_floats(static_cast<int>(K), static_cast<int>(K)))));
}

}  // namespace

size_t fisher_fit_workspace(int64_t n, int64_t K) { return split_bytes(K, n); }

// Two thirds of it (8 rows' planes at least).
size_t fisher_fit_least(int64_t n, int64_t K) {
  return std::max(split_bytes(K, std::min<int64_t>(n, 8)), split_bytes(K, n) * 2 / 3);
}

cudaError_t launch_fisher_fit(const float* x, int n, int K, int64_t ldx, float* r, int64_t ldr,
                              void* ws, size_t ws_bytes, int* status, int sms, cudaStream_t s) {
  // as many rows at a time as the workspace holds: all of them in the queried size
  int part = n;
  if (split_bytes(K, n) > ws_bytes)
    part = static_cast<int>(ws_bytes / split_bytes(K, 8)) * 8;
  for (int i0 = 0; i0 < n; i0 += part) {
    const int rows = std::min(part, n - i0);
    size_t off = 0;
    const SplitOperand xt = take_split(static_cast<uint8_t*>(ws), &off, K, rows);
    cudaError_t e = launch_transpose_split(x + i0 * ldx, rows, K, ldx, xt, s);
    if (e != cudaSuccess) return e;
    SquareArgs a;
    a.x = xt;
    a.y = xt;
    a.symmetric = true;
    a.accumulate = i0 > 0;
    a.alpha = 1.0f / static_cast<float>(n);
    a.c = r;
    a.ldc = ldr;
    a.status = status;
    if ((e = launch_square(&a, 1, sms, s)) != cudaSuccess) return e;
  }
  return cudaSuccess;
}

namespace {

size_t power_bytes(int64_t K, int splits, int matrices) {
  return splits * split_bytes(K, K) +
         matrices * round_up256(static_cast<size_t>(K) * K * sizeof(float)) +
         round_up256(part_floats(K) * sizeof(float)) + kScalBytes;
}
size_t full_bytes(int64_t K) { return power_bytes(K, 4, 2); }

}  // namespace

size_t fisher_power_least(int64_t K) { return power_bytes(K, 3, 1); }

size_t fisher_power_workspace(int64_t K) {
  return K <= kFullK ? full_bytes(K) : fisher_power_least(K);
}

// Full layout (32 K^2 bytes): the splits of Z, Y, T and T^T and the fp32 Z and Y
// products, which go in one launch, as do the passes over them.
// Lean (22 K^2): T^T is transposed from T's split into Z's room once the Z product
// has read that, and the Y product takes T's room.  Same results, a launch and a
// transposition more an update, and two products' last rounds instead of one.
cudaError_t launch_fisher_power(const float* r1, const float* r2, int K, int64_t ldr, float lam,
                                float damping, int inverse, int iterations, float tol,
                                float* residuals, int* iterations_done, float* m, int64_t ldm,
                                void* ws, size_t ws_bytes, int* status, int sms, cudaStream_t s) {
  const bool full = ws_bytes >= full_bytes(K);
  uint8_t* base = static_cast<uint8_t*>(ws);
  const size_t kk = round_up256(static_cast<size_t>(K) * K * sizeof(float));
  size_t off = 0;
  const SplitOperand zs = take_split(base, &off, K, K);
  const SplitOperand ys = take_split(base, &off, K, K);
  const SplitOperand ts = take_split(base, &off, K, K);
  const SplitOperand tts = full ? take_split(base, &off, K, K) : zs;
  float* zf = reinterpret_cast<float*>(base + off);
  off += kk;
  float* yf = reinterpret_cast<float*>(full ? base + off : reinterpret_cast<uint8_t*>(ts.planes));
  if (full) off += kk;
  float* part = reinterpret_cast<float*>(base + off);
  off += round_up256(part_floats(K) * sizeof(float));
  float* scal = reinterpret_cast<float*>(base + off);  // trace, c, 1/c, 1/sqrt(c), 1/c, -, stop
  int* stop = reinterpret_cast<int*>(scal + 6);
  auto product = [&](const SplitOperand& x, const SplitOperand& y, float* c) {
    SquareArgs a;
    a.x = x;
    a.y = y;
    a.c = c;
    a.ldc = K;
    a.stop = stop;
    a.status = status;
    return a;
  };
  auto sym_pass = [&](const float* c, const SplitOperand& o) {
    SquarePassArgs a;
    a.c = c;
    a.sym = o;
    return a;
  };
  const bool track = residuals != nullptr || tol > 0.0f;
  if (iterations_done != nullptr) *iterations_done = 0;
  mixed_trace_kernel<<<1, 1024, 0, s>>>(r1, r2, ldr, K, lam, scal);
  mix_kernel<<<std::min(K, 4096), 256, 0, s>>>(r1, r2, ldr, K, lam, damping, scal, yf, part);
  frob_final_kernel<<<1, 1024, 0, s>>>(part, K, scal, stop);
  const int t64 = (K + 63) / 64;
  ns_first_kernel<<<dim3(t64, t64), 256, 0, s>>>(yf, K, scal, zf, part);
  cudaError_t e = cudaGetLastError();
  if (e != cudaSuccess) return e;
  const int n_part = square_part_count(K, K, sms);
  int updates = 0;               // updates applied (Z is still I at 0)
  int read = 0;                  // residuals read back
  for (int it = 0;; ++it) {
    if (!track && it == iterations) {
      updates = it;
      break;
    }
    // T = 1.5 I - 0.5 Z Y;  Z <- T Z;  Y <- Y T.
    // Z Y is not symmetric in floating point, so T != T^T: the Y update must
    // use T itself.  The products are NT (C = A B^T), so T Z = nt(T, Z) (Z is
    // symmetric) and Y T = nt(Y, T^T): T is split both ways.
    // (Taking Y T^T instead is unstable: to first order, a symmetric
    // perturbation of the iterates along eigenvectors i, j of R grows by
    // (rho - 1) / 2 per step, rho = (s_i / s_j + s_j / s_i) / 2 with s the
    // eigenvalues of R^1/2, so once R's condition number exceeds ~34
    // (s_i / s_j > 3 + sqrt(8)) the converged iterates drift away again.
    // With Y T the same perturbation maps to a fixed point: stable.)
    if (it > 0) {
      SquareArgs t;
      t.x = zs;
      t.y = ys;
      t.alpha = -0.5f;
      t.gamma = 1.5f;
      t.row_out = ts;
      if (full) t.col_out = tts;
      t.part = track ? part : nullptr;
      t.stop = stop;
      t.status = status;
      if ((e = launch_square(&t, 1, sms, s)) != cudaSuccess) return e;
    }
    if (track) {
      // ||I - Z Y||_F / sqrt(K) = 2 ||T - I||_F / sqrt(K): the current iterate's
      // residual (Z Y = Z (R/c) Z = M R M while the iteration keeps Y = (R/c) Z).
      e = launch_dependent(frob_norm_kernel, dim3(1), dim3(1024), 0, s,
                           static_cast<const float*>(part), it == 0 ? t64 * t64 : n_part,
                           2.0f / sqrtf(static_cast<float>(K)), tol, scal + 8 + it, stop);
      if (e != cudaSuccess) return e;
      if (it == iterations || it % kItersPerSync == kItersPerSync - 1) {
        float res[kItersPerSync];
        const int n = it + 1 - read;
        if ((e = cudaMemcpyAsync(res, scal + 8 + read, n * sizeof(float), cudaMemcpyDeviceToHost,
                                 s)) != cudaSuccess ||
            (e = cudaStreamSynchronize(s)) != cudaSuccess)
          return e;
        bool done = it == iterations;
        updates = it;
        for (int i = 0; i < n; ++i) {
          if (residuals != nullptr) residuals[read + i] = res[i];
          if (res[i] <= tol) {
            updates = read + i;
            done = true;
            break;
          }
        }
        read = it + 1;
        if (done) break;
      }
    }
    if (it == 0) {
      // zf holds T0^T, and Z1 = T0: no product; Y1 = Y0 T0
      SquarePassArgs a[2];
      a[0] = sym_pass(zf, zs);
      a[0].row = tts;
      a[1].c = yf;
      a[1].row = ys;
      if (full) {
        const SquareArgs y1 = product(ys, tts, yf);
        const SquarePassArgs yp = sym_pass(yf, ys);
        if ((e = launch_square_pass(a, 2, K, stop, s)) != cudaSuccess ||
            (e = launch_square(&y1, 1, sms, s)) != cudaSuccess ||
            (e = launch_square_pass(&yp, 1, K, stop, s)) != cudaSuccess)
          return e;
      } else {
        // Y0 leaves T's room for T0^T, and Y1 goes to Z's until that is split
        float* y1f = reinterpret_cast<float*>(zs.planes);
        SquarePassArgs t0;
        t0.c = zf;
        t0.row = ts;
        const SquareArgs y1 = product(ys, ts, y1f);
        const SquarePassArgs yp = sym_pass(y1f, ys), zp = sym_pass(zf, zs);
        if ((e = launch_square_pass(a + 1, 1, K, stop, s)) != cudaSuccess ||
            (e = launch_square_pass(&t0, 1, K, stop, s)) != cudaSuccess ||
            (e = launch_square(&y1, 1, sms, s)) != cudaSuccess ||
            (e = launch_square_pass(&yp, 1, K, stop, s)) != cudaSuccess ||
            (e = launch_square_pass(&zp, 1, K, stop, s)) != cudaSuccess)
          return e;
      }
    } else {
      const SquareArgs zy[2] = {product(ts, zs, zf), product(ys, tts, yf)};
      const SquarePassArgs ps[2] = {sym_pass(zf, zs), sym_pass(yf, ys)};
      if ((e = launch_square(zy, full ? 2 : 1, sms, s)) != cudaSuccess ||
          (!full && ((e = launch_split_transpose(ts, tts, stop, s)) != cudaSuccess ||
                     (e = launch_square(zy + 1, 1, sms, s)) != cudaSuccess)) ||
          (e = launch_square_pass(ps, 2, K, stop, s)) != cudaSuccess)
        return e;
    }
  }
  if (iterations_done != nullptr) *iterations_done = updates;
  // Z ~ (R/c)^-1/2:  R^-1/2 = Z / sqrt(c);  R^-1 = Z Z / c
  if (updates == 0) {
    scaled_identity_kernel<<<std::min(K, 4096), 256, 0, s>>>(K, inverse ? scal + 4 : scal + 3, m,
                                                             ldm);
    return cudaGetLastError();
  }
  if (!inverse) return launch_symmetric_scale(zf, K, K, scal + 3, m, ldm, s);
  SquareArgs a;
  a.x = zs;
  a.y = zs;
  a.symmetric = true;
  a.alpha_s = scal + 4;
  a.c = m;
  a.ldc = ldm;
  a.status = status;
  return launch_square(&a, 1, sms, s);
}

}  // namespace bergson
