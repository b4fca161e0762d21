// Tiled SIMT GEMM for the FP32 and FP64 paths (CUDA cores, no tensor cores).
//
//   C(m, n) = epilogue(m, n, sum_k op(A(m, k), B(k, n)))
//
// A and B are read through small loader functors, so one kernel serves
// x W^T (forward), dY W (input gradient), dY^T X (weight gradient) and the
// energy matrices (op = product, squared difference or absolute difference).
#pragma once

#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "trace.h"

namespace crl {

enum class InnerOp { kMul, kSqDiff, kAbsDiff };

template <typename T, InnerOp OP>
__device__ __forceinline__ T inner(T a, T b) {
  if constexpr (OP == InnerOp::kMul) return a * b;
  else if constexpr (OP == InnerOp::kSqDiff) { const T d = a - b; return d * d; }
  else return fabs(a - b);
}

// Tile BM x BN (64 x 64 or 32 x 32), 32-deep k slices, 256 threads, each
// thread TM x TN outputs strided by 16 rows / columns (conflict-free shared
// reads).  The next slice is prefetched into registers while the current one
// is multiplied out of the other shared-memory buffer, so each slice costs one
// barrier and the global-load latency overlaps the arithmetic.
template <typename T, InnerOp OP, int BM, int BN, class LA, class LB, class EP>
__global__ void __launch_bounds__(256) gemm_tile_kernel(int M, int N, int K, LA la, LB lb, EP ep) {
  pdl_enter();
  constexpr int BK = 32;
  constexpr int TM = BM / 16, TN = BN / 16;
  constexpr int LDA = BM * BK / 256, LDB = BN * BK / 256;  // elements each thread loads per slice
  __shared__ T As[2][BK][BM + 1];
  __shared__ T Bs[2][BK][BN + 1];
  const int tid = threadIdx.x;
  const int tx = tid % 16, ty = tid / 16;
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  T acc[TM][TN];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) acc[i][j] = T(0);

  T ra[LDA], rb[LDB];
  auto load = [&](int k0) {
#pragma unroll
    for (int r = 0; r < LDA; ++r) {
      const int e = tid + r * 256;
      int mm, kk;
      if constexpr (LA::kContigK) { kk = e % BK; mm = e / BK; }
      else { mm = e % BM; kk = e / BM; }
      const int m = m0 + mm, k = k0 + kk;
      ra[r] = (m < M && k < K) ? la(m, k) : T(0);
    }
#pragma unroll
    for (int r = 0; r < LDB; ++r) {
      const int e = tid + r * 256;
      int nn, kk;
      if constexpr (LB::kContigK) { kk = e % BK; nn = e / BK; }
      else { nn = e % BN; kk = e / BN; }
      const int n = n0 + nn, k = k0 + kk;
      rb[r] = (n < N && k < K) ? lb(k, n) : T(0);
    }
  };
  auto store = [&](int buf) {
#pragma unroll
    for (int r = 0; r < LDA; ++r) {
      const int e = tid + r * 256;
      int mm, kk;
      if constexpr (LA::kContigK) { kk = e % BK; mm = e / BK; }
      else { mm = e % BM; kk = e / BM; }
      As[buf][kk][mm] = ra[r];
    }
#pragma unroll
    for (int r = 0; r < LDB; ++r) {
      const int e = tid + r * 256;
      int nn, kk;
      if constexpr (LB::kContigK) { kk = e % BK; nn = e / BK; }
      else { nn = e % BN; kk = e / BN; }
      Bs[buf][kk][nn] = rb[r];
    }
  };

  load(0);
  store(0);
  __syncthreads();
  int buf = 0;
  for (int k0 = 0; k0 < K; k0 += BK) {
    const bool more = k0 + BK < K;
    if (more) load(k0 + BK);
    // Padded k entries are zero on both sides, so they add 0 for every inner op.
#pragma unroll 8
    for (int kk = 0; kk < BK; ++kk) {
      T a[TM], b[TN];
#pragma unroll
      for (int i = 0; i < TM; ++i) a[i] = As[buf][kk][ty + 16 * i];
#pragma unroll
      for (int j = 0; j < TN; ++j) b[j] = Bs[buf][kk][tx + 16 * j];
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN; ++j) acc[i][j] += inner<T, OP>(a[i], b[j]);
    }
    if (more) store(buf ^ 1);
    __syncthreads();
    buf ^= 1;
  }
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int m = m0 + ty + 16 * i, n = n0 + tx + 16 * j;
      if (m < M && n < N) ep(m, n, acc[i][j]);
    }
}

// ---- FP32 kernel ---------------------------------------------------------------
// The same product for FP32 operands.  The 2 x 2 and 4 x 4 outputs per thread of
// the kernel above take one 4-byte shared read per operand value: at 32 x 32 tiles
// the shared-memory pipe, not the FMA pipe, set the pace (1024 x 256 x 256: 10 us
// against 1.7 us of FMAs).  Here a thread owns TM x TN neighbouring outputs, reads
// its operands 8 or 16 bytes at a time and multiplies two columns per instruction;
// slices of 16 k arrive through a four-deep ring of asynchronous copies.  Every
// output is the same chain of fused multiply-adds over k in order, so it has the
// bits of the kernel above, whatever the tile.
__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool live) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(live ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool live) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.cg.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(live ? 16 : 0) : "memory");
}

template <int N>
__device__ __forceinline__ void lds_row(const float* p, float (&v)[N]) {
  if constexpr (N == 4) {
    const float4 t = *reinterpret_cast<const float4*>(p);
    v[0] = t.x, v[1] = t.y, v[2] = t.z, v[3] = t.w;
  } else {
    const float2 t = *reinterpret_cast<const float2*>(p);
    v[0] = t.x, v[1] = t.y;
  }
}

template <InnerOp OP, int BM, int BN, int TM, int TN, class LA, class LB, class EP>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
    gemm_f32_kernel(int M, int N, int K, LA la, LB lb, EP ep, int vec_a, int vec_b) {
  constexpr int BK = 16, kStages = 4, kThreads = (BM / TM) * (BN / TN);
  constexpr int LDA = BM + 4, LDB = BN + 4;   // rows stay 16-byte aligned
  static_assert((BM * BK) % (4 * kThreads) == 0 || BM * BK / 4 < kThreads, "A copies per thread");
  __shared__ __align__(16) float As[kStages][BK][LDA];
  __shared__ __align__(16) float Bs[kStages][BK][LDB];
  pdl_enter();
  const int tid = threadIdx.x;
  const int tx = tid % (BN / TN), ty = tid / (BN / TN);
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  auto load = [&](int buf, int k0) {
    if (!LA::kContigK && vec_a) {   // 4 m of one k per copy
      for (int e = tid; e < BM * BK / 4; e += kThreads) {
        const int mm = 4 * (e % (BM / 4)), kk = e / (BM / 4), m = m0 + mm, k = k0 + kk;
        const bool live = m < M && k < K;
        cp_async16(&As[buf][kk][mm], la.addr(live ? m : 0, live ? k : 0), live);
      }
    } else {
#pragma unroll
      for (int r = 0; r < (BM * BK + kThreads - 1) / kThreads; ++r) {
        const int e = tid + r * kThreads;
        const int mm = LA::kContigK ? e / BK : e % BM, kk = LA::kContigK ? e % BK : e / BM;
        const int m = m0 + mm, k = k0 + kk;
        const bool live = m < M && k < K;
        cp_async4(&As[buf][kk][mm], la.addr(live ? m : 0, live ? k : 0), live);
      }
    }
    if (!LB::kContigK && vec_b) {
      for (int e = tid; e < BN * BK / 4; e += kThreads) {
        const int nn = 4 * (e % (BN / 4)), kk = e / (BN / 4), n = n0 + nn, k = k0 + kk;
        const bool live = n < N && k < K;
        cp_async16(&Bs[buf][kk][nn], lb.addr(live ? k : 0, live ? n : 0), live);
      }
    } else {
#pragma unroll
      for (int r = 0; r < (BN * BK + kThreads - 1) / kThreads; ++r) {
        const int e = tid + r * kThreads;
        const int nn = LB::kContigK ? e / BK : e % BN, kk = LB::kContigK ? e % BK : e / BN;
        const int n = n0 + nn, k = k0 + kk;
        const bool live = n < N && k < K;
        cp_async4(&Bs[buf][kk][nn], lb.addr(live ? k : 0, live ? n : 0), live);
      }
    }
  };
  float2 acc[TM][TN / 2];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc[i][j] = make_float2(0.f, 0.f);
  const int nk = (K + BK - 1) / BK;
#pragma unroll
  for (int s = 0; s < kStages - 1; ++s) {
    if (s < nk) load(s, s * BK);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int t = 0; t < nk; ++t) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kStages - 2) : "memory");
    __syncthreads();   // slice t has landed for every thread, and slice t - 1 has been read
    if (t + kStages - 1 < nk) load((t + kStages - 1) % kStages, (t + kStages - 1) * BK);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const float* as = &As[t % kStages][0][TM * ty];
    const float* bs = &Bs[t % kStages][0][TN * tx];
    // (padded k are zero on both sides: they add 0 for every inner op)
#pragma unroll
    for (int kk = 0; kk < BK; ++kk) {
      float a[TM], b[TN];
      lds_row<TM>(as + kk * LDA, a);
      lds_row<TN>(bs + kk * LDB, b);
#pragma unroll
      for (int i = 0; i < TM; ++i)
#pragma unroll
        for (int j = 0; j < TN / 2; ++j) {
          const float2 aa = make_float2(a[i], a[i]), bb = make_float2(b[2 * j], b[2 * j + 1]);
          if constexpr (OP == InnerOp::kMul) {
            acc[i][j] = fma_x2(aa, bb, acc[i][j]);
          } else {
            const float2 d = fma_x2(bb, make_float2(-1.f, -1.f), aa);   // a - b
            if constexpr (OP == InnerOp::kSqDiff) acc[i][j] = fma_x2(d, d, acc[i][j]);
            else acc[i][j] = add_x2(acc[i][j], make_float2(fabsf(d.x), fabsf(d.y)));
          }
        }
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int m = m0 + TM * ty + i, n = n0 + TN * tx + j;
      if (m < M && n < N) ep(m, n, (j & 1) ? acc[i][j / 2].y : acc[i][j / 2].x);
    }
}

template <InnerOp OP, int BM, int BN, int TM, int TN, class LA, class LB, class EP>
void launch_gemm_f32(int M, int N, int K, const LA& la, const LB& lb, const EP& ep, cudaStream_t st) {
  launch_k(gemm_f32_kernel<OP, BM, BN, TM, TN, LA, LB, EP>, dim3(ceil_div(N, BN), ceil_div(M, BM)),
           dim3((BM / TM) * (BN / TN)), 0, st, M, N, K, la, lb, ep, la.vec4(M) ? 1 : 0, lb.vec4(N) ? 1 : 0);
}

// Launch; traced as class `cls` (CRL_TRACE_*) with 2 M N K flops of work.  FP32
// takes the tile whose waves over the 152 SMs cost least: outputs per SM, weighted
// by the shared reads per FMA of its thread tile (a 2 x 2 tile reads twice what a
// 4 x 4 tile does).  FP64 keeps the 32 x 32 tile of the kernel above.
template <typename T, InnerOp OP = InnerOp::kMul, class LA, class LB, class EP>
void gemm(int M, int N, int K, const LA& la, const LB& lb, const EP& ep, cudaStream_t st, int cls = CRL_TRACE_GEMM) {
  if (M <= 0 || N <= 0) return;
  TraceLaunch tr(cls, st, 2.0 * M * N * K);
  if constexpr (sizeof(T) == 8) {
    // (its 64 x 64 double buffers would exceed 48 KiB of static shared memory)
    dim3 grid(ceil_div(N, 32), ceil_div(M, 32));
    launch_k(gemm_tile_kernel<T, OP, 32, 32, LA, LB, EP>, dim3(grid), dim3(256), 0, st, M, N, K, la, lb, ep);
  } else {
    auto cost = [&](int bm, int bn, double w) {
      if (bm < 64 && ceil_div(M, bm) > 65535) return 1e300;   // grid.y
      const long long ctas = (long long)ceil_div(M, bm) * ceil_div(N, bn);
      return (double)((ctas + 151) / 152) * bm * bn * w;
    };
    const double c64 = cost(64, 64, 1.0), c32w = cost(32, 64, 1.05), c32 = cost(32, 32, 1.2), c16 = cost(16, 32, 1.5);
    const double best = std::min(std::min(c64, c32w), std::min(c32, c16));
    if (best == c64) launch_gemm_f32<OP, 64, 64, 4, 4>(M, N, K, la, lb, ep, st);
    else if (best == c32w) launch_gemm_f32<OP, 32, 64, 4, 4>(M, N, K, la, lb, ep, st);
    else if (best == c32) launch_gemm_f32<OP, 32, 32, 2, 4>(M, N, K, la, lb, ep, st);
    else launch_gemm_f32<OP, 16, 32, 2, 2>(M, N, K, la, lb, ep, st);
  }
}

// ---- loaders ---------------------------------------------------------------
// A(m, k) = concat(x0[m][0:split], x1[m][0:K-split])[k]  (row-major, k contiguous)
template <typename T, typename T0, typename T1>
struct LoadRowsSplit {
  static constexpr bool kContigK = true;
  const T0* p0;
  const T1* p1;
  int ld0, ld1, split;
  __device__ T operator()(int m, int k) const {
    return k < split ? T(p0[(size_t)m * ld0 + k]) : T(p1[(size_t)m * ld1 + (k - split)]);
  }
  __device__ const T* addr(int m, int k) const {
    return k < split ? p0 + (size_t)m * ld0 + k : p1 + (size_t)m * ld1 + (k - split);
  }
  bool vec4(int) const { return false; }
};
// B(k, n) = X[k][n] split by columns (row-major X, n contiguous): weight gradient dY^T X.
template <typename T, typename T0, typename T1>
struct LoadColsSplit {
  static constexpr bool kContigK = false;
  const T0* p0;
  const T1* p1;
  int ld0, ld1, split;
  __device__ T operator()(int k, int n) const {
    return n < split ? T(p0[(size_t)k * ld0 + n]) : T(p1[(size_t)k * ld1 + (n - split)]);
  }
  __device__ const T* addr(int k, int n) const {
    return n < split ? p0 + (size_t)k * ld0 + n : p1 + (size_t)k * ld1 + (n - split);
  }
  // 16-byte pieces: one source, aligned rows, whole pieces
  bool vec4(int n) const {
    return n == split && (reinterpret_cast<uintptr_t>(p0) & 15) == 0 && (ld0 & 3) == 0 && (n & 3) == 0;
  }
};
// B(k, n) = W[n][k]: the weight of x W^T (k contiguous).
template <typename T>
struct LoadNK {
  static constexpr bool kContigK = true;
  const T* p;
  int ld;
  __device__ T operator()(int k, int n) const { return p[(size_t)n * ld + k]; }
  __device__ const T* addr(int k, int n) const { return p + (size_t)n * ld + k; }
  bool vec4(int) const { return false; }
};
// B(k, n) = W[k][n] (n contiguous).
template <typename T>
struct LoadKN {
  static constexpr bool kContigK = false;
  const T* p;
  int ld;
  __device__ T operator()(int k, int n) const { return p[(size_t)k * ld + n]; }
  __device__ const T* addr(int k, int n) const { return p + (size_t)k * ld + n; }
  bool vec4(int n) const { return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld & 3) == 0 && (n & 3) == 0; }
};
// A(m, k) = X[k][m]: the transposed operand of dY^T X (m contiguous).
template <typename T>
struct LoadTrans {
  static constexpr bool kContigK = false;
  const T* p;
  int ld;
  __device__ T operator()(int m, int k) const { return p[(size_t)k * ld + m]; }
  __device__ const T* addr(int m, int k) const { return p + (size_t)k * ld + m; }
  bool vec4(int m) const { return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld & 3) == 0 && (m & 3) == 0; }
};
// A(m, k) = X[m][k] (k contiguous).
template <typename T>
struct LoadMK {
  static constexpr bool kContigK = true;
  const T* p;
  int ld;
  __device__ T operator()(int m, int k) const { return p[(size_t)m * ld + k]; }
  __device__ const T* addr(int m, int k) const { return p + (size_t)m * ld + k; }
  bool vec4(int) const { return false; }
};

// ---- epilogues -------------------------------------------------------------
// C = act(acc + bias[n])
template <typename T>
struct EpiBias {
  T* C;
  int ldc;
  const T* bias;
  int relu;
  __device__ void operator()(int m, int n, T acc) const {
    T v = acc + (bias ? bias[n] : T(0));
    if (relu) v = v > T(0) ? v : T(0);
    C[(size_t)m * ldc + n] = v;
  }
};
// C = alpha * acc
template <typename T>
struct EpiScale {
  T* C;
  int ldc;
  T alpha;
  __device__ void operator()(int m, int n, T acc) const { C[(size_t)m * ldc + n] = alpha * acc; }
};
// v = acc * [mask[m][n] > 0]; written to c0 (n < split) or c1 (n >= split), either may be null.
template <typename T>
struct EpiMaskSplit {
  T* c0;
  T* c1;
  int ld0, ld1, split;
  const T* mask;
  int ldm;
  __device__ void operator()(int m, int n, T acc) const {
    T v = acc;
    if (mask && !(mask[(size_t)m * ldm + n] > T(0))) v = T(0);
    if (n < split) {
      if (c0) c0[(size_t)m * ld0 + n] = v;
    } else if (c1) {
      c1[(size_t)m * ld1 + (n - split)] = v;
    }
  }
};
// C = alpha * acc - s[m] * X[m][n]
template <typename T>
struct EpiSubRowScaled {
  T* C;
  int ldc;
  T alpha;
  const T* s;
  const T* X;
  int ldx;
  __device__ void operator()(int m, int n, T acc) const {
    C[(size_t)m * ldc + n] = alpha * acc - s[m] * X[(size_t)m * ldx + n];
  }
};

}  // namespace crl
