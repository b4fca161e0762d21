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
// The same product for FP32 operands.  The kernel above takes one 4-byte shared
// read per operand value: at 32 x 32 tiles the shared-memory pipe, not the FMA pipe,
// set the pace (1024 x 256 x 256: 10 us against 1.7 us of FMAs).  Here every shared
// read is 8 or 16 bytes, and slices of 16 k arrive through a four-deep ring of
// asynchronous copies (16 bytes each where the rows allow it).  An operand stays in
// the order it has in memory: k along rows ([m][16 + 4]: the pitch and the strided
// rows of a thread, ty, ty + BM / TM, ..., make the reads conflict-free), or m / n
// along rows ([k][BM + 4], a thread's neighbouring columns, two per instruction).
// Every output is the same chain of fused multiply-adds over k in order, so it has
// the bits of the kernel above, whatever the tile and the orders.
__device__ __forceinline__ void cp_async4(float* dst, const float* src, bool live) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 4, %2;" ::"r"(d), "l"(src), "r"(live ? 4 : 0) : "memory");
}
__device__ __forceinline__ void cp_async16(float* dst, const float* src, bool live) {
  const uint32_t d = static_cast<uint32_t>(__cvta_generic_to_shared(dst));
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;" ::"r"(d), "l"(src), "r"(live ? 16 : 0) : "memory");
}

constexpr int kF32K = 16, kF32Stages = 4;

// One operand's ring: R rows or columns of the tile, T of them per thread.
// KC: k is contiguous in memory (and in the ring).
template <bool KC, int R, int T>
struct F32Ring {
  static constexpr int kPitch = KC ? kF32K + 4 : R + 4;
  static constexpr int kRows = KC ? R : kF32K;
  float v[kF32Stages][kRows][kPitch];
  // copy slice k0 .. k0 + 15; at(i, k): element address; rows [r0, n) and k < K live
  template <int THREADS, class AT>
  __device__ __forceinline__ void load(int buf, int k0, int r0, int n, int K, bool vec, const AT& at) {
    const int tid = threadIdx.x;
    if (vec) {   // 4 consecutive elements of a row per copy, wholly inside or outside
#pragma unroll
      for (int e0 = 0; e0 < R * kF32K / 4; e0 += THREADS) {
        const int e = e0 + tid;
        if (R * kF32K / 4 % THREADS != 0 && e >= R * kF32K / 4) break;
        const int r = KC ? e / (kF32K / 4) : 4 * (e % (R / 4)), kk = KC ? 4 * (e % (kF32K / 4)) : e / (R / 4);
        const bool live = r0 + r < n && k0 + kk < K;
        cp_async16(KC ? &v[buf][r][kk] : &v[buf][kk][r], at(live ? r0 + r : 0, live ? k0 + kk : 0), live);
      }
    } else {
#pragma unroll
      for (int e0 = 0; e0 < R * kF32K; e0 += THREADS) {
        const int e = e0 + tid;
        const int r = KC ? e / kF32K : e % R, kk = KC ? e % kF32K : e / R;
        const bool live = r0 + r < n && k0 + kk < K;
        cp_async4(KC ? &v[buf][r][kk] : &v[buf][kk][r], at(live ? r0 + r : 0, live ? k0 + kk : 0), live);
      }
    }
  }
  // this thread's i-th row / column of the tile
  static __device__ __forceinline__ int index(int t, int i) { return KC ? t + (R / T) * i : T * t + i; }
  // its T values at k = k4 .. k4 + 3
  __device__ __forceinline__ void read(int buf, int t, int k4, float (&x)[4][T]) const {
    if constexpr (KC) {
#pragma unroll
      for (int i = 0; i < T; ++i) {
        const float4 f = *reinterpret_cast<const float4*>(&v[buf][index(t, i)][k4]);
        x[0][i] = f.x, x[1][i] = f.y, x[2][i] = f.z, x[3][i] = f.w;
      }
    } else {
#pragma unroll
      for (int q = 0; q < 4; ++q) {
        if constexpr (T == 4) {
          const float4 f = *reinterpret_cast<const float4*>(&v[buf][k4 + q][T * t]);
          x[q][0] = f.x, x[q][1] = f.y, x[q][2] = f.z, x[q][3] = f.w;
        } else {
          const float2 f = *reinterpret_cast<const float2*>(&v[buf][k4 + q][T * t]);
          x[q][0] = f.x, x[q][1] = f.y;
        }
      }
    }
  }
};

// One product; a launch takes one or two that do not depend on each other (the two
// networks of the critic: blockIdx.z).  At its sizes a product is a few tiles per SM
// at most, and half the launches halve the time.
template <class LA, class LB, class EP>
struct GemmSet {
  int M, N, K;
  LA la;
  LB lb;
  EP ep;
  int vec_a = 0, vec_b = 0;   // 16-byte copies (set by the launch)
};
template <class LA, class LB, class EP>
struct GemmSets {
  GemmSet<LA, LB, EP> s[2];
};

template <InnerOp OP, int BM, int BN, int TM, int TN, class LA, class LB, class EP>
__global__ void __launch_bounds__((BM / TM) * (BN / TN))
    gemm_f32_kernel(const __grid_constant__ GemmSets<LA, LB, EP> sets) {
  constexpr int kThreads = (BM / TM) * (BN / TN);
  static_assert(BM * kF32K % kThreads == 0 && BN * kF32K % kThreads == 0, "copies per thread");
  using RA = F32Ring<LA::kContigK, BM, TM>;
  using RB = F32Ring<LB::kContigK, BN, TN>;
  __shared__ __align__(16) RA As;
  __shared__ __align__(16) RB Bs;
  pdl_enter();
  const GemmSet<LA, LB, EP>& set = sets.s[blockIdx.z];
  const int M = set.M, N = set.N, K = set.K, vec_a = set.vec_a, vec_b = set.vec_b;
  const LA la = set.la;
  const LB lb = set.lb;
  const EP ep = set.ep;
  const int tid = threadIdx.x;
  const int tx = tid % (BN / TN), ty = tid / (BN / TN);
  const int m0 = blockIdx.y * BM, n0 = blockIdx.x * BN;
  if (m0 >= M || n0 >= N) return;   // (the grid covers the larger product)
  auto load = [&](int buf, int k0) {
    As.template load<kThreads>(buf, k0, m0, M, K, vec_a != 0, [&](int m, int k) { return la.addr(m, k); });
    Bs.template load<kThreads>(buf, k0, n0, N, K, vec_b != 0, [&](int n, int k) { return lb.addr(k, n); });
  };
  float2 acc[TM][TN / 2];
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN / 2; ++j) acc[i][j] = make_float2(0.f, 0.f);
  const int nk = (K + kF32K - 1) / kF32K;
#pragma unroll
  for (int s = 0; s < kF32Stages - 1; ++s) {
    if (s < nk) load(s, s * kF32K);
    asm volatile("cp.async.commit_group;" ::: "memory");
  }
  for (int t = 0; t < nk; ++t) {
    asm volatile("cp.async.wait_group %0;" ::"n"(kF32Stages - 2) : "memory");
    __syncthreads();   // slice t has landed for every thread, and slice t - 1 has been read
    if (t + kF32Stages - 1 < nk) load((t + kF32Stages - 1) % kF32Stages, (t + kF32Stages - 1) * kF32K);
    asm volatile("cp.async.commit_group;" ::: "memory");
    const int buf = t % kF32Stages;
    // (padded k are zero on both sides: they add 0 for every inner op)
#pragma unroll
    for (int k4 = 0; k4 < kF32K; k4 += 4) {
      float a[4][TM], b[4][TN];
      As.read(buf, ty, k4, a);
      Bs.read(buf, tx, k4, b);
#pragma unroll
      for (int q = 0; q < 4; ++q)
#pragma unroll
        for (int i = 0; i < TM; ++i)
#pragma unroll
          for (int j = 0; j < TN / 2; ++j) {
            const float x = a[q][i], y0 = b[q][2 * j], y1 = b[q][2 * j + 1];
            if constexpr (!LB::kContigK && OP == InnerOp::kMul) {   // neighbouring columns: two per instruction
              acc[i][j] = fma_x2(make_float2(x, x), make_float2(y0, y1), acc[i][j]);
            } else if constexpr (OP == InnerOp::kMul) {
              acc[i][j].x = fmaf(x, y0, acc[i][j].x);
              acc[i][j].y = fmaf(x, y1, acc[i][j].y);
            } else {
              const float d0 = x - y0, d1 = x - y1;
              if constexpr (OP == InnerOp::kSqDiff) {
                acc[i][j].x = fmaf(d0, d0, acc[i][j].x);
                acc[i][j].y = fmaf(d1, d1, acc[i][j].y);
              } else {
                acc[i][j].x += fabsf(d0);
                acc[i][j].y += fabsf(d1);
              }
            }
          }
    }
  }
#pragma unroll
  for (int i = 0; i < TM; ++i)
#pragma unroll
    for (int j = 0; j < TN; ++j) {
      const int m = m0 + RA::index(ty, i), n = n0 + RB::index(tx, j);
      if (m < M && n < N) ep(m, n, (j & 1) ? acc[i][j / 2].y : acc[i][j / 2].x);
    }
}

template <InnerOp OP, int BM, int BN, int TM, int TN, class LA, class LB, class EP>
void launch_gemm_f32(const GemmSets<LA, LB, EP>& g, int n, int M, int N, cudaStream_t st) {
  static std::atomic<uint64_t> allowed{0};
  const auto kernel = gemm_f32_kernel<OP, BM, BN, TM, TN, LA, LB, EP>;
  const dim3 grid(ceil_div(N, BN), ceil_div(M, BM), n);
  constexpr size_t kFixed = sizeof(F32Ring<LA::kContigK, BM, TM>) + sizeof(F32Ring<LB::kContigK, BN, TN>);
  launch_k(kernel, grid, dim3((BM / TM) * (BN / TN)), spread_smem(kernel, allowed, kFixed, (long long)grid.x * grid.y * n),
           st, g);
}

// The FP32 tiles, widest first, with the cost of an output relative to the first.
struct F32Tile {
  int bm, bn;
  double w;
};
constexpr F32Tile kF32Tiles[4] = {{64, 64, 1.0}, {32, 64, 1.05}, {32, 32, 1.2}, {16, 32, 1.5}};
inline double f32_tile_cost(const F32Tile& t, long long ctas) { return (double)((ctas + 151) / 152) * t.bm * t.bn * t.w; }

// Launch of n products (one or two); traced as class `cls` (CRL_TRACE_*) with
// 2 M N K flops of work each.  FP32 takes the tile whose waves over the 152 SMs cost
// least: outputs per SM, weighted by the shared reads per FMA of its thread tile (a
// 2 x 2 tile reads twice what a 4 x 4 tile does).  FP64 keeps the 32 x 32 tile of the
// kernel above, a launch per product.
template <typename T, InnerOp OP = InnerOp::kMul, class LA, class LB, class EP>
void gemm_sets(const GemmSet<LA, LB, EP>* set, int n, cudaStream_t st, int cls = CRL_TRACE_GEMM) {
  if constexpr (sizeof(T) == 8) {
    for (int i = 0; i < n; ++i) {
      const GemmSet<LA, LB, EP>& p = set[i];
      if (p.M <= 0 || p.N <= 0) continue;
      TraceLaunch tr(cls, st, 2.0 * p.M * p.N * p.K);
      // (its 64 x 64 double buffers would exceed 48 KiB of static shared memory)
      dim3 grid(ceil_div(p.N, 32), ceil_div(p.M, 32));
      launch_k(gemm_tile_kernel<T, OP, 32, 32, LA, LB, EP>, dim3(grid), dim3(256), 0, st, p.M, p.N, p.K, p.la, p.lb, p.ep);
    }
  } else {
    GemmSets<LA, LB, EP> g;
    int live = 0, M = 0, N = 0;
    double flops = 0;
    for (int i = 0; i < n; ++i) {
      if (set[i].M <= 0 || set[i].N <= 0) continue;
      GemmSet<LA, LB, EP>& p = g.s[live++];
      p = set[i];
      p.vec_a = p.la.vec4(p.M, p.K) ? 1 : 0;
      p.vec_b = p.lb.vec4(p.N, p.K) ? 1 : 0;
      M = std::max(M, p.M), N = std::max(N, p.N);
      flops += 2.0 * p.M * p.N * p.K;
    }
    if (live == 0) return;
    if (live == 1) g.s[1] = g.s[0];
    TraceLaunch tr(cls, st, flops);
    int pick = 0;
    double best = 0;
    for (int q = 0; q < 4; ++q) {
      const F32Tile& t = kF32Tiles[q];
      if (t.bm < 64 && ceil_div(M, t.bm) > 65535) continue;   // grid.y
      long long ctas = 0;
      for (int i = 0; i < live; ++i) ctas += (long long)ceil_div(g.s[i].M, t.bm) * ceil_div(g.s[i].N, t.bn);
      const double c = f32_tile_cost(t, ctas);
      if (q == 0 || c < best) best = c, pick = q;
    }
    if (pick == 0) launch_gemm_f32<OP, 64, 64, 4, 4>(g, live, M, N, st);
    else if (pick == 1) launch_gemm_f32<OP, 32, 64, 4, 4>(g, live, M, N, st);
    else if (pick == 2) launch_gemm_f32<OP, 32, 32, 2, 4>(g, live, M, N, st);
    else launch_gemm_f32<OP, 16, 32, 2, 2>(g, live, M, N, st);
  }
}
template <typename T, InnerOp OP = InnerOp::kMul, class LA, class LB, class EP>
void gemm(int M, int N, int K, const LA& la, const LB& lb, const EP& ep, cudaStream_t st, int cls = CRL_TRACE_GEMM) {
  const GemmSet<LA, LB, EP> one{M, N, K, la, lb, ep};
  gemm_sets<T, OP>(&one, 1, st, cls);
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
  // 16-byte pieces along k: one source, aligned rows, whole pieces
  bool vec4(int, int K) const {
    return K == split && (reinterpret_cast<uintptr_t>(p0) & 15) == 0 && (ld0 & 3) == 0 && (K & 3) == 0;
  }
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
  // the same along n
  bool vec4(int n, int) const {
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
  bool vec4(int, int K) const { return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld & 3) == 0 && (K & 3) == 0; }
};
// B(k, n) = W[k][n] (n contiguous).
template <typename T>
struct LoadKN {
  static constexpr bool kContigK = false;
  const T* p;
  int ld;
  __device__ T operator()(int k, int n) const { return p[(size_t)k * ld + n]; }
  __device__ const T* addr(int k, int n) const { return p + (size_t)k * ld + n; }
  bool vec4(int n, int) const { return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld & 3) == 0 && (n & 3) == 0; }
};
// A(m, k) = X[k][m]: the transposed operand of dY^T X (m contiguous).
template <typename T>
struct LoadTrans {
  static constexpr bool kContigK = false;
  const T* p;
  int ld;
  __device__ T operator()(int m, int k) const { return p[(size_t)k * ld + m]; }
  __device__ const T* addr(int m, int k) const { return p + (size_t)k * ld + m; }
  bool vec4(int m, int) const { return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld & 3) == 0 && (m & 3) == 0; }
};
// A(m, k) = X[m][k] (k contiguous).
template <typename T>
struct LoadMK {
  static constexpr bool kContigK = true;
  const T* p;
  int ld;
  __device__ T operator()(int m, int k) const { return p[(size_t)m * ld + k]; }
  __device__ const T* addr(int m, int k) const { return p + (size_t)m * ld + k; }
  bool vec4(int, int K) const { return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld & 3) == 0 && (K & 3) == 0; }
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
