// Grouped BF16 tensor-core GEMM on tcgen05 with TMEM accumulators and TMA
// operand loads.  One launch runs a list of independent problems
//
//   C_p(m, n) = epilogue_p(m, n, sum_k A_p[m][k] * B_p[n][k])      A, B: BF16, K-major
//
// (the same layer of several networks, or all weight gradients of a network),
// each split into 128 x BN tiles; CTA t finds its problem by a binary search of
// the tiles' prefix sums in the problem table.  The table (tensor maps,
// sizes, epilogue descriptor) lives in device memory and is never written
// while kernels run.
//
// One CTA computes one 128 x BN tile (BN in {64, 128, 256}); 256 threads:
//   warp 0 / lane 0 -- TMA producer: 64-wide K slices of A and B (as 64-row
//                      boxes: every tensor map has box {64, 64}) into a
//                      STAGES-deep shared-memory ring (128-byte swizzle);
//   warp 1 / lane 0 -- MMA issuer: 4 x tcgen05.mma (K = 16 each) per slice
//                      into the FP32 accumulator in TMEM (128 lanes x BN cols);
//   all 8 warps     -- epilogue: warp w reads TMEM lanes 32 (w % 4) .. (rows)
//                      of every second 32-column step and applies the problem's
//                      epilogue (whole row segments, through shared memory).
// Either operand may be stored MN-major instead (the weight gradients read the
// activations and output gradients as they are stored: the batch is K).
// Out-of-range rows and columns of the operands are zero-filled by TMA; the
// epilogue clips its stores to M x N.
#pragma once

#include <cuda_bf16.h>

#include "common.cuh"
#include "tc_common.cuh"

namespace crl {
namespace tc {

constexpr int kBM = 128;
constexpr int kBK = 64;

// What the FP32 accumulator tile of a problem becomes.
enum EpiKind : int {
  kEpiFwdHidden = 0,  // h = ReLU(acc + b) as BF16 hi / lo parts: h_hi [M][ld0] columns [0, N), h_lo = bf16(h -
                      // h_hi) at columns [c0, c0 + N) of the same rows
  kEpiFwdPreLN = 1,   // z = acc + b: FP32 [M][ld0] (LayerNorm follows)
  kEpiFwdOut = 2,     // y = acc + b: FP32 [M][ld0]
  kEpiBwdDX = 3,      // dz = acc * [mask > 0]: BF16 dz [M][ld0]
  kEpiBwdDXLN = 4,    // du = acc * [mask > 0]: FP32 [M][ld0]
  kEpiBwdDW = 5,      // dW [M][kin] (columns < kin), db [M] (column kin: the ones row)
  kEpiBwdDW0 = 6,     // split first layer: dW[m][c] = acc[2c] + acc[2c+1], db[m] = acc[2 kin]
  kEpiDX0 = 7,        // dx [M][nc] = acc columns [c0, c0 + nc)
  kEpiFwdOutEnergy = 8,  // output layer feeding the fused energy: y = acc + b FP32 [M][ld0], the BF16
                         // energy operand x = y * s [M][N] (out1), aux [M];
                         // s = 1 / |y| and aux = s for the cosine energy, else s = 1 and aux = |bf16(y)|^2.
                         // The tile must span the whole row (the launch picks BN >= N).
};

struct EpiDesc {
  int kind, ld0, ld1, kin, c0, nc, ldm, energy;
  const float* bias;
  const __nv_bfloat16* mask;  // [M][ldm], BF16 post-ReLU activation (> 0 where the unit is active)
  void* out0;
  void* out1;
  void* out2;
  float* aux;
};

struct GemmProblem {   // 128-byte aligned by its tensor maps
  CUtensorMap a, b;
  CUtensorMap o0, o1;   // tma_out: output maps, boxes of 32 rows x 128 bytes (o1: the lo part of a hidden layer)
  int M, N, K, nkA;   // nkA > 0: split-weight product (see tc_gemm_kernel)
  int a_mn, b_mn;     // operand stored MN-major ([K][M] / [K][N], the M / N index contiguous): its
                      // tensor map's inner dimension is M / N, boxes {64 MN, 64 K}
  int a_gap, a_skip;  // a_gap > 0 (K-major A): A's K slices from a_gap on sit a_skip 64-column blocks further
  int tiles_n, tile_begin;
  int ksplit;         // > 1: K is split over ksplit CTAs per output tile (one-tile kernel only)
  int ksplit_cap;     // the most splits the problem's buffers hold (the launch picks ksplit <= it)
  int tma_out, pad_;
  EpiDesc epi;
  float* part;        // split-K partial tiles [tile][ksplit][128][BN] (FP32)
  unsigned* tickets;  // split-K arrival count per output tile (zero between launches)
};
static_assert(alignof(GemmProblem) >= 64 && sizeof(GemmProblem) % 64 == 0, "problem tables hold aligned tensor maps");

// Ring depth STAGES: deep rings keep a whole 512-deep product in flight at
// once (latency-bound small problems); shallow ones leave room for two CTAs
// per SM, one's epilogue overlapping the other's main loop (large problems).
constexpr int kTileThreads = 256;        // one-tile kernel: 8 warps
constexpr int kPersistentThreads = 320;  // persistent kernel: producer, issuer, 8 epilogue warps
constexpr int kPairThreads = 320;        // CTA-pair kernel: producer, issuer, 8 epilogue warps
template <int BN, int STAGES>
struct GemmSmem {
  static constexpr uint32_t kABytes = kBM * kBK * 2;   // 16 KiB
  static constexpr uint32_t kBBytes = BN * kBK * 2;    // BN * 128 B
  static constexpr uint32_t kStageBytes = kABytes + kBBytes;
  static constexpr int kStages = STAGES;
  // operand ring + barriers (full[S], empty[S], done) + TMEM slot, plus 1 KiB for alignment
  static constexpr uint32_t kBytes = kStages * kStageBytes + 1024 + 256;
  // the persistent kernel's epilogue runs beside the ring and has staging blocks of its own
  static constexpr uint32_t kPersistentBytes = kBytes + 8 * 4096;
  static constexpr uint32_t kTmemCols = BN;
  static_assert(BN % 64 == 0 && BN <= 256, "BN must be 64, 128 or 256");
  static_assert(kBytes <= 227 * 1024, "shared memory per CTA");
  static_assert(kStages * kStageBytes >= 8 * 4096, "the one-tile kernel stages its epilogue in the ring");
};

__device__ __forceinline__ void load_bias32(const float* b, float (&x)[32]) {
  const float4* s = reinterpret_cast<const float4*>(b);
#pragma unroll
  for (int q = 0; q < 8; ++q) {
    const float4 t = __ldg(s + q);
    x[4 * q] = t.x;
    x[4 * q + 1] = t.y;
    x[4 * q + 2] = t.z;
    x[4 * q + 3] = t.w;
  }
}

// L2 prefetch of a tile's B operand (the weight side of every product here),
// issued before pdl_wait so that its DRAM reads overlap the predecessor's
// tail.  The predecessor never writes it: B holds weights (written by the
// Adam step of an earlier launch) or activations of an earlier layer.
template <int BN>
__device__ __forceinline__ void prefetch_b_tile(const CUtensorMap* tmB, int K, int N, int n0) {
  const int nk = (K + kBK - 1) / kBK;
  for (int kb = 0; kb < nk && kb < 64; ++kb)
#pragma unroll
    for (int r = 0; r < BN / 64; ++r)
      if (n0 + 64 * r < N) tma_prefetch_2d(tmB, kb * kBK, n0 + 64 * r);
}

// L2 prefetch of a tile's B operand in either storage order.
template <int BN>
__device__ __forceinline__ void prefetch_b(const GemmProblem* P, int n0) {
  if (!P->b_mn) {
    prefetch_b_tile<BN>(&P->b, P->K, P->N, n0);
    return;
  }
  const int nk = (P->K + kBK - 1) / kBK;
  for (int kb = 0; kb < nk && kb < 64; ++kb)
#pragma unroll
    for (int r = 0; r < BN / 64; ++r)
      if (n0 + 64 * r < P->N) tma_prefetch_2d(&P->b, n0 + 64 * r, kb * kBK);
}

// TMA loads of K slice kb: 128 rows of A from row m0 and NB 64-row boxes of B
// from row n0, each box landing 8 KiB after the previous.  K-major operands
// come as {64 K, 64 rows} boxes (the slice's 128-byte rows), MN-major ones as
// {64 MN, 64 K} boxes (64 K rows of 128 bytes per 64 M or N): in both cases a
// box is an 8 KiB 128-byte-swizzled block.
// The operand description of a problem, read into registers once per tile
// (the loads' asm statements would otherwise force a reread per slice).
struct SliceSrc {
  const CUtensorMap* a;
  const CUtensorMap* b;
  int a_mn, b_mn, nkA, a_gap, a_skip;
};
__device__ __forceinline__ SliceSrc slice_src(const GemmProblem* P) {
  return SliceSrc{&P->a, &P->b, P->a_mn, P->b_mn, P->nkA, P->a_gap, P->a_skip};
}
template <int NB>
__device__ __forceinline__ void load_slice(const SliceSrc& P, uint8_t* a_dst, uint8_t* b_dst, uint64_t* bar, int kb,
                                           int m0, int n0) {
  const CUtensorMap* tmA = P.a;
  const CUtensorMap* tmB = P.b;
  if (P.a_mn) {
#pragma unroll
    for (int r = 0; r < kBM / 64; ++r) tma_load_2d(a_dst + r * 8192, tmA, bar, m0 + 64 * r, kb * kBK);
  } else {
    const int ka = P.nkA > 0 ? kb % P.nkA : kb;
    const int kx = (P.a_gap > 0 && ka >= P.a_gap) ? ka + P.a_skip : ka;
#pragma unroll
    for (int r = 0; r < kBM / 64; ++r) tma_load_2d(a_dst + r * 8192, tmA, bar, kx * kBK, m0 + 64 * r);
  }
  if (P.b_mn) {
#pragma unroll
    for (int r = 0; r < NB; ++r) tma_load_2d(b_dst + r * 8192, tmB, bar, n0 + 64 * r, kb * kBK);
  } else {
#pragma unroll
    for (int r = 0; r < NB; ++r) tma_load_2d(b_dst + r * 8192, tmB, bar, kb * kBK, n0 + 64 * r);
  }
}

// Shared-memory descriptor of a slice's operand tile (K step 0) and the
// increment of its address field per K step of 16: K-major +32 bytes along the
// 128-byte rows, MN-major 16 K rows further (2 KiB; 64-element MN blocks 8 KiB
// apart).  The MMA issuer adds k * step: no per-MMA descriptor arithmetic.
__device__ __forceinline__ uint64_t slice_desc(const uint8_t* tile, bool mn) {
  return mn ? sdesc_mnmajor_sw128(tile, 8192) : sdesc_kmajor_sw128(tile);
}
__device__ __forceinline__ uint32_t slice_step(bool mn) { return mn ? 2048u >> 4 : 32u >> 4; }
// The instruction descriptor's operand-order bits (A: bit 15, B: bit 16; 1 = MN-major).
__device__ __forceinline__ uint32_t idesc_major(uint32_t idesc, const GemmProblem* P) {
  return idesc | ((P->a_mn ? 1u : 0u) << 15) | ((P->b_mn ? 1u : 0u) << 16);
}

// ---- epilogue -----------------------------------------------------------------
// Eight warps: warp (eg, half) reads TMEM lanes (rows) 32 eg .. 32 eg + 31 and
// every second column step of the tile.  A thread holds one row's columns, so
// a direct 16-byte store per thread touches 32 rows: 32 L1 wavefronts and 32
// half-used lines per instruction (measured 2.7 TB/s into L2 against 4.9-6.0
// for whole rows).  Each warp therefore turns its block round in 4 KiB of shared
// memory of its own and stores whole 64- or 128-byte row segments; the ReLU
// masks of the input gradients are read in that layout too.
constexpr int kEpiWarps = 8;
constexpr uint32_t kStageWarpBytes = 4096;
constexpr uint32_t kStageBytesAll = kEpiWarps * kStageWarpBytes;
// Columns per step: 64 with the 256-wide tiles (whole 128-byte BF16 lines that
// leave as TMA stores), 32 with the narrower ones, whose segments the warps store
// themselves.  Measured at 3 x [8192 x 512] hidden outputs, K = 384 (persistent
// kernel): 256-wide 25.6 -> 18.9 us with TMA stores, 128-wide 28.6 -> 34.
template <int BN>
constexpr int kStepCols = BN == 256 ? 64 : 32;

// Byte offset of the 16-byte chunk `ch` of row `row` in a warp's staging block:
// rows of 128 bytes (8 chunks) or of 64 bytes (4 chunks), XOR-swizzled so that
// both the row-per-thread writes and the segment reads are conflict-free.
__device__ __forceinline__ uint32_t stage128(int row, int ch) { return row * 128 + ((ch ^ (row & 7)) << 4); }
__device__ __forceinline__ uint32_t stage64(int row, int ch) { return row * 64 + ((ch ^ ((row >> 1) & 3)) << 4); }

__device__ __forceinline__ uint4 pack_bf16x8(const float* x) {
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(x[2 * i], x[2 * i + 1]);
    w[i] = *reinterpret_cast<const uint32_t*>(&p);
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// 32 FP32 columns of the warp's 32 rows through the staging block:
// f(row, column, float4) for 4 rows of 128 bytes per instruction.
template <class F>
__device__ __forceinline__ void emit_f32x4(uint8_t* st, int lane, const float* v, F&& f) {
#pragma unroll
  for (int q = 0; q < 8; ++q)
    *reinterpret_cast<float4*>(st + stage128(lane, q)) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
  __syncwarp();
  const int ch = lane & 7;
#pragma unroll
  for (int j = 0; j < 8; ++j) {
    const int row = 4 * j + (lane >> 3);
    f(row, 4 * ch, *reinterpret_cast<const float4*>(st + stage128(row, ch)));
  }
  __syncwarp();
}
// The same, one row of 32 columns per instruction (rows without 16-byte alignment): f(row, column, float).
template <class F>
__device__ __forceinline__ void emit_f32(uint8_t* st, int lane, const float* v, F&& f) {
#pragma unroll
  for (int q = 0; q < 8; ++q)
    *reinterpret_cast<float4*>(st + stage128(lane, q)) = make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
  __syncwarp();
#pragma unroll 8
  for (int row = 0; row < 32; ++row)
    f(row, lane, *reinterpret_cast<const float*>(st + stage128(row, lane >> 2) + 4 * (lane & 3)));
  __syncwarp();
}
// NC (64 or 32) BF16 columns: f(j, row, column, uint4 of 8 columns), j = 0 .. NC / 8 - 1.
template <int NC, class F>
__device__ __forceinline__ void emit_bf16(uint8_t* st, int lane, const float* v, F&& f) {
  constexpr int kCh = NC / 8;
#pragma unroll
  for (int q = 0; q < kCh; ++q)
    *reinterpret_cast<uint4*>(st + (NC == 64 ? stage128(lane, q) : stage64(lane, q))) = pack_bf16x8(v + 8 * q);
  __syncwarp();
  const int ch = lane % kCh;
#pragma unroll
  for (int j = 0; j < kCh; ++j) {
    const int row = (32 / kCh) * j + lane / kCh;
    f(j, row, 8 * ch, *reinterpret_cast<const uint4*>(st + (NC == 64 ? stage128(row, ch) : stage64(row, ch))));
  }
  __syncwarp();
}

// Zero the BF16 halves of x whose unit is inactive (mask m <= 0: the post-ReLU
// activations are never negative, so a live unit is one that is not +-0).
__device__ __forceinline__ uint32_t mask_pair(uint32_t x, uint32_t m) {
  const __nv_bfloat162 p = *reinterpret_cast<const __nv_bfloat162*>(&m);
  const uint32_t lo = __low2float(p) > 0.f ? 0x0000FFFFu : 0u, hi = __high2float(p) > 0.f ? 0xFFFF0000u : 0u;
  return x & (lo | hi);
}

// FP32 rows that take 16-byte accesses: the callers' own arrays (an op-level output
// or gradient) may start on any 4-byte boundary.
__device__ __forceinline__ bool rows_aligned16(const float* p, int ld) {
  return (reinterpret_cast<uintptr_t>(p) & 15) == 0 && (ld & 3) == 0;
}

// 32 columns of a gradient output (weights, split first-layer weights, first-layer inputs).
__device__ __forceinline__ void epilogue_grad32(const EpiDesc& e, uint8_t* st, int row0, int lane, const float* v,
                                                int col0, int M, int N) {
  const int row = row0 + lane;   // v: this row's columns
  switch (e.kind) {
    case kEpiBwdDW: {
      float* dW = static_cast<float*>(e.out0);
      if (col0 < e.kin) {
        if (rows_aligned16(dW, e.kin))
          emit_f32x4(st, lane, v, [&](int r, int k, float4 x) {
            if (row0 + r < M && col0 + k < e.kin)
              *reinterpret_cast<float4*>(dW + (size_t)(row0 + r) * e.kin + col0 + k) = x;
          });
        else
          emit_f32(st, lane, v, [&](int r, int k, float x) {
            if (row0 + r < M && col0 + k < e.kin) dW[(size_t)(row0 + r) * e.kin + col0 + k] = x;
          });
      }
      if (row < M && e.kin >= col0 && e.kin < col0 + 32) {
        float* db = static_cast<float*>(e.out1);
#pragma unroll
        for (int i = 0; i < 32; ++i)
          if (col0 + i == e.kin) db[row] = v[i];
      }
      break;
    }
    case kEpiBwdDW0: {
      float* dW = static_cast<float*>(e.out0);
      // 16 summed columns per row, turned round so that 16 lanes store a row's segment
#pragma unroll
      for (int q = 0; q < 4; ++q)
        *reinterpret_cast<float4*>(st + stage64(lane, q)) =
            make_float4(v[8 * q] + v[8 * q + 1], v[8 * q + 2] + v[8 * q + 3], v[8 * q + 4] + v[8 * q + 5],
                        v[8 * q + 6] + v[8 * q + 7]);
      __syncwarp();
      const int k = lane & 15, c = col0 / 2 + k;
#pragma unroll 8
      for (int j = 0; j < 16; ++j) {
        const int r = 2 * j + (lane >> 4);
        const float x = *reinterpret_cast<const float*>(st + stage64(r, k >> 2) + 4 * (k & 3));
        if (row0 + r < M && c < e.kin) dW[(size_t)(row0 + r) * e.kin + c] = x;
      }
      __syncwarp();
      if (row < M && 2 * e.kin >= col0 && 2 * e.kin < col0 + 32) {
        float* db = static_cast<float*>(e.out1);
#pragma unroll
        for (int i = 0; i < 32; i += 2)
          if (col0 + i == 2 * e.kin) db[row] = v[i];
      }
      break;
    }
    default: {  // kEpiDX0
      float* dx = static_cast<float*>(e.out0);
      if (col0 + 32 <= e.c0 || col0 >= e.c0 + e.nc) break;
      emit_f32(st, lane, v, [&](int r, int k, float x) {
        const int c = col0 + k - e.c0;
        if (row0 + r < M && col0 + k < N && c >= 0 && c < e.nc) dx[(size_t)(row0 + r) * e.nc + c] = x;
      });
      break;
    }
  }
}

// The bias of 32 columns (every lane reads the same 16 bytes; the lines were touched ahead, see touch_bias).
__device__ __forceinline__ void bias_cols32(const EpiDesc& e, int col0, int N, float (&x)[32]) {
  if (col0 + 32 <= N) {
    load_bias32(e.bias + col0, x);
  } else {
#pragma unroll
    for (int i = 0; i < 32; ++i) x[i] = col0 + i < N ? __ldg(e.bias + col0 + i) : 0.f;
  }
}

// ---- TMA stores of staged blocks
// A staged block (32 rows of 128 bytes, stage128) leaves as one box of the
// problem's output map: one instruction, no address arithmetic, and the warp
// goes on while the copy engine writes whole lines.  The map clips rows >= M and
// columns >= N.
__device__ __forceinline__ void stage_publish(const CUtensorMap* map, const uint8_t* st, int lane, int x, int y) {
  asm volatile("fence.proxy.async.shared::cta;" ::: "memory");   // this lane's writes, before the copy reads them
  __syncwarp();
  if (lane == 0) {
    asm volatile("cp.async.bulk.tensor.2d.global.shared::cta.bulk_group [%0, {%2, %3}], [%1];" ::"l"(
                     reinterpret_cast<uint64_t>(map)),
                 "r"(smem_u32(st)), "r"(x), "r"(y)
                 : "memory");
    asm volatile("cp.async.bulk.commit_group;" ::: "memory");
  }
}
// The warp's earlier stores have read the staging block: it may be written again.
__device__ __forceinline__ void stage_reclaim(int lane) {
  if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
  __syncwarp();
}

// 32 columns of an FP32 output.
__device__ __forceinline__ void epilogue_f32x32(const GemmProblem* P, const EpiDesc& e, uint8_t* st, bool tma, int row0,
                                                int lane, uint32_t taddr, int col0, int M, int N) {
  float v[32];
  switch (e.kind) {
    case kEpiFwdPreLN:
    case kEpiFwdOut: {
      tmem_ldn(taddr, v);
      float* z = static_cast<float*>(e.out0);
      float b[32];
      bias_cols32(e, col0, N, b);
#pragma unroll
      for (int i = 0; i < 32; ++i) v[i] += b[i];
      if (tma) {
        stage_reclaim(lane);
#pragma unroll
        for (int q = 0; q < 8; ++q)
          *reinterpret_cast<float4*>(st + stage128(lane, q)) =
              make_float4(v[4 * q], v[4 * q + 1], v[4 * q + 2], v[4 * q + 3]);
        stage_publish(&P->o0, st, lane, col0, row0);
      } else if (rows_aligned16(z, e.ld0) && (N & 3) == 0) {
        emit_f32x4(st, lane, v, [&](int r, int k, float4 x) {
          if (row0 + r < M && col0 + k < N) *reinterpret_cast<float4*>(z + (size_t)(row0 + r) * e.ld0 + col0 + k) = x;
        });
      } else {
        emit_f32(st, lane, v, [&](int r, int k, float x) {
          if (row0 + r < M && col0 + k < N) z[(size_t)(row0 + r) * e.ld0 + col0 + k] = x;
        });
      }
      break;
    }
    case kEpiBwdDXLN: {
      // the masks of the segments this lane will store, in flight during the TMEM read
      uint2 m[8];
#pragma unroll
      for (int j = 0; j < 8; ++j) {
        const int r = row0 + 4 * j + (lane >> 3), c = col0 + 4 * (lane & 7);
        m[j] = (r < M && c < N) ? *reinterpret_cast<const uint2*>(e.mask + (size_t)r * e.ldm + c) : make_uint2(0u, 0u);
      }
      tmem_ldn(taddr, v);
      float* du = static_cast<float*>(e.out0);
      emit_f32x4(st, lane, v, [&](int r, int k, float4 x) {
        const uint2 mm = m[(r - (lane >> 3)) / 4];
        const __nv_bfloat162 a = *reinterpret_cast<const __nv_bfloat162*>(&mm.x);
        const __nv_bfloat162 b = *reinterpret_cast<const __nv_bfloat162*>(&mm.y);
        if (row0 + r < M && col0 + k < N)
          *reinterpret_cast<float4*>(du + (size_t)(row0 + r) * e.ld0 + col0 + k) =
              make_float4(__low2float(a) > 0.f ? x.x : 0.f, __high2float(a) > 0.f ? x.y : 0.f,
                          __low2float(b) > 0.f ? x.z : 0.f, __high2float(b) > 0.f ? x.w : 0.f);
      });
      break;
    }
    default:
      tmem_ldn(taddr, v);
      epilogue_grad32(e, st, row0, lane, v, col0, M, N);
      break;
  }
}

// Eight BF16 hi parts of v (returned), v left as the remainders v - hi.
__device__ __forceinline__ uint4 split_bf16x8(float* v) {
  uint32_t w[4];
#pragma unroll
  for (int i = 0; i < 4; ++i) {
    const __nv_bfloat162 p = __floats2bfloat162_rn(v[2 * i], v[2 * i + 1]);
    w[i] = *reinterpret_cast<const uint32_t*>(&p);
    // v - hi, one rounding (two columns per instruction)
    const float2 r = fma_x2(make_float2(__uint_as_float(w[i] << 16), __uint_as_float(w[i] & 0xFFFF0000u)),
                            make_float2(-1.f, -1.f), make_float2(v[2 * i], v[2 * i + 1]));
    v[2 * i] = r.x;
    v[2 * i + 1] = r.y;
  }
  return make_uint4(w[0], w[1], w[2], w[3]);
}

// One step: NC (32 or 64) columns from col0 of the warp's rows row0 .. row0 + 31.
// Hidden widths are multiples of 8 (their BF16 rows need 16-byte TMA strides),
// so an 8-column chunk of a BF16 output lies wholly inside or outside the
// problem; FP32 rows without 16-byte alignment (odd widths) take 4-byte stores.
template <int NC>
__device__ __forceinline__ void epilogue_step(const GemmProblem* P, const EpiDesc& e, uint8_t* st, bool tma, int row0,
                                              int lane, uint32_t taddr, int col0, int M, int N) {
  using bf16 = __nv_bfloat16;
  switch (e.kind) {
    case kEpiFwdHidden: {
      float v[NC];
      tmem_ldn(taddr, v);
#pragma unroll
      for (int c = 0; c < NC; c += 32) {
        float b[32];
        bias_cols32(e, col0 + c, N, b);
#pragma unroll
        for (int i = 0; i < 32; i += 2) {
          const float2 t = add_x2(make_float2(v[c + i], v[c + i + 1]), make_float2(b[i], b[i + 1]));
          v[c + i] = fmaxf(t.x, 0.f);
          v[c + i + 1] = fmaxf(t.y, 0.f);
        }
      }
      if constexpr (NC == 64) {
        // hi block, then lo block, each leaving as one TMA store
        stage_reclaim(lane);
#pragma unroll
        for (int q = 0; q < 8; ++q) *reinterpret_cast<uint4*>(st + stage128(lane, q)) = split_bf16x8(v + 8 * q);
        stage_publish(&P->o0, st, lane, col0, row0);
        uint4 w[8];
#pragma unroll
        for (int q = 0; q < 8; ++q) w[q] = pack_bf16x8(v + 8 * q);
        stage_reclaim(lane);
#pragma unroll
        for (int q = 0; q < 8; ++q) *reinterpret_cast<uint4*>(st + stage128(lane, q)) = w[q];
        stage_publish(&P->o1, st, lane, col0, row0);
      } else {
        // narrow tiles: hi and lo halves of a row side by side in the staging block, 64-byte segments
        bf16* h = static_cast<bf16*>(e.out0);
#pragma unroll
        for (int q = 0; q < 4; ++q) {
          *reinterpret_cast<uint4*>(st + stage128(lane, q)) = split_bf16x8(v + 8 * q);
          *reinterpret_cast<uint4*>(st + stage128(lane, 4 + q)) = pack_bf16x8(v + 8 * q);
        }
        __syncwarp();
        const int ch = lane & 7, c = 8 * (ch & 3);
        bf16* base = h + (ch < 4 ? 0 : e.c0) + col0 + c;
#pragma unroll
        for (int j = 0; j < 8; ++j) {
          const int r = 4 * j + (lane >> 3);
          const uint4 x = *reinterpret_cast<const uint4*>(st + stage128(r, ch));
          if (row0 + r < M && col0 + c < N) *reinterpret_cast<uint4*>(base + (size_t)(row0 + r) * e.ld0) = x;
        }
        __syncwarp();
      }
      break;
    }
    case kEpiBwdDX: {
      // the masks of the segments this lane will store, in flight during the TMEM read
      constexpr int kCh = NC / 8;
      const int mc = col0 + 8 * (lane % kCh);
      uint4 m[kCh];
#pragma unroll
      for (int j = 0; j < kCh; ++j) {
        const int r = row0 + (32 / kCh) * j + lane / kCh;
        m[j] = (r < M && mc < N) ? *reinterpret_cast<const uint4*>(e.mask + (size_t)r * e.ldm + mc)
                                 : make_uint4(0u, 0u, 0u, 0u);
      }
      float v[NC];
      tmem_ldn(taddr, v);
      bf16* dz = static_cast<bf16*>(e.out0);
      emit_bf16<NC>(st, lane, v, [&](int j, int r, int c, uint4 x) {
        if (row0 + r < M && col0 + c < N)
          *reinterpret_cast<uint4*>(dz + (size_t)(row0 + r) * e.ld0 + col0 + c) =
              make_uint4(mask_pair(x.x, m[j].x), mask_pair(x.y, m[j].y), mask_pair(x.z, m[j].z),
                         mask_pair(x.w, m[j].w));
      });
      break;
    }
    default: {
      // FP32 outputs, 32 columns at a time
#pragma unroll 1
      for (int c = 0; c < NC && col0 + c < N; c += 32)
        epilogue_f32x32(P, e, st, tma, row0, lane, taddr + c, col0 + c, M, N);
      break;
    }
  }
}

// The output layer feeding the fused energy (kEpiFwdOutEnergy): two passes over
// this thread's row in TMEM (the tile holds all N columns, a multiple of 64):
// the squared norm of the whole row (both half warps of a row block form it, in
// column order), then the FP32 output and the scaled BF16 operand of this warp's
// 32-column chunks.
__device__ __forceinline__ void epilogue_energy(const EpiDesc& e, uint8_t* st, int row0, int lane, int half,
                                                uint32_t lane_base, int N, int M) {
  using bf16 = __nv_bfloat16;
  const bool cosine = e.energy == CRL_ENERGY_COS;
  float q = 0.f;
#pragma unroll 1
  for (int c = 0; c < N; c += 32) {
    float v[32], b[32];
    tmem_ldn(lane_base + c, v);
    load_bias32(e.bias + c, b);
#pragma unroll
    for (int i = 0; i < 32; ++i) {
      v[i] += b[i];
      const float r = cosine ? v[i] : __bfloat162float(__float2bfloat16_rn(v[i]));
      q += r * r;
    }
  }
  const float scale = cosine ? rsqrtf(q) : 1.f;
  if (half == 0 && row0 + lane < M) e.aux[row0 + lane] = cosine ? scale : q;
  float* y = static_cast<float*>(e.out0);
  bf16* X = static_cast<bf16*>(e.out1);
#pragma unroll 1
  for (int c = 32 * half; c < N; c += 64) {
    float v[32], b[32];
    tmem_ldn(lane_base + c, v);
    load_bias32(e.bias + c, b);
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] += b[i];
    emit_f32x4(st, lane, v, [&](int r, int k, float4 x) {
      if (row0 + r < M) *reinterpret_cast<float4*>(y + (size_t)(row0 + r) * e.ld0 + c + k) = x;
    });
#pragma unroll
    for (int i = 0; i < 32; ++i) v[i] *= scale;
    emit_bf16<32>(st, lane, v, [&](int, int r, int k, uint4 x) {
      if (row0 + r < M) *reinterpret_cast<uint4*>(X + (size_t)(row0 + r) * N + c + k) = x;
    });
  }
}

// The warp's share of a 128 x BN tile at (m0, n0), accumulator at `acc`: rows
// m0 + 32 eg .., every second step of NC columns.
template <int BN, int NC>
__device__ __forceinline__ void epilogue_tile(const GemmProblem* P, const EpiDesc& e, uint8_t* st, uint32_t acc, int eg,
                                              int half, int lane, int m0, int n0, int M, int N) {
  static_assert(BN % (2 * NC) == 0, "two half warps share the tile's steps");
  const int row0 = m0 + 32 * eg;
  if (row0 >= M) return;
  const uint32_t lane_base = acc + ((uint32_t)(32 * eg) << 16);
  const bool tma = NC == 64 && P->tma_out != 0;
  // The staging block may still belong to the copies of the warp's last tile (in the
  // kernels that walk a list: a policy's output that left as TMA stores, then an
  // encoder's, or a policy's whose rows TMA does not take).  The steps that store
  // through TMA wait for that before each write; nothing else does.
  if (NC == 64 && !tma) stage_reclaim(lane);
  if (e.kind == kEpiFwdOutEnergy) {
    epilogue_energy(e, st, row0, lane, half, lane_base, N, M);
    return;
  }
  const int ncol = (N - n0 < BN) ? N - n0 : BN;
#pragma unroll 1
  for (int c = NC * half; c < ncol; c += 2 * NC)
    epilogue_step<NC>(P, e, st, tma, row0, lane, lane_base + c, n0 + c, M, N);
}

// Before the accumulator is ready: the bias lines of the warp's columns into L1
// (a first touch costs an L2 round trip that would otherwise stand in every
// tile's epilogue), and the tensor-map proxy's view of the output maps.
template <int BN, int NC>
__device__ __forceinline__ void epilogue_ahead(const GemmProblem* P, int half, int lane, int n0) {
  if (P->epi.bias != nullptr && 4 * lane < BN / 2) {
    const int k = 4 * lane, c = n0 + NC * half + 2 * NC * (k / NC) + k % NC;   // the warp's k-th column
    if (c < P->N) {
      float x;
      asm volatile("ld.global.f32 %0, [%1];" : "=f"(x) : "l"(P->epi.bias + c));
    }
  }
  if (NC == 64 && lane == 0 && P->tma_out) {
    tmap_acquire(&P->o0);
    if (P->epi.kind == kEpiFwdHidden) tmap_acquire(&P->o1);
  }
}
// After the warp's last tile: its stores have read the staging block.
__device__ __forceinline__ void epilogue_end(int lane) {
  if (lane == 0) asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

// nkA > 0: A has only nkA K-slices and slice kb of B multiplies slice kb % nkA of
// A -- B holds the weight pair along K ([W_hi | W_lo], or [W_hi | W_hi | W_lo]
// against A = [h_hi | h_lo]) and each A tile is used against several parts.
template <int BN, int STAGES>
__global__ void __launch_bounds__(kTileThreads, (GemmSmem<BN, STAGES>::kBytes <= 113 * 1024) ? 2 : 1)
    tc_gemm_kernel(const GemmProblem* __restrict__ probs, int nprob, unsigned* status) {
  using S = GemmSmem<BN, STAGES>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  uint8_t* sA = smem;
  uint8_t* sB = smem + S::kStages * S::kABytes;
  uint64_t* full = reinterpret_cast<uint64_t*>(smem + S::kStages * S::kStageBytes);
  uint64_t* empty = full + S::kStages;
  uint64_t* done = empty + S::kStages;
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(done + 1);

  // problem of this CTA: the last p with tile_begin <= blockIdx.x (the table is immutable)
  int lo = 0, hi = nprob - 1;
  const int t = blockIdx.x;
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (probs[mid].tile_begin <= t) lo = mid;
    else hi = mid - 1;
  }
  const GemmProblem* P = probs + lo;
  // split-K: ksplit consecutive CTAs share one output tile, each a K range
  const int ksplit = P->ksplit > 1 ? P->ksplit : 1;
  const int lt = (t - P->tile_begin) / ksplit, split = (t - P->tile_begin) % ksplit;
  const int M = P->M, N = P->N, K = P->K, nkA = P->nkA;
  const int m0 = (lt / P->tiles_n) * kBM, n0 = (lt % P->tiles_n) * BN;
  const CUtensorMap* tmA = &P->a;
  const CUtensorMap* tmB = &P->b;
  const EpiDesc e = P->epi;   // (immutable: read ahead of the predecessor's end, not at the epilogue's start)

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  const int nk_all = (K + kBK - 1) / kBK;
  const int kb0 = split * nk_all / ksplit, nk = (split + 1) * nk_all / ksplit - kb0;

  if (threadIdx.x == 0) {
    tmap_acquire(tmA);
    tmap_acquire(tmB);
    prefetch_tmap(tmA);
    prefetch_tmap(tmB);
    prefetch_b<BN>(P, n0);
    for (int s = 0; s < S::kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    mbar_init(done, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(tmem_slot, S::kTmemCols);
    tmem_relinquish();
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  // operands come from the predecessor; the epilogue may overwrite what it read
  pdl_wait();
  pdl_trigger();
  const unsigned long long lim = wait_limit(status);

  if (warp == 0 && lane == 0) {
    // TMA producer
    const SliceSrc src = slice_src(P);
    int issued = 0;
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % S::kStages;
      if (kb >= S::kStages && !mbar_wait(&empty[s], ((kb / S::kStages) & 1) ^ 1, lim)) {
        atomicOr(status, CRL_STATUS_TIMEOUT);
        break;
      }
      ++issued;
      mbar_arrive_expect_tx(&full[s], S::kStageBytes);
      // operands arrive as 64-row boxes (8 KiB each); stacked along rows they
      // form the same 128-byte-swizzled K-major tile as one tall box
      load_slice<BN / 64>(src, sA + s * S::kABytes, sB + s * S::kBBytes, &full[s], kb0 + kb, m0, n0);
    }
    // nothing may land in this CTA's shared memory after it exits
    drain_ring(full, S::kStages, issued);
  } else if (warp == 1 && lane == 0) {
    // MMA issuer
    const uint32_t idesc = idesc_major(idesc_bf16_f32(kBM, BN), P);
    const bool amn = P->a_mn != 0, bmn = P->b_mn != 0;
    const uint32_t sa = slice_step(amn), sb = slice_step(bmn);
    for (int kb = 0; kb < nk; ++kb) {
      const int s = kb % S::kStages;
      if (!mbar_wait(&full[s], (kb / S::kStages) & 1, lim)) {
        atomicOr(status, CRL_STATUS_TIMEOUT);
        break;
      }
      fence_after_sync();
      const uint64_t da = slice_desc(sA + s * S::kABytes, amn), db = slice_desc(sB + s * S::kBBytes, bmn);
#pragma unroll
      for (int k = 0; k < kBK / 16; ++k)
        mma_bf16(tmem, da + sa * k, db + sb * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
      mma_commit(&empty[s]);
    }
    // always: `done` completes once every MMA issued here has (after a timeout
    // the accumulator is incomplete, and the status word says so)
    mma_commit(done);
  }
  __syncwarp();

  // epilogue (tcgen05.ld is warp-collective: keep the decision warp-uniform).
  // Every MMA has completed, so the operand ring is free: it becomes the warps'
  // staging blocks.
  const int eg = warp & 3, half = warp >> 2;
  constexpr int NC = kStepCols<BN>;
  epilogue_ahead<BN, NC>(P, half, lane, n0);
  const bool ok = __all_sync(0xffffffffu, mbar_wait(done, 0, lim) ? 1 : 0) != 0;
  fence_after_sync();
  uint8_t* stage = smem + warp * kStageWarpBytes;
  if (ok && ksplit > 1) {
    // split-K: store this split's FP32 partial tile; the last CTA of the tile to
    // arrive adds the ksplit partials in split order (its own included) and runs
    // the epilogue, so the result does not depend on which CTA is last.  A
    // partial is [BN / 4][128 rows] 16-byte pieces: a warp's accesses are
    // contiguous (row-major partials cost 32 lines per instruction both ways).
    __shared__ int s_last;
    const int r = eg * 32 + lane;
    const uint32_t lane_base = tmem + ((uint32_t)(eg * 32) << 16);
    const int ncol = (N - n0 < BN) ? N - n0 : BN;
    float4* part = reinterpret_cast<float4*>(P->part + (size_t)lt * ksplit * kBM * BN) + r;
    constexpr size_t kPart = (size_t)kBM * BN / 4;   // 16-byte pieces per partial tile
#pragma unroll 1
    for (int c = 32 * half; c < ncol; c += 64) {
      float v[32];
      tmem_ldn(lane_base + c, v);
#pragma unroll
      for (int i = 0; i < 8; ++i)
        __stcg(part + split * kPart + (size_t)(c / 4 + i) * kBM,
               make_float4(v[4 * i], v[4 * i + 1], v[4 * i + 2], v[4 * i + 3]));
    }
    __threadfence();
    __syncthreads();
    if (threadIdx.x == 0) s_last = (atomicAdd(P->tickets + lt, 1u) == (unsigned)ksplit - 1u) ? 1 : 0;
    __syncthreads();
    if (s_last) {
      __threadfence();
#pragma unroll 1
      for (int c = 32 * half; c < ncol; c += 64) {
        float v[32];
#pragma unroll
        for (int i = 0; i < 32; ++i) v[i] = 0.f;
#pragma unroll 2
        for (int q = 0; q < ksplit; ++q) {
#pragma unroll
          for (int i = 0; i < 8; ++i) {
            const float4 x = __ldcg(part + q * kPart + (size_t)(c / 4 + i) * kBM);
            v[4 * i] += x.x;
            v[4 * i + 1] += x.y;
            v[4 * i + 2] += x.z;
            v[4 * i + 3] += x.w;
          }
        }
        if (m0 + 32 * eg < M) epilogue_grad32(e, stage, m0 + 32 * eg, lane, v, n0 + c, M, N);
      }
      if (threadIdx.x == 0) P->tickets[lt] = 0u;
    }
  } else if (ok) {
    epilogue_tile<BN, NC>(P, e, stage, tmem, eg, half, lane, m0, n0, M, N);
    if (NC == 64) epilogue_end(lane);
  } else if (threadIdx.x == 0) {
    atomicOr(status, CRL_STATUS_TIMEOUT);
  }
  // the accumulator is freed only after every MMA writing it has completed
  if (!ok && threadIdx.x == 0) mbar_wait(done, 0, kDrainLimitNs);
  fence_before_sync();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, S::kTmemCols);
}

// The problem of tile t: the last p with tile_begin <= t (the table is immutable).
__device__ __forceinline__ const GemmProblem* find_problem(const GemmProblem* __restrict__ probs, int nprob, int t) {
  int lo = 0, hi = nprob - 1;
  while (lo < hi) {
    const int mid = (lo + hi + 1) / 2;
    if (probs[mid].tile_begin <= t) lo = mid;
    else hi = mid - 1;
  }
  return probs + lo;
}

// Persistent variant: gridDim.x CTAs (one per SM at most) walk the tiles
// t = blockIdx.x, blockIdx.x + gridDim.x, ... of the whole problem list.
// 320 threads:
//   warp 0 / lane 0 -- TMA producer over all of the CTA's tiles: the operand
//                      ring runs on across tile boundaries;
//   warp 1 / lane 0 -- MMA issuer: tile i accumulates into TMEM buffer i % 2
//                      (2 x BN columns), once the epilogue has released it;
//   warps 2..9      -- epilogue of tile i from buffer i % 2 while the MMAs of
//                      tile i + 1 fill the other one (warp w reads TMEM lanes
//                      32 (w % 4) .., every second column step).
// The epilogue is the same as the one-tile kernel's, so both give identical
// outputs.
template <int BN, int STAGES>
__global__ void __launch_bounds__(kPersistentThreads, 1)
    tc_gemm_persistent_kernel(const GemmProblem* __restrict__ probs, int nprob, int total, unsigned* status) {
  using S = GemmSmem<BN, STAGES>;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  uint8_t* sA = smem;
  uint8_t* sB = smem + S::kStages * S::kABytes;
  uint8_t* sE = smem + S::kStages * S::kStageBytes;   // epilogue staging, 4 KiB per warp
  uint64_t* full = reinterpret_cast<uint64_t*>(sE + kStageBytesAll);
  uint64_t* empty = full + S::kStages;
  uint64_t* accf = empty + S::kStages;  // [2] accumulator buffer ready (MMA -> epilogue)
  uint64_t* acce = accf + 2;            // [2] accumulator buffer free (epilogue -> MMA), 8 arrivals
  uint64_t* drain = acce + 2;           // every MMA of this CTA has completed (teardown)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);

  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (threadIdx.x == 0) {
    if ((int)blockIdx.x < total) {   // the first tile's B operand
      const GemmProblem* P = find_problem(probs, nprob, blockIdx.x);
      tmap_acquire(&P->b);
      prefetch_b<BN>(P, (((int)blockIdx.x - P->tile_begin) % P->tiles_n) * BN);
    }
    for (int s = 0; s < S::kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], kEpiWarps);
    }
    mbar_init(drain, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc(tmem_slot, 2 * BN);
    tmem_relinquish();
  }
  fence_before_sync();
  __syncthreads();
  fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();
  pdl_trigger();
  const unsigned long long lim = wait_limit(status);

  if (warp == 0) {
    if (lane == 0) {
      // TMA producer; `it` counts K-slices over all tiles of this CTA
      int it = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < total && ok; t += gridDim.x) {
        const GemmProblem* P = find_problem(probs, nprob, t);
        const int lt = t - P->tile_begin;
        const int m0 = (lt / P->tiles_n) * kBM, n0 = (lt % P->tiles_n) * BN;
        const int nk = (P->K + kBK - 1) / kBK;
        tmap_acquire(&P->a);
        tmap_acquire(&P->b);
        const SliceSrc src = slice_src(P);
        for (int kb = 0; kb < nk; ++kb, ++it) {
          const int s = it % S::kStages;
          if (it >= S::kStages && !mbar_wait(&empty[s], ((it / S::kStages) & 1) ^ 1, lim)) {
            atomicOr(status, CRL_STATUS_TIMEOUT);
            ok = false;
            break;
          }
          mbar_arrive_expect_tx(&full[s], S::kStageBytes);
          load_slice<BN / 64>(src, sA + s * S::kABytes, sB + s * S::kBBytes, &full[s], kb, m0, n0);
        }
      }
      // `it` slices were issued (a timed-out one was not): let them all land
      drain_ring(full, S::kStages, it);
    }
  } else if (warp == 1) {
    if (lane == 0) {
      // MMA issuer
      int it = 0, i = 0;
      bool ok = true;
      for (int t = blockIdx.x; t < total && ok; t += gridDim.x, ++i) {
        const GemmProblem* P = find_problem(probs, nprob, t);
        const int nk = (P->K + kBK - 1) / kBK;
        const uint32_t idesc = idesc_major(idesc_bf16_f32(kBM, BN), P);
        const bool amn = P->a_mn != 0, bmn = P->b_mn != 0;
        const uint32_t sa = slice_step(amn), sb = slice_step(bmn);
        const int buf = i & 1, use = i >> 1;
        // the epilogue of tile i - 2 must have read this buffer out
        if (use > 0 && !mbar_wait(&acce[buf], (use - 1) & 1, lim)) {
          atomicOr(status, CRL_STATUS_TIMEOUT);
          break;
        }
        fence_after_sync();
        const uint32_t d = tmem + (uint32_t)(buf * BN);
        for (int kb = 0; kb < nk; ++kb, ++it) {
          const int s = it % S::kStages;
          if (!mbar_wait(&full[s], (it / S::kStages) & 1, lim)) {
            atomicOr(status, CRL_STATUS_TIMEOUT);
            ok = false;
            break;
          }
          fence_after_sync();
          const uint64_t da = slice_desc(sA + s * S::kABytes, amn), db = slice_desc(sB + s * S::kBBytes, bmn);
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k) mma_bf16(d, da + sa * k, db + sb * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
          mma_commit(&empty[s]);
        }
        if (ok) mma_commit(&accf[buf]);
      }
      mma_commit(drain);   // completes once every MMA issued above has
    }
  } else {
    // epilogue warps (tcgen05.ld is warp-collective: decisions stay warp-uniform)
    constexpr int NC = kStepCols<BN>;
    const int eg = warp & 3, ew = warp - 2, half = ew >> 2;
    int i = 0;
    for (int t = blockIdx.x; t < total; t += gridDim.x, ++i) {
      const int buf = i & 1, use = i >> 1;
      // everything the epilogue reads of its problem, before the accumulator is ready
      const GemmProblem* P = find_problem(probs, nprob, t);
      const int lt = t - P->tile_begin;
      const int m0 = (lt / P->tiles_n) * kBM, n0 = (lt % P->tiles_n) * BN;
      const int M = P->M, N = P->N;
      const EpiDesc& e = P->epi;   // fields read where used (L1): the steps need the registers
      epilogue_ahead<BN, NC>(P, half, lane, n0);
      const bool ok = __all_sync(0xffffffffu, mbar_wait(&accf[buf], use & 1, lim) ? 1 : 0) != 0;
      if (!ok) {
        if (lane == 0) atomicOr(status, CRL_STATUS_TIMEOUT);
        break;
      }
      fence_after_sync();
      epilogue_tile<BN, NC>(P, e, sE + ew * kStageWarpBytes, tmem + (uint32_t)(buf * BN), eg, half, lane, m0, n0, M, N);
      // release the buffer to the MMA issuer
      fence_before_sync();
      __syncwarp();
      if (lane == 0) mbar_arrive(&acce[buf]);
    }
    if (NC == 64) epilogue_end(lane);
  }
  // no MMA may still write the accumulators when they are freed
  if (threadIdx.x == 0) mbar_wait(drain, 0, kDrainLimitNs);
  fence_before_sync();
  __syncthreads();
  if (warp == 0) tmem_dealloc(tmem, 2 * BN);
}

// CTA-pair variant: a cluster of two CTAs (on one TPC) computes 256 x BN
// tiles with tcgen05.mma.cta_group::2, walking the tiles t = cluster,
// cluster + clusters, ... like the persistent kernel.  Each CTA loads its own
// operands into its own ring: 128 rows of A (the pair's rows 128 r ..) and
// BN / 2 rows of B (columns BN / 2 r .. of the tile), so a pair moves half the
// operand bytes of two one-SM tiles of the same work.  The even CTA issues
// every MMA; its accumulator rows live in the even CTA's TMEM, the others in
// the odd CTA's.  No operand load is multicast; the CTAs exchange mbarrier
// arrivals, the MMA commits among them on both CTAs' barriers at once.
//   warp 0 / lane 0 -- TMA producer of this CTA's ring;
//   warp 1 / lane 0 -- even CTA: MMA issuer.  It waits for its own slot and the
//                      odd CTA's `pfull` arrival; its commits free each slot
//                      (`empty`) and announce each finished accumulator (`accf`)
//                      in both CTAs (a relay warp cost about 0.5 us per slot:
//                      more than one slot's MMA time).  Odd CTA: reports each
//                      landed slot to the even CTA's `pfull`;
//   warps 2..9      -- epilogue of this CTA's 128 rows from TMEM buffer i % 2;
//                      the pair's sixteen warps release it on the even CTA's `acce`.
// The epilogue is the one-tile kernel's, so every kernel gives identical outputs
// where the MMA sums each K = 16 slice the same way.
template <int BN, int STAGES>
struct GemmPairSmem {
  static constexpr uint32_t kABytes = kBM * kBK * 2;         // 16 KiB: this CTA's 128 rows of A
  static constexpr uint32_t kBBytes = (BN / 2) * kBK * 2;    // this CTA's BN / 2 rows of B
  static constexpr uint32_t kStageBytes = kABytes + kBBytes;
  static constexpr int kStages = STAGES;
  // ring, the epilogue's staging blocks, barriers (full, empty, pfull [S]; accf, acce [2]; drain) +
  // TMEM slot, plus 1 KiB for alignment (the last slot's B rows plus BN / 2 rows stay inside this
  // CTA's shared memory)
  static constexpr uint32_t kBytes = kStages * kStageBytes + 8 * 4096 + 1024 + 512;
  static_assert(kBBytes <= 8 * 4096, "the staging blocks cover one more B half behind the ring");
  static constexpr uint32_t kTmemCols = 2 * BN;   // two accumulator buffers
  static_assert(BN == 128 || BN == 256, "pair tiles are 256 x 128 or 256 x 256");
  static_assert(kTmemCols <= 512, "TMEM columns");
  static_assert(kBytes <= 227 * 1024, "shared memory per CTA");
};

template <int BN, int STAGES>
__global__ void __cluster_dims__(2, 1, 1) __launch_bounds__(kPairThreads, 1)
    tc_gemm_pair_kernel(const GemmProblem* __restrict__ probs, int nprob, int total, unsigned* status) {
  using S = GemmPairSmem<BN, STAGES>;
  constexpr int kPairM = 2 * kBM;
  extern __shared__ uint8_t smem_raw[];
  uint8_t* smem = align1024(smem_raw);
  uint8_t* sA = smem;
  uint8_t* sB = smem + S::kStages * S::kABytes;
  uint8_t* sE = smem + S::kStages * S::kStageBytes;   // epilogue staging, 4 KiB per warp
  uint64_t* full = reinterpret_cast<uint64_t*>(sE + kStageBytesAll);
  uint64_t* empty = full + S::kStages;
  uint64_t* pfull = empty + S::kStages;  // even CTA: the odd CTA's slot has landed
  uint64_t* accf = pfull + S::kStages;   // [2] accumulator buffer ready
  uint64_t* acce = accf + 2;             // [2] even CTA: buffer read out by all 16 epilogue warps
  uint64_t* drain = acce + 2;            // every MMA of the pair has completed (teardown)
  uint32_t* tmem_slot = reinterpret_cast<uint32_t*>(drain + 1);

  const uint32_t rank = cluster_ctarank();
  const bool even = rank == 0;
  const int cl = blockIdx.x / 2, ncl = gridDim.x / 2;
  const int warp = threadIdx.x / 32, lane = threadIdx.x % 32;
  if (threadIdx.x == 0) {
    if (cl < total) {   // the first tile's B rows of this CTA
      const GemmProblem* P = find_problem(probs, nprob, cl);
      tmap_acquire(&P->b);
      prefetch_b<BN / 2>(P, ((cl - P->tile_begin) % P->tiles_n) * BN + (BN / 2) * rank);
    }
    for (int s = 0; s < S::kStages; ++s) {
      mbar_init(&full[s], 1);
      mbar_init(&empty[s], 1);
      mbar_init(&pfull[s], 1);
    }
    for (int b = 0; b < 2; ++b) {
      mbar_init(&accf[b], 1);
      mbar_init(&acce[b], 2 * kEpiWarps);
    }
    mbar_init(drain, 1);
    fence_mbar_init();
  }
  if (warp == 0) {
    tmem_alloc_pair(tmem_slot, S::kTmemCols);
    tmem_relinquish_pair();
  }
  fence_before_sync();
  cluster_sync();   // both CTAs' barriers are initialised before any remote arrival
  fence_after_sync();
  const uint32_t tmem = *tmem_slot;
  pdl_wait();
  pdl_trigger();
  const unsigned long long lim = wait_limit(status);

  if (warp == 0) {
    if (lane == 0) {
      // TMA producer; `it` counts K-slices over all tiles of this pair
      int it = 0;
      bool ok = true;
      for (int t = cl; t < total && ok; t += ncl) {
        const GemmProblem* P = find_problem(probs, nprob, t);
        const int lt = t - P->tile_begin;
        const int m0 = (lt / P->tiles_n) * kPairM + kBM * (int)rank;
        const int n0 = (lt % P->tiles_n) * BN + (BN / 2) * (int)rank;
        const int nk = (P->K + kBK - 1) / kBK;
        tmap_acquire(&P->a);
        tmap_acquire(&P->b);
        const SliceSrc src = slice_src(P);
        for (int kb = 0; kb < nk; ++kb, ++it) {
          const int s = it % S::kStages;
          if (it >= S::kStages) {
            const bool got = even ? mbar_wait(&empty[s], ((it / S::kStages) & 1) ^ 1, lim)
                                  : mbar_wait_cluster(&empty[s], ((it / S::kStages) & 1) ^ 1, lim);
            if (!got) {
              atomicOr(status, CRL_STATUS_TIMEOUT);
              ok = false;
              break;
            }
          }
          mbar_arrive_expect_tx(&full[s], S::kStageBytes);
          load_slice<BN / 128>(src, sA + s * S::kABytes, sB + s * S::kBBytes, &full[s], kb, m0, n0);
        }
      }
      drain_ring(full, S::kStages, it);
    }
  } else if (warp == 1) {
    if (lane == 0 && even) {
      // MMA issuer of the pair
      int it = 0, i = 0;
      bool ok = true;
      for (int t = cl; t < total && ok; t += ncl, ++i) {
        const GemmProblem* P = find_problem(probs, nprob, t);
        const int nk = (P->K + kBK - 1) / kBK;
        const uint32_t idesc = idesc_major(idesc_bf16_f32(kPairM, BN), P);
        const bool amn = P->a_mn != 0, bmn = P->b_mn != 0;
        const uint32_t sa = slice_step(amn), sb = slice_step(bmn);
        const int buf = i & 1, use = i >> 1;
        // all sixteen epilogue warps must have read out this buffer (tile i - 2)
        if (use > 0 && !mbar_wait_cluster(&acce[buf], (use - 1) & 1, lim)) {
          atomicOr(status, CRL_STATUS_TIMEOUT);
          break;
        }
        fence_after_sync();
        const uint32_t d = tmem + (uint32_t)(buf * BN);
        for (int kb = 0; kb < nk; ++kb, ++it) {
          const int s = it % S::kStages;
          const uint32_t par = (it / S::kStages) & 1;
          if (!mbar_wait(&full[s], par, lim) || !mbar_wait_cluster(&pfull[s], par, lim)) {
            atomicOr(status, CRL_STATUS_TIMEOUT);
            ok = false;
            break;
          }
          fence_after_sync();
          const uint64_t da = slice_desc(sA + s * S::kABytes, amn), db = slice_desc(sB + s * S::kBBytes, bmn);
#pragma unroll
          for (int k = 0; k < kBK / 16; ++k)
            mma_bf16_pair(d, da + sa * k, db + sb * k, idesc, (kb > 0 || k > 0) ? 1u : 0u);
          mma_commit_both(&empty[s]);
        }
        if (ok) mma_commit_both(&accf[buf]);
      }
      mma_commit_pair(drain);   // completes once every MMA issued above has
    } else if (lane == 0) {
      // odd CTA: report each landed slot to the MMA issuer
      int it = 0;
      bool ok = true;
      for (int t = cl; t < total && ok; t += ncl) {
        const GemmProblem* P = find_problem(probs, nprob, t);
        const int nk = (P->K + kBK - 1) / kBK;
        for (int kb = 0; kb < nk; ++kb, ++it) {
          const int s = it % S::kStages;
          if (!mbar_wait(&full[s], (it / S::kStages) & 1, lim)) {
            atomicOr(status, CRL_STATUS_TIMEOUT);
            ok = false;
            break;
          }
          mbar_arrive_remote(mapa_shared(&pfull[s], 0));
        }
      }
    }
  } else {
    // epilogue warps: this CTA's 128 rows of the pair's tile
    constexpr int NC = kStepCols<BN>;
    const int eg = warp & 3, ew = warp - 2, half = ew >> 2;
    int i = 0;
    for (int t = cl; t < total; t += ncl, ++i) {
      const int buf = i & 1, use = i >> 1;
      // everything the epilogue reads of its problem, before the accumulator is ready
      const GemmProblem* P = find_problem(probs, nprob, t);
      const int lt = t - P->tile_begin;
      const int m0 = (lt / P->tiles_n) * kPairM + kBM * (int)rank, n0 = (lt % P->tiles_n) * BN;
      const int M = P->M, N = P->N;
      const EpiDesc& e = P->epi;   // fields read where used (L1): the steps need the registers
      epilogue_ahead<BN, NC>(P, half, lane, n0);
      const bool got = even ? mbar_wait(&accf[buf], use & 1, lim) : mbar_wait_cluster(&accf[buf], use & 1, lim);
      const bool ok = __all_sync(0xffffffffu, got ? 1 : 0) != 0;
      if (!ok) {
        if (lane == 0) atomicOr(status, CRL_STATUS_TIMEOUT);
        break;
      }
      fence_after_sync();
      epilogue_tile<BN, NC>(P, e, sE + ew * kStageWarpBytes, tmem + (uint32_t)(buf * BN), eg, half, lane, m0, n0, M, N);
      // release the buffer to the MMA issuer
      fence_before_sync();
      __syncwarp();
      if (lane == 0) {
        if (even) mbar_arrive(&acce[buf]);
        else mbar_arrive_remote(mapa_shared(&acce[buf], 0));
      }
    }
    if (NC == 64) epilogue_end(lane);
  }
  // teardown: no MMA may still write either CTA's accumulators when they are
  // freed, and no remote arrival may reach a CTA that has left
  fence_before_sync();
  __syncthreads();
  if (threadIdx.x == 0) {
    if (even) {
      mbar_wait(drain, 0, kDrainLimitNs);
      mbar_arrive_remote(mapa_shared(drain, 1));
    } else {
      mbar_wait_cluster(drain, 0, kDrainLimitNs);
    }
  }
  fence_before_sync();
  cluster_sync();
  fence_after_sync();
  if (warp == 0) tmem_dealloc_pair(tmem, S::kTmemCols);
}

}  // namespace tc
}  // namespace crl
