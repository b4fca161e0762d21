// Collection side of Algorithm 1 (the loop over environments) with synthetic
// dynamics standing in for the simulator, which is outside this library: it
// lets the update-to-data loop run end to end on the device (§5.6 studies the
// ratio of gradient updates to environment steps; App. B.3 fixes 1024
// environments and 1000-step episodes for Ant).
//
// Per environment step, for all E environments at once:
//   1. (mu, l) = pi(concat(s, g)), a = tanh(mu + e^clip(l) eps)   (the actor's
//      policy head; eps from Philox stream word 2 at the collection step);
//   2. the slice (s, a, done) goes into the replay buffer, done = the episode's
//      last step (t = episode_length - 1);
//   3. s' = s + 0.1 xi + 0.05 a[d mod A] with xi ~ N(0, I) (stream word 3), or,
//      after the last step of an episode, a fresh state s' ~ N(0, I) (word 4)
//      and a fresh commanded goal g' ~ N(0, I) (word 5).
// The first call draws every environment's first state and goal as a reset at
// the counter value 2^64 - 1.  All draws are Box-Muller on Philox4x64-10 blocks
// (step, env, word, d / 4) keyed (seed, agent), the same construction as the
// actor's noise.
#include <cuda_bf16.h>

#include <algorithm>
#include <cmath>

#include "actor_head.cuh"
#include "common.cuh"
#include "ctx.h"
#include "gemm_simt.cuh"
#include "internal.h"
#include "philox.cuh"
#include "tc_common.cuh"
#include "trace.h"

namespace crl {

namespace {

constexpr unsigned long long kInitStep = ~0ull;

// First states and goals of every environment.  One warp per environment.
__global__ void __launch_bounds__(256) env_init_kernel(int E, int D, int G, float* __restrict__ s,
                                                      float* __restrict__ g, int32_t* __restrict__ t,
                                                      unsigned long long seed, unsigned long long agent) {
  pdl_enter();
  const int lane = threadIdx.x % kWarp;
  const int e = blockIdx.x * (blockDim.x / kWarp) + threadIdx.x / kWarp;
  if (e >= E) return;
  for (int d = lane; d < D; d += kWarp) s[(size_t)e * D + d] = philox_normal<float>(kInitStep, e, 4ull, d, seed, agent);
  for (int d = lane; d < G; d += kWarp) g[(size_t)e * G + d] = philox_normal<float>(kInitStep, e, 5ull, d, seed, agent);
  if (lane == 0) t[e] = 0;
}

// One environment step after the policy's forward, one warp per environment: the
// action from the policy's output (step 1), the slice written straight into the
// replay buffer with the episode it closes stamped (step 2: what a one-slice
// insert does), and the dynamics (step 3).  As four launches (head, step, counter,
// insert) with a staged slice between them these took 10 us of a 43 us step and
// most of the host's time; nothing but this warp reads the environment's values
// in between.
template <typename T>
struct CollectArgs {
  BufferDev bd;
  long long total_before;   // steps inserted before this one
  int G, episode_length;
  float* s;                 // [E][D]
  float* g;                 // [E][G]
  int32_t* t;               // [E]
  const T* pi_out;          // [E][2 A]
  T* a;                     // [E][A]
  const unsigned long long* step_dev;
  unsigned long long i;     // steps of this call before this one (the counter advances once per call)
  float* obs_out;           // this step's [E][D], [E][A], [E] or null
  float* act_out;
  uint8_t* done_out;
  unsigned long long seed, agent;
};

template <typename T>
__global__ void __launch_bounds__(256) collect_step_kernel(const __grid_constant__ CollectArgs<T> p) {
  pdl_enter();
  const BufferDev& bd = p.bd;
  const int D = bd.D, A = bd.A;
  const int lane = threadIdx.x % kWarp;
  const int e = blockIdx.x * (blockDim.x / kWarp) + threadIdx.x / kWarp;
  const long long total_after = p.total_before + 1;
  const long long size_after = total_after < bd.T ? total_after : bd.T;
  if (blockIdx.x == 0 && threadIdx.x == 0) {
    bd.state[0] = (int32_t)size_after;
    bd.state[1] = (int32_t)total_after;
  }
  if (e >= bd.E) return;
  const unsigned long long k = *p.step_dev + p.i;
  const int te = p.t[e];
  const bool last = te >= p.episode_length - 1;
  float* dst = bd.rows + ((size_t)e * bd.T + (size_t)(p.total_before % bd.T)) * bd.W;
  T* ae = p.a + (size_t)e * A;
  for (int d = lane; d < A; d += kWarp) {
    const T mu = p.pi_out[(size_t)e * 2 * A + d];
    const T lraw = p.pi_out[(size_t)e * 2 * A + A + d];
    const T l = fmin(fmax(lraw, T(kLogStdMin)), T(kLogStdMax));
    const T n = philox_normal<T>(k, e, 2ull, d, p.seed, p.agent);
    const T u = mu + dev_exp(l) * n;
    const T act = dev_tanh(u);
    ae[d] = act;
    dst[D + d] = (float)act;
    if (p.act_out) p.act_out[(size_t)e * A + d] = (float)act;
  }
  __syncwarp();   // the dynamics read the warp's actions
  float* se = p.s + (size_t)e * D;
  for (int d = lane; d < D; d += kWarp) {
    const float x = se[d];
    dst[d] = x;
    if (p.obs_out) p.obs_out[(size_t)e * D + d] = x;
    float nx;
    if (last) {
      nx = philox_normal<float>(k, e, 4ull, d, p.seed, p.agent);
    } else {
      const float xi = philox_normal<float>(k, e, 3ull, d, p.seed, p.agent);
      nx = x + 0.1f * xi + 0.05f * (float)ae[d % A];
    }
    se[d] = nx;
  }
  for (int c = D + A + lane; c < bd.W; c += kWarp) dst[c] = c == D + A ? __int_as_float(-1) : 0.f;
  if (last) {
    for (int d = lane; d < p.G; d += kWarp)
      p.g[(size_t)e * p.G + d] = philox_normal<float>(k, e, 5ull, d, p.seed, p.agent);
    __syncwarp();   // this row's open mark precedes its stamp
    const long long win_lo = total_after - size_after, start = bd.ep_start[e];
    for (long long a = (start > win_lo ? start : win_lo) + lane; a <= p.total_before; a += kWarp)
      bd.rows[((size_t)e * bd.T + (size_t)(a % bd.T)) * bd.W + D + A] = __int_as_float((int)p.total_before);
    __syncwarp();   // every lane has read the episode's start
  }
  if (lane == 0) {
    if (p.done_out) p.done_out[e] = last ? 1 : 0;
    p.t[e] = last ? 0 : te + 1;
    if (last) bd.ep_start[e] = (int32_t)total_after;
  }
}

__global__ void advance_kernel(unsigned long long* c, unsigned long long n) {
  pdl_enter();
  *c += n;
}

// ---- the whole unroll in one launch ---------------------------------------------
// The policy does not change during a call and environments do not touch each
// other, so one cluster of C CTAs carries ME environments through all n steps
// without leaving shared memory.  Launched layer by layer, a step of 1024
// environments with two layers of 256 takes 25 us for 2.2 us of FMAs (launches,
// reloading the weights, and 64 to 128 threads' worth of work per SM in between);
// here it takes 9.2 us (62 steps: 1921 -> 569 us), of which 4.1 are the second
// layer's products, 1.2 the output layer's chains and 1.3 the barriers.
//
// Split: CTA `rank` keeps columns [rank nc, rank nc + nc) of every hidden layer
// ([k][nc], transposed once per launch) and the whole output layer.  Activations
// are [k][env] for all ME environments of the cluster in every CTA: a CTA writes
// its columns into every CTA's copy, and a cluster barrier separates the layers.
// Two buffers suffice: a layer writes the one that was last read before the
// barrier in front of it.  The output layer, the action, the slice and the
// dynamics are done by the CTA that owns the environment (ME / C of them), which
// sends the next state to its peers.
//
// Warps 0 to 3 multiply: 4 columns x 4 environments per thread, 8 x 4 threads per
// warp, so that a k step is two conflict-free 16-byte shared reads for 16 FMAs
// (8 two-lane instructions).  Warps 4 to 7 draw
// the step's noise meanwhile.  Every output is the chain of fused multiply-adds
// over k in order that the layer-by-layer products have, and LayerNorm and the
// step use the same expressions, so both paths give the same bits.
constexpr int kUnrollThreads = 256, kUnrollGemmWarps = 4;
constexpr int kUnrollSteps = 1024;   // steps per launch at most (about 10 ms)
constexpr int kUnrollSmem = 227 * 1024;

struct UnrollArgs {
  BufferDev bd;
  long long total_before;
  int n, G, episode_length;
  int layers, H, in, layernorm;
  int C, ME, nc, pitch;
  const float* params;
  int64_t W[CRL_MAX_LAYERS + 1], b[CRL_MAX_LAYERS + 1], g[CRL_MAX_LAYERS], beta[CRL_MAX_LAYERS];
  float *s, *gs;
  int32_t* t;
  const unsigned long long* step_dev;
  unsigned long long i0;   // steps of this call before this launch
  float* obs_out;          // [n][E][D], [n][E][A], [n][E] or null
  float* act_out;
  uint8_t* done_out;
  unsigned long long seed, agent;
};

// Shared-memory pieces in floats, in this order; every piece starts on 16 bytes.
struct UnrollSmem {
  int w, wo, wo_pitch, bias, bo, ln, buf, s, g, act, noise, out, t, fin, total;
};
__host__ __device__ inline UnrollSmem unroll_smem(int layers, int in, int H, int D, int A, int G, int layernorm, int C,
                                                  int ME, int nc, int pitch) {
  UnrollSmem u;
  int at = 0;
  auto take = [&](int n) {
    const int o = at;
    at += (n + 3) / 4 * 4;
    return o;
  };
  const int own = ME / C;
  u.w = take((in + (layers - 1) * H) * nc);   // layer after layer
  // output weights [column][k]: an odd multiple of 16 bytes apart
  u.wo_pitch = (H + 3) / 4 * 4;
  if (u.wo_pitch / 4 % 2 == 0) u.wo_pitch += 4;
  u.wo = take(u.wo_pitch * 2 * A);
  u.bias = take(layers * nc);
  u.bo = take(2 * A);
  u.ln = take(layernorm ? layers * 2 * H : 0);
  u.buf = take(2 * (in > H ? in : H) * pitch);
  u.s = take(own * D);
  u.g = take(own * G);
  u.act = take(own * A);
  u.noise = take(own * (A + D));
  u.out = take(own * 2 * A);
  u.t = take(own);
  u.fin = take(own);
  u.total = at;
  return u;
}

__device__ __forceinline__ void st_cluster4(uint32_t a, float4 v) {
  asm volatile("st.shared::cluster.v4.f32 [%0], {%1, %2, %3, %4};" ::"r"(a), "f"(v.x), "f"(v.y), "f"(v.z), "f"(v.w)
               : "memory");
}
__device__ __forceinline__ void st_cluster1(uint32_t a, float v) {
  asm volatile("st.shared::cluster.f32 [%0], %1;" ::"r"(a), "f"(v) : "memory");
}

__global__ void __launch_bounds__(kUnrollThreads, 1) unroll_kernel(const __grid_constant__ UnrollArgs p) {
  extern __shared__ __align__(16) float sm[];
  pdl_enter();
  const BufferDev& bd = p.bd;
  const int D = bd.D, A = bd.A, G = p.G, H = p.H, A2 = 2 * A;
  const int C = p.C, ME = p.ME, nc = p.nc, pitch = p.pitch, own = ME / C;
  const int tid = threadIdx.x, lane = tid % kWarp, wid = tid / kWarp;
  const int rank = (int)(blockIdx.x % C), e0 = (int)(blockIdx.x / C) * ME;
  const UnrollSmem u = unroll_smem(p.layers, p.in, H, D, A, G, p.layernorm, C, ME, nc, pitch);
  const int n0 = rank * nc, size = (p.in > H ? p.in : H) * pitch;   // size: floats of one buffer
  int32_t* st = reinterpret_cast<int32_t*>(sm + u.t);
  int32_t* fin = reinterpret_cast<int32_t*>(sm + u.fin);   // the step ended its episode

  // weights: 8 rows x 16 k per warp (64-byte pieces of a row; 4-way shared stores)
  for (int l = 0; l < p.layers; ++l) {
    const int K = l == 0 ? p.in : H, kb = (K + 15) / 16, nb = (nc + 7) / 8;
    const float* Wg = p.params + p.W[l];
    const bool vec = (K & 3) == 0;   // tensors start 256 bytes apart in a 16-byte aligned array
    for (int b = wid; b < kb * nb; b += kUnrollThreads / kWarp) {
      const int n = 8 * (b % nb) + lane % 8, k = 16 * (b / nb) + 4 * (lane / 8);
      if (n >= nc || k >= K) continue;
      float4 v = make_float4(0.f, 0.f, 0.f, 0.f);
      if (n0 + n < H) {
        const float* src = Wg + (size_t)(n0 + n) * K + k;
        if (vec) {
          v = *reinterpret_cast<const float4*>(src);
        } else {
          v.x = src[0];
          if (k + 1 < K) v.y = src[1];
          if (k + 2 < K) v.z = src[2];
          if (k + 3 < K) v.w = src[3];
        }
      }
      float* dst = sm + u.w + (l == 0 ? 0 : p.in + (l - 1) * H) * nc + k * nc + n;
      dst[0] = v.x;
      if (k + 1 < K) dst[nc] = v.y;
      if (k + 2 < K) dst[2 * nc] = v.z;
      if (k + 3 < K) dst[3 * nc] = v.w;
    }
    for (int n = tid; n < nc; n += kUnrollThreads) sm[u.bias + l * nc + n] = n0 + n < H ? p.params[p.b[l] + n0 + n] : 0.f;
    if (p.layernorm)
      for (int n = tid; n < H; n += kUnrollThreads) {
        sm[u.ln + 2 * l * H + n] = p.params[p.g[l] + n];
        sm[u.ln + (2 * l + 1) * H + n] = p.params[p.beta[l] + n];
      }
  }
  for (int q = tid; q < A2 * H; q += kUnrollThreads) {
    const int j = q / H, k = q % H;
    sm[u.wo + j * u.wo_pitch + k] = p.params[p.W[p.layers] + q];
  }
  for (int j = tid; j < A2; j += kUnrollThreads) sm[u.bo + j] = p.params[p.b[p.layers] + j];
  // the environments this CTA owns
  const int first = e0 + rank * own;
  for (int q = tid; q < own * D; q += kUnrollThreads)
    sm[u.s + q] = first + q / D < bd.E ? p.s[(size_t)first * D + q] : 0.f;
  for (int q = tid; q < own * G; q += kUnrollThreads)
    sm[u.g + q] = first + q / G < bd.E ? p.gs[(size_t)first * G + q] : 0.f;
  for (int q = tid; q < own; q += kUnrollThreads) st[q] = first + q < bd.E ? p.t[first + q] : 0;
  const unsigned long long step0 = *p.step_dev + p.i0;
  __syncthreads();
  tc::cluster_sync();   // every CTA of the cluster runs: its shared memory may be written
  // one environment's policy input (s, g) into buffer `buf` of every CTA of the cluster; one warp
  auto send_input = [&](int q, int buf) {
    float* here = sm + u.buf + buf * size + rank * own + q;
    for (int d = lane; d < D + G; d += kWarp) {
      const float v = d < D ? sm[u.s + q * D + d] : sm[u.g + q * G + (d - D)];
      here[d * pitch] = v;
      for (int r = 1; r < C; ++r) st_cluster1(tc::mapa_shared(here + d * pitch, (rank + r) & (C - 1)), v);
    }
  };
  for (int q = wid; q < own; q += kUnrollThreads / kWarp) send_input(q, 0);
  __syncwarp();
  tc::cluster_sync();

  const int lane_mod = lane % A, warp_mod = kWarp % A;
  const int oq = tid / A2, oj = tid % A2;   // this thread's first output
  int slot = (int)(p.total_before % bd.T);   // the ring's row of this step
  // this warp's first block of 8 x 4 thread tiles
  const int nct = nc / 4, net = ME / 4, nbx = (nct + 7) / 8, nby = (net + 3) / 4;
  const int bx0 = wid % nbx, by0 = wid / nbx;
  // step j's slice (buffer row `row`) into the replay buffer; warps 4 to 7, during
  // the next step's first product
  auto write_slice = [&](int j, int row) {
    const long long total_before = p.total_before + j, total_after = total_before + 1;
    for (int q = wid - kUnrollGemmWarps; q < own; q += kUnrollThreads / kWarp - kUnrollGemmWarps) {
      const int e = first + q;
      if (e >= bd.E) break;
      const bool last = fin[q] != 0;
      const size_t at = (size_t)j * bd.E + e;
      float* dst = bd.rows + ((size_t)e * bd.T + row) * bd.W;
      const float* x = sm + u.noise + q * (A + D) + A;
      const float* ae = sm + u.act + q * A;
      for (int d = lane; d < D; d += kWarp) {
        dst[d] = x[d];
        if (p.obs_out) p.obs_out[at * D + d] = x[d];
      }
      for (int d = lane; d < A; d += kWarp) {
        dst[D + d] = ae[d];
        if (p.act_out) p.act_out[at * A + d] = ae[d];
      }
      for (int c = D + A + lane; c < bd.W; c += kWarp) dst[c] = c == D + A ? __int_as_float(-1) : 0.f;
      if (lane == 0 && p.done_out) p.done_out[at] = last ? 1 : 0;
      if (last) {
        __syncwarp();   // this row's open mark precedes its stamp
        const long long win_lo = total_after - (total_after < bd.T ? total_after : bd.T), start = bd.ep_start[e];
        for (long long a = (start > win_lo ? start : win_lo) + lane; a <= total_before; a += kWarp)
          bd.rows[((size_t)e * bd.T + (size_t)(a % bd.T)) * bd.W + D + A] = __int_as_float((int)total_before);
        __syncwarp();   // every lane has read the episode's start
        if (lane == 0) bd.ep_start[e] = (int32_t)total_after;
      }
    }
  };
  int cur = 0, row = 0;   // row: the slice not yet written
  for (int i = 0; i < p.n; ++i, slot = slot + 1 == bd.T ? 0 : slot + 1) {
    const unsigned long long k = step0 + (unsigned long long)i;
    const float* wl = sm + u.w;
    for (int l = 0; l < p.layers; ++l) {
      const int K = l == 0 ? p.in : H;
      if (wid < kUnrollGemmWarps) {
        for (int bx = bx0, by = by0; by < nby;) {
          const int ct = 8 * bx + lane % 8, et = 4 * by + lane / 8;
          for (bx += kUnrollGemmWarps; bx >= nbx; bx -= nbx) ++by;
          if (ct >= nct || et >= net) continue;
          const float* w = wl + 4 * ct;
          const float* x = sm + u.buf + cur * size + 4 * et;
          float2 acc[4][2];
#pragma unroll
          for (int a = 0; a < 4; ++a) acc[a][0] = acc[a][1] = make_float2(0.f, 0.f);
          auto eight = [&](int k0, bool guard) {
#pragma unroll
            for (int r = 0; r < 8; ++r) {
              float4 wv = make_float4(0.f, 0.f, 0.f, 0.f), xv = wv;   // (zeros past K on both sides add nothing)
              if (!guard || k0 + r < K) {
                wv = *reinterpret_cast<const float4*>(w + (k0 + r) * nc);
                xv = *reinterpret_cast<const float4*>(x + (k0 + r) * pitch);
              }
              const float xs[4] = {xv.x, xv.y, xv.z, xv.w};
#pragma unroll
              for (int a = 0; a < 4; ++a) {
                acc[a][0] = fma_x2(make_float2(xs[a], xs[a]), make_float2(wv.x, wv.y), acc[a][0]);
                acc[a][1] = fma_x2(make_float2(xs[a], xs[a]), make_float2(wv.z, wv.w), acc[a][1]);
              }
            }
          };
          int k0 = 0;
#pragma unroll 2
          for (; k0 + 8 <= K; k0 += 8) eight(k0, false);
          if (k0 < K) eight(k0, true);
          const float4 bv = *reinterpret_cast<const float4*>(sm + u.bias + l * nc + 4 * ct);
          const float bs[4] = {bv.x, bv.y, bv.z, bv.w};
          float* base = sm + u.buf + (cur ^ 1) * size + (n0 + 4 * ct) * pitch + 4 * et;
#pragma unroll
          for (int j = 0; j < 4; ++j) {
            if (n0 + 4 * ct + j >= H) break;
            float v[4];
#pragma unroll
            for (int a = 0; a < 4; ++a) {
              v[a] = ((j & 1) ? acc[a][j / 2].y : acc[a][j / 2].x) + bs[j];
              if (!p.layernorm) v[a] = v[a] > 0.f ? v[a] : 0.f;
            }
            const float4 f = make_float4(v[0], v[1], v[2], v[3]);
            *reinterpret_cast<float4*>(base + j * pitch) = f;
            for (int r = 1; r < C; ++r) st_cluster4(tc::mapa_shared(base + j * pitch, (rank + r) & (C - 1)), f);
          }
        }
      }
      __syncwarp();
      tc::cluster_arrive();
      if (l == 0 && i > 0 && wid >= kUnrollGemmWarps) {
        write_slice(i - 1, row);
        // (its state is read before the noise takes its place)
        asm volatile("bar.sync 1, %0;" ::"n"(kUnrollThreads - kUnrollGemmWarps * kWarp) : "memory");
      }
      if (l == p.layers - 1 && wid >= kUnrollGemmWarps) {
        // the step's noise: two neighbouring elements per thread; a reset draws its state instead
        const int pa = (A + 1) / 2, pd = (D + 1) / 2;
        for (int q = tid - kUnrollGemmWarps * kWarp; q < own * (pa + pd); q += kUnrollThreads - kUnrollGemmWarps * kWarp) {
          const int q0 = q / (pa + pd), r = q % (pa + pd);
          const bool act = r < pa;
          const int pr = act ? r : r - pa, lim = act ? A : D;
          const unsigned long long word = act ? 2ull : (st[q0] >= p.episode_length - 1 ? 4ull : 3ull);
          const float2 z = philox_normal_pair(k, first + q0, word, pr, p.seed, p.agent);
          float* dst = sm + u.noise + q0 * (A + D) + (act ? 0 : A) + 2 * pr;
          dst[0] = z.x;
          if (2 * pr + 1 < lim) dst[1] = z.y;
        }
        __syncwarp();
      }
      tc::cluster_wait();
      cur ^= 1;
      wl += K * nc;
      if (p.layernorm) {
        // every CTA normalises its own copy: one warp per environment
        const float* gain = sm + u.ln + 2 * l * H;
        const float* bias = gain + H;
        for (int q = wid; q < ME; q += kUnrollThreads / kWarp) {
          float* z = sm + u.buf + cur * size + q;
          float sum = 0;
          for (int c = lane; c < H; c += kWarp) sum += z[c * pitch];
          const float mean = warp_sum(sum) / float(H);
          float sq = 0;
          for (int c = lane; c < H; c += kWarp) {
            const float d = z[c * pitch] - mean;
            sq += d * d;
          }
          const float var = warp_sum(sq) / float(H);
          const float rs = 1.f / sqrtf(var + float(kLnEps));
          for (int c = lane; c < H; c += kWarp) {
            const float zh = (z[c * pitch] - mean) * rs;
            const float v = zh * gain[c] + bias[c];
            z[c * pitch] = v > 0.f ? v : 0.f;
          }
        }
        __syncthreads();
      }
    }
    __syncthreads();   // the noise
    // The output layer, one output per thread: the chain of dependent FMAs is the
    // time, so sixteen k are read ahead of it in two sets of registers (one column's
    // weights 16 bytes at a time).  Unrolled reads alone took 13 clocks per k.
    for (int o = tid, q = oq, j = oj; o < own * A2; o += kUnrollThreads) {
      const float* x = sm + u.buf + cur * size + rank * own + q;
      const float* w = sm + u.wo + j * u.wo_pitch;
      float acc = 0.f, xa[8], xb[8];
      float4 wa[2], wb[2];
      auto read = [&](int kk, float (&xs)[8], float4 (&ws)[2]) {
#pragma unroll
        for (int r = 0; r < 8; ++r) xs[r] = x[(kk + r) * pitch];
        ws[0] = *reinterpret_cast<const float4*>(w + kk);
        ws[1] = *reinterpret_cast<const float4*>(w + kk + 4);
      };
      auto chain = [&](const float (&xs)[8], const float4 (&ws)[2]) {
#pragma unroll
        for (int r = 0; r < 2; ++r) {
          acc = fmaf(xs[4 * r], ws[r].x, acc);
          acc = fmaf(xs[4 * r + 1], ws[r].y, acc);
          acc = fmaf(xs[4 * r + 2], ws[r].z, acc);
          acc = fmaf(xs[4 * r + 3], ws[r].w, acc);
        }
      };
      int kk = 0;
      if (H >= 16) {
        read(0, xa, wa);
        for (; kk + 16 <= H; kk += 16) {
          read(kk + 8, xb, wb);
          chain(xa, wa);
          read(kk + 24 <= H ? kk + 16 : kk, xa, wa);
          chain(xb, wb);
        }
      }
      for (; kk < H; ++kk) acc = fmaf(x[kk * pitch], w[kk], acc);
      sm[u.out + o] = acc + sm[u.bo + j];
      q += kUnrollThreads / A2, j += kUnrollThreads % A2;
      if (j >= A2) j -= A2, ++q;
    }
    __syncthreads();
    // The action and the next state, to every CTA.  Nothing goes to global memory here:
    // the barrier's release would wait for it.
    for (int q = wid; q < own; q += kUnrollThreads / kWarp) {
      const int e = first + q;
      if (e >= bd.E) break;
      const int te = st[q];
      const bool last = te >= p.episode_length - 1;
      float* nz = sm + u.noise + q * (A + D);
      float* ae = sm + u.act + q * A;
      for (int d = lane; d < A; d += kWarp) {
        const float mu = sm[u.out + q * A2 + d];
        const float l = fmin(fmax(sm[u.out + q * A2 + A + d], float(kLogStdMin)), float(kLogStdMax));
        const float un = mu + dev_exp(l) * nz[d];
        ae[d] = dev_tanh(un);
      }
      __syncwarp();   // the dynamics read the warp's actions
      for (int d = lane, am = lane_mod; d < D; d += kWarp) {
        const float x = sm[u.s + q * D + d], xi = nz[A + d];
        sm[u.s + q * D + d] = last ? xi : x + 0.1f * xi + 0.05f * ae[am];
        nz[A + d] = x;   // (kept for the slice)
        am += warp_mod;   // am = d % A
        if (am >= A) am -= A;
      }
      if (last)
        for (int d = lane; d < G; d += kWarp) sm[u.g + q * G + d] = philox_normal<float>(k, e, 5ull, d, p.seed, p.agent);
      __syncwarp();   // every lane has read the episode's step
      if (lane == 0) {
        st[q] = last ? 0 : te + 1;
        fin[q] = last ? 1 : 0;
      }
      send_input(q, cur ^ 1);
    }
    __syncwarp();
    tc::cluster_sync();
    __syncthreads();   // st, fin and the actions
    row = slot;
    cur ^= 1;
  }
  if (wid >= kUnrollGemmWarps) write_slice(p.n - 1, row);
  for (int q = tid; q < own * D; q += kUnrollThreads)
    if (first + q / D < bd.E) p.s[(size_t)first * D + q] = sm[u.s + q];
  for (int q = tid; q < own * G; q += kUnrollThreads)
    if (first + q / G < bd.E) p.gs[(size_t)first * G + q] = sm[u.g + q];
  for (int q = tid; q < own; q += kUnrollThreads)
    if (first + q < bd.E) p.t[first + q] = st[q];
  if (blockIdx.x == 0 && tid == 0) {
    const long long total = p.total_before + p.n;
    bd.state[0] = (int32_t)(total < bd.T ? total : bd.T);
    bd.state[1] = (int32_t)total;
  }
}

// ---- which path a call takes ------------------------------------------------------
// Modelled us, fits to both paths' times at 252 policies and sizes (D 3 to 500, hidden 32
// to 512, one to four layers, with and without LayerNorm; E 1 to 16,000) and calls of 1
// to 62 steps.  A call of n steps is the one launch's where setup + n step < n layers.
// The one launch fills its shared memory in every wave of clusters, so a call of one or
// two steps of many environments is the layers'.  us per call, D 29, A 8, two layers of
// 256, layers / one launch:
//   E          n = 1       n = 2       n = 8        n = 62
//   1          17 / 25     32 / 32     127 / 79     970 / 499
//   1024       26 / 27     52 / 36     204 / 90     1567 / 569
//   8192       76 / 132    150 / 191   599 / 547    4626 / 3742
//   16000      122 / 256   243 / 374   976 / 1081   7562 / 7445
// Over those 1,512 calls the choice takes 0.8 % more than the faster path on average and
// at most 19 % (17 us) more than the layers; 24 calls, most of one or two steps, take more
// than 5 % more.
// Beyond kUnrollEnvs environments the products fill the SMs by themselves.
constexpr int kUnrollEnvs = 16384;

// One step layer by layer: the launches, the tiles' waves of every product, LayerNorm,
// the step kernel.
double layers_step_us(const crl_config& cf, const MlpShape& s) {
  const double E = cf.E, D = cf.D, H = s.hidden;
  double us = 4.0 + 1.24e-3 * E + 1.26e-5 * E * D + 7.3e-3 * std::sqrt(E * D) + 0.0325 * D;
  for (int l = 0; l <= s.layers; ++l) {
    const int K = l == 0 ? s.in() : s.hidden, N = l == s.layers ? s.out : s.hidden;
    double tiles = 0;
    for (const F32Tile& t : kF32Tiles) {
      const double c = f32_tile_cost(t, (long long)ceil_div(cf.E, t.bm) * ceil_div(N, t.bn));
      if (tiles == 0 || c < tiles) tiles = c;
    }
    us += 1.31 + K * (0.004 + 7.08e-6 * tiles + 2.37e-4 * std::sqrt(tiles));
  }
  return us + (s.layernorm ? s.layers * (2.3 + 7.6e-7 * E * H + 8.1e-4 * std::sqrt(E * H)) : 0.0);
}

// The one launch, `waves` of clusters after one another.  Clocks of a step: the products
// of 8 x 4 blocks of thread tiles, beside them the slice in the first layer and the noise
// in the last; the barriers; the output chains; the dynamics and the pieces sent to the
// peers.  Set-up: the weights and the environments' state.
void unroll_model(const crl_config& cf, const MlpShape& s, int waves, UnrollPlan* q) {
  const int H = s.hidden, in = s.in(), own = q->ME / q->C;
  const int rounds = ceil_div(ceil_div(q->nc / 4, 8) * ceil_div(q->ME / 4, 4), kUnrollGemmWarps);
  const double noise = 1710.0 + 1445.0 * ceil_div(own * (ceil_div(cf.A, 2) + ceil_div(cf.D, 2)), 128);
  const double slice = 76.0 * ceil_div(own, 4) * (ceil_div(cf.D, 32) + ceil_div(cf.A, 32) + 1);
  double clocks = H * (1.8 + 2.63 * ceil_div(own * 2 * cf.A, 32)) +
                  ceil_div(own, 8) * (1650.0 + ceil_div(in, 32) * (337.0 + 68.0 * (q->C - 1)));
  for (int l = 0; l < s.layers; ++l)
    clocks += std::max(rounds * (22.3 * (l == 0 ? in : H) + 1167.0),
                       (l == 0 ? slice : 0.0) + (l == s.layers - 1 ? noise : 0.0)) +
              475.0 * q->C;
  if (s.layernorm) clocks += s.layers * ceil_div(q->ME, 8) * (3.79 * H + 1060.0);
  const double w = waves * (0.99 + 0.01 * waves);   // (waves fill the SMs a little less well than one)
  q->step = w * clocks / 1920.0;
  q->setup = 0.8 + w * (5.75 + 3.16e-4 * (in + (s.layers - 1.0) * H) * q->nc + 2.4e-4 * cf.A * H +
                            1.2e-3 * own * cf.D + 0.004 * ceil_div(own, 8) * ceil_div(in, 32) * q->C);
}

// The cluster size and environments per cluster that fit with the least waves x clocks
// per step (a ranking of the forms of one policy: the terms that differ little between
// them are left out, so its values are good to a factor of 1.5 only).  C = 0: nothing fits.
UnrollPlan unroll_plan(const crl_config& cf, const MlpShape& s) {
  UnrollPlan best;
  double least = 0;
  int waves = 0;
  const int H = s.hidden, in = s.in();
  if (in != cf.D + cf.G || s.out != 2 * cf.A || cf.E > kUnrollEnvs) return best;
  CRL_CHECK_CUDA(cudaFuncSetAttribute(unroll_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kUnrollSmem));
  for (int C = 1; C <= 8; C *= 2) {
    const int nc = round_up(ceil_div(H, C), 4);
    if ((C - 1) * nc >= H) continue;   // a CTA without columns
    // clusters at a time: 152, 76, 36 and 15
    cudaLaunchAttribute attr;
    attr.id = cudaLaunchAttributeClusterDimension;
    attr.val.clusterDim.x = C;
    attr.val.clusterDim.y = attr.val.clusterDim.z = 1;
    cudaLaunchConfig_t lc = {};
    lc.gridDim = dim3(C);
    lc.blockDim = dim3(kUnrollThreads);
    lc.dynamicSmemBytes = kUnrollSmem;
    lc.attrs = &attr;
    lc.numAttrs = 1;
    int resident = 0;
    if (cudaOccupancyMaxActiveClusters(&resident, unroll_kernel, &lc) != cudaSuccess || resident < 1) {
      cudaGetLastError();
      continue;
    }
    const int unit = C < 4 ? 4 : C;
    for (int ME = unit; ME <= 64; ME += unit) {
      int pitch = ME;
      if (pitch / 4 % 2 == 0) pitch += 4;   // (an odd multiple of 16 bytes)
      const UnrollSmem u = unroll_smem(s.layers, in, H, cf.D, cf.A, cf.G, s.layernorm, C, ME, nc, pitch);
      const size_t bytes = (size_t)u.total * sizeof(float);
      if (bytes > kUnrollSmem) break;
      const int clusters = ceil_div(cf.E, ME), w = ceil_div(clusters, resident), own = ME / C;
      const int rounds = ceil_div(ceil_div(nc / 4, 8) * ceil_div(ME / 4, 4), kUnrollGemmWarps);
      const double clocks = 26.5 * rounds * (in + (s.layers - 1) * (double)H) + 2600.0 * s.layers +
                            10.0 * H * ceil_div(own * 2 * cf.A, kUnrollThreads) + 1200.0 * ceil_div(own, 8) + 1500.0 +
                            50.0 * C * s.layers +
                            (s.layernorm ? s.layers * ceil_div(ME, 8) * (H / 32 * 60.0 + 250.0) : 0.0);
      if (best.C == 0 || w * clocks < least) {
        best.C = C, best.ME = ME, best.nc = nc, best.pitch = pitch, best.clusters = clusters, best.smem = bytes;
        least = w * clocks;
        waves = w;
      }
    }
  }
  if (best.C) {
    unroll_model(cf, s, waves, &best);
    best.layers_step = layers_step_us(cf, s);
  }
  return best;
}

// Whether a call of n steps is the one launch's.
bool unroll_pays(const UnrollPlan& q, int n) {
  return q.C != 0 && ceil_div(n, kUnrollSteps) * q.setup + n * q.step < n * q.layers_step;
}

// All n steps of one call (as many as the step counter has room for).
int collect_unroll(crl_ctx* c, const UnrollPlan& q, int n, int episode_length, float* obs_out, float* act_out,
                   uint8_t* done_out, cudaStream_t st) {
  const crl_config& cf = c->cfg;
  const MlpShape& s = c->shapes[CRL_NET_PI];
  LayerOffsets lay[CRL_MAX_LAYERS + 1];
  mlp_layout(s, lay);
  UnrollArgs a;
  a.bd = c->bd;
  a.G = cf.G;
  a.episode_length = episode_length;
  a.layers = s.layers, a.H = s.hidden, a.in = s.in(), a.layernorm = s.layernorm;
  a.C = q.C, a.ME = q.ME, a.nc = q.nc, a.pitch = q.pitch;
  a.params = static_cast<const float*>(c->nets[CRL_NET_PI].params);
  double flops = 0;
  for (int l = 0; l <= s.layers; ++l) {
    a.W[l] = lay[l].W, a.b[l] = lay[l].b;
    if (l < s.layers) a.g[l] = lay[l].g, a.beta[l] = lay[l].beta;
    flops += 2.0 * cf.E * lay[l].in * lay[l].out;
  }
  a.s = c->env.s, a.gs = c->env.g, a.t = c->env.t;
  a.step_dev = c->env.step;
  a.seed = cf.seed, a.agent = cf.agent;
  int i = 0;
  while (i < n && c->total_host + 1 < ((int64_t)1 << 31) - 1) {
    const int64_t room = ((int64_t)1 << 31) - 2 - c->total_host;
    a.n = (int)std::min<int64_t>(std::min(n - i, kUnrollSteps), room);
    a.total_before = c->total_host;
    a.i0 = (unsigned long long)i;
    a.obs_out = obs_out ? obs_out + (size_t)i * cf.E * cf.D : nullptr;
    a.act_out = act_out ? act_out + (size_t)i * cf.E * cf.A : nullptr;
    a.done_out = done_out ? done_out + (size_t)i * cf.E : nullptr;
    TraceLaunch tr(CRL_TRACE_GEMM, st, flops * a.n);
    launch_k_cluster(unroll_kernel, dim3(q.clusters * q.C), dim3(kUnrollThreads), q.smem, st, (unsigned)q.C, a);
    i += a.n;
    c->total_host += a.n;
    c->size_host = (int32_t)(c->total_host < cf.T ? c->total_host : cf.T);
  }
  return i;
}

template <typename T>
void collect_steps(crl_ctx* c, int n, int episode_length, float* obs_out, float* act_out, uint8_t* done_out,
                   cudaStream_t st) {
  const crl_config& cf = c->cfg;
  crl_ctx::Envs& v = c->env;
  const int E = cf.E;
  const T* params = static_cast<const T*>(c->nets[CRL_NET_PI].params);
  int i = 0;
  if (sizeof(T) == 4 && !v.planned) {   // (the configuration decides: once per context)
    v.plan = unroll_plan(cf, c->shapes[CRL_NET_PI]);
    v.planned = true;
  }
  const bool one = sizeof(T) == 4 && unroll_pays(v.plan, n);
  if (one) i = collect_unroll(c, v.plan, n, episode_length, obs_out, act_out, done_out, st);
  for (; !one && i < n && c->total_host + 1 < ((int64_t)1 << 31) - 1; ++i) {
    mlp_forward<T, float>(c->shapes[CRL_NET_PI], params, v.s, v.g, E, static_cast<T*>(v.pi_out), v.saved, st);
    CollectArgs<T> a;
    a.bd = c->bd;
    a.total_before = c->total_host;
    a.G = cf.G;
    a.episode_length = episode_length;
    a.s = v.s;
    a.g = v.g;
    a.t = v.t;
    a.pi_out = static_cast<const T*>(v.pi_out);
    a.a = static_cast<T*>(v.a);
    a.step_dev = v.step;
    a.i = (unsigned long long)i;
    a.obs_out = obs_out ? obs_out + (size_t)i * E * cf.D : nullptr;
    a.act_out = act_out ? act_out + (size_t)i * E * cf.A : nullptr;
    a.done_out = done_out ? done_out + (size_t)i * E : nullptr;
    a.seed = cf.seed;
    a.agent = cf.agent;
    TraceLaunch tr(CRL_TRACE_AUX, st, (double)E * (3.0 * cf.D * 4 + cf.A * (2.0 * sizeof(T) + 4)));
    launch_k(collect_step_kernel<T>, dim3(ceil_div(E, 8)), dim3(256), 0, st, a);
    c->total_host += 1;
    c->size_host = (int32_t)(c->total_host < cf.T ? c->total_host : cf.T);
  }
  launch_k(advance_kernel, dim3(1), dim3(1), 0, st, v.step, (unsigned long long)i);
  CRL_REQUIRE(i == n, CRL_E_INVALID_ARG, "more than 2^31 - 2 steps inserted per environment");
}

}  // namespace

// Allocates the collection stub's environments and staging and resets every
// environment (episode starts drawn from the collection stream at step 0).
void collect_alloc(crl_ctx* ctx, cudaStream_t st) {
  const crl_config& cf = ctx->cfg;
  crl_ctx::Envs& v = ctx->env;
  const size_t es = ctx->esz;
  const int E = cf.E;
  v.s = static_cast<float*>(ctx->dalloc((size_t)E * cf.D * sizeof(float)));
  v.g = static_cast<float*>(ctx->dalloc((size_t)E * cf.G * sizeof(float)));
  v.t = static_cast<int32_t*>(ctx->dalloc((size_t)E * sizeof(int32_t)));
  v.step = static_cast<unsigned long long*>(ctx->dalloc(sizeof(unsigned long long)));
  v.pi_out = ctx->dalloc((size_t)E * 2 * cf.A * es);
  v.a = ctx->dalloc((size_t)E * cf.A * es);
  v.saved = ctx->dalloc(mlp_saved_bytes(ctx->shapes[CRL_NET_PI], E, es));
  CRL_CHECK_CUDA(cudaMemsetAsync(v.step, 0, sizeof(unsigned long long), st));
  launch_k(env_init_kernel, dim3(ceil_div(E, 8)), dim3(256), 0, st, E, cf.D, cf.G, v.s, v.g, v.t,
           (unsigned long long)cf.seed, (unsigned long long)cf.agent);
  v.ready = true;
}

}  // namespace crl

extern "C" int crl_collect(crl_ctx* ctx, int32_t n_steps, int32_t episode_length, float* obs_out, float* act_out,
                           uint8_t* done_out, void* stream) {
  using namespace crl;
  NvtxRange nvtx("crl_collect");
  return guarded(ctx, [&] {
    CRL_REQUIRE(ctx, CRL_E_INVALID_ARG, "null context");
    CRL_REQUIRE(ctx->bound, CRL_E_NOT_BOUND, "crl_bind_params has not been called");
    CRL_REQUIRE(n_steps >= 1, CRL_E_INVALID_ARG, "n_steps must be >= 1");
    CRL_REQUIRE(episode_length >= 1, CRL_E_INVALID_ARG, "episode_length must be >= 1");
    CRL_REQUIRE(!obs_out || !is_host_pointer(obs_out), CRL_E_INVALID_ARG, "obs_out must be device memory");
    CRL_REQUIRE(!act_out || !is_host_pointer(act_out), CRL_E_INVALID_ARG, "act_out must be device memory");
    CRL_REQUIRE(!done_out || !is_host_pointer(done_out), CRL_E_INVALID_ARG, "done_out must be device memory");
    const crl_config& cf = ctx->cfg;
    cudaStream_t st = static_cast<cudaStream_t>(stream);
    if (!ctx->env.ready) collect_alloc(ctx, st);
    if (cf.precision == CRL_PREC_FP64)
      collect_steps<double>(ctx, n_steps, episode_length, obs_out, act_out, done_out, st);
    else
      collect_steps<float>(ctx, n_steps, episode_length, obs_out, act_out, done_out, st);
    check_launch("collect");
  });
}
