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

#include "actor_head.cuh"
#include "common.cuh"
#include "ctx.h"
#include "internal.h"
#include "philox.cuh"
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

template <typename T>
void collect_steps(crl_ctx* c, int n, int episode_length, float* obs_out, float* act_out, uint8_t* done_out,
                   cudaStream_t st) {
  const crl_config& cf = c->cfg;
  crl_ctx::Envs& v = c->env;
  const int E = cf.E;
  const T* params = static_cast<const T*>(c->nets[CRL_NET_PI].params);
  int i = 0;
  for (; i < n && c->total_host + 1 < ((int64_t)1 << 31) - 1; ++i) {
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
