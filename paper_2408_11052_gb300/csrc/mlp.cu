// Encoder / actor MLPs of the CRL update step, forward and hand-written backward
// (FP32 and FP64 SIMT path).
//
// A network (arXiv 2408.11052 §3.1 phi(s,a) and psi(g); §3.2 the policy; App. B.3
// hidden [256, 256], repr 64; §5.4 LayerNorm before every activation for the
// 4 x 1024 networks) is
//     h_0 = concat(x0, x1);  z_l = h_{l-1} W_l^T + b_l;  u_l = LN(z_l) or z_l;
//     h_l = ReLU(u_l);  y = h_L W_out^T + b_out.
// LayerNorm: biased variance, eps 1e-6, learned gain and bias.
//
// Saved activations per hidden layer (for the backward): h_l [M][H] and, with
// LayerNorm, zhat_l [M][H] and rstd_l [M].  The backward scratch (three
// [M][H] buffers) follows them in the same workspace.
#include "common.cuh"
#include "gemm_simt.cuh"
#include "internal.h"
#include "trace.h"

namespace crl {


int64_t mlp_layout(const MlpShape& s, LayerOffsets* lay) {
  int64_t off = 0;
  auto take = [&](int64_t n) {
    const int64_t o = off;
    off += round_up(n, 64);
    return o;
  };
  for (int l = 0; l <= s.layers; ++l) {
    const int in = (l == 0) ? s.in() : s.hidden;
    const int out = (l == s.layers) ? s.out : s.hidden;
    LayerOffsets& L = lay[l];
    L.in = in;
    L.out = out;
    L.W = take((int64_t)in * out);
    L.b = take(out);
    if (s.layernorm && l < s.layers) {
      L.g = take(out);
      L.beta = take(out);
    } else {
      L.g = L.beta = -1;
    }
  }
  return off;
}

size_t mlp_saved_bytes(const MlpShape& s, int M, size_t elem) {
  size_t n = (size_t)s.layers * M * s.hidden;                 // h_l
  if (s.layernorm) n += (size_t)s.layers * ((size_t)M * s.hidden + M);  // zhat_l, rstd_l
  n += 3 * (size_t)M * s.hidden;                              // backward scratch
  return n * elem;
}

namespace {

template <typename T>
struct Saved {
  T* h[CRL_MAX_LAYERS];
  T* zhat[CRL_MAX_LAYERS];
  T* rstd[CRL_MAX_LAYERS];
  T* scratch[3];
};

template <typename T>
Saved<T> carve(const MlpShape& s, int M, void* base) {
  Saved<T> sv{};
  T* p = static_cast<T*>(base);
  const size_t mh = (size_t)M * s.hidden;
  for (int l = 0; l < s.layers; ++l) {
    sv.h[l] = p;
    p += mh;
  }
  if (s.layernorm) {
    for (int l = 0; l < s.layers; ++l) {
      sv.zhat[l] = p;
      p += mh;
      sv.rstd[l] = p;
      p += M;
    }
  }
  for (int i = 0; i < 3; ++i) {
    sv.scratch[i] = p;
    p += mh;
  }
  return sv;
}

// Row-wise LayerNorm + ReLU: z (in zhat, overwritten by zhat), rstd, h = ReLU(zhat*g + beta).
// One warp per row.
template <typename T>
struct LnFwd {   // one network's; blockIdx.y picks the network
  int M, N;
  T *zhat, *rstd, *h;
  const T *gain, *bias;
};
template <typename T>
struct LnFwds {
  LnFwd<T> a[2];
};
template <typename T>
__global__ void __launch_bounds__(256) layernorm_relu_kernel(const __grid_constant__ LnFwds<T> args) {
  pdl_enter();
  const LnFwd<T>& p = args.a[blockIdx.y];
  const int M = p.M, N = p.N;
  T* __restrict__ zhat = p.zhat;
  T* __restrict__ rstd = p.rstd;
  T* __restrict__ h = p.h;
  const T* __restrict__ gain = p.gain;
  const T* __restrict__ bias = p.bias;
  const int lane = threadIdx.x % kWarp;
  const int row = blockIdx.x * (blockDim.x / kWarp) + threadIdx.x / kWarp;
  if (row >= M) return;
  T* z = zhat + (size_t)row * N;
  T sum = 0;
  for (int c = lane; c < N; c += kWarp) sum += z[c];
  const T mean = warp_sum(sum) / T(N);
  T sq = 0;
  for (int c = lane; c < N; c += kWarp) {
    const T d = z[c] - mean;
    sq += d * d;
  }
  const T var = warp_sum(sq) / T(N);
  const T rs = T(1) / dev_sqrt(var + T(kLnEps));
  for (int c = lane; c < N; c += kWarp) {
    const T zh = (z[c] - mean) * rs;
    z[c] = zh;
    const T u = zh * gain[c] + bias[c];
    h[(size_t)row * N + c] = u > T(0) ? u : T(0);
  }
  if (lane == 0) rstd[row] = rs;
}

// Row-wise LayerNorm backward: du (already masked by ReLU) -> dz.
template <typename T>
struct LnBwd {
  int M, N;
  const T *du, *zhat, *rstd, *gain;
  T* dz;
};
template <typename T>
struct LnBwds {
  LnBwd<T> a[2];
};
template <typename T>
__global__ void __launch_bounds__(256) layernorm_bwd_kernel(const __grid_constant__ LnBwds<T> args) {
  pdl_enter();
  const LnBwd<T>& p = args.a[blockIdx.y];
  const int M = p.M, N = p.N;
  const T* __restrict__ du = p.du;
  const T* __restrict__ zhat = p.zhat;
  const T* __restrict__ rstd = p.rstd;
  const T* __restrict__ gain = p.gain;
  T* __restrict__ dz = p.dz;
  const int lane = threadIdx.x % kWarp;
  const int row = blockIdx.x * (blockDim.x / kWarp) + threadIdx.x / kWarp;
  if (row >= M) return;
  const T* d = du + (size_t)row * N;
  const T* zh = zhat + (size_t)row * N;
  T s1 = 0, s2 = 0;
  for (int c = lane; c < N; c += kWarp) {
    const T dzh = d[c] * gain[c];
    s1 += dzh;
    s2 += dzh * zh[c];
  }
  s1 = warp_sum(s1) / T(N);
  s2 = warp_sum(s2) / T(N);
  const T rs = rstd[row];
  for (int c = lane; c < N; c += kWarp) {
    const T dzh = d[c] * gain[c];
    dz[(size_t)row * N + c] = rs * (dzh - s1 - zh[c] * s2);
  }
}

// Column sums over M rows: out1[n] = sum X, out2[n] = sum X*Y (Y optional).  Block =
// 32 columns x 32 row groups (eight groups left M / 8 dependent loads per thread: 9 us
// at M = 256 against 4 now); eight groups in FP64, whose additions are slow enough
// that merging 32 costs more than the shorter chains save (a backward of 2 x 128 with
// LayerNorm at 64 rows: 143 us with 32, 134 with 8; from 512 rows on within 1 %).
template <typename T>
constexpr int kSumRows = sizeof(T) == 8 ? 8 : 32;
template <typename T>
struct ColSum {
  int M, N;
  const T *X, *Y;
  T *out1, *out2;
};
template <typename T>
struct ColSums {
  ColSum<T> a[2];
};
template <typename T>
__global__ void __launch_bounds__(32 * kSumRows<T>) colsum_kernel(const __grid_constant__ ColSums<T> args) {
  pdl_enter();
  const ColSum<T>& p = args.a[blockIdx.y];
  const int M = p.M, N = p.N;
  const T* __restrict__ X = p.X;
  const T* __restrict__ Y = p.Y;
  T* __restrict__ out1 = p.out1;
  T* __restrict__ out2 = p.out2;
  __shared__ T sm[2][kSumRows<T>][33];
  const int cx = threadIdx.x % 32, ry = threadIdx.x / 32;
  const int n = blockIdx.x * 32 + cx;
  T a1 = 0, a2 = 0;
  if (n < N) {
#pragma unroll 4
    for (int m = ry; m < M; m += kSumRows<T>) {
      const size_t o = (size_t)m * N + n;
      const T x = X[o];
      a1 += x;
      if (Y) a2 += x * Y[o];
    }
  }
  sm[0][ry][cx] = a1;
  sm[1][ry][cx] = a2;
  __syncthreads();
  if (ry == 0 && n < N) {
    T s1 = 0, s2 = 0;
#pragma unroll 8
    for (int r = 0; r < kSumRows<T>; ++r) {
      s1 += sm[0][r][cx];
      s2 += sm[1][r][cx];
    }
    if (out1) out1[n] = s1;
    if (out2) out2[n] = s2;
  }
}

template <typename T>
void colsum(const ColSum<T>* c, int n, cudaStream_t st) {
  ColSums<T> a;
  double bytes = 0;
  int N = 0;
  for (int i = 0; i < 2; ++i) {
    a.a[i] = c[i < n ? i : 0];
    if (i >= n) continue;
    bytes += (double)c[i].M * c[i].N * sizeof(T) * (1 + (c[i].Y != nullptr));
    N = std::max(N, c[i].N);
  }
  TraceLaunch tr(CRL_TRACE_AUX, st, bytes);
  launch_k(colsum_kernel<T>, dim3(ceil_div(N, 32), n), dim3(32 * kSumRows<T>), 0, st, a);
}

}  // namespace

// Networks of one call share each launch (blockIdx.z of a product, blockIdx.y of the
// others); they need the same number of layers and the same LayerNorm setting.
template <typename T, typename TX1>
void mlp_forward(const MlpForward<T, TX1>* net, int n, cudaStream_t st) {
  const int layers = net[0].s->layers, layernorm = net[0].s->layernorm;
  if (n == 2 && (net[1].s->layers != layers || net[1].s->layernorm != layernorm)) {
    mlp_forward<T, TX1>(net, 1, st);
    mlp_forward<T, TX1>(net + 1, 1, st);
    return;
  }
  LayerOffsets lay[2][CRL_MAX_LAYERS + 1];
  Saved<T> sv[2];
  for (int i = 0; i < n; ++i) {
    mlp_layout(*net[i].s, lay[i]);
    sv[i] = carve<T>(*net[i].s, net[i].M, net[i].saved);
  }
  for (int l = 0; l <= layers; ++l) {
    const bool last = (l == layers);
    GemmSet<LoadRowsSplit<T, float, TX1>, LoadNK<T>, EpiBias<T>> first[2];
    GemmSet<LoadRowsSplit<T, T, T>, LoadNK<T>, EpiBias<T>> later[2];
    for (int i = 0; i < n; ++i) {
      const MlpForward<T, TX1>& p = net[i];
      const LayerOffsets& L = lay[i][l];
      const int H = p.s->hidden;
      T* out = last ? p.y : (layernorm ? sv[i].zhat[l] : sv[i].h[l]);
      const int ldo = last ? p.s->out : H;
      const EpiBias<T> ep{out, ldo, p.params + L.b, (!last && !layernorm) ? 1 : 0};
      const LoadNK<T> lb{p.params + L.W, L.in};
      if (l == 0)
        first[i] = {p.M, L.out, L.in, LoadRowsSplit<T, float, TX1>{p.x0, p.x1, p.s->in0, p.s->in1, p.s->in0}, lb, ep};
      else
        later[i] = {p.M, L.out, L.in, LoadRowsSplit<T, T, T>{sv[i].h[l - 1], nullptr, H, 0, H}, lb, ep};
    }
    if (l == 0) gemm_sets<T>(first, n, st);
    else gemm_sets<T>(later, n, st);
    if (!last && layernorm) {
      LnFwds<T> a;
      double bytes = 0;
      int M = 0;
      for (int i = 0; i < 2; ++i) {
        const int k = i < n ? i : 0;
        const MlpForward<T, TX1>& p = net[k];
        const LayerOffsets& L = lay[k][l];
        a.a[i] = {p.M, p.s->hidden, sv[k].zhat[l], sv[k].rstd[l], sv[k].h[l], p.params + L.g, p.params + L.beta};
        if (i < n) bytes += 4.0 * p.M * p.s->hidden * sizeof(T), M = std::max(M, p.M);
      }
      TraceLaunch tr(CRL_TRACE_AUX, st, bytes);
      launch_k(layernorm_relu_kernel<T>, dim3(ceil_div(M, 8), n), dim3(256), 0, st, a);
    }
  }
}

template <typename T, typename TX1>
void mlp_backward(const MlpBackward<T, TX1>* net, int n, cudaStream_t st) {
  const int layers = net[0].s->layers, layernorm = net[0].s->layernorm;
  const bool grads = net[0].dparams != nullptr;
  const bool dx = net[0].dx0 || net[0].dx1;
  if (n == 2 && (net[1].s->layers != layers || net[1].s->layernorm != layernorm ||
                 (net[1].dparams != nullptr) != grads || (net[1].dx0 || net[1].dx1) != dx)) {
    mlp_backward<T, TX1>(net, 1, st);
    mlp_backward<T, TX1>(net + 1, 1, st);
    return;
  }
  LayerOffsets lay[2][CRL_MAX_LAYERS + 1];
  Saved<T> sv[2];
  const T* dcur[2];   // dZ of the layer being processed ([M][out_l])
  for (int i = 0; i < n; ++i) {
    mlp_layout(*net[i].s, lay[i]);
    sv[i] = carve<T>(*net[i].s, net[i].M, const_cast<void*>(net[i].saved));
    dcur[i] = net[i].dy;
  }
  int bufi = 0;
  for (int l = layers; l >= 0; --l) {
    if (grads) {
      // db_l = colsum(dZ_l);  dW_l[n][k] = sum_m dZ_l[m][n] * in_l[m][k]
      ColSum<T> db[2];
      GemmSet<LoadTrans<T>, LoadColsSplit<T, float, TX1>, EpiScale<T>> first[2];
      GemmSet<LoadTrans<T>, LoadColsSplit<T, T, T>, EpiScale<T>> later[2];
      for (int i = 0; i < n; ++i) {
        const MlpBackward<T, TX1>& p = net[i];
        const LayerOffsets& L = lay[i][l];
        const int H = p.s->hidden;
        db[i] = {p.M, L.out, dcur[i], nullptr, p.dparams + L.b, nullptr};
        const LoadTrans<T> la{dcur[i], L.out};
        const EpiScale<T> ep{p.dparams + L.W, L.in, T(1)};
        if (l == 0)
          first[i] = {L.out, L.in, p.M, la, LoadColsSplit<T, float, TX1>{p.x0, p.x1, p.s->in0, p.s->in1, p.s->in0}, ep};
        else
          later[i] = {L.out, L.in, p.M, la, LoadColsSplit<T, T, T>{sv[i].h[l - 1], nullptr, H, 0, H}, ep};
      }
      colsum<T>(db, n, st);
      if (l == 0) gemm_sets<T>(first, n, st);
      else gemm_sets<T>(later, n, st);
    }
    if (l == 0 && !dx) break;
    // dU_{l-1} = (dZ_l W_l) * [h_{l-1} > 0], or the input gradients
    GemmSet<LoadMK<T>, LoadKN<T>, EpiMaskSplit<T>> prod[2];
    for (int i = 0; i < n; ++i) {
      const MlpBackward<T, TX1>& p = net[i];
      const LayerOffsets& L = lay[i][l];
      const int H = p.s->hidden;
      const LoadMK<T> la{dcur[i], L.out};
      const LoadKN<T> lb{p.params + L.W, L.in};
      if (l == 0)
        prod[i] = {p.M, L.in, L.out, la, lb, EpiMaskSplit<T>{p.dx0, p.dx1, p.s->in0, p.s->in1, p.s->in0, nullptr, 0}};
      else
        prod[i] = {p.M, H, L.out, la, lb,
                   EpiMaskSplit<T>{sv[i].scratch[bufi], nullptr, H, 0, H, sv[i].h[l - 1], H}};
    }
    gemm_sets<T>(prod, n, st);
    if (l == 0) break;
    if (layernorm) {
      LnBwds<T> a;
      ColSum<T> dg[2];
      double bytes = 0;
      int M = 0;
      for (int i = 0; i < 2; ++i) {
        const int k = i < n ? i : 0;
        const MlpBackward<T, TX1>& p = net[k];
        const LayerOffsets& P = lay[k][l - 1];
        T* du = sv[k].scratch[bufi];
        a.a[i] = {p.M, p.s->hidden, du, sv[k].zhat[l - 1], sv[k].rstd[l - 1], p.params + P.g, sv[k].scratch[2]};
        if (i >= n) continue;
        dg[i] = {p.M, p.s->hidden, du, sv[i].zhat[l - 1], grads ? p.dparams + P.beta : nullptr,
                 grads ? p.dparams + P.g : nullptr};
        bytes += 3.0 * p.M * p.s->hidden * sizeof(T);
        M = std::max(M, p.M);
        // the next product reads dz (scratch[2]) and writes the other ping-pong buffer: no overlap
        dcur[i] = sv[i].scratch[2];
      }
      {
        TraceLaunch tr(CRL_TRACE_AUX, st, bytes);
        launch_k(layernorm_bwd_kernel<T>, dim3(ceil_div(M, 8), n), dim3(256), 0, st, a);
      }
      if (grads) colsum<T>(dg, n, st);
    } else {
      for (int i = 0; i < n; ++i) dcur[i] = sv[i].scratch[bufi];
    }
    bufi = (bufi + 1) % 2;
  }
}

template void mlp_forward<float, float>(const MlpForward<float, float>*, int, cudaStream_t);
template void mlp_forward<double, float>(const MlpForward<double, float>*, int, cudaStream_t);
template void mlp_forward<double, double>(const MlpForward<double, double>*, int, cudaStream_t);
template void mlp_backward<float, float>(const MlpBackward<float, float>*, int, cudaStream_t);
template void mlp_backward<double, float>(const MlpBackward<double, float>*, int, cudaStream_t);
template void mlp_backward<double, double>(const MlpBackward<double, double>*, int, cudaStream_t);

}  // namespace crl
