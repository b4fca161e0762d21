// Adam update for the CRL networks (Kingma & Ba, 2015; bias-corrected, no
// weight decay).  arXiv 2408.11052 App. B.3 gives the learning rates (critic
// 3e-4, policy 6e-4) without naming the optimiser; Adam is the reading taken.
//
// The step number t is read from device memory (so the update can be replayed
// inside a CUDA graph while the counter advances) or passed by value.
#include <algorithm>

#include "common.cuh"
#include "internal.h"
#include "trace.h"

namespace crl {

namespace {

template <typename T>
struct AdamPair {
  AdamArrays<T> a[2];
};
// blockIdx.y: the network.
template <typename T>
__global__ void __launch_bounds__(256) adam_kernel(const __grid_constant__ AdamPair<T> pair,
                                                  const int* __restrict__ t_dev, int t_host, float lr, float b1,
                                                  float b2, float eps) {
  pdl_enter();
  T* __restrict__ p = pair.a[blockIdx.y].p;
  const T* __restrict__ g = pair.a[blockIdx.y].g;
  T* __restrict__ m = pair.a[blockIdx.y].m;
  T* __restrict__ v = pair.a[blockIdx.y].v;
  const long long n = pair.a[blockIdx.y].n;
  // Bias corrections in double (1 - b^t loses most of its digits in float for
  // small t), computed once per block.
  // b^t by repeated squaring (at most 31 double products; pow() took several us of
  // the FP64 pipe before every block's first load), one thread per power.
  __shared__ double s_corr[2];
  if (threadIdx.x == 0 || threadIdx.x == kWarp) {
    double x = threadIdx.x == 0 ? (double)b1 : (double)b2, bt = 1.0;
    for (int t = t_dev ? *t_dev : t_host; t > 0; t >>= 1) {
      if (t & 1) bt *= x;
      x *= x;
    }
    if (threadIdx.x == 0) s_corr[0] = (double)lr / (1.0 - bt);
    else s_corr[1] = 1.0 / (1.0 - bt);
  }
  __syncthreads();
  const T step = T(s_corr[0]);
  const T ibc2 = T(s_corr[1]);
  const T tb1 = T(b1), tb2 = T(b2), one = T(1);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += (long long)gridDim.x * blockDim.x) {
    const T gi = g[i];
    const T mi = tb1 * m[i] + (one - tb1) * gi;
    const T vi = tb2 * v[i] + (one - tb2) * gi * gi;
    m[i] = mi;
    v[i] = vi;
    p[i] -= step * mi / (dev_sqrt(vi * ibc2) + T(eps));
  }
}

}  // namespace

template <typename T>
void adam_update(const AdamArrays<T>* a, int count, const int* t_dev, int t_host, float lr, float b1, float b2,
                 float eps, cudaStream_t st) {
  AdamPair<T> pair;
  int64_t longest = 0, total = 0;
  int live = 0;
  for (int i = 0; i < count; ++i) {
    if (a[i].n <= 0) continue;
    pair.a[live++] = a[i];
    longest = std::max(longest, a[i].n);
    total += a[i].n;
  }
  if (live == 0) return;
  if (live == 1) pair.a[1] = pair.a[0];
  const int blocks = (int)std::min<int64_t>(ceil_div(longest, 256), 152 * 8 / live);
  TraceLaunch tr(CRL_TRACE_ADAM, st, 7.0 * sizeof(T) * total);  // read p, g, m, v; write p, m, v
  launch_k(adam_kernel<T>, dim3(blocks, live), dim3(256), 0, st, pair, t_dev, t_host, lr, b1, b2, eps);
}

template void adam_update<float>(const AdamArrays<float>*, int, const int*, int, float, float, float, float,
                                 cudaStream_t);
template void adam_update<double>(const AdamArrays<double>*, int, const int*, int, float, float, float, float,
                                  cudaStream_t);

}  // namespace crl
