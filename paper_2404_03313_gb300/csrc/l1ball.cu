// Projection onto the l1 ball {x : ||x||_1 <= r} (Alg. 1 steps 3-4; the paper
// cites Condat's fast l1-ball projection and gives it O(N log N) in Table II).
//
// The projection is sign(x) max(|x| - tau, 0) with the unique tau >= 0 solving
// h(tau) = sum_i max(|x_i| - tau, 0) = r (tau = 0 when ||x||_1 <= r).  Instead of
// sorting, the threshold is found by radix selection over the 31 magnitude bits
// of the FP32 values, which orders them exactly like their values: three
// histogram passes (11, 11 and 9 bits) each keep the bin whose lower edge is the
// last one with h >= r.  After the third level every bin holds a single value,
// the active set {|x| > tau} is exactly the elements above the chosen bin, and
// tau = (sum of the active |x| - r) / (their count), evaluated in FP64.
// The CTA of a histogram pass that finishes last narrows the threshold
// (l1_select.cuh): one launch per level.
#include <math.h>
#include "l1_select.cuh"

namespace s3ttv {
namespace {

template <int LEVEL, bool VEC>
__global__ void __launch_bounds__(kSelThreads, 3) l1_hist_kernel(L1Args a) {
  __shared__ BinSums s_hist;
  chained();
  const int pb = blockIdx.y;
  if (a.sc->done) return;
  const L1State st = a.sc->l1[pb];
  if (LEVEL > 1 && st.mode != 0) return;  // decided at an earlier level
  l1_hist<LEVEL, VEC>(a, st, pb, (long long)blockIdx.x * kSelThreads + threadIdx.x,
                      (long long)gridDim.x * kSelThreads, s_hist);
  if (last_cta(&a.sc->ticket[pb], gridDim.x)) l1_scan_level<LEVEL>(a, pb);
}

// x and out may be the same buffer (an in-place projection): each element is
// read and written by the same thread, and the pointers carry no __restrict__.
__global__ void soft_threshold_kernel(const float *x, float *out, long long n, const Scalars *sc, int prob) {
  const float tau = sc->l1[prob].tau, tau_lo = sc->l1[prob].tau_lo;
  const long long stride = (long long)gridDim.x * blockDim.x;
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < n; i += stride)
    out[i] = soft_threshold(x[i], tau, tau_lo);
}

}  // namespace

cudaError_t launch_l1_level(const L1Args &a, int level, int grid, cudaStream_t st) {
  const auto aligned = [](const float *x) { return (reinterpret_cast<uintptr_t>(x) & 15) == 0; };
  const bool vec = a.n % 4 == 0 && aligned(a.x[0]) && (a.nprob < 2 || aligned(a.x[1]));
  const dim3 g(grid, a.nprob);
  const auto kernel = level == 1   ? (vec ? l1_hist_kernel<1, true> : l1_hist_kernel<1, false>)
                      : level == 2 ? (vec ? l1_hist_kernel<2, true> : l1_hist_kernel<2, false>)
                                   : (vec ? l1_hist_kernel<3, true> : l1_hist_kernel<3, false>);
  return launch_chained(kernel, g, kSelThreads, 0, st, a);
}

cudaError_t launch_soft_threshold(const float *x, float *out, long long n, const Scalars *sc, int prob,
                                  cudaStream_t st) {
  long long g = (n + 255) / 256;
  if (g < 1) g = 1;
  if (g > 4096) g = 4096;
  soft_threshold_kernel<<<(int)g, 256, 0, st>>>(x, out, n, sc, prob);
  return cudaGetLastError();
}

}  // namespace s3ttv
