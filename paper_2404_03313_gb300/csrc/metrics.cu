// Evaluation of a restored cube (Sec. IV-A) and the objective value of
// Prob. (S3TTV_denoising): the reductions behind s3ttv_quality and
// s3ttv_objective.  Cubes here are the caller's plain layout [N1][N2][N3]
// (band fastest).
// Every sum accumulates in FP64.
#include <math.h>

#include "s3ttv_internal.cuh"

namespace s3ttv {
namespace {

// Per-band sums of (u - ref)^2: thread t of a block owns bands t, t + 256, ...
// and walks the block's pixels, so a warp reads consecutive bands.
__global__ void __launch_bounds__(256) band_sqerr_kernel(const float *u, const float *ref, long long P, int N3,
                                                        long long chunk, double *out) {
  const long long p0 = blockIdx.x * chunk, p1 = p0 + chunk < P ? p0 + chunk : P;
  for (int b = threadIdx.x; b < N3; b += blockDim.x) {
    double s = 0.0;
    for (long long p = p0; p < p1; ++p) {
      const double d = (double)u[p * N3 + b] - (double)ref[p * N3 + b];
      s = fma(d, d, s);
    }
    if (p1 > p0) atomicAdd(out + b, s);
  }
}

// Spectral angle at every pixel: lanes stride over the bands of one pixel after the
// other, each keeping the sums of one of ppw <= 32 consecutive pixels, and then take
// one angle per lane: acos of the clipped normalized inner product (pi / 2 if one
// spectrum is zero, 0 if both are).  GB300 does about two FP64 operations a cycle
// and SM, whatever the number of active lanes, so an angle per warp (its square
// roots, division and acos for one pixel) cost more than the sums over the bands:
// 364 -> 172 us at 256 x 256 x 128.
__global__ void __launch_bounds__(256) sam_kernel(const float *u, const float *ref, long long P, int N3, int ppw,
                                                 float *map, double *sum) {
  __shared__ double red[8];
  const int lane = threadIdx.x & 31, warp = threadIdx.x >> 5;
  double acc = 0.0;
  for (long long p0 = (blockIdx.x * 8LL + warp) * ppw; p0 < P; p0 += gridDim.x * 8LL * ppw) {
    const int np = (int)min((long long)ppw, P - p0);
    double mdot = 0.0, mnu = 0.0, mnr = 0.0;
    for (int i = 0; i < np; ++i) {
      const float *pu = u + (p0 + i) * N3, *pr = ref + (p0 + i) * N3;
      double dot = 0.0, nu = 0.0, nr = 0.0;
      for (int b = lane; b < N3; b += 32) {
        const double x = pu[b], y = pr[b];
        dot = fma(x, y, dot);
        nu = fma(x, x, nu);
        nr = fma(y, y, nr);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) {
        dot += __shfl_xor_sync(kFull, dot, o);
        nu += __shfl_xor_sync(kFull, nu, o);
        nr += __shfl_xor_sync(kFull, nr, o);
      }
      if (lane == i) {
        mdot = dot;
        mnu = nu;
        mnr = nr;
      }
    }
    double ang;
    if (mnu > 0.0 && mnr > 0.0) {
      double c = mdot / (sqrt(mnu) * sqrt(mnr));
      c = c > 1.0 ? 1.0 : (c < -1.0 ? -1.0 : c);
      ang = acos(c);
    } else {
      ang = (mnu > 0.0 || mnr > 0.0) ? 1.5707963267948966 : 0.0;
    }
    if (lane < np) {
      if (map) map[p0 + lane] = (float)ang;
      acc += ang;
    }
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
  if (lane == 0) red[warp] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double s = 0.0;
    for (int w = 0; w < 8; ++w) s += red[w];
    atomicAdd(sum, s);
  }
}

// SSIM map of every band at every pixel whose 11 x 11 window lies inside the image,
// summed per band.  The Gaussian window is separable: a CTA takes 32 bands (a lane
// each) and kSsimCols output columns (a warp each) and walks down the rows.  Each
// row's x + y, x - y and their squares go through shared memory in FP64, are
// filtered along the row (11 products per moment), and added into the 11 output
// rows they reach (11 more), held in registers.  The four moments of the sum and the
// difference stand for the five of x and y: mx my = (p^2 - m^2) / 4,
// mx^2 + my^2 = (p^2 + m^2) / 2, and likewise for the (co)variances.
// Bound by the FP64 rate: about 92 operations and one division per voxel in place
// of 121 taps of seven; 15.98 -> 2.35 ms at 256 x 256 x 128.  Where fewer than
// kSsimCols output columns are left, the warps without one only help to fill the rows
// (400000 x 11 x 32: 65 -> 13.7 ms, 200000 x 12 x 4: 32.8 -> 7.7 ms with it and with
// as many row chunks as fill the SMs).
// A CTA is one group of bands, then one tile of columns, then one chunk of rows, all
// on grid.x: the other grid dimensions end at 65535, which a wide image exceeds.
constexpr int kSsimCols = 8;
constexpr int kSsimRowCols = kSsimCols + kSsimTaps - 1;
struct SsimWeights {
  double w[kSsimTaps];
};

__global__ void __launch_bounds__(32 * kSsimCols, 2) ssim_kernel(const float *u, const float *ref, int N1, int N2, int N3,
                                                               int b0, int nb, int rows, int gx, int gy, SsimWeights sw,
                                                               double *out) {
  __shared__ double row[2][kSsimRowCols][4][32];
  const int lane = threadIdx.x & 31, wp = threadIdx.x >> 5;
  const int Hv = N1 - kSsimTaps + 1, Wv = N2 - kSsimTaps + 1;
  const int xg = blockIdx.x % gx, xr = blockIdx.x / gx;
  const int b = min(b0 + xg * 32 + lane, b0 + nb - 1);  // lanes past the last band repeat it
  const int j0 = xr % gy * kSsimCols, i0 = xr / gy * rows;
  const int ncol = min(kSsimRowCols, N2 - j0);  // input columns of this CTA
  const bool mine = j0 + wp < Wv;               // this warp has an output column
  const int nout = min(rows, Hv - i0), nin = nout + kSsimTaps - 1;  // output and input rows of this CTA
  constexpr int LD = (kSsimRowCols + kSsimCols - 1) / kSsimCols;
  float xs[LD], ys[LD];
  auto fetch = [&](int r) {  // this warp's columns of input row r
#pragma unroll
    for (int e = 0; e < LD; ++e) {
      const int c = wp + e * kSsimCols;
      xs[e] = ys[e] = 0.f;
      if (c < ncol && r < nin) {
        const size_t o = ((size_t)(i0 + r) * N2 + j0 + c) * N3 + b;
        xs[e] = ref[o];
        ys[e] = u[o];
      }
    }
  };
  double acc[kSsimTaps][4] = {};  // partial windows of the 11 output rows a row reaches
  double total = 0.0;
  fetch(0);
  for (int base = 0; base < nin; base += kSsimTaps) {
#pragma unroll
    for (int ph = 0; ph < kSsimTaps; ++ph) {
      const int r = base + ph;
      if (r < nin) {  // CTA-uniform
        double(*buf)[4][32] = row[r & 1];
#pragma unroll
        for (int e = 0; e < LD; ++e) {
          const int c = wp + e * kSsimCols;
          if (c < ncol) {
            const double x = xs[e], y = ys[e], p = x + y, m = x - y;
            buf[c][0][lane] = p;
            buf[c][1][lane] = m;
            buf[c][2][lane] = p * p;
            buf[c][3][lane] = m * m;
          }
        }
        fetch(r + 1);
        __syncthreads();
        if (!mine) continue;  // (to the next row's barrier)
        double h[4] = {0.0, 0.0, 0.0, 0.0};
#pragma unroll
        for (int c = 0; c < kSsimTaps; ++c)
#pragma unroll
          for (int q = 0; q < 4; ++q) h[q] = fma(sw.w[c], buf[wp + c][q][lane], h[q]);
        // output row o sits in slot o mod 11 and takes input row r with weight r - o
#pragma unroll
        for (int k = 0; k < kSsimTaps; ++k) {
          if ((unsigned)(r - k) >= (unsigned)nout) continue;  // not an output row of this CTA
          const int s = (ph - k + kSsimTaps) % kSsimTaps;
#pragma unroll
          for (int q = 0; q < 4; ++q) acc[s][q] = k == 0 ? sw.w[0] * h[q] : fma(sw.w[k], h[q], acc[s][q]);
        }
        if (r >= kSsimTaps - 1) {  // output row r - 10 is whole
          const double *A = acc[(ph + 1) % kSsimTaps];
          const double p2 = A[0] * A[0], m2 = A[1] * A[1], vp = A[2] - p2, vm = A[3] - m2;
          const double C1 = 1e-4, C2 = 9e-4;  // (0.01 L)^2, (0.03 L)^2 with L = 1
          const double num = (0.5 * (p2 - m2) + C1) * (0.5 * (vp - vm) + C2);
          const double den = (0.5 * (p2 + m2) + C1) * (0.5 * (vp + vm) + C2);
          total += num / den;
        }
      }
    }
  }
  __syncthreads();
  double *red = &row[0][0][0][0];
  red[wp * 32 + lane] = total;  // (zero without a column)
  __syncthreads();
  if (wp == 0 && xg * 32 + lane < nb) {
    double s = 0.0;
    for (int w = 0; w < kSsimCols; ++w) s += red[w * 32 + lane];
    atomicAdd(out + (b - b0), s);
  }
}

// S3TTV(u) = sum_l ||X_l||_*, X_l the k^2 x 2N3 structure tensor of block l
// (eq. SSST: row a k + c is pixel ((p+a) mod N1, (q+c) mod N2), column 2b its
// D_v D_s u and 2b+1 its D_h D_s u at band b, periodic differences).  One CTA
// per block, all in FP64: the entries of X_l from the FP32 cube, the Gram
// G = X_l X_l^T accumulated in shared memory over chunks of kObjCW columns,
// then a one-sided (Hestenes) Jacobi on the rows of G (round-robin pairs, eight
// lanes per pair) until they are orthogonal: row r becomes lambda_r u_r^T, so
// sigma_r = sqrt(|row r|).  Rows below 1e-14 ||G||_F are numerical zeros.  The sigma of every block are summed into *out.
constexpr int kObjCW = 32;

__global__ void __launch_bounds__(256) objective_kernel(const float *u, int N1, int N2, int N3, int k, int stacked,
                                                       int open_s, int first_order, int parts, double tol,
                                                       int max_sweeps, double *out, unsigned *nonconv) {
  extern __shared__ double dsm[];
  const int n = stacked ? 2 * k * k : k * k, NP = n + (n & 1), W = stacked ? N3 : parts * N3;
  double *G = dsm;                 // NP x n
  double *X = dsm + (size_t)NP * n;  // n x kObjCW
  __shared__ double nrm[kMaxLargeK * kMaxLargeK];  // >= 2 kMaxStackedK^2 rows too
  __shared__ double s_fro2;
  const int tid = threadIdx.x, lane = tid & 31, warp = tid >> 5;
  const long long L = (long long)N1 * N2;
  double total = 0.0;
  for (long long l = blockIdx.x; l < L; l += gridDim.x) {
    const int p = (int)(l / N2), q = (int)(l - (long long)p * N2);
    for (int e = tid; e < NP * n; e += 256) G[e] = 0.0;
    for (int c0 = 0; c0 < W; c0 += kObjCW) {
      __syncthreads();
      for (int e = tid; e < n * kObjCW; e += 256) {
        const int r = e / kObjCW, cc = e - r * kObjCW, col = c0 + cc;
        double x = 0.0;
        // paper layout: row r is window pixel r, column parts * b + o; stacked:
        // row 2r + o is pixel r, column b; o = 0 vertical, 1 horizontal, 2
        // spectral (SSST)
        const int pr = stacked ? r >> 1 : r, o = stacked ? r & 1 : col % parts, b = stacked ? col : col / parts;
        if (col < W && !(open_s && b == N3 - 1)) {
          const int a = pr / k, c = pr - a * k;
          const int i = (p + a) % N1, j = (q + c) % N2;
          const int i1 = i + 1 == N1 ? 0 : i + 1, j1 = j + 1 == N2 ? 0 : j + 1, b1 = b + 1 == N3 ? 0 : b + 1;
          const size_t s00 = ((size_t)i * N2 + j) * N3;
          const size_t s10 = o ? ((size_t)i * N2 + j1) * N3 : ((size_t)i1 * N2 + j) * N3;
          if (o == 2) {  // SSST: D_s u
            x = (double)u[s00 + b1] - (double)u[s00 + b];
          } else if (first_order) {  // STV, SSST: D_v u or D_h u
            x = (double)u[s10 + b] - (double)u[s00 + b];
          } else {
            const double ds0 = (double)u[s00 + b1] - (double)u[s00 + b];
            const double ds1 = (double)u[s10 + b1] - (double)u[s10 + b];
            x = ds1 - ds0;
          }
        }
        X[r * kObjCW + cc] = x;
      }
      __syncthreads();
      for (int e = tid; e < n * n; e += 256) {
        const int i = e / n, j = e - i * n;
        if (j < i) continue;
        double s = 0.0;
        for (int c = 0; c < kObjCW; ++c) s = fma(X[i * kObjCW + c], X[j * kObjCW + c], s);
        G[i * n + j] += s;
      }
    }
    __syncthreads();
    if (tid == 0) s_fro2 = 0.0;
    __syncthreads();
    {
      double f2 = 0.0;
      for (int e = tid; e < n * n; e += 256) {
        const int i = e / n, j = e - i * n;
        if (j < i) G[i * n + j] = G[j * n + i];
        const double g = G[j <= i ? j * n + i : i * n + j];
        f2 = fma(g, g, f2);
      }
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) f2 += __shfl_xor_sync(kFull, f2, o);
      if (lane == 0) atomicAdd(&s_fro2, f2);
    }
    __syncthreads();
    // rows below 1e-14 ||G||_F are numerically zero (their sigma is below
    // 1e-7 sqrt(||G||_F)): they take part in no rotation and count as zero
    const double floor2 = 1e-28 * s_fro2;
    // one-sided Jacobi on the rows of G (row NP - 1 is zero when n is odd)
    bool converged = false;
    for (int sw = 0; sw < max_sweeps && !converged; ++sw) {
      int rotated = 0;
      for (int step = 0; step < NP - 1; ++step) {
        for (int base = 0; base < NP / 2; base += 32) {
          const int i = base + (tid >> 3), gl = tid & 7;
          const bool act = i < NP / 2;
          const int pa = act ? i : 0, pb = NP - 1 - pa;
          int xa = pa - 1 + step, xb = pb - 1 + step;
          xa -= xa >= NP - 1 ? NP - 1 : 0;
          xb -= xb >= NP - 1 ? NP - 1 : 0;
          const int ra = pa == 0 ? 0 : 1 + xa, rb = 1 + xb;
          double *A = G + (size_t)ra * n, *B = G + (size_t)rb * n;
          double d = 0.0, na = 0.0, nb = 0.0;
          if (act)
            for (int c = gl; c < n; c += 8) {
              d = fma(A[c], B[c], d);
              na = fma(A[c], A[c], na);
              nb = fma(B[c], B[c], nb);
            }
#pragma unroll
          for (int o = 4; o > 0; o >>= 1) {
            d += __shfl_xor_sync(kFull, d, o);
            na += __shfl_xor_sync(kFull, na, o);
            nb += __shfl_xor_sync(kFull, nb, o);
          }
          if (act && fmin(na, nb) > floor2 && fabs(d) > tol * sqrt(na * nb)) {
            // rotation that makes rows A and B orthogonal (Hestenes)
            const double zeta = (nb - na) / (2.0 * d);
            const double t = copysign(1.0, zeta) / (fabs(zeta) + sqrt(1.0 + zeta * zeta));
            const double cs = 1.0 / sqrt(1.0 + t * t), sn = cs * t;
            for (int c = gl; c < n; c += 8) {
              const double x = A[c], y = B[c];
              A[c] = cs * x - sn * y;
              B[c] = sn * x + cs * y;
            }
            rotated = 1;
          }
        }
        __syncthreads();
      }
      converged = !__syncthreads_or(rotated);
    }
    if (!converged && tid == 0) atomicAdd(nonconv, 1u);
    for (int r = warp; r < n; r += 8) {
      double s = 0.0;
      for (int c = lane; c < n; c += 32) s = fma(G[r * n + c], G[r * n + c], s);
#pragma unroll
      for (int o = 16; o > 0; o >>= 1) s += __shfl_xor_sync(kFull, s, o);
      if (lane == 0) nrm[r] = s > floor2 ? sqrt(sqrt(s)) : 0.0;  // |row r| = lambda_r; sigma_r = sqrt(lambda_r)
    }
    __syncthreads();
    if (tid == 0)
      for (int r = 0; r < n; ++r) total += nrm[r];
    __syncthreads();
  }
  if (tid == 0) atomicAdd(out, total);
}

// SSTV's objective ||D D_s u||_1 = sum |D_v D_s u| + |D_h D_s u| (periodic), FP64
__global__ void __launch_bounds__(256) sstv_l1_kernel(const float *u, int N1, int N2, int N3, double *out) {
  __shared__ double red[8];
  const long long N = (long long)N1 * N2 * N3;
  double acc = 0.0;
  for (long long e = blockIdx.x * 256LL + threadIdx.x; e < N; e += gridDim.x * 256LL) {
    const int b = (int)(e % N3);
    const long long pix = e / N3;
    const int i = (int)(pix / N2), j = (int)(pix % N2);
    const int i1 = i + 1 == N1 ? 0 : i + 1, j1 = j + 1 == N2 ? 0 : j + 1, b1 = b + 1 == N3 ? 0 : b + 1;
    const size_t p0 = (size_t)pix * N3, pv = ((size_t)i1 * N2 + j) * N3, ph = ((size_t)i * N2 + j1) * N3;
    const double ds0 = (double)u[p0 + b1] - (double)u[p0 + b];
    acc += fabs(((double)u[pv + b1] - (double)u[pv + b]) - ds0) + fabs(((double)u[ph + b1] - (double)u[ph + b]) - ds0);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    atomicAdd(out, t);
  }
}

// HSSTV's objective: || (D_v D_s u, D_h D_s u, omega D_v u, omega D_h u) || summed
// over voxels, l1 (l12 = 0) or the l2 norm of each voxel's four entries (l12 = 1)
__global__ void __launch_bounds__(256) hsstv_norm_kernel(const float *u, int N1, int N2, int N3, double omega, int l12,
                                                        double *out) {
  __shared__ double red[8];
  const long long N = (long long)N1 * N2 * N3;
  double acc = 0.0;
  for (long long e = blockIdx.x * 256LL + threadIdx.x; e < N; e += gridDim.x * 256LL) {
    const int b = (int)(e % N3);
    const long long pix = e / N3;
    const int i = (int)(pix / N2), j = (int)(pix % N2);
    const int i1 = i + 1 == N1 ? 0 : i + 1, j1 = j + 1 == N2 ? 0 : j + 1, b1 = b + 1 == N3 ? 0 : b + 1;
    const size_t p0 = (size_t)pix * N3, pv = ((size_t)i1 * N2 + j) * N3, ph = ((size_t)i * N2 + j1) * N3;
    const double ds0 = (double)u[p0 + b1] - (double)u[p0 + b];
    const double a0 = ((double)u[pv + b1] - (double)u[pv + b]) - ds0;
    const double a1 = ((double)u[ph + b1] - (double)u[ph + b]) - ds0;
    const double a2 = omega * ((double)u[pv + b] - (double)u[p0 + b]);
    const double a3 = omega * ((double)u[ph + b] - (double)u[p0 + b]);
    acc += l12 ? sqrt(a0 * a0 + a1 * a1 + a2 * a2 + a3 * a3) : fabs(a0) + fabs(a1) + fabs(a2) + fabs(a3);
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) acc += __shfl_xor_sync(kFull, acc, o);
  if ((threadIdx.x & 31) == 0) red[threadIdx.x >> 5] = acc;
  __syncthreads();
  if (threadIdx.x == 0) {
    double t = 0.0;
    for (int w = 0; w < 8; ++w) t += red[w];
    atomicAdd(out, t);
  }
}

}  // namespace

cudaError_t launch_hsstv_norm(const float *u, int N1, int N2, int N3, double omega, int l12, double *out, int grid,
                              cudaStream_t st) {
  hsstv_norm_kernel<<<grid, 256, 0, st>>>(u, N1, N2, N3, omega, l12, out);
  return cudaGetLastError();
}

cudaError_t launch_sstv_l1(const float *u, int N1, int N2, int N3, double *out, int grid, cudaStream_t st) {
  sstv_l1_kernel<<<grid, 256, 0, st>>>(u, N1, N2, N3, out);
  return cudaGetLastError();
}

cudaError_t launch_band_sqerr(const float *u, const float *ref, long long P, int N3, double *out, int grid,
                              cudaStream_t st) {
  const long long chunk = (P + grid - 1) / grid;
  band_sqerr_kernel<<<(unsigned)((P + chunk - 1) / chunk), 256, 0, st>>>(u, ref, P, N3, chunk, out);
  return cudaGetLastError();
}

cudaError_t launch_sam(const float *u, const float *ref, long long P, int N3, float *map, double *sum, int grid,
                       cudaStream_t st) {
  // 32 pixels a warp where that still gives every SM eight warps (grid: 8 CTAs per SM)
  long long ppw = (P + grid - 1) / grid;
  ppw = ppw < 1 ? 1 : ppw > 32 ? 32 : ppw;
  long long g = (P + 8 * ppw - 1) / (8 * ppw);
  if (g > grid) g = grid;
  sam_kernel<<<(unsigned)g, 256, 0, st>>>(u, ref, P, N3, (int)ppw, map, sum);
  return cudaGetLastError();
}

cudaError_t launch_ssim(const float *u, const float *ref, int N1, int N2, int N3, int b0, int nb, double *out,
                        int num_sms, cudaStream_t st) {
  // the Gaussian window of [Wang et al. 2004]: standard deviation 1.5, 11 x 11, sum 1
  SsimWeights sw;
  double tot = 0.0;
  for (int a = 0; a < kSsimTaps; ++a) {
    const double x = a - kSsimTaps / 2;
    sw.w[a] = exp(-(x * x) / (2.0 * 1.5 * 1.5));
    tot += sw.w[a];
  }
  for (double &x : sw.w) x /= tot;
  const int Hv = N1 - kSsimTaps + 1, Wv = N2 - kSsimTaps + 1;
  const int gx = (nb + 31) / 32, gy = (Wv + kSsimCols - 1) / kSsimCols;
  // rows per CTA: the fewest row steps of the busiest SM (two CTAs each); a CTA's
  // first 10 rows only feed its windows, at a bit over half a row's work
  int rows = Hv;
  double best = 1e300;
  const long long tiles = (long long)gx * gy, slots = 2LL * num_sms;
  for (long long n = 1; n <= Hv && (n == 1 || tiles * n <= 16 * slots); n += n < 64 ? 1 : n / 16) {
    const int r = (int)((Hv + n - 1) / n);
    const long long ctas = tiles * ((Hv + r - 1) / r);
    const double cost = (double)((ctas + slots - 1) / slots) * (r + 6.0);
    if (cost < best) {
      best = cost;
      rows = r;
    }
  }
  const long long ctas = tiles * ((Hv + rows - 1) / rows);
  if (ctas > 0x7fffffffLL) return cudaErrorInvalidValue;
  ssim_kernel<<<(unsigned)ctas, 32 * kSsimCols, 0, st>>>(u, ref, N1, N2, N3, b0, nb, rows, gx, gy, sw, out);
  return cudaGetLastError();
}

size_t objective_smem_bytes(int k, int stacked) {
  const int n = stacked ? 2 * k * k : k * k, NP = n + (n & 1);
  return sizeof(double) * ((size_t)NP * n + (size_t)n * kObjCW);
}

cudaError_t launch_objective(const float *u, int N1, int N2, int N3, int k, int stacked, int open_s,
                             int first_order, double *out, unsigned *nonconv, int grid, cudaStream_t st,
                             int parts) {
  const size_t smem = objective_smem_bytes(k, stacked);
  cudaError_t e = cudaFuncSetAttribute(objective_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)smem);
  if (e != cudaSuccess) return e;
  const long long L = (long long)N1 * N2;
  objective_kernel<<<(unsigned)(L < grid ? L : grid), 256, smem, st>>>(u, N1, N2, N3, k, stacked, open_s, first_order,
                                                                       parts, 1e-13, 60, out, nonconv);
  return cudaGetLastError();
}

}  // namespace s3ttv
