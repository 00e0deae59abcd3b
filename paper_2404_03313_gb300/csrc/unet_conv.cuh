// The 3 x 3 x 3 convolution of the warm-start network on the tcgen05 tensor
// cores (unet_conv.cu), as unet.cu calls it.
#pragma once
#include <cuda_bf16.h>
#include <cuda_runtime.h>

namespace s3ttv_net_detail {

typedef __nv_bfloat16 bf16;

constexpr unsigned long long kWaitNs = 4000000000ull;  // the waits' default time limit

struct Vol {
  int B, D, H, W;
};
__host__ __device__ inline int nvox(const Vol &g) { return g.B * g.D * g.H * g.W; }

// Output channels of one packed weight tile: the channels one work unit computes.
__host__ __device__ constexpr int conv_tile_n(int cout) { return cout % 64 == 0 ? 64 : 32; }

// Position of weight (output n, tap, input c) in the packed image that
// conv_launch reads: [n / NP][dy, dx][c / 8][2 - tz][n % NP][c % 8], so the bytes
// of one pipeline stage are contiguous and already in the shared-memory layout
// of the tensor cores' B operand.
__host__ __device__ inline long long conv_pack_index(int cin, int cout, int n, int tap, int c) {
  const int np = conv_tile_n(cout), tz = tap / 9, yx = tap - 9 * tz;
  return (((((long long)(n / np) * 9 + yx) * (cin / 8) + c / 8) * 3 + (2 - tz)) * np + n % np) * 8 + c % 8;
}

struct ConvArgs {
  const bf16 *x0;     // [V][c0], same size as the output
  const bf16 *x1;     // [V / 8][c1] read through nearest upsampling, its channels first; null: none
  const bf16 *w;      // packed weights (conv_pack_index)
  const float *bias;  // [cout] or null
  const bf16 *mask;   // [V][cout] or null: output zeroed where mask <= 0
  bf16 *y;            // [V][cout]
  int c0, c1, cout, relu;
  Vol g;
  int *err, *bad;     // host and device memory; set when a wait inside the kernel ran out
  unsigned long long wait_ns;  // time limit of such a wait (0: none is sat out)
  // With 32 output channels, optionally the network's head on the rounded outputs
  // f: h = Wh f + bh, (u, s, t) = (v + h0, h1, h2); hp holds Wh[3][32], then bh[3].
  // y may be null then: the layer's output is not stored.
  const float *hp = nullptr, *hv = nullptr;
  float *hu = nullptr, *hs = nullptr, *ht = nullptr;
};

// Opt in to the kernels' shared memory (once per device before conv_launch).
cudaError_t conv_prepare();
// y = conv(x) on `stream`.  Input channel counts (c0, c1): (32, 0), (64, 0),
// (128, 0), (64, 128), (32, 64); cout a multiple of 32.
cudaError_t conv_launch(const ConvArgs &a, int num_sms, cudaStream_t stream);

// dw[o][tap][c] += sum_p g[p][o] x[p + delta_tap][c] and db[o] += sum_p g[p][o], x the concatenation of x1
// (through nearest upsampling, its channels first) and x0 as in ConvArgs; channel
// counts multiples of 32.
struct WgradTcArgs {
  const bf16 *g;      // [V][cout]
  const bf16 *x0, *x1;
  float *dw;          // [cout][27][c1 + c0]
  float *db;          // [cout]
  int c0, c1, cout;
  Vol vol;
  int *err, *bad;
  unsigned long long wait_ns;
};
cudaError_t wgrad_prepare();
cudaError_t wgrad_launch(const WgradTcArgs &a, int num_sms, cudaStream_t stream);

}  // namespace s3ttv_net_detail
