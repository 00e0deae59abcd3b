// 3 x 3 x 3 convolution (zero padding, channels-last, BF16 in and out, FP32
// accumulation) of the warm-start network, forward and input gradient, as an
// implicit GEMM on the tcgen05 tensor cores: Y[p, n] = sum_{tap, c} X[p + delta_tap, c] W[n, tap, c].
//
// A CTA owns a column of the volume, 8 voxels along x (W) by 16 J along y (H),
// and marches along z (D).  Each plane of the column is copied into shared memory
// once, with its one-voxel halo, as [c / 8][y][x] pieces of 8 channels (16 bytes):
// the no-swizzle K-major operand layout, in which an 8-row core matrix is 8
// voxels of a row of x, the next one is the next y (SBO = one halo row), and a
// tap's shift in y and x is an offset of the descriptor's start address.  So the
// 27 neighbours of a voxel cost no copies and no address arithmetic.
//
// Plane p serves three output planes: z = p - 1 with the taps dz = +1, z = p with
// dz = 0, z = p + 1 with dz = -1.  The three have the same A operand for equal
// (dy, dx), so one tcgen05.mma covers them with N = 3 NT columns: the TMEM
// accumulators of consecutive z sit in consecutive column slots (a ring; where it
// wraps, the instruction is split in two) and the B operand holds the three taps'
// weights one below the other.  That triples the work per byte of A that the
// tensor cores read from shared memory, which is what bounds M = 128 with N = 32.
// Every accumulator still sums its products tap by tap and channel by channel.
//
// Volumes that do not fill their tiles (fewer than 8 voxels along x or 16 along y: small
// crops, whose coarse levels are 1 to 4 voxels wide) share them: a unit then takes a
// mosaic of mx by my pieces, a piece being a chunk of planes of one volume, laid side by
// side with one column or row of zeros between, which is the zero padding of both.
// Every voxel sums the same products in the same order.  16384 crops of 4^3: forward 6.44
// -> 0.68 ms, training gradient 27.0 -> 3.1 (2.23 and 11.5 by gathering kernels, which
// packed voxels across volumes); 4096 of 8^3: 3.36 -> 1.02 and 14.8 -> 4.6.
//
// Roles: warps 0-7 read finished accumulators (two warps per quarter of the TMEM
// lanes, taking turns at blocks of 32 columns), apply bias, ReLU and mask and store
// BF16; warps 8 and 9 issue the MMAs, one per 128-voxel tile (with one warp for both,
// issuing took longer than the products: 3500 cycles per plane of 256 voxels and 32
// channels); warp 10 copies weights (cp.async.bulk, a ring of (dy, dx, channel
// slice) stages; with 32 input channels all of them once, a CTA keeps its tile of
// output channels); warps 11-18 copy planes (cp.async with zero fill outside the volume, nearest upsampling
// by halving the coordinates).  Every wait has a time limit, after which the CTA
// ends its roles, waits for its MMAs and copies in flight, frees its TMEM, sets the
// error flags and ends.
#include "unet_conv.cuh"

#include "chain.cuh"

#include <stdint.h>

#include <type_traits>

namespace s3ttv_net_detail {
using s3ttv::chained;
using s3ttv::launch_chained;
namespace {

constexpr int kEpiWarps = 8, kMmaWarp = 8, kWWarp = 10, kLoadWarp0 = 11, kLoadWarps = 8;
constexpr int kThreads = (kLoadWarp0 + kLoadWarps) * 32;
constexpr int kTX = 8, kTY = 16;   // a 128-voxel tile: x by y
constexpr int kPX = kTX + 2;       // halo row
constexpr int kMaxAStages = 4, kMaxWStages = 16, kMaxSlots = 8;
constexpr int kTmemCols = 512;
constexpr int kSmemMax = 227 * 1024 - 2048;
constexpr int kSmemMin = 120 * 1024;  // one CTA per SM: each takes all of TMEM

// Input channels per weight stage, and whether a CTA keeps all its weights in
// shared memory (9 stages of 6 or 12 KB at 32 input channels).
__host__ __device__ constexpr int stage_channels(int cin) { return cin > 96 ? 64 : cin; }
__host__ __device__ constexpr bool weights_resident(int cin) { return cin == 32; }

struct Plan {
  int J;               // 128-voxel tiles along y per unit
  int nt, slots, sh;   // output channels per unit, accumulator slots of the TMEM ring (1 << sh)
  int lz, nzc;         // output planes per unit, units along z
  int mx, my;          // pieces along x and y that share a unit's tiles (1, 1: none do)
  int tx, ty, nn;      // tiles along x, y; channel tiles
  int units;           // spatial units; each is computed once per channel tile
  int a_stages, w_stages;
  int lbo;             // bytes between the 8-channel pieces of a plane
  int smem;
};

__device__ __forceinline__ uint32_t smem_u32(const void *p) { return (uint32_t)__cvta_generic_to_shared(p); }

__device__ __forceinline__ void mbar_init(uint32_t bar, int count) {
  asm volatile("mbarrier.init.shared::cta.b64 [%0], %1;\n" ::"r"(bar), "r"(count) : "memory");
}
__device__ __forceinline__ void mbar_arrive(uint32_t bar) {
  asm volatile("mbarrier.arrive.shared::cta.b64 _, [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void mbar_expect(uint32_t bar, uint32_t bytes) {
  asm volatile("mbarrier.arrive.expect_tx.shared::cta.b64 _, [%0], %1;\n" ::"r"(bar), "r"(bytes) : "memory");
}
__device__ __forceinline__ bool mbar_try(uint32_t bar, uint32_t parity) {
  uint32_t ok;
  asm volatile(
      "{\n .reg .pred p;\n mbarrier.try_wait.parity.shared::cta.b64 p, [%1], %2;\n selp.b32 %0, 1, 0, p;\n}\n"
      : "=r"(ok)
      : "r"(bar), "r"(parity)
      : "memory");
  return ok != 0;
}
__device__ __forceinline__ unsigned long long now_ns() {
  unsigned long long t;
  asm volatile("mov.u64 %0, %globaltimer;" : "=l"(t));
  return t;
}
// Wait for a barrier's phase; false when the time limit (in ns) or another role's
// failure (stop) ends the wait.
__device__ __forceinline__ bool mbar_wait(uint32_t bar, uint32_t parity, volatile int *stop, unsigned long long limit) {
  if (mbar_try(bar, parity)) return true;
  const unsigned long long t0 = now_ns();
  while (true) {
#pragma unroll 1  // (unrolled into every role's loops, the tries crowd the instruction cache)
    for (int i = 0; i < 32; ++i)
      if (mbar_try(bar, parity)) return true;
    if (*stop) return false;
    if (now_ns() - t0 > limit) {
      *stop = 1;
      return false;
    }
  }
}

// (.ca: through L1.  With .cg the copies backed up in the load/store unit and held up
// the epilogue's stores as well: 580 against 470 us for the 192-channel layer.)
__device__ __forceinline__ void cp16(uint32_t smem, const void *gmem, int bytes) {
  asm volatile("cp.async.ca.shared.global [%0], [%1], 16, %2;\n" ::"r"(smem), "l"(gmem), "r"(bytes));
}
__device__ __forceinline__ void bulk_copy(uint32_t smem, const void *gmem, uint32_t bytes, uint32_t bar) {
  asm volatile("cp.async.bulk.shared::cluster.global.mbarrier::complete_tx::bytes [%0], [%1], %2, [%3];\n" ::"r"(smem),
               "l"(gmem), "r"(bytes), "r"(bar)
               : "memory");
}
// A value that is the same in every lane, as the compiler can see it: operands of
// tcgen05.mma live in uniform registers, and moving each one there before every
// instruction cost more than the instruction (130 against 56 cycles at N = 96).
__device__ __forceinline__ uint32_t uniform(uint32_t x) { return __shfl_sync(0xffffffffu, x, 0); }

// One lane of a converged warp (the same one each time).
__device__ __forceinline__ bool elect_one() {
  uint32_t r;
  asm volatile("{\n .reg .pred p;\n elect.sync _|p, 0xffffffff;\n selp.b32 %0, 1, 0, p;\n}\n" : "=r"(r));
  return r != 0;
}
// Wait for what is in flight, so that no MMA or copy outlives the CTA, its shared
// memory or its TMEM, whichever role failed.
__device__ __forceinline__ void mbar_drain(uint32_t bar, uint32_t parity, volatile int *stop) {
  for (int i = 0; i < 32; ++i)
    if (mbar_try(bar, parity)) return;
  const unsigned long long t0 = now_ns();  // (reading the clock takes about a microsecond)
  while (!mbar_try(bar, parity))
    if (now_ns() - t0 > kWaitNs) {
      *stop = 1;
      return;
    }
}
// The operand descriptors come as their low and high words: the high words are
// constants and only the low ones (start address) move.  add = 0: D = A B, else
// D += A B.
__device__ __forceinline__ void mma_f16(uint32_t d, uint32_t alo, uint32_t ahi, uint32_t blo, uint32_t bhi,
                                        uint32_t idesc, uint32_t add = 1u) {
  asm volatile(
      "{\n .reg .pred p;\n .reg .b64 a, b;\n setp.ne.b32 p, %6, 0;\n mov.b64 a, {%1, %2};\n mov.b64 b, {%3, %4};\n"
      " tcgen05.mma.cta_group::1.kind::f16 [%0], a, b, %5, p;\n}\n" ::"r"(d),
      "r"(alo), "r"(ahi), "r"(blo), "r"(bhi), "r"(idesc), "r"(add)
      : "memory");
}
__device__ __forceinline__ void mma_commit(uint32_t bar) {
  asm volatile("tcgen05.commit.cta_group::1.mbarrier::arrive::one.shared::cluster.b64 [%0];\n" ::"r"(bar) : "memory");
}
__device__ __forceinline__ void tmem_ld32(uint32_t (&v)[32], uint32_t addr) {
  asm volatile(
      "tcgen05.ld.sync.aligned.32x32b.x32.b32 "
      "{%0,%1,%2,%3,%4,%5,%6,%7,%8,%9,%10,%11,%12,%13,%14,%15,%16,%17,%18,%19,%20,%21,%22,%23,%24,%25,%26,%27,%28,%29,"
      "%30,%31}, [%32];\n"
      : "=r"(v[0]), "=r"(v[1]), "=r"(v[2]), "=r"(v[3]), "=r"(v[4]), "=r"(v[5]), "=r"(v[6]), "=r"(v[7]), "=r"(v[8]),
        "=r"(v[9]), "=r"(v[10]), "=r"(v[11]), "=r"(v[12]), "=r"(v[13]), "=r"(v[14]), "=r"(v[15]), "=r"(v[16]),
        "=r"(v[17]), "=r"(v[18]), "=r"(v[19]), "=r"(v[20]), "=r"(v[21]), "=r"(v[22]), "=r"(v[23]), "=r"(v[24]),
        "=r"(v[25]), "=r"(v[26]), "=r"(v[27]), "=r"(v[28]), "=r"(v[29]), "=r"(v[30]), "=r"(v[31])
      : "r"(addr));
  asm volatile("tcgen05.wait::ld.sync.aligned;\n" ::: "memory");
}
__device__ __forceinline__ void fence_before() { asm volatile("tcgen05.fence::before_thread_sync;\n" ::: "memory"); }
__device__ __forceinline__ void fence_after() { asm volatile("tcgen05.fence::after_thread_sync;\n" ::: "memory"); }

// No-swizzle K-major operand descriptor.  Low word: start address and the bytes
// between the two 8-channel halves of a K = 16 step (lbo); high word: the bytes
// between 8-row groups (sbo) and the descriptor version.
__device__ __forceinline__ uint32_t desc_lo(uint32_t addr, uint32_t lbo) {
  return ((lbo >> 4) << 16) | ((addr & 0x3ffffu) >> 4);
}
__device__ __forceinline__ uint32_t desc_hi(uint32_t sbo) { return (1u << 14) | (sbo >> 4); }

// 32 bytes (a whole L2 sector) in one store
__device__ __forceinline__ void st_sector(void *p, const uint32_t *v) {
  asm volatile("st.global.v8.b32 [%0], {%1, %2, %3, %4, %5, %6, %7, %8};\n" ::"l"(p), "r"(v[0]), "r"(v[1]), "r"(v[2]),
               "r"(v[3]), "r"(v[4]), "r"(v[5]), "r"(v[6]), "r"(v[7])
               : "memory");
}

// One work unit: an (x, y) column and a chunk of z of a volume, or of a mosaic of
// pieces, whose planes count from each piece's first.
struct Unit {
  int b, x0, y0, z0, z1;  // the volume, or a mosaic's first piece; output planes [z0, z1)
  int p0, p1;             // input planes [p0, p1]
};
template <bool MOSAIC>
__device__ __forceinline__ Unit unit_at(int u, const Plan &pl, const Vol &g) {
  Unit t;
  t.x0 = (u % pl.tx) * kTX;
  u /= pl.tx;
  t.y0 = (u % pl.ty) * kTY * pl.J;
  u /= pl.ty;
  if (MOSAIC) {  // (lz divides D)
    t.b = u * pl.mx * pl.my;
    t.z0 = 0;
    t.z1 = pl.lz;
    t.p0 = pl.nzc > 1 ? -1 : 0;
    t.p1 = pl.nzc > 1 ? pl.lz : pl.lz - 1;
  } else {
    t.z0 = (u % pl.nzc) * pl.lz;
    t.b = u / pl.nzc;
    t.z1 = min(t.z0 + pl.lz, g.D);
    t.p0 = max(t.z0 - 1, 0);
    t.p1 = min(t.z1, g.D - 1);
  }
  return t;
}
// The piece and the position in it of column x and row y of the mosaic of piece q on;
// false between pieces and outside.
__device__ __forceinline__ bool in_mosaic(int q, int mx, int my, int pieces, const Vol &g, int &piece, int &y, int &x) {
  const int cx = (unsigned)x / (unsigned)(g.W + 1), cy = (unsigned)y / (unsigned)(g.H + 1);  // (-1: not below mx, my)
  piece = q + cy * mx + cx;
  x -= cx * (g.W + 1);
  y -= cy * (g.H + 1);
  return cx < mx && cx >= 0 && cy < my && cy >= 0 && x >= 0 && x < g.W && y >= 0 && y < g.H && piece < pieces;
}

template <int C0, int C1, int J, bool MOSAIC>
__global__ void __launch_bounds__(kThreads, 1) conv_tc_kernel(ConvArgs a, Plan pl) {
  chained();
  constexpr int CIN = C0 + C1, NQ = CIN / 8;
  constexpr int CS = stage_channels(CIN), NS = CIN / CS;  // channels per weight stage
  constexpr bool RES = weights_resident(CIN);
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t bars[2 * kMaxAStages + 2 * kMaxWStages + 2 * kMaxSlots + 2];
  __shared__ __align__(16) float s_bias[192];
  __shared__ __align__(16) float s_head[100];  // the head's weights and biases
  __shared__ uint32_t s_tmem;
  __shared__ int s_stop[2];  // a wait has run out; the weight copies have ended
  const int tid = threadIdx.x, lane = tid & 31;
  // broadcasts, so that the compiler knows the role and TMEM address as warp-uniform
  // and keeps the MMA loop's operands in uniform registers
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const Vol g = a.g;
  const int NT = pl.nt, S = pl.slots, nt_tile = blockIdx.x % pl.nn;  // this CTA's tile of output channels
  const int u0 = blockIdx.x / pl.nn, du = gridDim.x / pl.nn;
  const uint32_t a_bytes = (uint32_t)pl.lbo * NQ, w_bytes = (uint32_t)(CS / 8) * 3 * NT * 16;
  const uint32_t sA = smem_u32(smem), sW = sA + a_bytes * pl.a_stages;
  const uint32_t bar0 = smem_u32(bars);
  auto a_full = [&](int s) { return bar0 + 8u * s; };
  auto a_empty = [&](int s) { return bar0 + 8u * (kMaxAStages + s); };
  auto w_full = [&](int s) { return bar0 + 8u * (2 * kMaxAStages + s); };
  auto w_empty = [&](int s) { return bar0 + 8u * (2 * kMaxAStages + kMaxWStages + s); };
  auto c_full = [&](int s) { return bar0 + 8u * (2 * kMaxAStages + 2 * kMaxWStages + s); };
  auto c_empty = [&](int s) { return bar0 + 8u * (2 * kMaxAStages + 2 * kMaxWStages + kMaxSlots + s); };
  const uint32_t drained = c_empty(kMaxSlots);  // (two): a tile's MMAs are done

  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&s_tmem)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (tid == kMmaWarp * 32) {
    for (int s = 0; s < kMaxAStages; ++s) {
      mbar_init(a_full(s), kLoadWarps);
      mbar_init(a_empty(s), J);
    }
    for (int s = 0; s < kMaxWStages; ++s) {
      mbar_init(w_full(s), 1);
      mbar_init(w_empty(s), J);
    }
    for (int s = 0; s < kMaxSlots; ++s) {
      mbar_init(c_full(s), J);
      mbar_init(c_empty(s), kEpiWarps);
    }
    mbar_init(drained, 1);
    mbar_init(drained + 8, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    s_stop[0] = a.wait_ns == 0;  // no wait is sat out
    s_stop[1] = 0;
  }
  for (int i = tid; i < a.cout; i += kThreads) s_bias[i] = a.bias ? a.bias[i] : 0.f;
  if (a.hp && tid < 99) s_head[tid] = a.hp[tid];
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);
  volatile int *stop = s_stop;
  const unsigned long long limit = a.wait_ns;

  if (warp < kEpiWarps) {
    // ---- epilogue: slot k of the ring holds output plane k, k + S, ... of this CTA ----
    const int quarter = warp & 3, turn = warp >> 2;
    const uint32_t lane_base = tmem + ((uint32_t)(quarter * 32) << 16);
    const int row = quarter * 32 + lane, ry = row >> 3, rx = row & 7, nblk = NT / 32;
    int slot = 0, job = 0;
    uint32_t phase = 0;
    bool ok = true;
    for (int u = u0; u < pl.units && ok; u += du) {
      const Unit t = unit_at<MOSAIC>(u, pl, g);
      int vox0[J];  // (MOSAIC) this thread's voxel in plane 0 of each tile, -1: none
      if (MOSAIC) {
#pragma unroll
        for (int sub = 0; sub < J; ++sub) {
          int y = t.y0 + sub * kTY + ry, x = t.x0 + rx, q;
          vox0[sub] = in_mosaic(t.b, pl.mx, pl.my, g.B * pl.nzc, g, q, y, x)
                          ? ((q / pl.nzc * g.D + q % pl.nzc * pl.lz) * g.H + y) * g.W + x
                          : -1;
        }
      }
      for (int z = t.z0; z < t.z1; ++z) {
        ok = __all_sync(0xffffffffu, mbar_wait(c_full(slot), phase, stop, limit));
        if (!ok) break;
        fence_after();
        // this warp's blocks of the tile are first, first + 2, ...; the slot is free
        // for the next tile as soon as the last one is in registers
        const int nb = J * nblk, first = (job & 1) ^ turn;
        job += nb;
        if (first >= nb) {
          if (lane == 0) mbar_arrive(c_empty(slot));
        }
        for (int e = first; e < nb; e += 2) {
          const int sub = e / nblk, c0 = (e - sub * nblk) * 32;
          const uint32_t col = lane_base + (uint32_t)((sub * S + slot) * NT + c0);
          uint32_t v[32];
          tmem_ld32(v, col);
          if (e + 2 >= nb) {
            fence_before();
            __syncwarp();
            if (lane == 0) mbar_arrive(c_empty(slot));
          }
          const int y = t.y0 + sub * kTY + ry, x = t.x0 + rx, v0 = MOSAIC ? (J == 2 && sub ? vox0[J - 1] : vox0[0]) : 0;
          if (MOSAIC ? v0 >= 0 : y < g.H && x < g.W) {
            const size_t vox = MOSAIC ? v0 + z * g.H * g.W : (((size_t)t.b * g.D + z) * g.H + y) * g.W + x;
            const int n0 = nt_tile * NT + c0;
            const size_t o = vox * a.cout + n0;
            uint32_t ow[16];
#pragma unroll
            for (int i = 0; i < 8; ++i) {
              const float4 b4 = *reinterpret_cast<const float4 *>(s_bias + n0 + 4 * i);
              float f[4] = {__uint_as_float(v[4 * i]) + b4.x, __uint_as_float(v[4 * i + 1]) + b4.y,
                            __uint_as_float(v[4 * i + 2]) + b4.z, __uint_as_float(v[4 * i + 3]) + b4.w};
              if (a.relu) {
#pragma unroll
                for (int j = 0; j < 4; ++j) f[j] = fmaxf(f[j], 0.f);
              }
              const __nv_bfloat162 h0 = __floats2bfloat162_rn(f[0], f[1]), h1 = __floats2bfloat162_rn(f[2], f[3]);
              ow[2 * i] = *reinterpret_cast<const uint32_t *>(&h0);
              ow[2 * i + 1] = *reinterpret_cast<const uint32_t *>(&h1);
            }
            if (a.mask) {
              const uint4 *mp = reinterpret_cast<const uint4 *>(a.mask + o);
#pragma unroll
              for (int q = 0; q < 4; ++q) {
                const uint4 m4 = mp[q];
                const uint32_t mw[4] = {m4.x, m4.y, m4.z, m4.w};
#pragma unroll
                for (int i = 0; i < 4; ++i) {
                  const __nv_bfloat162 m = *reinterpret_cast<const __nv_bfloat162 *>(&mw[i]);
                  ow[4 * q + i] &= (__bfloat162float(m.x) > 0.f ? 0xffffu : 0u) |
                                   (__bfloat162float(m.y) > 0.f ? 0xffff0000u : 0u);
                }
              }
            }
            if (a.y) {
              st_sector(a.y + o, ow);
              st_sector(a.y + o + 16, ow + 8);
            }
            if (a.hp) {  // channel by channel, as a kernel of its own would sum
              float h0 = s_head[96], h1 = s_head[97], h2 = s_head[98];
#pragma unroll
              for (int i = 0; i < 8; ++i) {
                const float4 w0 = *reinterpret_cast<const float4 *>(s_head + 4 * i);
                const float4 w1 = *reinterpret_cast<const float4 *>(s_head + 32 + 4 * i);
                const float4 w2 = *reinterpret_cast<const float4 *>(s_head + 64 + 4 * i);
                const float2 fa = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&ow[2 * i]));
                const float2 fb = __bfloat1622float2(*reinterpret_cast<const __nv_bfloat162 *>(&ow[2 * i + 1]));
                h0 = fmaf(w0.w, fb.y, fmaf(w0.z, fb.x, fmaf(w0.y, fa.y, fmaf(w0.x, fa.x, h0))));
                h1 = fmaf(w1.w, fb.y, fmaf(w1.z, fb.x, fmaf(w1.y, fa.y, fmaf(w1.x, fa.x, h1))));
                h2 = fmaf(w2.w, fb.y, fmaf(w2.z, fb.x, fmaf(w2.y, fa.y, fmaf(w2.x, fa.x, h2))));
              }
              a.hu[vox] = a.hv[vox] + h0;
              a.hs[vox] = h1;
              a.ht[vox] = h2;
            }
          }
          __syncwarp();
        }
        if (++slot == S) {
          slot = 0;
          phase ^= 1;
        }
      }
    }
  } else if (warp < kMmaWarp + 2) {
    // ---- MMA issue: the whole warp runs the (uniform) loop, one lane issues ----
    if (warp - kMmaWarp < J) {
      const int sub = warp - kMmaWarp;  // this warp's 128-voxel tile
      const uint32_t idesc0 = (1u << 4) | (1u << 7) | (1u << 10) | (8u << 24);  // F32 <- BF16 x BF16, M = 128
      const uint32_t id0 = idesc0 | ((uint32_t)(NT >> 3) << 17);
      const uint32_t b_lbo = 3u * NT * 16, ahi = desc_hi(kPX * 16), bhi = desc_hi(128);
      const uint32_t ak = 2u * pl.lbo >> 4, bk = 2u * b_lbo >> 4;  // descriptor steps of 16 channels
      const uint32_t wstep = w_bytes >> 4;                          // and of a weight stage
      const uint32_t dsub = tmem + (uint32_t)(sub * S * NT);       // the tile's accumulator ring
      const bool issue = elect_one();
      int as = 0, ws = 0, slot0 = 0;        // slot0: the slot of the unit's first output plane
      uint32_t aph = 0, wph = 0, cph = 1;   // cph: the parity to wait for in the ring turn slot0 is in
      bool ok = true;
      // (a wait for weights that fails ends this loop at its next other wait, or lets it run
      // on to its end over whatever lies there: the result is reported as failed)
      if (RES)
        for (int st = 0; st < 9; ++st) mbar_wait(w_full(st), 0, stop, limit);
      for (int u = u0; u < pl.units && ok; u += du) {
        const Unit t = unit_at<MOSAIC>(u, pl, g);
        const int bottom = MOSAIC ? t.p0 : 0, top = MOSAIC ? t.p1 : g.D - 1;  // outermost planes there are
        for (int p = t.p0; p <= t.p1; ++p) {
          const int zlo = max(p - 1, t.z0), zhi = min(p + 1, t.z1 - 1), n = zhi - zlo + 1;
          bool got = true;
          for (int z = zlo; z <= zhi; ++z) {
            if (p != max(z - 1, bottom)) continue;  // not the first plane that adds into z
            // c_empty(s) completes its phase k - 1 when the slot is free for its k-th use
            const int k = slot0 + (z - t.z0);
            got = mbar_wait(c_empty(k & (S - 1)), cph ^ (uint32_t)((k >> pl.sh) & 1), stop, limit) && got;
          }
          got = mbar_wait(a_full(as), aph, stop, limit) && got;
          ok = __all_sync(0xffffffffu, got);
          if (!ok) break;
          fence_after();
          const int s0 = (slot0 + zlo - t.z0) & (S - 1), n1 = min(n, S - s0);
          // (uniform() tells the compiler what it cannot see through the divisions)
          const bool wrap = uniform(n1 < n ? 1u : 0u) != 0u;
          const uint32_t id1 = uniform(idesc0 | ((uint32_t)(n1 * NT >> 3) << 17));
          const uint32_t id2 = uniform(idesc0 | ((uint32_t)((n - n1) * NT >> 3) << 17));
          const uint32_t alo = uniform(desc_lo(sA + a_bytes * as + (uint32_t)(sub * kTY * kPX) * 16, pl.lbo));
          // rows of B: the lowest output plane's block first (block 0 is dz = +1)
          const uint32_t blo0 = uniform(desc_lo(sW + (uint32_t)((zlo - (p - 1)) * NT) * 16, b_lbo));
          const uint32_t d1 = uniform(dsub + (uint32_t)(s0 * NT)), bw = uniform((uint32_t)(n1 * NT));
          uint32_t tap = alo;  // the A descriptor of the tap's shift in y and x
          // (rolled: straight-line code for nine taps outruns the instruction cache)
#pragma unroll 1
          for (int yx = 0; yx < 9; ++yx) {
#pragma unroll
            for (int sl = 0; sl < NS; ++sl) {
              // (a failed wait for weights still sits the copy out, unless none will come: its
              // stage may not be armed again before it lands; nothing else is checked here, where
              // a vote or a flag carried along cost 2 to 10%)
              if (!RES && !mbar_wait(w_full(ws), wph, stop, limit))
                for (unsigned i = 0; i < (1u << 26) && !mbar_try(w_full(ws), wph) && !stop[1]; ++i) {
                }
              const uint32_t blo = RES ? blo0 + wstep * yx : uniform(blo0 + wstep * ws);
              const uint32_t a0 = tap + (uint32_t)(sl * (CS / 16)) * ak;
              if (issue) {
                const bool start = sl == 0 && yx == 0;
                if (start)
                  // the plane's first step, output plane by output plane: one that no
                  // plane has added into yet is written instead of added to
                  for (int i = 0; i < n; ++i)
                    mma_f16(dsub + (uint32_t)(((s0 + i) & (S - 1)) * NT), a0, ahi, blo + i * NT, bhi, id0,
                            p == max(zlo + i - 1, bottom) ? 0u : 1u);
#pragma unroll
                for (int kk = 0; kk < CS / 16; ++kk)
                  if (kk > 0 || !start) mma_f16(d1, a0 + kk * ak, ahi, blo + kk * bk, bhi, id1);
                if (wrap) {
#pragma unroll
                  for (int kk = 0; kk < CS / 16; ++kk)
                    if (kk > 0 || !start) mma_f16(dsub, a0 + kk * ak, ahi, blo + kk * bk + bw, bhi, id2);
                }
                if (!RES) mma_commit(w_empty(ws));
              }
              __syncwarp();
              if (!RES && ++ws == pl.w_stages) {
                ws = 0;
                wph ^= 1;
              }
            }
            tap += yx % 3 == 2 ? kPX - 2 : 1;
          }
          if (issue) {
            mma_commit(a_empty(as));
            // the planes that p completes: p - 1, and p itself if it is the last
            for (int z = zlo; z <= zhi; ++z)
              if (min(z + 1, top) == p) mma_commit(c_full((slot0 + z - t.z0) & (S - 1)));
          }
          __syncwarp();
          if (++as == pl.a_stages) {
            as = 0;
            aph ^= 1;
          }
        }
        const int k = slot0 + (t.z1 - t.z0);
        cph ^= (uint32_t)((k >> pl.sh) & 1);
        slot0 = k & (S - 1);
      }
      if (issue) mma_commit(drained + 8u * sub);
    }
  } else if (warp == kWWarp) {
    if (lane == 0) {
      // ---- weight copies ----
      int ws = 0;
      uint32_t ph = 1;
      bool ok = true;
      unsigned issued = 0;
      auto stage_src = [&](int yx, int sl) {
        return a.w + (((size_t)(nt_tile * 9 + yx) * NQ + sl * (CS / 8)) * 3) * NT * 8;
      };
      if (RES) {
        for (int st = 0; st < 9 * NS; ++st) {
          mbar_expect(w_full(st), w_bytes);
          bulk_copy(sW + w_bytes * st, stage_src(st / NS, st % NS), w_bytes, w_full(st));
          ++issued;
        }
      } else {
        for (int u = u0; u < pl.units && ok; u += du) {
          const Unit t = unit_at<MOSAIC>(u, pl, g);
          for (int p = t.p0; p <= t.p1 && ok; ++p)
            for (int st = 0; st < 9 * NS; ++st) {
              ok = mbar_wait(w_empty(ws), ph, stop, limit);
              if (!ok) break;
              mbar_expect(w_full(ws), w_bytes);
              bulk_copy(sW + w_bytes * ws, stage_src(st / NS, st % NS), w_bytes, w_full(ws));
              ++issued;
              if (++ws == pl.w_stages) {
                ws = 0;
                ph ^= 1;
              }
            }
        }
      }
      for (unsigned i = issued > (unsigned)pl.w_stages ? issued - pl.w_stages : 0u; i < issued; ++i)
        mbar_drain(w_full(i % pl.w_stages), (i / pl.w_stages) & 1, stop);
      stop[1] = 1;
    }
  } else {
    // ---- plane copies ----
    // A thread keeps its 8-channel piece q and its NI voxels of the plane, whose
    // offsets (-1 outside the volume) it computes once per unit.
    constexpr int LT = (kLoadWarps * 32) / NQ * NQ, VS = LT / NQ, NV = kPX * (kTY * J + 2), NI = (NV + VS - 1) / VS;
    const int lt = tid - kLoadWarp0 * 32, q = lt % NQ, v0 = lt < LT ? lt / NQ : NV;
    const bool half = C1 && q < C1 / 8;  // this piece comes from the half-size input
    const int hs = half ? 1 : 0, C = half ? C1 : C0, Hs = g.H >> hs, Ws = g.W >> hs, Ds = g.D >> hs;
    const bf16 *base = half ? a.x1 + q * 8 : a.x0 + (q * 8 - C1);
    auto landed = [&](int s) {  // this warp's copies into stage s are visible to the tensor cores
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(a_full(s));
    };
    int as = 0, prev = -1;  // prev: a stage whose copies are in flight
    uint32_t ph = 1;
    bool ok = true;
    for (int u = u0; u < pl.units && ok; u += du) {
      const Unit t = unit_at<MOSAIC>(u, pl, g);
      int off[NI];
      using Mask = typename std::conditional<(NI > 32), unsigned long long, unsigned>::type;
      Mask zfirst = 0, zlast = 0;  // (MOSAIC) the voxels of pieces that start, end their volume
#pragma unroll
      for (int i = 0; i < NI; ++i) {
        const int v = v0 + i * VS, vy = v / kPX, vx = v - vy * kPX;
        int y = t.y0 + vy - 1, x = t.x0 + vx - 1;
        if (MOSAIC) {
          int q;
          const bool in = in_mosaic(t.b, pl.mx, pl.my, g.B * pl.nzc, g, q, y, x);
          const int zc = q % pl.nzc, z = q / pl.nzc * Ds + (zc * pl.lz >> hs);  // (zc lz is even where hs is 1)
          off[i] = in ? ((z * Hs + (y >> hs)) * Ws + (x >> hs)) * C : -1;
          zfirst |= (Mask)(zc == 0) << i;
          zlast |= (Mask)(zc == pl.nzc - 1) << i;
        } else {
          const bool in = (unsigned)y < (unsigned)g.H && (unsigned)x < (unsigned)g.W;
          off[i] = in ? ((y >> hs) * Ws + (x >> hs)) * C : -1;
        }
      }
      for (int p = t.p0; p <= t.p1; ++p) {
        ok = __all_sync(0xffffffffu, mbar_wait(a_empty(as), ph, stop, limit));
        if (!ok) break;
        const uint32_t dst = sA + a_bytes * as + (uint32_t)q * pl.lbo + (uint32_t)v0 * 16;
        if (MOSAIC) {
          const Mask out = p < 0 ? zfirst : p >= t.z1 ? zlast : (Mask)0;
          const bf16 *plane = base + (long long)(p >> hs) * Hs * Ws * C;
#pragma unroll
          for (int i = 0; i < NI; ++i)
            if (lt < LT && ((i + 1) * VS <= NV || v0 + i * VS < NV)) {
              const bool in = off[i] >= 0 && !(out >> i & 1);
              cp16(dst + (uint32_t)(i * VS) * 16, in ? plane + off[i] : base, in ? 16 : 0);
            }
        } else {
          const bf16 *plane = base + ((size_t)t.b * Ds + (p >> hs)) * Hs * Ws * C;
#pragma unroll
          for (int i = 0; i < NI; ++i)
            if (lt < LT && ((i + 1) * VS <= NV || v0 + i * VS < NV))
              cp16(dst + (uint32_t)(i * VS) * 16, plane + max(off[i], 0), off[i] >= 0 ? 16 : 0);
        }
        asm volatile("cp.async.commit_group;\n" ::: "memory");
        // With three stages or more, the next plane's copies are issued before this one's
        // are waited for (with two, their stage is the one the tensor cores are reading).
        if (prev >= 0) {
          asm volatile("cp.async.wait_group 1;\n" ::: "memory");
          landed(prev);
        }
        prev = as;
        if (pl.a_stages < 3) {
          asm volatile("cp.async.wait_group 0;\n" ::: "memory");
          landed(prev);
          prev = -1;
        }
        if (++as == pl.a_stages) {
          as = 0;
          ph ^= 1;
        }
      }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    if (prev >= 0) landed(prev);
  }
  __syncwarp();
  fence_before();
  __syncthreads();
  if (warp == 0) {
    if (*stop)  // (otherwise the accumulators read out say as much)
      for (int j = 0; j < J; ++j) mbar_drain(drained + 8u * j, 0, stop);
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kTmemCols));
  }
  if (tid == 0 && *stop) {
    *reinterpret_cast<volatile int *>(a.err) = 1;
    *a.bad = 1;
  }
}

// ---------------------------------------------------------------- weight gradient
// dW[o, tap, c] = sum_p G[p, o] X[p + delta_tap, c] for 32 input channels (a slice)
// and 32 output channels per CTA: the voxels are the K dimension, so both operands
// are read voxel-major (MN-major descriptors: a core matrix is 8 voxels of x by 8
// channels, the layout of the forward kernel's planes).  M = 128 rows are the slice's
// channels of the planes z - 1, z and z + 1 of X and a fourth plane of zeros; N = 32
// are the output channels of plane z of G.  One tcgen05.mma per 16 voxels thus covers
// the taps dz = -1, 0, +1 of one (dy, dx).  The 27 x 32 x 32 gradients stay in TMEM,
// nine accumulators of 32 columns, over several of a CTA's bricks (8 x 16 voxels of one
// plane), and are then added into dW, 32 consecutive channels per instruction.
//
// The tensor cores cut off what of a product lies below the running sum, so a sum's
// error grows with the number of products added one after the other (WPlan::group).
// The bias gradients are summed in FP32, a brick's values first and the bricks with the
// additions' rounding errors kept: as a fourth plane of ones they came along with the
// products, 3e-4 of themselves off (values of one sign, 256 x 256 x 128, 96 -> 32; now
// 1e-7), and summed by the loading threads they held up the copies.
// The largest error of a weight gradient of one sign there, with chains of a whole CTA's
// bricks and now: 32 -> 32 1.2e-4, 4e-6; 96 -> 32 3.3e-4, 3e-6; 192 -> 64 2.1e-4, 1.1e-5
// (with the mma.sync kernels 1.3e-4, 3.3e-4, 5.7e-5).
//
// Bound by the 40 cycles that M = 128, N = 32, K = 16 takes (its operand reads).  Against
// the mma.sync kernels and column sums that it replaces (a tap per warp, every tap
// gathering X again), four 32^3 crops, a layer with its bias gradient: 32 -> 32 at 32^3
// 71 us before, 24 now; 96 -> 32 185 and 47; 192 -> 64 at 16^3 86 and 29; 64 -> 64 46 and 16
// (the training gradient 1080 -> 690 us).  The issue of the MMAs keeps pace only without
// divisions between them: with the bricks' rows known to be whole, the gradient at 256 x
// 256 x 128 14.75 -> 14.26 ms.
constexpr int kWX = (kPX * (kTY + 2) + 6) * 16;         // bytes of a plane's 8-channel piece of X (padded: 2 mod 8 pieces)
constexpr int kWG = (kTX * kTY + 2) * 16;               // and of G
constexpr int kWStage = 4 * 4 * kWX + 4 * kWG;
constexpr int kWStages = 4;
// 8 loading warps, 1 for the MMAs, 4 for the sums: one per quarter of the TMEM lanes, of
// which the zero plane's sums G for the bias gradient
constexpr int kWThreads = (kLoadWarps + 5) * 32;

struct WPlan {
  int nsl, nt;         // slices of input channels, tiles of output channels
  int per;             // CTAs per (slice, tile)
  int mx, my;          // planes along x and y that share bricks (1, 1: none do)
  int hm;              // rows of a plane, or of a mosaic of planes
  int tx, ty;          // bricks along x, y
  int bricks;
  int group;           // bricks summed in TMEM before they are added into dW
};

// Add x into the sum hi + lo, keeping the rounding error in lo.
__device__ __forceinline__ void two_sum(float &hi, float &lo, float x) {
  const float s = hi + x, b = s - hi;
  lo += (hi - (s - b)) + (x - b);
  hi = s;
}

__global__ void __launch_bounds__(kWThreads, 1) wgrad_tc_kernel(WgradTcArgs a, WPlan pl) {
  chained();
  extern __shared__ __align__(128) unsigned char smem[];
  __shared__ __align__(8) uint64_t bars[2 * kWStages + 3];
  __shared__ uint32_t s_tmem;
  __shared__ int s_stop;
  const int tid = threadIdx.x, lane = tid & 31;
  const int warp = __shfl_sync(0xffffffffu, tid >> 5, 0);
  const Vol g = a.vol;
  const int combo = blockIdx.x % (pl.nsl * pl.nt), first = blockIdx.x / (pl.nsl * pl.nt);
  const int sl = combo % pl.nsl, nt = combo / pl.nsl;
  const uint32_t base = smem_u32(smem), bar0 = smem_u32(bars);
  auto full = [&](int s) { return bar0 + 8u * s; };
  auto empty = [&](int s) { return bar0 + 8u * (kWStages + s); };
  // the accumulators hold a group's sums, have been read; all MMAs are done
  const uint32_t acc_full = empty(kWStages), acc_empty = acc_full + 8, done = acc_full + 16;
  if (warp == 0) {
    asm volatile("tcgen05.alloc.cta_group::1.sync.aligned.shared::cta.b32 [%0], %1;\n" ::"r"(smem_u32(&s_tmem)),
                 "r"(kTmemCols)
                 : "memory");
    asm volatile("tcgen05.relinquish_alloc_permit.cta_group::1.sync.aligned;\n");
  }
  if (tid == kLoadWarps * 32) {
    for (int s = 0; s < kWStages; ++s) {
      mbar_init(full(s), kLoadWarps);
      mbar_init(empty(s), sl == 0 ? 2 : 1);  // the MMAs, the bias gradients
    }
    mbar_init(acc_full, 1);
    mbar_init(acc_empty, 3);
    mbar_init(done, 1);
    asm volatile("fence.mbarrier_init.release.cluster;\n" ::: "memory");
    s_stop = a.wait_ns == 0;  // no wait is sat out
  }
  // the fourth plane of every stage
  for (int i = tid; i < kWStages * 4 * (kWX / 16); i += kWThreads) {
    const int st = i / (4 * (kWX / 16)), e = i - st * 4 * (kWX / 16);
    *reinterpret_cast<uint4 *>(smem + st * kWStage + 3 * 4 * kWX + e * 16) = make_uint4(0u, 0u, 0u, 0u);
  }
  asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
  fence_before();
  __syncthreads();
  fence_after();
  const uint32_t tmem = __shfl_sync(0xffffffffu, s_tmem, 0);
  volatile int *stop = &s_stop;
  const unsigned long long limit = a.wait_ns;

  if (warp < kLoadWarps) {
    // ---- brick copies: thread t keeps the 8-channel piece t mod 4 and steps over voxels ----
    constexpr int VS = kLoadWarps * 8, NVX = kPX * (kTY + 2), NX = (NVX + VS - 1) / VS, NG = kTX * kTY / VS;
    const int q = tid & 3, v0 = tid >> 2;
    const int cb = sl * 32;
    const bool half = cb < a.c1;
    const int hs = half ? 1 : 0, C = half ? a.c1 : a.c0, Hs = g.H >> hs, Ws = g.W >> hs, Ds = g.D >> hs;
    const bf16 *xb = (half ? a.x1 + cb : a.x0 + (cb - a.c1)) + q * 8;
    const bf16 *gb = a.g + nt * 32 + q * 8;
    auto landed = [&](int st) {  // this warp's copies into stage st are visible to the tensor cores
      asm volatile("fence.proxy.async.shared::cta;\n" ::: "memory");
      __syncwarp();
      if (lane == 0) mbar_arrive(full(st));
    };
    int s = 0, prev = -1;
    uint32_t ph = 1;
    for (int u = first; u < pl.bricks; u += pl.per) {
      const int x0 = u % pl.tx * kTX, y0 = u / pl.tx % pl.ty * kTY, m = u / pl.tx / pl.ty;
      if (!__all_sync(0xffffffffu, mbar_wait(empty(s), ph, stop, limit))) break;
      const uint32_t sx = base + kWStage * s + q * kWX, sg = base + kWStage * s + 4 * 4 * kWX + q * kWG;
      if (pl.mx * pl.my > 1) {  // a mosaic of planes (b, z), m its number
        const int q0 = m * pl.mx * pl.my, nq = g.B * g.D;
#pragma unroll
        for (int i = 0; i < NX; ++i) {
          const int v = v0 + i * VS, vy = v / kPX, vx = v - vy * kPX;
          int y = y0 + vy - 1, x = x0 + vx - 1, piece;
          const bool in = in_mosaic(q0, pl.mx, pl.my, nq, g, piece, y, x);
          const int b = piece / g.D, z0 = piece - b * g.D, yx = (y >> hs) * Ws + (x >> hs);
#pragma unroll
          for (int j = 0; j < 3; ++j) {
            const int z = z0 + j - 1;
            const bool inz = in && z >= 0 && z < g.D;
            if (v < NVX)
              cp16(sx + j * 4 * kWX + v * 16, inz ? xb + ((b * Ds + (z >> hs)) * Hs * Ws + yx) * C : xb, inz ? 16 : 0);
          }
        }
#pragma unroll
        for (int i = 0; i < NG; ++i) {
          const int v = v0 + i * VS;
          int y = y0 + v / kTX, x = x0 + v % kTX, piece;
          const bool in = in_mosaic(q0, pl.mx, pl.my, nq, g, piece, y, x);
          cp16(sg + v * 16, in ? gb + (size_t)((piece * g.H + y) * g.W + x) * a.cout : gb, in ? 16 : 0);
        }
      } else {
        const int b = m / g.D, z0 = m - b * g.D;
        int off[NX];
#pragma unroll
        for (int i = 0; i < NX; ++i) {
          const int v = v0 + i * VS, vy = v / kPX, vx = v - vy * kPX, y = y0 + vy - 1, x = x0 + vx - 1;
          off[i] = (unsigned)y < (unsigned)g.H && (unsigned)x < (unsigned)g.W ? ((y >> hs) * Ws + (x >> hs)) * C : -1;
        }
#pragma unroll
        for (int j = 0; j < 3; ++j) {
          const int z = z0 + j - 1;
          const bool inz = z >= 0 && z < g.D;
          const bf16 *plane = xb + ((size_t)b * Ds + (inz ? z >> hs : 0)) * Hs * Ws * C;
#pragma unroll
          for (int i = 0; i < NX; ++i) {
            const int v = v0 + i * VS;
            if (v < NVX)
              cp16(sx + j * 4 * kWX + v * 16, plane + max(off[i], 0), inz && off[i] >= 0 ? 16 : 0);
          }
        }
#pragma unroll
        for (int i = 0; i < NG; ++i) {
          const int v = v0 + i * VS, y = y0 + v / kTX, x = x0 + v % kTX;
          const bool in = y < g.H && x < g.W;
          const size_t vox = (((size_t)b * g.D + z0) * g.H + (in ? y : 0)) * g.W + (in ? x : 0);
          cp16(sg + v * 16, gb + vox * a.cout, in ? 16 : 0);
        }
      }
      asm volatile("cp.async.commit_group;\n" ::: "memory");
      if (prev >= 0) {  // the next brick's copies are issued before this one's are waited for
        asm volatile("cp.async.wait_group 1;\n" ::: "memory");
        landed(prev);
      }
      prev = s;
      if (++s == kWStages) {
        s = 0;
        ph ^= 1;
      }
    }
    asm volatile("cp.async.wait_group 0;\n" ::: "memory");
    if (prev >= 0) landed(prev);
  } else if (warp == kLoadWarps) {
    // ---- MMA issue ----
    // F32 <- BF16 x BF16, A and B MN-major (bits 15, 16), N = 32, M = 128
    const uint32_t idesc = (1u << 4) | (1u << 7) | (1u << 10) | (1u << 15) | (1u << 16) | (4u << 17) | (8u << 24);
    // MN-major: the stride word is between 8-channel pieces, the leading word between 8-voxel groups of K
    const uint32_t ahi = desc_hi(kWX), bhi = desc_hi(kWG);
    const bool issue = elect_one(), ragged = pl.hm % kTY != 0;
    int s = 0;
    uint32_t ph = 0, gph = 1;  // gph: the parity of acc_empty that frees the accumulators for the group
    bool ok = true;
    // (a loop per group: bookkeeping in the loop over the bricks, where the issue of the
    // MMAs bounds the kernel, cost 4% of it)
    for (int u = first; u < pl.bricks && ok;) {
      ok = __all_sync(0xffffffffu, mbar_wait(acc_empty, gph, stop, limit));
      gph ^= 1;
      uint32_t add = 0;
      const int end = min(pl.bricks, u + pl.group * pl.per);
      for (; u < end && ok; u += pl.per) {
        // 16-voxel steps (two rows of y); no divisions where every brick is whole
        int nk = kTY / 2;
        if (ragged) nk = min(nk, (pl.hm - u / pl.tx % pl.ty * kTY + 1) / 2);
        ok = __all_sync(0xffffffffu, mbar_wait(full(s), ph, stop, limit));
        if (!ok) break;
        fence_after();
        const uint32_t blo = uniform(desc_lo(base + kWStage * s + 4 * 4 * kWX, kTX * 16));
        const uint32_t acc = uniform(add);
        uint32_t tap = uniform(desc_lo(base + kWStage * s, kPX * 16)), d = tmem;
#pragma unroll 1
        for (int yx = 0; yx < 9; ++yx) {
          if (issue) {
#pragma unroll
            for (int ks = 0; ks < kTY / 2; ++ks)
              if (ks < nk) mma_f16(d, tap + ks * 2 * kPX, ahi, blo + ks * 2 * kTX, bhi, idesc, ks ? 1u : acc);
          }
          __syncwarp();
          tap += yx % 3 == 2 ? kPX - 2 : 1;
          d += 32;
        }
        add = 1;
        if (issue) mma_commit(empty(s));
        __syncwarp();
        if (++s == kWStages) {
          s = 0;
          ph ^= 1;
        }
      }
      if (issue && ok) mma_commit(acc_full);
    }
    if (issue) mma_commit(done);
    __syncwarp();
  } else if ((warp & 3) == 3) {
    // ---- bias gradients: lane t sums the 8-channel piece t mod 4 of every 8th voxel ----
    if (sl == 0) {
      const int q = lane & 3, v0 = lane >> 2;
      float hi[8], lo[8];
#pragma unroll
      for (int i = 0; i < 8; ++i) hi[i] = lo[i] = 0.f;
      int s = 0;
      uint32_t ph = 0;
      for (int u = first; u < pl.bricks; u += pl.per) {
        if (!__all_sync(0xffffffffu, mbar_wait(full(s), ph, stop, limit))) break;
        const unsigned char *sg = smem + kWStage * s + 4 * 4 * kWX + q * kWG + v0 * 16;
        float x[8];
#pragma unroll
        for (int i = 0; i < 8; ++i) x[i] = 0.f;
#pragma unroll 8
        for (int i = 0; i < kTX * kTY / 8; ++i) {
          const uint4 w = *reinterpret_cast<const uint4 *>(sg + i * 128);
          const uint32_t p[4] = {w.x, w.y, w.z, w.w};
#pragma unroll
          for (int e = 0; e < 4; ++e) {  // (a BF16 value is the upper half of its FP32 value)
            x[2 * e] += __uint_as_float(p[e] << 16);
            x[2 * e + 1] += __uint_as_float(p[e] & 0xffff0000u);
          }
        }
        __syncwarp();
        if (lane == 0) mbar_arrive(empty(s));
#pragma unroll
        for (int i = 0; i < 8; ++i) two_sum(hi[i], lo[i], x[i]);
        if (++s == kWStages) {
          s = 0;
          ph ^= 1;
        }
      }
#pragma unroll
      for (int i = 0; i < 8; ++i) {
        float x = hi[i] + lo[i];
#pragma unroll
        for (int o = 4; o < 32; o <<= 1) x += __shfl_xor_sync(0xffffffffu, x, o);
        if (lane < 4) atomicAdd(a.db + nt * 32 + lane * 8 + i, x);
      }
    }
  } else {
    // ---- a group's sums into dW: quarter w of the TMEM lanes holds tap plane dz = w - 1, a
    // lane one input channel of the slice ----
    const int w = warp & 3, cin = a.c0 + a.c1, nb = (pl.bricks - first + pl.per - 1) / pl.per;
    const uint32_t rows = tmem + ((uint32_t)(w * 32) << 16);
    float *dst = a.dw + (size_t)(nt * 32) * 27 * cin + (size_t)(w * 9) * cin + sl * 32 + lane;
    uint32_t ph = 0;
    for (int i = 0; i < nb; i += pl.group) {
      if (!__all_sync(0xffffffffu, mbar_wait(acc_full, ph, stop, limit))) break;
      ph ^= 1;
      fence_after();
#pragma unroll 3
      for (int yx = 0; yx < 9; ++yx) {
        uint32_t v[32];
        tmem_ld32(v, rows + yx * 32);
        if (yx == 8) {  // the next group's products may overwrite the accumulators
          fence_before();
          __syncwarp();
          if (lane == 0) mbar_arrive(acc_empty);
        }
#pragma unroll
        for (int o = 0; o < 32; ++o) atomicAdd(dst + ((size_t)o * 27 + yx) * cin, __uint_as_float(v[o]));
      }
    }
  }
  __syncwarp();
  fence_before();
  __syncthreads();
  if (warp == 0) {
    if (*stop) mbar_drain(done, 0, stop);  // (otherwise the last sums read out say as much)
    fence_after();
    asm volatile("tcgen05.dealloc.cta_group::1.sync.aligned.b32 %0, %1;\n" ::"r"(tmem), "r"(kTmemCols));
  }
  if (tid == 0 && *stop) {
    *reinterpret_cast<volatile int *>(a.err) = 1;
    *a.bad = 1;
  }
}

// Tensor-core cycles of one plane that serves n output planes (per 16-channel
// step, 128-voxel tile and (dy, dx)): the products at N / 2 cycles for M = 128,
// K = 16, or the operands' 128-byte shared-memory reads, whichever is longer.
double step_cycles(int n, int nt) {
  const double products = 0.5 * n * nt, reads = 32.0 + 0.25 * n * nt;
  return products > reads ? products : reads;
}

bool fit(Plan &pl, int cin) {
  const int nq = cin / 8, cs = stage_channels(cin), nst = 9 * (cin / cs);
  const int nvp = kPX * (kTY * pl.J + 2);
  // 16-byte pieces of 8 consecutive lanes fall into different banks: 4 pieces of
  // 2 voxels (32 channels) or the 8 and more pieces of one voxel
  const int want = nq == 4 ? 2 : 1;
  pl.lbo = (nvp + ((want - nvp % 8) + 8) % 8) * 16;
  const int ab = pl.lbo * nq, wb = cs / 8 * 3 * pl.nt * 16;
  if (weights_resident(cin)) {
    pl.w_stages = nst;
    pl.a_stages = 2;
  } else {
    pl.a_stages = 2 * ab + 2 * wb <= kSmemMax ? 2 : 1;
    pl.w_stages = (kSmemMax - pl.a_stages * ab) / wb;
    if (pl.w_stages > 8) pl.w_stages = 8;
    if (pl.w_stages < 2) return false;
  }
  if (pl.w_stages > kMaxWStages || pl.a_stages * ab + pl.w_stages * wb > kSmemMax) return false;
  while (pl.a_stages < kMaxAStages && (pl.a_stages + 1) * ab + pl.w_stages * wb <= kSmemMax) ++pl.a_stages;
  pl.smem = pl.a_stages * ab + pl.w_stages * wb;
  if (pl.smem < kSmemMin) pl.smem = kSmemMin;
  return true;
}

// Pieces of W x H voxels, n in all, that share tiles of kTX x rows voxels: the mosaic
// (mx, my) with the fewest tiles per piece, one zero column or row between neighbours.
void choose_mosaic(const Vol &g, long long n, int rows, int *mx, int *my) {
  *mx = *my = 1;
  auto tiles = [](int m, int side, int tile) { return (m * (side + 1) - 1 + tile - 1) / tile; };
  if (g.W < kTX)
    for (int m = 2; m <= 8 && m <= n; ++m)
      if (tiles(m, g.W, kTX) * *mx < tiles(*mx, g.W, kTX) * m) *mx = m;
  const long long left = (n + *mx - 1) / *mx;
  if (g.H < rows)
    for (int m = 2; m <= 16 && m <= left; ++m)
      if (tiles(m, g.H, rows) * *my < tiles(*my, g.H, rows) * m) *my = m;
}

// The split of the volume into work units: tiles along y per unit and planes per
// unit, by the tensor-core time of the busiest CTA (a plane at either end of a
// unit serves one or two output planes instead of three, so longer units cost
// less, but the units have to fill the SMs).  Mosaics only where there is more than one
// unit to a CTA and they take three quarters of the time or less: their set-up per unit
// is longer (64 crops of 20^3: forward 0.542 ms without, 0.564 where any gain counted).
bool make_plan(const ConvArgs &a, int num_sms, Plan *best) {
  const int cin = a.c0 + a.c1;
  double best_cost = 1e300;
  auto consider = [&](int J, int lz, bool mosaic) {
    Plan pl;
    pl.J = J;
    pl.nt = conv_tile_n(a.cout);
    pl.nn = a.cout / pl.nt;
    pl.sh = J * pl.nt > 64 ? 2 : 3;  // 4 slots of 2 x 64 columns, else 8
    pl.slots = 1 << pl.sh;
    pl.lz = lz;
    pl.nzc = (a.g.D + lz - 1) / lz;
    const long long pieces = (long long)a.g.B * pl.nzc;
    pl.mx = pl.my = 1;
    if (mosaic) choose_mosaic(a.g, pieces, kTY * J, &pl.mx, &pl.my);
    const int per = pl.mx * pl.my, wm = pl.mx * (a.g.W + 1) - 1, hm = pl.my * (a.g.H + 1) - 1;
    if ((mosaic && per == 1) || (J == 2 && hm <= kTY)) return;
    pl.tx = (wm + kTX - 1) / kTX;
    pl.ty = (hm + kTY * J - 1) / (kTY * J);
    const long long units = (pieces + per - 1) / per * pl.ty * pl.tx;
    if (units > (1 << 30)) return;
    pl.units = (int)units;
    const long long ctas = num_sms > pl.nn ? num_sms / pl.nn : 1, waves = (units + ctas - 1) / ctas;
    const double c1 = step_cycles(1, pl.nt), c2 = step_cycles(2, pl.nt), c3 = step_cycles(3, pl.nt);
    const double unit = lz == 1 ? 3 * c1 : 2 * c1 + 2 * c2 + (lz - 2) * c3;
    const double cost = waves * (9.0 * (cin / 16) * J * unit + 250.0 * (lz + 2) + 1500.0);
    if (cost < best_cost && fit(pl, cin)) {
      best_cost = cost;
      *best = pl;
    }
  };
  for (int J = 1; J <= 2; ++J)
    for (int lz = 1; lz <= a.g.D; lz = lz < 8 ? lz + 1 : lz + (lz + 3) / 4) consider(J, lz, false);
  if (best_cost < 1e300 && (a.g.W < kTX || a.g.H < kTY) && (long long)best->units * best->nn > num_sms) {
    best_cost *= 0.75;
    for (int J = 1; J <= 2; ++J)  // whole chunks of planes; of an even count where an input is read at half size
      for (int lz = 1; lz <= a.g.D; ++lz)
        if (a.g.D % lz == 0 && (lz % 2 == 0 || !a.c1 || lz == a.g.D)) consider(J, lz, true);
  }
  return best_cost < 1e300;
}

template <int C0, int C1>
cudaError_t launch(const ConvArgs &a, const Plan &pl, int num_sms, cudaStream_t stream) {
  const int ctas = num_sms > pl.nn ? num_sms / pl.nn : 1, grid = pl.nn * (pl.units < ctas ? pl.units : ctas);
  const bool mosaic = pl.mx * pl.my > 1;
  const auto kernel = pl.J == 2 ? (mosaic ? conv_tc_kernel<C0, C1, 2, true> : conv_tc_kernel<C0, C1, 2, false>)
                                : (mosaic ? conv_tc_kernel<C0, C1, 1, true> : conv_tc_kernel<C0, C1, 1, false>);
  return launch_chained(kernel, grid, kThreads, pl.smem, stream, a, pl);
}

template <int C0, int C1>
cudaError_t prepare() {
  for (const auto kernel : {conv_tc_kernel<C0, C1, 1, false>, conv_tc_kernel<C0, C1, 2, false>,
                            conv_tc_kernel<C0, C1, 1, true>, conv_tc_kernel<C0, C1, 2, true>}) {
    const cudaError_t e = cudaFuncSetAttribute(kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kSmemMax);
    if (e != cudaSuccess) return e;
  }
  return cudaSuccess;
}

}  // namespace

cudaError_t conv_prepare() {
  cudaError_t e = prepare<32, 0>();
  if (e == cudaSuccess) e = prepare<64, 0>();
  if (e == cudaSuccess) e = prepare<128, 0>();
  if (e == cudaSuccess) e = prepare<64, 128>();
  if (e == cudaSuccess) e = prepare<32, 64>();
  return e;
}

cudaError_t wgrad_prepare() {
  return cudaFuncSetAttribute(wgrad_tc_kernel, cudaFuncAttributeMaxDynamicSharedMemorySize, kWStages * kWStage);
}

cudaError_t wgrad_launch(const WgradTcArgs &a, int num_sms, cudaStream_t stream) {
  if (a.c0 % 32 || a.c1 % 32 || a.cout % 32) return cudaErrorInvalidValue;
  WPlan pl;
  pl.nsl = (a.c0 + a.c1) / 32;
  pl.nt = a.cout / 32;
  const int most_per = num_sms / (pl.nsl * pl.nt) > 1 ? num_sms / (pl.nsl * pl.nt) : 1;
  auto split = [&](int mx, int my) {
    const int planes = a.vol.B * a.vol.D;
    pl.mx = mx;
    pl.my = my;
    pl.hm = my * (a.vol.H + 1) - 1;
    pl.tx = (mx * (a.vol.W + 1) - 1 + kTX - 1) / kTX;
    pl.ty = (pl.hm + kTY - 1) / kTY;
    pl.bricks = (planes + mx * my - 1) / (mx * my) * pl.tx * pl.ty;
    pl.per = most_per < pl.bricks ? most_per : pl.bricks;
    return (pl.bricks + pl.per - 1) / pl.per;  // of a CTA
  };
  const int alone = split(1, 1);
  if (alone > 1) {
    int mx, my;
    choose_mosaic(a.vol, (long long)a.vol.B * a.vol.D, kTY, &mx, &my);
    if (mx * my > 1 && split(mx, my) >= alone) split(1, 1);
  }
  // Products added one after the other in TMEM: an eighth of a CTA's, but at least 192 and
  // at most 1024 steps of 16 voxels (a group's end takes 3 us or so, 192 steps 33).
  const int per_brick = pl.hm < kTY ? (pl.hm + 1) / 2 : kTY / 2;
  const int own = (pl.bricks + pl.per - 1) / pl.per, steps = own * per_brick;
  const int most = steps / 8 < 192 ? 192 : (steps / 8 > 1024 ? 1024 : steps / 8), groups = (steps + most - 1) / most;
  pl.group = (own + groups - 1) / groups;
  return launch_chained(wgrad_tc_kernel, pl.nsl * pl.nt * pl.per, kWThreads, kWStages * kWStage, stream, a, pl);
}

cudaError_t conv_launch(const ConvArgs &a, int num_sms, cudaStream_t stream) {
  Plan pl;
  if (a.cout % 32 || a.cout > 192 || (a.hp && a.cout != 32) || !make_plan(a, num_sms, &pl)) return cudaErrorInvalidValue;
  if (a.c0 == 32 && a.c1 == 0) return launch<32, 0>(a, pl, num_sms, stream);
  if (a.c0 == 64 && a.c1 == 0) return launch<64, 0>(a, pl, num_sms, stream);
  if (a.c0 == 128 && a.c1 == 0) return launch<128, 0>(a, pl, num_sms, stream);
  if (a.c0 == 64 && a.c1 == 128) return launch<64, 128>(a, pl, num_sms, stream);
  if (a.c0 == 32 && a.c1 == 64) return launch<32, 64>(a, pl, num_sms, stream);
  return cudaErrorInvalidValue;
}

}  // namespace s3ttv_net_detail
