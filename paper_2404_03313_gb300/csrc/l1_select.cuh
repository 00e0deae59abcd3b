// Device code of the l1-ball threshold search (l1ball.cu), shared with the
// kernels that take a level of it along: the primal step builds the first
// histogram, and whichever CTA of a kernel finishes last narrows the threshold.
// (As kernels of their own the three scans and the scalar finish of a pass took
// 4-8 and 7-11 us each, nearly all of it launch and latency: 27 of 65 us per pass
// of a 32 x 32 x 16 cube.)
#pragma once
#include <math.h>
#include "s3ttv_internal.cuh"

namespace s3ttv {

// CTA size of every kernel that scans: few, large CTAs, because each adds its
// histogram into the global one, and the FP64 atomics of 1216 CTAs on the same few
// cache lines took 10 us
constexpr int kSelThreads = 512;

// True in the CTA of this grid that calls it last (all its threads); every CTA's
// global writes before the call are visible to that CTA.  The counter is back at
// zero afterwards.
__device__ __forceinline__ bool last_cta(unsigned *counter, unsigned ctas) {
  __shared__ int s_last;
  __threadfence();
  __syncthreads();
  if (threadIdx.x == 0) {
    s_last = atomicAdd(counter, 1u) == ctas - 1u;
    if (s_last) *counter = 0u;
  }
  __syncthreads();
  if (s_last) __threadfence();
  return s_last != 0;
}

// Narrow problem pb's threshold by one radix level from its histogram and clear
// the histogram, by a team of kTeam threads (team t: threads t kTeam .. of the CTA,
// barrier 1 + t), PER bins each.  Teams of 128, because FP64 runs at two operations a
// cycle and SM whatever it is spread over: with all 512 threads taking part the scan
// took 8 us, most of it in the adds of the cross-warp sums.
constexpr int kTeam = 128, kTeams = 2;
template <int PER>
__device__ void l1_scan(Scalars *sc, unsigned *cnt, double *sum, int pb, int level, int team) {
  constexpr int NW = kTeam / 32;
  __shared__ unsigned long long s_wc[kTeams][NW], s_suf[kTeams][PER + 1];
  __shared__ double s_ws[kTeams][NW], s_ssf[kTeams][PER + 1];
  __shared__ int s_first[kTeams][NW];
  const int tid = threadIdx.x - team * kTeam, lane = tid & 31, w = tid >> 5;
  auto sync = [&]() { asm volatile("bar.sync %0, %1;\n" ::"r"(1 + team), "n"(kTeam) : "memory"); };
  constexpr int nb = PER * kTeam;
  const int bits = l1_level_bits(level), shift = l1_level_shift(level);
  L1State st = sc->l1[pb];
  if (level == 1) {
    st.S_above = 0.0;
    st.C_above = 0ull;
    st.prefix = 0u;
    st.mode = 0;
    st.tau = 0.f;
    st.tau_lo = 0.f;
  }
  // thread tid owns the PER bins below bin top (counted from the top)
  const int top = nb - 1 - PER * tid;
  unsigned c[PER];
  double sm[PER];
#pragma unroll
  for (int e = 0; e < PER; ++e) {
    c[e] = __ldcg(cnt + top - e);
    sm[e] = __ldcg(sum + top - e);
  }
  unsigned long long own_c = 0ull;
  double own_s = 0.0;
#pragma unroll
  for (int e = 0; e < PER; ++e) {
    cnt[top - e] = 0u;
    sum[top - e] = 0.0;
    own_c += c[e];
    own_s += sm[e];
  }
  // inclusive scan from the top: sums over all bins down to this thread's last
  unsigned long long ci = own_c;
  double si = own_s;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long cu = __shfl_up_sync(kFull, ci, o);
    const double su = __shfl_up_sync(kFull, si, o);
    if (lane >= o) {
      ci += cu;
      si += su;
    }
  }
  if (lane == 31) {
    s_wc[team][w] = ci;
    s_ws[team][w] = si;
  }
  sync();
  for (int i = 0; i < w; ++i) {  // warp-uniform
    ci += s_wc[team][i];
    si += s_ws[team][i];
  }
  const double r = st.radius;
  if (level == 1) {
    double total = 0.0;
    for (int i = 0; i < NW; ++i) total += s_ws[team][i];
    if (total <= r || r <= 0.0) {  // team-uniform
      if (tid == 0) {
        st.mode = total <= r ? 1 : 2;
        st.tau = total <= r ? 0.f : INFINITY;
        sc->l1[pb] = st;
      }
      return;
    }
  }
  const int pshift = bits + shift;
  const unsigned pre = level == 1 ? 0u : st.prefix;
  // h at the lower edge of a bin, from the totals down to it; h falls as the edge rises
  auto h_at = [&](int bin, unsigned long long cc, double ss) {
    const unsigned lob = (pshift >= 32 ? 0u : (pre << pshift)) | ((unsigned)bin << shift);
    return st.S_above + ss - (double)__uint_as_float(lob) * (double)(st.C_above + cc);
  };
  // The bin sought is the highest with h >= r (h(0) >= r holds by construction): it
  // belongs to the first thread whose lowest bin has h >= r; that thread's bins are
  // then looked at by a lane each.
  const bool mine = h_at(top - (PER - 1), ci, si) >= r || tid == kTeam - 1;
  const unsigned ball = __ballot_sync(kFull, mine);
  if (lane == 0) s_first[team][w] = ball ? w * 32 + __ffs(ball) - 1 : kTeam;
  sync();
  int owner = kTeam;
#pragma unroll
  for (int i = 0; i < NW; ++i) owner = min(owner, s_first[team][i]);
  if (tid == owner) {
    unsigned long long suf = ci - own_c;
    double ssf = si - own_s;
#pragma unroll
    for (int e = 0; e < PER; ++e) {  // totals strictly above bin top - e
      s_suf[team][e] = suf;
      s_ssf[team][e] = ssf;
      suf += c[e];
      ssf += sm[e];
    }
    s_suf[team][PER] = suf;
    s_ssf[team][PER] = ssf;
  }
  sync();
  if (w == 0) {
    const int otop = nb - 1 - PER * owner, e = min(lane, PER - 1);
    const unsigned hit = __ballot_sync(kFull, e == PER - 1 || h_at(otop - e, s_suf[team][e + 1], s_ssf[team][e + 1]) >= r);
    const int best = __ffs(hit) - 1;
    if (lane == 0) {
      st.C_above += s_suf[team][best];
      st.S_above += s_ssf[team][best];
      st.prefix = (pre << bits) | (unsigned)(otop - best);
      if (level == 3) {
        st.mode = 3;
        const double tau = st.C_above > 0 ? (st.S_above - r) / (double)st.C_above : 0.0;
        st.tau = (float)tau;
        st.tau_lo = (float)(tau - (double)st.tau);
      }
      sc->l1[pb] = st;
    }
  }
}

// (a CTA's first team)
template <int LEVEL>
__device__ __forceinline__ void l1_scan_level(const L1Args &a, int pb) {
  if (threadIdx.x < kTeam)
    l1_scan<(LEVEL == 3 ? 1 << 9 : kHistBins) / kTeam>(a.sc, a.hcnt + pb * kHistBins, a.hsum + pb * kHistBins, pb, LEVEL,
                                                       0);
}

// A radix level's histogram of |z| in shared memory, in integers: within a bin only
// the bits below the level differ (20, 9 or none of them), so the bin's sum follows
// exactly from its count and the sum of those bits (level 1: of their two halves).
// Shared memory adds integers natively but floats by compare-and-swap, and
// neighbouring values crowd a few bins: with float sums the primal step took 109 us
// at 256 x 256 x 128 once both projections were active, with these 67.  (The sums
// stay below 2^32 up to 4 M elements per CTA: elementwise_ctas().)
struct BinSums {
  unsigned cnt[kHistBins], hi[kHistBins], lo[kHistBins];
};
template <int LEVEL>
__device__ __forceinline__ void hist_add(BinSums &h, unsigned prefix, float z) {
  constexpr int bits = LEVEL == 3 ? 9 : 11, shift = LEVEL == 1 ? 20 : (LEVEL == 2 ? 9 : 0);
  const unsigned ub = __float_as_uint(z) & 0x7fffffffu;
  if (ub == 0u || (LEVEL > 1 && (ub >> (bits + shift)) != prefix)) return;  // zeros never enter the active set
  const unsigned key = (ub >> shift) & ((1u << bits) - 1u);
  atomicAdd(&h.cnt[key], 1u);
  if (LEVEL == 1) atomicAdd(&h.hi[key], (ub >> 10) & 1023u);
  if (LEVEL == 1) atomicAdd(&h.lo[key], ub & 1023u);
  if (LEVEL == 2) atomicAdd(&h.lo[key], ub & 511u);
}
// The sum of the values of bin key: their common upper bits once per value, and the rest.
template <int LEVEL>
__device__ __forceinline__ double bin_sum(const BinSums &h, unsigned prefix, unsigned key) {
  constexpr int bits = LEVEL == 3 ? 9 : 11, shift = LEVEL == 1 ? 20 : (LEVEL == 2 ? 9 : 0);
  const unsigned base = (LEVEL == 1 ? 0u : prefix << (bits + shift)) | key << shift, e = base >> 23;
  unsigned long long low = 0ull;
  if (LEVEL == 1) low = ((unsigned long long)h.hi[key] << 10) + h.lo[key];
  if (LEVEL == 2) low = h.lo[key];
  if (e == 255u) return low || (base & 0x7fffffu) ? __longlong_as_double(0x7ff8000000000000ll) : (double)INFINITY;
  const unsigned long long mant = (e ? 1u << 23 : 0u) | (base & 0x7fffffu);
  const int p2 = (int)(e ? e : 1u) - 150;  // value = mantissa 2^p2
  return (double)(h.cnt[key] * mant + low) * __longlong_as_double((long long)(p2 + 1023) << 52);
}

// One radix level's histogram of problem pb over elements first, first + stride, ...
// (float4 pieces where VEC: n a multiple of 4 and x 16-byte aligned), by one CTA.
template <int LEVEL, bool VEC>
__device__ void l1_hist(const L1Args &a, const L1State &st, int pb, long long first, long long stride, BinSums &h) {
  constexpr int nb = LEVEL == 3 ? 1 << 9 : kHistBins;
  for (int i = threadIdx.x; i < nb; i += kSelThreads) h.cnt[i] = h.hi[i] = h.lo[i] = 0u;
  __syncthreads();
  const unsigned prefix = LEVEL == 1 ? 0u : st.prefix;
  const float *x = a.x[pb];
  if (VEC) {
    // four pieces in flight per thread: the loop was bound by the latency of one
    const long long n4 = a.n >> 2;
    const float4 *x4 = reinterpret_cast<const float4 *>(x);
    for (long long i = first; i < n4; i += 4 * stride) {
      float4 z[4];
#pragma unroll
      for (int e = 0; e < 4; ++e)
        z[e] = i + e * stride < n4 ? __ldg(x4 + i + e * stride) : make_float4(0.f, 0.f, 0.f, 0.f);
#pragma unroll
      for (int e = 0; e < 4; ++e) {
        hist_add<LEVEL>(h, prefix, z[e].x);
        hist_add<LEVEL>(h, prefix, z[e].y);
        hist_add<LEVEL>(h, prefix, z[e].z);
        hist_add<LEVEL>(h, prefix, z[e].w);
      }
    }
  } else {
    for (long long i = first; i < a.n; i += stride) hist_add<LEVEL>(h, prefix, x[i]);
  }
  __syncthreads();
  for (int i = threadIdx.x; i < nb; i += kSelThreads) {
    const unsigned c = h.cnt[i];
    if (c) {
      atomicAdd(&a.hcnt[pb * kHistBins + i], c);
      atomicAdd(&a.hsum[pb * kHistBins + i], bin_sum<LEVEL>(h, prefix, i));
    }
  }
}

}  // namespace s3ttv
