// Global systematic resampling on the GPU: the exact integer rule's building blocks, shared by
// dpf_resample and by the outer stage of a step: the quantised counts, the number of systematic
// points below a cumulative count, the CTAs' prefixes, and the scatter of one CTA's ancestors.
#pragma once

#include <cuda/atomic>
#include <cstring>
#include <type_traits>

#include "dpf_common.cuh"
#include "dpf_internal.h"

namespace dpf {

constexpr int SPIN_LIMIT = 1 << 22;  // bounded wait at the outer stage's grid barrier (~0.3 s with the back-off)

typedef unsigned __int128 u128;

template <typename T>
__device__ __forceinline__ T pow2_t(int e);
template <>
__device__ __forceinline__ float pow2_t<float>(int e) { return __int_as_float((127 + e) << 23); }
template <>
__device__ __forceinline__ double pow2_t<double>(int e) {
  return __longlong_as_double((long long)(1023 + e) << 52);
}

// K(c) = #{ k in [0, n) : (k 2^32 + u) C < c n 2^32 }, the number of systematic
// points below the cumulative count c (global rule). The
// condition falls as k grows, so K is the first k where it fails: an estimate
// c n / C - u 2^-32 (single precision up to n = 2^24, whose error is a few units;
// double beyond) is settled by exact 128-bit comparisons.
__device__ __forceinline__ int points_below_est(unsigned long long c, long long n, uint32_t u,
                                                unsigned long long C) {
  if (c == 0) return 0;
  const u128 X = ((u128)c * (u128)(unsigned long long)n) << 32;
  long long k;
  if (n <= (1ll << 24)) {
    const float e = __fdividef((float)c, (float)C) * (float)n - (float)u * 0x1p-32f;
    k = e > 0.f ? (long long)ceilf(e) : 0;
  } else {
    const double e = (double)c / (double)C * (double)n - (double)u * 0x1p-32;
    k = e > 0.0 ? (long long)ceil(e) : 0;
  }
  if (k > n) k = n;
  while (k > 0 && !((u128)((unsigned long long)(k - 1) << 32 | u) * C < X)) --k;
  while (k < n && (u128)((unsigned long long)k << 32 | u) * C < X) ++k;
  return (int)k;
}

// The same count by one 64-bit product for almost every c. With P = c n / C (so K(c) =
// ceil(P - u 2^-32)) and F = floor(n 2^(64+f) / C), m = floor(c F 2^-64) satisfies
// P 2^f in [m, m + 1.5) (c < 2^63), and U = floor(u 2^(f-32)) satisfies u 2^(f-32) in [U, U + 1);
// so (P - u 2^-32) 2^f lies in (d - 1, d + 1.5), d = m - U, and its ceiling in units of 2^f is
// certain unless that interval meets a multiple of 2^f: 2.5 in 2^f of the values, which take
// the exact comparisons. Both scales are computed once a CTA.
struct PointScale {
  unsigned long long F;
  int f;  // < 0: no scale (C / n below 2^9)
};
__device__ __forceinline__ PointScale point_scale(long long n, unsigned long long C) {
  PointScale p{0ull, -1};
  const unsigned long long q = C / (unsigned long long)n;
  const int f = q ? 62 - __clzll((long long)q) : -1;  // n 2^f < C
  if (f < 8) return p;
  p.f = f < 32 ? f : 32;
  p.F = (unsigned long long)(((u128)(unsigned long long)n << (64 + p.f)) / C);
  return p;
}
__device__ __forceinline__ int points_below(unsigned long long c, long long n, uint32_t u, unsigned long long C,
                                            const PointScale& p) {
  if (c == 0) return 0;
  if (p.f > 0) {
    const long long d = (long long)__umul64hi(c, p.F) - (long long)((unsigned long long)u >> (32 - p.f));
    if (d >= 1) {
      const long long r = (d - 1) & ((1ll << p.f) - 1), k = ((d - 1) >> p.f) + 1;
      if (r + 3 <= (1ll << p.f)) return (int)(k < n ? k : n);
    } else if (d <= -2) {
      return 0;
    }
  }
  return points_below_est(c, n, u, C);
}

template <typename T>
__device__ __forceinline__ T exp_t(T v);
template <>
__device__ __forceinline__ float exp_t<float>(float v) { return expf(v); }
template <>
__device__ __forceinline__ double exp_t<double>(double v) { return exp(v); }

// c = floor(W 2^shift) as a 64-bit count (exact: power-of-two scaling, floor). The scaling is two
// products by powers of two, each of half the exponent (|shift| <= 211 in FP32, 1136 in FP64, so
// both factors are normal numbers): where the result is at least 1, W, the product between and the
// result are ordered in magnitude, so both products are exact, as ldexp is; below 1 the floor is 0.
template <typename T>
__device__ __forceinline__ unsigned long long quantize_u64(T W, int shift) {
  const int h = shift / 2;
  return (unsigned long long)floor(W * pow2_t<T>(h) * pow2_t<T>(shift - h));
}

// Q consecutive weights from w[i], zeros past n: 16-byte loads where `vec` (w on 16 bytes, i a
// multiple of Q). Plain loads: the weights may have been written earlier in the same kernel.
template <typename T, int Q>
__device__ __forceinline__ void load_weights(const T* w, long long i, long long n, bool vec, T (&v)[Q]) {
  if (vec && i + Q <= n) {
    constexpr int V = 16 / (int)sizeof(T);
#pragma unroll
    for (int q = 0; q < Q / V; ++q) {
      const uint4 b = reinterpret_cast<const uint4*>(w + i)[q];
      memcpy(&v[q * V], &b, 16);
    }
  } else {
#pragma unroll
    for (int q = 0; q < Q; ++q) v[q] = i + q < n ? w[i + q] : T(0);
  }
}

// The exclusive prefix of CTA `bid`'s count total and the total C of the `nb` CTAs of OF_NT
// threads, once every CTA's total is in place (block-wide: every thread receives both).
__device__ __forceinline__ void count_prefix(const unsigned long long* ctot, int bid, int nb,
                                             unsigned long long& pre, unsigned long long& C) {
  constexpr int NW = OF_NT / 32;
  __shared__ unsigned long long su[2][NW];
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  unsigned long long p = 0, t = 0;
  for (int b = tid; b < nb; b += OF_NT) {
    const unsigned long long c = __ldcg(ctot + b);
    t += c;
    if (b < bid) p += c;
  }
  p = warp_sum(p);
  t = warp_sum(t);
  __syncthreads();
  if (lane == 0) {
    su[0][w] = p;
    su[1][w] = t;
  }
  __syncthreads();
  pre = 0;
  C = 0;
#pragma unroll
  for (int r = 0; r < NW; ++r) {
    pre += su[0][r];
    C += su[1][r];
  }
}

// The outputs of one CTA (OF_NT threads): items i0 .. iend - 1 of n, the CTAs before it holding `pre`
// of the total count C > 0. Chunk by chunk (IPT consecutive items a thread): the items' counts
// (load(i, W) gives a thread's weights, zeros past iend; quant the count of one), their scan, the
// number of systematic points below each cumulative count, and then output k takes the item j with
// K[j] <= k < K[j + 1]. That last step is a warp's own: its 32 IPT items own a contiguous range of
// outputs, taken in windows of 32 IPT; every item with outputs marks its first one, a maximum scan
// over the window (eight slots a lane, then shuffles) carries the marks forward, and the window
// leaves in whole lines. What bounds it is shared memory and latency: a binary search among the
// block's counts read 11 words an output, one after another, where this moves about one and a half,
// and it has no block barrier (a particle filter's step at N = 8,454,144: 303 us, now 275; dpf_resample
// at n = 1,000,003, with its grid of four CTAs an SM: 80 us, now 68). slots: OF_NT IPT ints on 16 bytes, su: OF_NT / 32 words of shared memory.
constexpr int SCATTER_IPT_LONG = 8;  // items a thread where a CTA owns many

// SCALED: by the 64-bit product (points_below); else by the estimate alone, kept to one copy of its
// 128-bit comparisons, which a kernel that runs once through its code has to fetch.
template <typename T, int IPT, bool SCALED, class Load, class Quant>
__device__ __forceinline__ void scatter_range(long long i0, long long iend, long long n, uint32_t u,
                                              unsigned long long pre, unsigned long long C, const PointScale ps,
                                              int32_t* out, int* slots, unsigned long long* su, Load load, Quant quant) {
  constexpr int NW = OF_NT / 32, CHUNK = OF_NT * IPT, WIN = 32 * IPT;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  int* const slot = slots + w * WIN;
  typedef typename std::conditional<IPT % 4 == 0, int4, int2>::type Vec;
  constexpr int VI = (int)sizeof(Vec) / 4;
  static_assert(IPT % VI == 0, "whole vectors a lane");
  unsigned long long run = pre;
  for (long long base = i0; base < iend; base += CHUNK) {
    unsigned long long c[IPT], ts = 0;
    T W[IPT];
    load(base + tid * IPT, W);
#pragma unroll
    for (int q = 0; q < IPT; ++q) {
      c[q] = quant(W[q]);
      ts += c[q];
    }
    // exclusive block scan of the per-thread sums
    unsigned long long incl = ts;
#pragma unroll
    for (int s = 1; s < 32; s <<= 1) {
      const unsigned long long m = __shfl_up_sync(FULL, incl, s);
      if (lane >= s) incl += m;
    }
    if (lane == 31) su[w] = incl;
    __syncthreads();
    unsigned long long wpre = 0, agg = 0;
#pragma unroll
    for (int r = 0; r < NW; ++r) {
      if (r < w) wpre += su[r];
      agg += su[r];
    }
    unsigned long long cum = run + wpre + incl - ts;
    int K[IPT + 1];  // points below each of the thread's items, and below the one after them
    K[0] = 0;
    if constexpr (SCALED) {
      if (lane == 0) K[0] = points_below(cum, n, u, C, ps);
#pragma unroll
      for (int q = 0; q < IPT; ++q) {
        cum += c[q];
        K[q + 1] = points_below(cum, n, u, C, ps);
      }
    } else {
      static_assert(IPT == 2, "the short form");
      const unsigned long long c0 = cum + c[0], c1 = c0 + c[1];
#pragma unroll 1
      for (int q = lane == 0 ? -1 : 0; q < 2; ++q) {
        const int v = points_below_est(q < 0 ? cum : q == 0 ? c0 : c1, n, u, C);
        if (q < 0) K[0] = v;
        else if (q == 0) K[1] = v;
        else K[2] = v;
      }
      __syncwarp();
    }
    {
      const int before = __shfl_up_sync(FULL, K[IPT], 1);
      if (lane > 0) K[0] = before;
    }
    const int kbeg = __shfl_sync(FULL, K[0], 0), kend = __shfl_sync(FULL, K[IPT], 31);
    int carry = -1;  // the item whose outputs reach into the window (the first window starts with a mark)
    for (int k0 = kbeg, left = kend - kbeg; left > 0; left -= WIN, k0 = (int)((unsigned)k0 + WIN)) {
      int v[IPT];
#pragma unroll
      for (int q = 0; q < IPT; ++q) v[q] = -1;
#pragma unroll
      for (int q = 0; q < IPT; q += VI) {
        Vec x;
        memcpy(&x, v + q, sizeof(Vec));
        *reinterpret_cast<Vec*>(slot + lane * IPT + q) = x;
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < IPT; ++q)
        if (K[q + 1] > K[q] && (unsigned)(K[q] - k0) < (unsigned)WIN) slot[K[q] - k0] = lane * IPT + q;
      __syncwarp();
#pragma unroll
      for (int q = 0; q < IPT; q += VI) {
        const Vec x = *reinterpret_cast<const Vec*>(slot + lane * IPT + q);
        memcpy(v + q, &x, sizeof(Vec));
      }
#pragma unroll
      for (int q = 1; q < IPT; ++q) v[q] = max(v[q], v[q - 1]);
      int m = max(v[IPT - 1], carry);
#pragma unroll
      for (int s = 1; s < 32; s <<= 1) {
        const int o = __shfl_up_sync(FULL, m, s);
        if (lane >= s) m = max(m, o);
      }
      const int o = __shfl_up_sync(FULL, m, 1), first = lane > 0 ? o : carry;
      carry = __shfl_sync(FULL, m, 31);
#pragma unroll
      for (int q = 0; q < IPT; ++q) v[q] = max(v[q], first);
#pragma unroll
      for (int q = 0; q < IPT; q += VI) {
        Vec x;
        memcpy(&x, v + q, sizeof(Vec));
        *reinterpret_cast<Vec*>(slot + lane * IPT + q) = x;
      }
      __syncwarp();
#pragma unroll
      for (int q = 0; q < IPT; ++q) {
        const int e = lane + 32 * q;
        if (e < left) out[k0 + e] = (int32_t)(base + w * WIN) + slot[e];
      }
      __syncwarp();  // the slots are written again by the next window
    }
    run += agg;
    __syncthreads();  // su is reused by the next chunk
  }
}

}  // namespace dpf
