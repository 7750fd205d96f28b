// Global systematic resampling on the GPU: a reduction for the quantised total
// C, then one pass that scans the quantised counts with a decoupled look-back
// (Merrill & Garland, "Single-pass Parallel Prefix Scan with Decoupled
// Look-back", 2016) and scatters each tile's share of the ancestor indices.
#pragma once

#include <cuda/atomic>
#include <cstring>

#include "dpf_common.cuh"
#include "dpf_internal.h"

namespace dpf {

constexpr int SPIN_LIMIT = 1 << 22;  // bounded look-back wait (~0.3 s with the back-off)

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

// Inputs of the scan-and-scatter pass: the weights W_i, with e = floor(log2 max W)
// given through the shift S - e.
template <typename T>
struct GlobalArgs {
  const T* w;              // n weights
  long long n;
  int shift;               // S - e
  const int* shift_dev;    // if non-null, read S - e from here instead
  const unsigned long long* C;  // device scalar: the quantised total
  const uint32_t* u_ptr;   // device scalar uniform word, or null
  Key key;                 // else u = rand_word(key, t, 0, P_OUTER, 0)
  uint32_t t;
  int32_t* out;
  ScanState st;
  unsigned long long ticket_base;
  uint32_t epoch;
  int* err;
  long long withhold;  // a tile that publishes nothing (a check of the bounded waits); -1: none
};

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
// multiple of Q).
template <typename T, int Q>
__device__ __forceinline__ void load_weights(const T* __restrict__ w, long long i, long long n, bool vec, T (&v)[Q]) {
  if (vec && i + Q <= n) {
    constexpr int V = 16 / (int)sizeof(T);
#pragma unroll
    for (int q = 0; q < Q / V; ++q) {
      const uint4 b = __ldg(reinterpret_cast<const uint4*>(w + i) + q);
      memcpy(&v[q * V], &b, 16);
    }
  } else {
#pragma unroll
    for (int q = 0; q < Q; ++q) v[q] = i + q < n ? w[i + q] : T(0);
  }
}

// One tile of the `ntiles` tiles of one resampling, the tile taken by ticket.
template <typename T>
__device__ __forceinline__ void global_scan_scatter_body(const GlobalArgs<T>& a, long long ntiles) {
  __shared__ int ks[SCAN_TILE + 1];  // systematic points below each item's cumulative count
  __shared__ unsigned long long wsum[SCAN_NT / 32];
  __shared__ unsigned long long s_prefix;
  __shared__ long long s_tile;
  const int tid = threadIdx.x, lane = tid & 31, wid = tid >> 5;

  if (tid == 0) {
    const unsigned long long tk = atomicAdd(a.st.ticket, 1ull) - a.ticket_base;
    s_tile = tk < (unsigned long long)ntiles ? (long long)tk : -1;
    if (s_tile < 0) atomicOr(a.err, ERR_BOUNDS);
  }
  __syncthreads();
  const long long tile = s_tile;
  if (tile < 0) return;
  const long long base = tile * SCAN_TILE;
  const unsigned long long C = *a.C;
  if (C == 0) return;  // no positive finite weight (flagged): in every tile, so none waits for another
  const int shift = a.shift_dev ? *a.shift_dev : a.shift;
  const uint32_t u = a.u_ptr ? *a.u_ptr : rand_word(a.key, a.t, 0, P_OUTER, 0);

  // quantise this thread's items (blocked arrangement) and sum them
  unsigned long long c[SCAN_IPT];
  unsigned long long tsum = 0;
  {
    T W[SCAN_IPT];
    load_weights<T, SCAN_IPT>(a.w, base + (long long)tid * SCAN_IPT, a.n, ((uintptr_t)a.w & 15) == 0, W);
#pragma unroll
    for (int q = 0; q < SCAN_IPT; ++q) {
      c[q] = quantize_u64(W[q], shift);
      tsum += c[q];
    }
  }
  // block exclusive scan of the per-thread sums
  unsigned long long v = tsum;
#pragma unroll
  for (int o = 1; o < 32; o <<= 1) {
    const unsigned long long nb = __shfl_up_sync(FULL, v, o);
    if (lane >= o) v += nb;
  }
  if (lane == 31) wsum[wid] = v;
  __syncthreads();
  unsigned long long wpre = 0, agg = 0;
#pragma unroll
  for (int q = 0; q < SCAN_NT / 32; ++q) {
    if (q < wid) wpre += wsum[q];
    agg += wsum[q];
  }
  const unsigned long long texcl = v - tsum + wpre;

  // decoupled look-back for the tile's exclusive prefix: warp 0 publishes the
  // tile's aggregate, then reads its predecessors' flags 32 at a time until it
  // meets an inclusive prefix (every wait is bounded)
  if (wid == 0) {
    const uint32_t ep = a.epoch & 0x3FFFFFFFu;
    unsigned long long prefix = 0;
    if (tile == a.withhold) {
      // publishes nothing: its successors' waits must run out and report
    } else if (tile == 0) {
      if (lane == 0) {
        a.st.incl[0] = agg;
        cuda::atomic_ref<uint32_t, cuda::thread_scope_device>(a.st.flags[0])
            .store((ep << 2) | 2u, cuda::memory_order_release);
      }
    } else {
      if (lane == 0) {
        a.st.agg[tile] = agg;
        cuda::atomic_ref<uint32_t, cuda::thread_scope_device>(a.st.flags[tile])
            .store((ep << 2) | 1u, cuda::memory_order_release);
      }
      long long hi = tile - 1;
      while (true) {
        const long long j = hi - lane;
        uint32_t fv = 0;
        bool ready = true;
        if (j >= 0) {
          cuda::atomic_ref<uint32_t, cuda::thread_scope_device> f(a.st.flags[j]);
          fv = f.load(cuda::memory_order_acquire);
          ready = (fv >> 2) == ep && (fv & 3u) != 0u;
          int spins = 0;
          while (!ready && spins < SPIN_LIMIT) {
            __nanosleep(64);
            fv = f.load(cuda::memory_order_acquire);
            ready = (fv >> 2) == ep && (fv & 3u) != 0u;
            ++spins;
          }
        }
        if (!__all_sync(FULL, ready)) {
          if (lane == 0) atomicOr(a.err, ERR_TIMEOUT);
          break;
        }
        const unsigned inc = __ballot_sync(FULL, j >= 0 && (fv & 3u) == 2u);
        const int first = inc ? __ffs(inc) - 1 : 32;
        unsigned long long val = 0;
        if (j >= 0 && lane <= first) val = lane == first ? a.st.incl[j] : a.st.agg[j];
#pragma unroll
        for (int o = 16; o > 0; o >>= 1) val += __shfl_xor_sync(FULL, val, o);
        prefix += val;
        if (inc || hi < 32) break;
        hi -= 32;
      }
      if (lane == 0) {
        a.st.incl[tile] = prefix + agg;
        cuda::atomic_ref<uint32_t, cuda::thread_scope_device>(a.st.flags[tile])
            .store((ep << 2) | 2u, cuda::memory_order_release);
      }
    }
    if (lane == 0) s_prefix = prefix;
  }
  __syncthreads();
  // scatter: output k takes the item j of this tile with ks[j] <= k < ks[j + 1]. The exact 128-bit
  // arithmetic is done once an item (the count of points below its cumulative count) and the
  // search compares 32-bit counts; a search on cumulative counts took eleven 128-bit products
  // an output (36 us of a call at n = 1,000,003)
  unsigned long long run = s_prefix + texcl;
  if (tid == 0) ks[0] = points_below_est(run, a.n, u, C);
#pragma unroll
  for (int q = 0; q < SCAN_IPT; ++q) {
    run += c[q];
    ks[tid * SCAN_IPT + q + 1] = points_below_est(run, a.n, u, C);
  }
  __syncthreads();
  const int khi = ks[SCAN_TILE];
  for (int k = ks[0] + tid; k < khi; k += SCAN_NT) {
    int lo = 0, hi = SCAN_TILE;
    while (hi - lo > 1) {
      const int mid = (lo + hi) >> 1;
      if (ks[mid] <= k)
        lo = mid;
      else
        hi = mid;
    }
    a.out[k] = (int32_t)(base + lo);
  }
}

template <typename T>
__global__ void __launch_bounds__(SCAN_NT) global_scan_scatter(GlobalArgs<T> a) {
  global_scan_scatter_body<T>(a, gridDim.x);
}

}  // namespace dpf
