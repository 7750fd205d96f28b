// The outer stage of one step: the evidence increment, the ESS and the filtered
// mean (eq. weightsopt), and the global systematic resampling of the N outer
// particles (Fig. 4 step 3).
//
// A single filter runs it in one cooperative launch (every CTA resident at
// once) with one grid-wide barrier:
//   A. each CTA sums W_i = exp(lw_i - max lw), W_i^2, W_i times the particle's
//      x and z means, and the quantised counts c_i = floor(W_i 2^S), over its
//      contiguous range of items;
//   B. the CTAs publish their count totals and wait for one another (a bounded
//      wait); each then reads the totals of the CTAs before it (its exclusive
//      prefix) and of all of them (the quantised total C);
//   C. each CTA scans its items' counts chunk by chunk, turns each cumulative
//      count into the number of systematic points below it, and writes the
//      ancestor of every point that falls in the chunk;
//   D. one CTA combines the partial sums into the statistics (an extra CTA with no
//      items where the grid has room for it, so that this serial double-precision
//      work overlaps the others' scatter), and the last CTA to finish resets the
//      counters for the next step.
// Many filters run the same phases in two ordinary launches (A, then B-D), the
// launch boundary standing in for the barrier, with each filter's partition
// unchanged, so their results are bit-identical to the single launch's.
// The integer rule is the one dpf_resample's global scan applies (S = 62 -
// ceil(log2 N); output k takes the first item with cum * N 2^32 > (k 2^32 + u) C),
// so the ancestors are the ones it would return for the same weights and word.
#pragma once

#include <cuda/atomic>

#include "dpf_common.cuh"
#include "dpf_internal.h"
#include "dpf_resample.cuh"
#include "dpf_step.cuh"

namespace dpf {

template <typename T>
struct FusedOuterArgs {
  OuterArgs<T> o;               // weights, means, statistics, counters
  T* w_out;                     // the W_i fed to the rule (may be null)
  int32_t* anc;                 // the N ancestors
  unsigned long long* ctot;     // one count total a CTA
  unsigned int* arrive;         // barrier arrivals, reset by the last CTA (null: no barrier)
  int nwork;                    // CTAs that own items; one more, if launched, only computes statistics
  int shift;                    // S = 62 - ceil(log2 N)
  double logN;                  // log N
  Key key;                      // u = rand_word(key, t, 0, P_OUTER, 0)
  uint32_t t;
  int withhold;                 // a CTA that never arrives (a check of the bounded wait); -1: none
  double* host_stats;           // a pinned host mirror of stats[0 .. 4 + d) and the error word, or null
};

// ---- A: the partial sums and the count total of CTA `bid` of the `nb` CTAs of one filter ----
// What only the bootstrap particle filter's outer stage does (PF; its sets are a hundred times
// larger and its step has the weighted sums already). The other filters' stage is a few microseconds
// of latency, most of it cold instruction fetches, so none of it is compiled into theirs.
// Whether a CTA owns at least two long chunks of the scatter.
template <typename T>
__device__ __forceinline__ bool long_ranges(const FusedOuterArgs<T>& a, int nb) {
  const long long nch = (a.o.N + OF_CHUNK - 1) / OF_CHUNK;
  return a.w_out && nch >= (long long)nb * 2 * SCATTER_IPT_LONG / OF_IPT;
}

// Whether the sums that came with the step serve (OuterArgs::npre): with the largest weight at
// least e^-20 of the reference its square is 4e-18, so single precision holds W'^2 and every
// weight of consequence beside it.
template <typename T>
__device__ __forceinline__ bool sums_given(const OuterArgs<T>& o, T lwmax) {
  return o.npre > 0 && lwmax >= o.lref - T(20) && lwmax <= o.lref + T(20);
}

template <typename T, int D1, int D2, bool PF>
__device__ __forceinline__ void outer_sums(const FusedOuterArgs<T>& a, int bid, int nb, T lwmax) {
  constexpr int NV = 2 + D1 + D2, NW = OF_NT / 32;
  __shared__ T sv[NV][NW];
  __shared__ unsigned long long su[NW];
  const OuterArgs<T>& o = a.o;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const long long N = o.N;
  const T sS = pow2_t<T>(a.shift);
  const long long nch = (N + OF_CHUNK - 1) / OF_CHUNK;
  const long long i0 = nch * bid / nb * OF_CHUNK, i1 = nch * (bid + 1) / nb * OF_CHUNK;
  const long long iend = i1 < N ? i1 : N;
  const bool given = PF && sums_given(o, lwmax), keep = PF && long_ranges(a, nb);  // uniform over the grid
  unsigned long long cc = 0;
  if (given) {
    for (long long i = i0 + tid; i < iend; i += OF_NT) {
      const T W = exp_t<T>(o.lw[i] - lwmax);
      if (keep) a.w_out[i] = W;
      cc += (unsigned long long)floor(W * sS);
    }
  } else {
    T v[NV];
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = T(0);
    for (long long i = i0 + tid; i < iend; i += OF_NT) {
      // every load of the item first (d of them in flight, not one product's at a time)
      T m[D1 + D2];
#pragma unroll
      for (int c = 0; c < D1; ++c) m[c] = PF ? o.xm[c * o.xc + i * o.xi] : o.xm[(long long)c * N + i];
#pragma unroll
      for (int c = 0; c < D2; ++c) m[D1 + c] = o.zm[(long long)c * N + i];
      const T W = exp_t<T>(o.lw[i] - lwmax);
      if (keep) a.w_out[i] = W;
      cc += (unsigned long long)floor(W * sS);  // exact: a power-of-two scaling, then a floor
      v[0] += W;
      v[1] += W * W;
#pragma unroll
      for (int c = 0; c < D1 + D2; ++c) v[2 + c] += W * m[c];
    }
#pragma unroll
    for (int q = 0; q < NV; ++q) v[q] = warp_sum(v[q]);
    if (lane == 0) {
#pragma unroll
      for (int q = 0; q < NV; ++q) sv[q][w] = v[q];
    }
  }
  cc = warp_sum(cc);
  if (lane == 0) su[w] = cc;
  __syncthreads();
  // the CTA's row, a thread a sum (the caller's barrier and its one thread's fence cover them all)
  if (!given && tid < NV) {
    T s = T(0);
#pragma unroll
    for (int r = 0; r < NW; ++r) s += sv[tid][r];
    o.partials[(long long)bid * NV + tid] = (double)s;
  }
  if (tid == OF_NT - 1) {
    unsigned long long s = 0;
#pragma unroll
    for (int r = 0; r < NW; ++r) s += su[r];
    a.ctot[bid] = s;
  }
}

// ---- C: the chunks' cumulative counts, the points below them, the ancestors (C > 0). A CTA of a
// large particle set (at least two long chunks each) reads back the weights the sums left in w_out
// and takes four times the items between barriers; else the weights are formed again from the
// log-weights, which the sums have just brought into the L1 cache ----
template <typename T, bool PF>
__device__ __forceinline__ void outer_scatter(const FusedOuterArgs<T>& a, int bid, int nb, T lwmax,
                                              unsigned long long pre, unsigned long long C) {
  __shared__ unsigned long long su[OF_NT / 32];
  __shared__ __align__(16) int slots[OF_NT * (PF ? SCATTER_IPT_LONG : OF_IPT)];
  const OuterArgs<T>& o = a.o;
  const long long N = o.N;
  const T sS = pow2_t<T>(a.shift);
  const long long nch = (N + OF_CHUNK - 1) / OF_CHUNK;
  const long long i0 = nch * bid / nb * OF_CHUNK, i1 = nch * (bid + 1) / nb * OF_CHUNK;
  const long long iend = i1 < N ? i1 : N;
  const uint32_t u = rand_word(a.key, a.t, 0, P_OUTER, 0);
  auto quant = [&](T W) { return (unsigned long long)floor(W * sS); };
  if constexpr (PF) {
    if (long_ranges(a, nb)) {
      __shared__ PointScale s_ps;
      if (threadIdx.x == 0) s_ps = point_scale(N, C);
      __syncthreads();
      auto load = [&](long long i, T (&W)[SCATTER_IPT_LONG]) {
        load_weights<T, SCATTER_IPT_LONG>(a.w_out, i, iend, true, W);
      };
      scatter_range<T, SCATTER_IPT_LONG, true>(i0, iend, N, u, pre, C, s_ps, a.anc, slots, su, load, quant);
      return;
    }
  }
  auto load = [&](long long i, T (&W)[OF_IPT]) {
#pragma unroll
    for (int q = 0; q < OF_IPT; ++q) {
      W[q] = T(0);
      if (i + q < iend) {
        W[q] = exp_t<T>(o.lw[i + q] - lwmax);
        if (a.w_out) a.w_out[i + q] = W[q];
      }
    }
  };
  scatter_range<T, OF_IPT, false>(i0, iend, N, u, pre, C, PointScale{0ull, -1}, a.anc, slots, su, load, quant);
}

// ---- D: the statistics from the `nb` CTAs' partial sums, by one CTA once they are
// all in place ----
template <typename T, bool PF>
__device__ __forceinline__ void outer_stats(const FusedOuterArgs<T>& a, int nb, T lwmax,
                                            unsigned long long C) {
  constexpr int NW = OF_NT / 32;
  __shared__ double sd[OF_MAX_NV];
  const OuterArgs<T>& o = a.o;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5;
  const int D = o.d1 + o.d2, NV = 2 + D;
  const bool given = PF && sums_given(o, lwmax);
  const int rows = given ? o.npre : nb;
  // a warp a sum; four of its rows in flight
  for (int q = w; q < NV; q += NW) {
    double s = 0.0;
#pragma unroll 4
    for (int b = lane; b < rows; b += 32) s += __ldcg(o.partials + (long long)b * NV + q);
    s = warp_sum(s);
    if (lane == 0) sd[q] = s;
  }
  __syncthreads();
  const double t1 = sd[0];
  for (int c = tid; c < D; c += OF_NT) {
    const double m = sd[2 + c] / t1;
    const int p = o.perm[c];
    o.stats[4 + p] = m;
    if (o.mean_out) o.mean_out[p] = m;
  }
  if (tid == 0) {
    const bool bad = !(lwmax > neg_inf<T>()) || lwmax != lwmax || !(t1 > 0) || C == 0;
    if (bad) atomicOr(o.err, ERR_NUMERIC);
    const double lz = (given ? (double)o.lref : (double)lwmax) + log(t1) - a.logN;
    o.stats[0] += lz;
    o.stats[1] = lz;
    o.stats[2] = t1 * t1 / sd[1];
    o.stats[3] = given ? t1 * exp((double)o.lref - (double)lwmax) : t1;
    if (o.logz_out) *o.logz_out = o.stats[0];
    *o.lwmax_t = lwmax;
    *o.Csum = C;
  }
  if (a.host_stats) {  // the mirror: the statistics as written above, then the error word
    __syncthreads();
    for (int q = tid; q < 4 + D; q += OF_NT) a.host_stats[q] = o.stats[q];
    if (tid == 0) a.host_stats[4 + D] = (double)*(volatile int*)o.err;
  }
}

// The last of the `nb` CTAs to get here resets the counters for the next step: by
// then every CTA has read the largest log-weight's key and passed the barrier.
template <typename T>
__device__ __forceinline__ void outer_done(const FusedOuterArgs<T>& a, int nb) {
  __syncthreads();
  if (threadIdx.x == 0 && atomicAdd(a.o.done, 1u) == (unsigned)nb - 1u) {
    *a.o.lwmax_key = 0ull;
    *a.o.done = 0u;
    if (a.arrive) *a.arrive = 0u;
  }
}

// One filter's outer stage in one cooperative launch (every CTA resident at once).
template <typename T, int D1, int D2, bool PF>
__global__ void __launch_bounds__(OF_NT) fused_outer_kernel(const __grid_constant__ FusedOuterArgs<T> a) {
  __shared__ int s_ok;
  const int tid = threadIdx.x, bid = blockIdx.x, nb = gridDim.x, nw = a.nwork;
  T lwmax;
  order_decode(*a.o.lwmax_key, lwmax);
  if (bid < nw) outer_sums<T, D1, D2, PF>(a, bid, nw, lwmax);
  __syncthreads();
  // grid-wide barrier: every CTA is resident, and the wait is bounded all the same
  if (tid == 0) {
    __threadfence();  // the CTA's partial row and count total, written before the barrier above
    cuda::atomic_ref<unsigned int, cuda::thread_scope_device> arr(*a.arrive);
    if (bid != a.withhold) arr.fetch_add(1u, cuda::memory_order_release);
    bool ok = arr.load(cuda::memory_order_acquire) >= (unsigned)nb;
    int spins = 0;
    while (!ok && spins < SPIN_LIMIT) {
      __nanosleep(64);
      ok = arr.load(cuda::memory_order_acquire) >= (unsigned)nb;
      ++spins;
    }
    s_ok = ok;
    if (!ok) atomicOr(a.o.err, ERR_TIMEOUT);
  }
  __syncthreads();
  unsigned long long pre, C;
  count_prefix(a.ctot, bid < nw ? bid : nw, nw, pre, C);
  if (bid == (nb > nw ? nw : nw - 1)) outer_stats<T, PF>(a, nw, lwmax, C);
  if (bid < nw && s_ok && C > 0) outer_scatter<T, PF>(a, bid, nw, lwmax, pre, C);  // else the ancestors stay
  outer_done<T>(a, nb);
}

// The same stage for many filters in two launches, CTAs cstart[f] .. cstart[f+1]-1
// serving filter f with the partition and arithmetic of its single launch: the
// sums, then (after the launch boundary) the prefix, the scatter and the statistics.
template <typename T, int D1, int D2>
__global__ void __launch_bounds__(OF_NT)
    outer_sums_batch_kernel(const FusedOuterArgs<T>* __restrict__ args, const int* __restrict__ cstart, int F) {
  __shared__ int s_f;
  if (threadIdx.x == 0) s_f = find_segment(cstart, F, (int)blockIdx.x);
  __syncthreads();
  const int f = s_f;
  const FusedOuterArgs<T>& a = args[f];
  T lwmax;
  order_decode(*a.o.lwmax_key, lwmax);
  outer_sums<T, D1, D2, false>(a, (int)blockIdx.x - cstart[f], cstart[f + 1] - cstart[f], lwmax);
}

template <typename T>
__global__ void __launch_bounds__(OF_NT)
    outer_scatter_batch_kernel(const FusedOuterArgs<T>* __restrict__ args, const int* __restrict__ cstart, int F) {
  __shared__ int s_f;
  if (threadIdx.x == 0) s_f = find_segment(cstart, F, (int)blockIdx.x);
  __syncthreads();
  const int f = s_f;
  const FusedOuterArgs<T>& a = args[f];
  const int bid = (int)blockIdx.x - cstart[f], nb = cstart[f + 1] - cstart[f];
  T lwmax;
  order_decode(*a.o.lwmax_key, lwmax);
  unsigned long long pre, C;
  count_prefix(a.ctot, bid, nb, pre, C);
  if (C > 0) outer_scatter<T, false>(a, bid, nb, lwmax, pre, C);
  if (bid == nb - 1) outer_stats<T, false>(a, nb, lwmax, C);
  outer_done<T>(a, nb);
}

// CTAs resident on the device at once for the single-filter launch.
template <typename T, int D1, int D2, bool PF = false>
int fused_outer_cap() {
  static const int cap = [] {
    int dev = 0, sms = 0, occ = 0;
    cudaGetDevice(&dev);
    cudaDeviceGetAttribute(&sms, cudaDevAttrMultiProcessorCount, dev);
    cudaOccupancyMaxActiveBlocksPerMultiprocessor(&occ, fused_outer_kernel<T, D1, D2, PF>, OF_NT, 0);
    const int c = occ * sms;
    return c < 2 ? 2 : c;
  }();
  return cap;
}

// CTAs that own items in a filter's outer stage over N items: one a chunk, at most
// OF_MAX_CTAS and one fewer than the resident capacity (the same in the single and
// batched forms, so that their partitions agree).
template <typename T, int D1, int D2, bool PF = false>
int fused_outer_grid(long long N) {
  const long long cap = fused_outer_cap<T, D1, D2, PF>() - 1;
  const long long lim = cap < OF_MAX_CTAS ? cap : OF_MAX_CTAS;
  const long long nch = (N + OF_CHUNK - 1) / OF_CHUNK;
  return (int)(nch < lim ? nch : lim);
}

// The single-filter launch: a.nwork CTAs with items and one for the statistics.
template <typename T, int D1, int D2, bool PF = false>
cudaError_t fused_outer_launch(const FusedOuterArgs<T>& a, cudaStream_t st) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3((unsigned)a.nwork + 1u);
  cfg.blockDim = dim3(OF_NT);
  cfg.dynamicSmemBytes = 0;
  cfg.stream = st;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeCooperative;
  at[0].val.cooperative = 1;
  cfg.attrs = at;
  cfg.numAttrs = 1;
  return cudaLaunchKernelEx(&cfg, fused_outer_kernel<T, D1, D2, PF>, a);
}

}  // namespace dpf
