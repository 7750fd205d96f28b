// dpf_resample: the standalone systematic-resampling entry point (global rule
// over one segment, or the local rule over many short segments).
#include <cuda_runtime.h>

#include <cmath>
#include <cstring>

#include "dpf_internal.h"
#include "dpf_resample.cuh"

namespace dpf {

// The global rule in three passes over the same partition (CTA b of nb owns a contiguous range of
// 512-item chunks): the largest weight, the counts' totals, and the scatter, whose prefix comes from
// the totals before it. The launch boundaries stand in for grid barriers; no CTA waits for another.
// (A single scan pass with decoupled look-back took 25 us at n = 1,000,003, of a call of 84,
// waiting along its chain of tiles; in three passes it took 78, and 68 with a warp's outputs by marks.)
constexpr int RS_Q = 8;  // weights a thread loads at once
constexpr unsigned long long RS_BAD = ~0ull;

struct RsRange {
  long long i0, iend;
};
__device__ __forceinline__ RsRange rs_range(long long n, int bid, int nb) {
  const long long nch = (n + 511) / 512;
  const long long i1 = nch * (bid + 1) / nb * 512;
  return RsRange{nch * bid / nb * 512, i1 < n ? i1 : n};
}

// keys[b]: the bits of CTA b's largest weight (weights are >= 0, so the IEEE bit pattern orders like
// the value), RS_BAD where a weight is negative, NaN or infinite.
template <typename T>
__global__ void __launch_bounds__(OF_NT) resample_max_kernel(const T* w, long long n, unsigned long long* keys) {
  __shared__ unsigned long long su[OF_NT / 32];
  const RsRange r = rs_range(n, blockIdx.x, gridDim.x);
  const bool vec = ((uintptr_t)w & 15) == 0;
  T best = T(0);
  bool bad = false;
  for (long long i = r.i0 + threadIdx.x * RS_Q; i < r.iend; i += OF_NT * RS_Q) {
    T W[RS_Q];
    load_weights<T, RS_Q>(w, i, r.iend, vec, W);
#pragma unroll
    for (int q = 0; q < RS_Q; ++q) {
      bad |= !(W[q] >= T(0)) || isinf(W[q]);
      best = fmax(best, W[q]);
    }
  }
  best = warp_max(best);
  bad = __any_sync(FULL, bad);
  if ((threadIdx.x & 31) == 0)
    su[threadIdx.x >> 5] = bad ? RS_BAD
                               : sizeof(T) == 8 ? (unsigned long long)__double_as_longlong((double)best)
                                                : (unsigned long long)__float_as_uint((float)best);
  __syncthreads();
  if (threadIdx.x == 0) {
    unsigned long long k = 0;
#pragma unroll
    for (int q = 0; q < OF_NT / 32; ++q) k = su[q] > k ? su[q] : k;
    keys[blockIdx.x] = k;
  }
}

// The shift S - e of the largest of the nb keys, with S = 62 - ceil(log2 n); false where no weight
// is positive or one is bad. Block-wide.
template <typename T>
__device__ __forceinline__ bool rs_shift(const unsigned long long* keys, int nb, long long n, int& shift) {
  __shared__ unsigned long long su[OF_NT / 32];
  unsigned long long k = 0;
  for (int b = threadIdx.x; b < nb; b += OF_NT) {
    const unsigned long long v = keys[b];
    k = v > k ? v : k;
  }
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const unsigned long long v = __shfl_xor_sync(FULL, k, o);
    k = v > k ? v : k;
  }
  if ((threadIdx.x & 31) == 0) su[threadIdx.x >> 5] = k;
  __syncthreads();
  k = su[0];
#pragma unroll
  for (int q = 1; q < OF_NT / 32; ++q) k = su[q] > k ? su[q] : k;
  if (k == 0 || k == RS_BAD) return false;
  const int e = sizeof(T) == 8 ? ilogb(__longlong_as_double((long long)k)) : ilogbf(__uint_as_float((uint32_t)k));
  shift = 62 - ceil_log2_i(n) - e;
  return true;
}

// totals[b] = sum of floor(W_i 2^(S - e)) over CTA b's weights.
template <typename T>
__global__ void __launch_bounds__(OF_NT)
    resample_sum_kernel(const T* w, long long n, const unsigned long long* keys, unsigned long long* totals) {
  __shared__ unsigned long long su[OF_NT / 32];
  int shift = 0;
  const bool ok = rs_shift<T>(keys, gridDim.x, n, shift);
  const RsRange r = rs_range(n, blockIdx.x, gridDim.x);
  const bool vec = ((uintptr_t)w & 15) == 0;
  unsigned long long s = 0;
  for (long long i = ok ? r.i0 + threadIdx.x * RS_Q : r.iend; i < r.iend; i += OF_NT * RS_Q) {
    T W[RS_Q];
    load_weights<T, RS_Q>(w, i, r.iend, vec, W);
#pragma unroll
    for (int q = 0; q < RS_Q; ++q) s += quantize_u64(W[q], shift);
  }
  s = warp_sum(s);
  if ((threadIdx.x & 31) == 0) su[threadIdx.x >> 5] = s;
  __syncthreads();
  if (threadIdx.x == 0) {
    s = 0;
#pragma unroll
    for (int q = 0; q < OF_NT / 32; ++q) s += su[q];
    totals[blockIdx.x] = s;
  }
}

// The ancestors; also the call's error word.
template <typename T>
__global__ void __launch_bounds__(OF_NT)
    resample_scatter_kernel(const T* w, long long n, const uint32_t* up, const unsigned long long* keys,
                            const unsigned long long* totals, int32_t* out, int* err) {
  __shared__ unsigned long long su[OF_NT / 32];
  __shared__ __align__(16) int slots[OF_NT * SCATTER_IPT_LONG];
  __shared__ PointScale s_ps;
  int shift = 0;
  const bool ok = rs_shift<T>(keys, gridDim.x, n, shift);
  unsigned long long pre, C;
  count_prefix(totals, blockIdx.x, gridDim.x, pre, C);
  if (blockIdx.x == 0 && threadIdx.x == 0) *err = ok && C > 0 ? 0 : ERR_NUMERIC;
  if (!ok || C == 0) return;
  const RsRange r = rs_range(n, blockIdx.x, gridDim.x);
  const bool vec = ((uintptr_t)w & 15) == 0;
  const bool scaled = n >= (1ll << 17);  // a division a CTA, repaid by a few hundred items
  if (threadIdx.x == 0) s_ps = scaled ? point_scale(n, C) : PointScale{0ull, -1};
  __syncthreads();
  auto quant = [&](T W) { return quantize_u64(W, shift); };
  if (r.iend - r.i0 > OF_CHUNK) {
    auto load = [&](long long i, T (&W)[SCATTER_IPT_LONG]) {
      load_weights<T, SCATTER_IPT_LONG>(w, i, r.iend, vec, W);
    };
    scatter_range<T, SCATTER_IPT_LONG, true>(r.i0, r.iend, n, *up, pre, C, s_ps, out, slots, su, load, quant);
  } else {
    auto load = [&](long long i, T (&W)[OF_IPT]) { load_weights<T, OF_IPT>(w, i, r.iend, false, W); };
    scatter_range<T, OF_IPT, false>(r.i0, r.iend, n, *up, pre, C, s_ps, out, slots, su, load, quant);
  }
}

// Local rule: one block per segment of n <= NT weights.
template <typename T, int NT>
__global__ void __launch_bounds__(NT) local_resample_kernel(const T* w, int n, const uint32_t* u,
                                                            int32_t* out, int* err) {
  __shared__ uint32_t cum[NT];
  __shared__ T redT[NT / 32];
  __shared__ uint32_t redU[NT / 32];
  const long long seg = blockIdx.x;
  const int j = threadIdx.x;
  T W = T(0);
  if (j < n) W = w[seg * n + j];
  const int bad = __syncthreads_or(j < n && (!(W >= T(0)) || isinf(W)));
  if (bad) {
    if (j == 0) atomicOr(err, ERR_NUMERIC);
    return;
  }
  const T mx = block_max<NT>(W, redT);
  if (!(mx > T(0))) {
    if (j == 0) atomicOr(err, ERR_NUMERIC);
    return;
  }
  const int e = sizeof(T) == 8 ? ilogb((double)mx) : ilogbf((float)mx);
  const int shift = (31 - ceil_log2_i(n)) - e;
  const uint32_t c = j < n ? quantize_u32(W, shift) : 0u;
  const uint32_t incl = block_incl_scan_u32<NT>(c, redU);
  cum[j] = incl;
  __syncthreads();
  const uint32_t C = cum[n - 1];
  if (j < n) out[seg * n + j] = sys_local_pick(cum, n, C, n, j, u[seg]);
}

template <typename T>
static dpf_status launch_local(const T* w, int n, long long nseg, const uint32_t* u, int32_t* out,
                               int* err, cudaStream_t s) {
#define DPF_LOCAL_CASE(NTV)                                                      \
  if (n <= NTV) {                                                                \
    local_resample_kernel<T, NTV><<<(unsigned)nseg, NTV, 0, s>>>(w, n, u, out, err); \
    return DPF_OK;                                                               \
  }
  DPF_LOCAL_CASE(32)
  DPF_LOCAL_CASE(64)
  DPF_LOCAL_CASE(128)
  DPF_LOCAL_CASE(256)
  DPF_LOCAL_CASE(512)
  DPF_LOCAL_CASE(1024)
#undef DPF_LOCAL_CASE
  return set_error(DPF_E_INVALID, "dpf_resample: local segments hold at most 1024 weights");
}

template <typename T>
static void launch_global(const T* w, long long n, const uint32_t* u, int32_t* out, Scratch& sc,
                          cudaStream_t s) {
  const int nb = resample_ctas(n);
  resample_max_kernel<T><<<nb, OF_NT, 0, s>>>(w, n, sc.keys);
  resample_sum_kernel<T><<<nb, OF_NT, 0, s>>>(w, n, sc.keys, sc.totals);
  resample_scatter_kernel<T><<<nb, OF_NT, 0, s>>>(w, n, u, sc.keys, sc.totals, out, sc.err);
}

// Launch the global-rule passes on scratch the caller has laid out.
void launch_global_on(const void* w, int32_t dtype, long long n, const uint32_t* u, int32_t* out,
                      Scratch& sc, cudaStream_t s) {
  if (dtype == DPF_F32)
    launch_global<float>((const float*)w, n, u, out, sc, s);
  else
    launch_global<double>((const double*)w, n, u, out, sc, s);
}

template <typename T>
__global__ void box_muller_kernel(const uint32_t* words, long long n_pairs, T* out) {
  for (long long p = blockIdx.x * (long long)blockDim.x + threadIdx.x; p < n_pairs;
       p += (long long)gridDim.x * blockDim.x) {
    T a, b;
    box_muller(words[2 * p], words[2 * p + 1], a, b);
    out[2 * p] = a;
    out[2 * p + 1] = b;
  }
}

}  // namespace dpf

using namespace dpf;

extern "C" dpf_status dpf_box_muller(const uint32_t* words, int64_t n_pairs, int32_t dtype,
                                     void* out, void* stream) {
  clear_error();
  if (n_pairs < 0 || (n_pairs > 0 && (!words || !out)))
    return set_error(DPF_E_INVALID, "dpf_box_muller: bad arguments");
  if (dtype != DPF_F32 && dtype != DPF_F64) return set_error(DPF_E_INVALID, "dpf_box_muller: dtype");
  if (n_pairs == 0) return DPF_OK;
  const int grid = (int)std::min<long long>((n_pairs + 255) / 256, 152 * 8);
  if (dtype == DPF_F32)
    box_muller_kernel<float><<<grid, 256, 0, (cudaStream_t)stream>>>(words, n_pairs, (float*)out);
  else
    box_muller_kernel<double><<<grid, 256, 0, (cudaStream_t)stream>>>(words, n_pairs, (double*)out);
  return cuda_error(cudaGetLastError(), "dpf_box_muller");
}

extern "C" dpf_status dpf_check_bounded_wait(void* stream) {
  clear_error();
  // a step's wait for staged rows that no copy brings
  dpf_status st = check_stage_wait((cudaStream_t)stream);
  if (st != DPF_E_TIMEOUT)
    return st ? st : set_error(DPF_E_CUDA, "dpf_check_bounded_wait: the wait for staged rows did not run out");
  // the grid barrier of a step's outer stage, which CTA 0 never reaches
  st = check_outer_barrier((cudaStream_t)stream);
  if (st != DPF_E_TIMEOUT)
    return st ? st : set_error(DPF_E_CUDA, "dpf_check_bounded_wait: the outer stage's barrier wait did not run out");
  return st;
}

extern "C" dpf_status dpf_resample(const void* w, int32_t dtype, int64_t n_total, int64_t n_seg,
                                   int32_t rule, const uint32_t* u, int32_t* out_idx,
                                   void* stream) {
  clear_error();
  if (n_total < 0 || n_seg < 1) return set_error(DPF_E_INVALID, "dpf_resample: bad sizes");
  if (n_total == 0) return DPF_OK;
  if (!w || !u || !out_idx) return set_error(DPF_E_INVALID, "dpf_resample: null pointer");
  if (dtype != DPF_F32 && dtype != DPF_F64) return set_error(DPF_E_INVALID, "dpf_resample: dtype");
  if (n_total % n_seg) return set_error(DPF_E_INVALID, "dpf_resample: n_seg must divide n_total");
  if (n_total >= (1ll << 31)) return set_error(DPF_E_INVALID, "dpf_resample: n_total >= 2^31");
  cudaStream_t s = (cudaStream_t)stream;
  const long long seglen = n_total / n_seg;
  if (rule == DPF_SYS_GLOBAL) {
    if (n_seg != 1) return set_error(DPF_E_INVALID, "dpf_resample: global rule needs n_seg == 1");
    Scratch sc;
    dpf_status st = scratch_alloc(sc, resample_ctas(n_total), s);
    if (st) return st;
    launch_global_on(w, dtype, n_total, u, out_idx, sc, s);
    return scratch_finish(sc, s, "dpf_resample");
  }
  if (rule != DPF_SYS_LOCAL) return set_error(DPF_E_INVALID, "dpf_resample: unknown rule");
  if (seglen > 1024) return set_error(DPF_E_INVALID, "dpf_resample: local segments hold <= 1024");
  Scratch sc;
  dpf_status st = scratch_alloc(sc, 0, s);
  if (st) return st;
  cudaMemsetAsync(sc.err, 0, sizeof(int), s);
  st = dtype == DPF_F32
           ? launch_local<float>((const float*)w, (int)seglen, n_seg, u, out_idx, sc.err, s)
           : launch_local<double>((const double*)w, (int)seglen, n_seg, u, out_idx, sc.err, s);
  if (st) {
    scratch_free(sc, s);
    return st;
  }
  return scratch_finish(sc, s, "dpf_resample");
}
