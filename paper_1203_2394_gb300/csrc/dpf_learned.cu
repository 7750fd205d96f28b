// The learned inner proposal: an MLP (3 hidden ReLU layers) with a Gaussian-mixture
// head, its training on the GPU (forward, backward and Adam kernels written here) and
// the packing of its weights for the tensor-core forward pass of the filter step.
//
// Parameters, one FP32 buffer in this order (row-major, W_l is out x in):
//   W1 (H x din), b1 (H), W2 (H x H), b2, W3 (H x H), b3, W4 (dout x H), b4 (dout),
// with dout = C (1 + 2 d2): logits, then the C x d2 means, then the C x d2 raw log
// standard deviations (clamped to [-7, 5] where used).
//
// Training minimises the weighted negative log-likelihood of the recorded
// (features, z) rows, sum_b w_b (-log q(z_b | f_b)) / sum_b w_b, per minibatch, with
// Adam (Kingma and Ba 2015). With bf16 on, the forward pass rounds the inputs, the
// weights and every hidden activation to bfloat16 as the tensor-core pass does
// (gradients pass the rounding straight through); off, it is plain FP32.
#include <cuda_bf16.h>
#include <cuda_runtime.h>

#include <algorithm>
#include <cmath>
#include <cstring>
#include <vector>

#include "dpf_learned.h"
#include "dpf_tc.cuh"

namespace dpf {

// ---- the training products: C[M x N] = op(A) op(B) with an epilogue ----
// A(m, k) = TA ? A[k lda + m] : A[m lda + k];  B(k, n) = TB ? B[n ldb + k] : B[k ldb + n].
// EPI: 0 store; 1 bias, ReLU and optional bfloat16 rounding; 2 bias; 3 multiply by
// (mask(m, n) > 0), mask with leading dimension ldc.
__device__ __forceinline__ float round_bf16(float v) { return __bfloat162float(__float2bfloat16_rn(v)); }

// On the tensor cores (tcgen05):
// One CTA of 512 threads per 128-row x npad-column tile of C (npad <= 64 columns of a
// TMEM accumulator in FP32) and one slice of K (the slices of a long K add their partial
// products into C, which the caller has zeroed: the plain-store epilogue only). The
// threads load op(A) and op(B)^T of a chunk of K from global memory, round them to the
// operand format and write them in the K-major layout without swizzle; one thread issues
// the MMAs (one per 32 bytes of K) and commits them to an mbarrier that every thread waits
// on (bounded; the CTA agrees on the outcome before it reuses the tiles); a warp then reads
// its 32 rows of the accumulator for the epilogue.
// PREC 0: BF16 operands (kind::f16), the forward pass's own rounding; PREC 1: 3xTF32
// (A_hi B_hi + A_hi B_lo + A_lo B_hi, kind::tf32), about FP32 accuracy.
//
// What bounds it: the latency of staging. A training minibatch (1024 rows, width 256) is
// 0.13 GFLOP a product, a microsecond of MMA work, so a CTA's time is the loads of its
// operands from L2. A thread therefore moves units of 8 consecutive K values of one row: two
// 16-byte loads (or, for an operand that is contiguous along its rows, 8 loads each coalesced
// over the warp's 32 rows), one rounding, one 16-byte store, which the 8 x 16-byte core
// matrices of consecutive rows take without bank conflicts; four units are in flight at once,
// and a chunk is as long as shared memory holds twice on an SM (256 BF16 or 64 TF32 values of
// K), so that a forward product is one round of loads, one of MMAs and one epilogue.
constexpr int TG_NT = 512;
constexpr int TG_SPIN = 1 << 22;
constexpr int TG_UNITS = 4;  // staging units a thread holds in flight
// A weight gradient's K is cut into slices. Its bias sums repeat bit for bit at every size, and the
// whole gradient below TG_REPEAT_ROWS rows: two slices may add into the zeroed result in any order
// (two addends onto zero commute), more leave theirs apart, for grad_tail_kernel.
constexpr int TG_MAX_SLICES = 64;
constexpr int TG_REPEAT_ROWS = 1024;
constexpr int TG_REPEAT_SLICES = 4;  // slices of 128 rows at least, their count doubled: fewer than 8 below that

template <int PREC>
__host__ __device__ constexpr int tg_chunk() { return PREC == 0 ? 256 : 64; }  // K values a chunk at most
template <int PREC>
__host__ __device__ constexpr int tg_kstep() { return PREC == 0 ? 16 : 8; }    // K values an MMA

// One product of a launch.
struct TgProb {
  const float* A;
  const float* B;
  float* C;
  const float* bias;
  const float* mask;
  // or null: asum[m] += sum_k op(A)(m, k), from the unrounded values (TA only), of one slice or two;
  // more slices set asum[slice apart + m]
  float* asum;
  int apart;
  long long cpart;  // > 0: slice s stores its tiles into C + s cpart (no atomics)
  int M, N, K, lda, ldb, ldc;
  int ta, tb, epi, round;
  int npad, mt, nt, ks, kslice;  // column tile, tiles, slices of K
  int va, vb, vc;                // rows of A, B, C start on 16 bytes
};
// Programmatic dependent launch, along the chain of small kernels of one minibatch: a kernel
// lets the next one start (its launch, its TMEM allocation and barrier set-up) as soon as every
// CTA of its own is running, and takes the previous one's results only after that one has
// completed. Without the launch attribute both are no-ops.
__device__ __forceinline__ void grid_launch_next() { asm volatile("griddepcontrol.launch_dependents;" ::: "memory"); }
__device__ __forceinline__ void grid_wait_previous() { asm volatile("griddepcontrol.wait;" ::: "memory"); }

template <class... KA, class... A>
static void launch_after(cudaStream_t s, bool overlap, unsigned grid, unsigned block, size_t smem,
                         void (*k)(KA...), A... args) {
  cudaLaunchConfig_t cfg = {};
  cfg.gridDim = dim3(grid);
  cfg.blockDim = dim3(block);
  cfg.dynamicSmemBytes = smem;
  cfg.stream = s;
  cudaLaunchAttribute at[1];
  at[0].id = cudaLaunchAttributeProgrammaticStreamSerialization;
  at[0].val.programmaticStreamSerializationAllowed = 1;
  cfg.attrs = at;
  cfg.numAttrs = overlap ? 1 : 0;
  cudaLaunchKernelEx(&cfg, k, KA(args)...);
}

// Up to two independent products in one launch: CTAs below `first` serve p[0].
struct TgLaunch {
  TgProb p[2];
  int first;
  int kc;          // K values a chunk (a multiple of the MMA's), for both
  uint32_t ncols;  // TMEM columns
  int* err;
};

// Stage R rows (row0 .. ; `rows` of them real) of op(X) for K values k0 .. k0 + kc - 1, where X
// is contiguous along its rows' index when `trans`, else along K. RS: R rounded up to a power
// of two that divides the block's threads, so that a thread stages one row. Returns the sum of
// the values this thread staged.
template <int PREC, int RS>
__device__ __forceinline__ float tg_stage(const float* __restrict__ X, int ld, bool trans, bool vec, int row0, int R,
                                          int rows, int k0, int kend, int kc, unsigned char* hi, unsigned char* lo) {
  constexpr int KS = tg_kstep<PREC>();
  const int left = kend - k0 < kc ? kend - k0 : kc;
  const int r = threadIdx.x % RS, step = TG_NT / RS, nu = (left + KS - 1) / KS * KS / 8;
  const int kc16 = PREC == 0 ? kc / 8 : kc / 4;
  const long long row = (long long)row0 + r;
  const bool live = row < rows;
  float sum = 0.f;
  if (r >= R) return sum;
  for (int u0 = threadIdx.x / RS; u0 < nu; u0 += step * TG_UNITS) {
    float v[TG_UNITS][8];
#pragma unroll
    for (int q = 0; q < TG_UNITS; ++q) {
      const int k = k0 + 8 * (u0 + q * step);
      const bool on = live && u0 + q * step < nu;
      if (!trans && vec && k + 8 <= kend) {
        float4 a = make_float4(0.f, 0.f, 0.f, 0.f), b = a;
        if (on) {
          const float4* src = reinterpret_cast<const float4*>(X + row * ld + k);
          a = src[0];
          b = src[1];
        }
        v[q][0] = a.x; v[q][1] = a.y; v[q][2] = a.z; v[q][3] = a.w;
        v[q][4] = b.x; v[q][5] = b.y; v[q][6] = b.z; v[q][7] = b.w;
      } else {
#pragma unroll
        for (int j = 0; j < 8; ++j)
          v[q][j] = on && k + j < kend ? (trans ? X[(long long)(k + j) * ld + row] : X[row * ld + k + j]) : 0.f;
      }
    }
#pragma unroll
    for (int q = 0; q < TG_UNITS; ++q) {
      const int u = u0 + q * step;
      if (u >= nu) break;
#pragma unroll
      for (int j = 0; j < 8; ++j) sum += v[q][j];
      if (PREC == 0) {
        __nv_bfloat162 h[4];
#pragma unroll
        for (int j = 0; j < 4; ++j) h[j] = __floats2bfloat162_rn(v[q][2 * j], v[q][2 * j + 1]);
        *reinterpret_cast<uint4*>(hi + tc::kmajor_offset(r, 16 * u, kc16)) = *reinterpret_cast<const uint4*>(h);
      } else {
        float h[8], l[8];
#pragma unroll
        for (int j = 0; j < 8; ++j) tc::split_tf32(v[q][j], h[j], l[j]);
#pragma unroll
        for (int j = 0; j < 2; ++j) {
          const uint32_t o = tc::kmajor_offset(r, 32 * u + 16 * j, kc16);
          *reinterpret_cast<float4*>(hi + o) = make_float4(h[4 * j], h[4 * j + 1], h[4 * j + 2], h[4 * j + 3]);
          *reinterpret_cast<float4*>(lo + o) = make_float4(l[4 * j], l[4 * j + 1], l[4 * j + 2], l[4 * j + 3]);
        }
      }
    }
  }
  return sum;
}

template <int PREC>
__global__ void __launch_bounds__(TG_NT, 2) tgemm_kernel(const __grid_constant__ TgLaunch g) {
  extern __shared__ __align__(1024) unsigned char sm[];
  __shared__ __align__(8) uint64_t bar;
  __shared__ uint32_t s_taddr;
  constexpr int KB = PREC == 0 ? 2 : 4;  // bytes of an operand value
  const int tid = threadIdx.x, w = tid >> 5;
  const bool second = (int)blockIdx.x >= g.first;
  const TgProb& p = g.p[second ? 1 : 0];
  const int bid = (int)blockIdx.x - (second ? g.first : 0);
  const int tm = bid % p.mt, tn = bid / p.mt % p.nt, tk = bid / p.mt / p.nt;
  const int npad = p.npad, kc = g.kc, kc16 = kc * KB / 16;
  const uint32_t a_bytes = 128u * kc * KB, b_bytes = (uint32_t)npad * kc * KB;
  unsigned char* a_hi = sm;
  unsigned char* b_hi = sm + a_bytes;
  unsigned char* a_lo = b_hi + b_bytes;  // 3xTF32 only
  unsigned char* b_lo = a_lo + a_bytes;
  const int m0 = tm * 128, n0 = tn * npad;  // this CTA's first row and column
  const int kbeg = tk * p.kslice;           // and its slice of K
  const int kend = kbeg + p.kslice < p.K ? kbeg + p.kslice : p.K;
  if (w == 0) {
    tc::tmem_alloc(&s_taddr, g.ncols);
    tc::tmem_relinquish();
  }
  if (tid == 0) {
    mbar_init(&bar, 1);
    mbar_fence_init();
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t taddr = s_taddr;
  grid_launch_next();
  grid_wait_previous();
  const uint32_t idesc = tc::instr_desc(PREC == 0 ? tc::FMT_BF16 : tc::FMT_TF32, 128, npad);
  int ok = 1;
  uint32_t phase = 0;
  float asum = 0.f;  // of row m0 + tid % 128
  for (int k0 = kbeg; k0 < kend && ok; k0 += kc) {
    asum += tg_stage<PREC, 128>(p.A, p.lda, p.ta, p.va, m0, 128, p.M, k0, kend, kc, a_hi, a_lo);
    tg_stage<PREC, 64>(p.B, p.ldb, !p.tb, p.vb, n0, npad, p.N, k0, kend, kc, b_hi, b_lo);
    tc::fence_proxy_async();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (tid == 0) {
      const uint32_t sah = smem_addr(a_hi), sbh = smem_addr(b_hi), sal = smem_addr(a_lo), sbl = smem_addr(b_lo);
      const int left = kend - k0, steps = ((left < kc ? left : kc) + tg_kstep<PREC>() - 1) / tg_kstep<PREC>();
      for (int ks = 0; ks < steps; ++ks) {
        const uint32_t off = (uint32_t)ks * 256;
        const uint32_t acc = (k0 > kbeg || ks > 0) ? 1u : 0u;
        if (PREC == 0) {
          tc::mma_f16(taddr, tc::smem_desc(sah + off, kc16), tc::smem_desc(sbh + off, kc16), idesc, acc);
        } else {  // small terms first, then the leading one
          tc::mma_tf32(taddr, tc::smem_desc(sal + off, kc16), tc::smem_desc(sbh + off, kc16), idesc, acc);
          tc::mma_tf32(taddr, tc::smem_desc(sah + off, kc16), tc::smem_desc(sbl + off, kc16), idesc, 1);
          tc::mma_tf32(taddr, tc::smem_desc(sah + off, kc16), tc::smem_desc(sbh + off, kc16), idesc, 1);
        }
      }
      tc::commit(&bar);
    }
    const bool done = tc::bar_wait(&bar, phase, TG_SPIN);
    phase ^= 1u;
    tc::fence_after();
    ok = __syncthreads_and(done ? 1 : 0);  // every thread saw the MMAs finish before the tiles change
  }
  if (!ok) {
    if (tid == 0) atomicOr(g.err, ERR_TIMEOUT);
    tc::bar_wait(&bar, phase ^ 1u, TG_SPIN);  // give MMAs still in flight a second bound
  } else {
    if (p.asum && tn == 0) {  // the four threads of a row, in their order
      float* red = reinterpret_cast<float*>(sm);  // (every MMA has read the tiles)
      red[tid] = asum;
      __syncthreads();
      if (tid < 128 && m0 + tid < p.M) {
        static_assert(TG_NT == 512, "four threads a row");
        const float t = ((red[tid] + red[tid + 128]) + red[tid + 256]) + red[tid + 384];
        if (p.ks > 2)
          p.asum[tk * p.apart + m0 + tid] = t;
        else
          atomicAdd(p.asum + m0 + tid, t);
      }
    }
    // warp w takes rows 32 (w mod 4) .. + 31 and the w / 4-th block of 16 columns
    const long long m = m0 + tid % 128;
    const bool split = p.ks > 1 && !p.cpart;
    for (int c0 = 16 * (w >> 2); c0 < npad; c0 += TG_NT / 8) {
      float v[16];
      tc::ld16(taddr + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)c0, v);
      if (m >= p.M) continue;
      const int n = n0 + c0;
      float* c = p.C + tk * p.cpart + m * p.ldc + n;
#pragma unroll
      for (int j = 0; j < 16; ++j) {
        if (n + j >= p.N) break;
        float x = v[j];
        if (p.epi == 1) {
          x = fmaxf(x + p.bias[n + j], 0.f);
          if (p.round) x = round_bf16(x);
        } else if (p.epi == 2) {
          x += p.bias[n + j];
        } else if (p.epi == 3) {
          x = p.mask[m * p.ldc + n + j] > 0.f ? x : 0.f;
        }
        v[j] = x;
      }
      if (p.vc && n + 16 <= p.N) {
#pragma unroll
        for (int j = 0; j < 4; ++j) {
          const float4 x = make_float4(v[4 * j], v[4 * j + 1], v[4 * j + 2], v[4 * j + 3]);
          if (split)
            atomicAdd(reinterpret_cast<float4*>(c) + j, x);
          else
            reinterpret_cast<float4*>(c)[j] = x;
        }
      } else {
#pragma unroll
        for (int j = 0; j < 16; ++j) {
          if (n + j >= p.N) break;
          if (split)
            atomicAdd(c + j, v[j]);
          else
            c[j] = v[j];
        }
      }
    }
  }
  tc::fence_before();
  __syncthreads();
  if (w == 0) tc::tmem_dealloc(taddr, g.ncols);
}

// Whether every row of q (ld floats) starts on 16 bytes.
static int tg_rows16(const float* q, int ld) { return ((uintptr_t)q | (uintptr_t)(4 * (size_t)ld)) % 16 == 0; }

// C = op(A) op(B) with the epilogue epi. A weight gradient (TA, epi 0) has the minibatch as its
// K and few tiles, so its K is split over CTAs that accumulate into C (zeroed by the caller).
static TgProb tg_prob(bool ta, bool tb, int epi, int M, int N, int K, const float* A, int lda, const float* B, int ldb,
                      float* C, int ldc, const float* bias = nullptr, const float* mask = nullptr, int round = 0) {
  TgProb p{};
  p.A = A; p.B = B; p.C = C; p.bias = bias; p.mask = mask;
  p.M = M; p.N = N; p.K = K; p.lda = lda; p.ldb = ldb; p.ldc = ldc;
  p.ta = ta; p.tb = tb; p.epi = epi; p.round = round;
  p.npad = std::min(64, (N + 15) / 16 * 16);
  p.mt = (M + 127) / 128;
  p.nt = (N + p.npad - 1) / p.npad;
  p.va = tg_rows16(A, lda);
  p.vb = tg_rows16(B, ldb);
  p.vc = tg_rows16(C, ldc);
  // slices of at least 128 rows, enough of them for about 96 CTAs: a longer slice leaves SMs
  // idle at minibatch sizes, a shorter one adds as many partial tiles into C as it saves loads
  // (the same rule at 16,384 rows: 8 slices of 2048, 64 CTAs a product, a gradient in 454 us)
  p.ks = 1;
  if (epi == 0)
    while (p.ks < TG_MAX_SLICES && (long long)p.mt * p.nt * p.ks * 2 <= 96 && K / (2 * p.ks) >= 128) p.ks *= 2;
  p.kslice = ((K + p.ks - 1) / p.ks + 15) / 16 * 16;
  p.ks = (K + p.kslice - 1) / p.kslice;  // every slice holds part of K
  return p;
}

template <int PREC>
static void tg_launch(cudaStream_t s, bool overlap, int* err, const TgProb& a, const TgProb* b) {
  TgLaunch g{};
  g.p[0] = a;
  g.p[1] = b ? *b : a;
  g.err = err;
  const long long n0 = (long long)a.mt * a.nt * a.ks, n1 = b ? (long long)b->mt * b->nt * b->ks : 0;
  g.first = (int)n0;
  const int longest = b ? std::max(std::min(a.K, a.kslice), std::min(b->K, b->kslice)) : std::min(a.K, a.kslice);
  const int step = tg_kstep<PREC>();
  g.kc = std::min(tg_chunk<PREC>(), (longest + step - 1) / step * step);
  const int npad = std::max(a.npad, b ? b->npad : 0);
  g.ncols = npad <= 32 ? 32u : 64u;
  // at most 512 / ncols CTAs can hold TMEM on an SM at once: a CTA asks for enough shared
  // memory that no more become resident (they would wait inside the allocation)
  const size_t floor_smem = g.ncols >= 64 ? 29 * 1024 : 0;
  const size_t smem = std::max((size_t)(128 + npad) * g.kc * (PREC == 0 ? 2 : 8), floor_smem);
  // (the attribute belongs to the kernel: the largest any launch asks for, not this one's)
  constexpr int most = (128 + 64) * tg_chunk<PREC>() * (PREC == 0 ? 2 : 8);
  cudaFuncSetAttribute(tgemm_kernel<PREC>, cudaFuncAttributeMaxDynamicSharedMemorySize, most);
  launch_after(s, overlap, (unsigned)(n0 + n1), TG_NT, smem, tgemm_kernel<PREC>, g);
}

// BF16 operands when the proposal trains in its BF16 form, 3xTF32 otherwise; b: a second,
// independent product in the same launch, or null. overlap: the launch before it on the stream
// is a kernel of the same chain.
static void tgemm(cudaStream_t s, bool bf16, bool overlap, int* err, const TgProb& a, const TgProb* b = nullptr) {
  if (bf16)
    tg_launch<0>(s, overlap, err, a, b);
  else
    tg_launch<1>(s, overlap, err, a, b);
}

// ---- the mixture head: loss and d(loss)/d(out) per row ----
struct HeadArgs {
  const float* out;  // n x dout
  const float* Z;    // n x d2
  const float* w;    // n
  const double* wsum;
  float* dout;       // n x dout
  double* loss;      // accumulated: sum_b w_b (-log q_b) / wsum
  int n, d2, C, dout_n;
};

// *loss += the sum of v over the warp's first `live` lanes (the calling ones): one atomic a warp.
__device__ __forceinline__ void add_loss(double* loss, double v, int live) {
  const int lane = threadIdx.x & 31;
  const unsigned mask = live >= 32 ? FULL : (1u << live) - 1u;
#pragma unroll
  for (int o = 16; o > 0; o >>= 1) {
    const double n = __shfl_down_sync(mask, v, o);
    if (lane + o < live) v += n;
  }
  if (lane == 0) atomicAdd(loss, v);
}

__global__ void head_loss_kernel(HeadArgs a) {
  grid_launch_next();
  grid_wait_previous();
  const int b = blockIdx.x * blockDim.x + threadIdx.x;
  const int live = __popc(__ballot_sync(FULL, b < a.n));  // the warp's rows: its first lanes
  if (b >= a.n) return;
  const int C = a.C, d2 = a.d2, D = a.dout_n;
  const float* o = a.out + (long long)b * D;
  const float* z = a.Z + (long long)b * d2;
  float* g = a.dout + (long long)b * D;
  // log softmax of the logits
  float lmax = -INFINITY;
  for (int c = 0; c < C; ++c) lmax = fmaxf(lmax, o[c]);
  float se = 0.f;
  for (int c = 0; c < C; ++c) se += expf(o[c] - lmax);
  const float lse_a = lmax + logf(se);
  float lc[kMaxComponents];
  float cmax = -INFINITY;
  const float HL2PI = 0.91893853320467274f;
  for (int c = 0; c < C; ++c) {
    float s = o[c] - lse_a;
    for (int d = 0; d < d2; ++d) {
      const float mu = o[C + c * d2 + d];
      const float ls = fminf(fmaxf(o[C + C * d2 + c * d2 + d], kLogSigMin), kLogSigMax);
      const float u = (z[d] - mu) * expf(-ls);
      s += -0.5f * u * u - ls - HL2PI;
    }
    lc[c] = s;
    cmax = fmaxf(cmax, s);
  }
  float sc = 0.f;
  for (int c = 0; c < C; ++c) sc += expf(lc[c] - cmax);
  const float lq = cmax + logf(sc);
  const float wn = (float)((double)a.w[b] / *a.wsum);
  add_loss(a.loss, -(double)wn * (double)lq, live);
  for (int c = 0; c < C; ++c) {
    const float gam = expf(lc[c] - lq);
    const float pi = expf(o[c] - lse_a);
    g[c] = wn * (pi - gam);
    for (int d = 0; d < d2; ++d) {
      const float mu = o[C + c * d2 + d];
      const float raw = o[C + C * d2 + c * d2 + d];
      const float ls = fminf(fmaxf(raw, kLogSigMin), kLogSigMax);
      const float is = expf(-ls);
      const float u = (z[d] - mu) * is;
      g[C + c * d2 + d] = -wn * gam * u * is;
      const bool inside = raw > kLogSigMin && raw < kLogSigMax;
      g[C + C * d2 + c * d2 + d] = inside ? -wn * gam * (u * u - 1.f) : 0.f;
    }
  }
}

// Affine (outer-amortised) head: out = (raw log s, c); Z row = (z, mu, m) (3 d2);
// zhat = m + (z - m - c) / s; -log q = 1/2 (zhat - mu)^T Q^-1 (zhat - mu) + sum log s + const.
struct AffineArgs {
  const float* out;
  const float* Z;
  const float* w;
  const double* wsum;
  float* dout;
  double* loss;
  int n, d2;
  const float* qinv;  // d2 x d2, row-major (device)
  float half_logdet;
};

// One warp a row, a lane for every 32nd coordinate; Q_z^-1 is staged in shared memory (rows one
// word longer, so that the lanes' rows fall on distinct banks). A thread a row kept its five
// d2-long arrays in local memory and walked d2 x d2 products alone.
constexpr int HA_WARPS = 8;
__global__ void __launch_bounds__(32 * HA_WARPS) head_affine_kernel(AffineArgs a) {
  __shared__ float q[kMaxD2Amortised * (kMaxD2Amortised + 1)];
  __shared__ float rs[HA_WARPS][kMaxD2Amortised];
  constexpr int NC = kMaxD2Amortised / 32;
  const int d2 = a.d2, lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  grid_launch_next();
  for (int e = threadIdx.x; e < d2 * d2; e += blockDim.x) q[e / d2 * (d2 + 1) + e % d2] = a.qinv[e];
  grid_wait_previous();
  __syncthreads();
  const int b = blockIdx.x * HA_WARPS + w;
  if (b >= a.n) return;  // whole warps
  const float* o = a.out + (long long)b * 2 * d2;
  const float* zr = a.Z + (long long)b * 3 * d2;
  float* g = a.dout + (long long)b * 2 * d2;
  float u[NC], ls[NC], raw[NC], r[NC];
  float sum_ls = 0.f, quad = 0.f;
#pragma unroll
  for (int p = 0; p < NC; ++p) {
    const int d = lane + 32 * p;
    u[p] = ls[p] = raw[p] = r[p] = 0.f;
    if (d < d2) {
      raw[p] = o[d];
      ls[p] = fminf(fmaxf(raw[p], kLogSigMin), kLogSigMax);
      u[p] = zr[d] - zr[2 * d2 + d] - o[d2 + d];  // z - m - c
      r[p] = zr[2 * d2 + d] + u[p] * expf(-ls[p]) - zr[d2 + d];
      rs[w][d] = r[p];
      sum_ls += ls[p];
    }
  }
  __syncwarp();
  const float wn = (float)((double)a.w[b] / *a.wsum);
#pragma unroll
  for (int p = 0; p < NC; ++p) {
    const int d = lane + 32 * p;
    if (d < d2) {
      float v = 0.f;
      for (int e = 0; e < d2; ++e) v += q[d * (d2 + 1) + e] * rs[w][e];
      quad += r[p] * v;
      const float is = expf(-ls[p]);
      const bool inside = raw[p] > kLogSigMin && raw[p] < kLogSigMax;
      g[d] = inside ? wn * (-v * u[p] * is + 1.f) : 0.f;
      g[d2 + d] = -wn * v * is;
    }
  }
  quad = warp_sum(quad);
  sum_ls = warp_sum(sum_ls);
  if (lane == 0) atomicAdd(a.loss, (double)wn * (0.5 * (double)quad + (double)sum_ls + (double)a.half_logdet));
}

// What a minibatch needs before its products: the sum of its weights (block 0, in a fixed
// order), the gradient set to zero (split products and the bias sums add into it) and, when
// `loss` is given, the loss too. One launch in the place of a launch and five memsets.
__global__ void __launch_bounds__(256)
    batch_prologue_kernel(const float* w, int n, double* wsum, float* grad, long long ngrad, double* loss) {
  grid_launch_next();
  const long long e = blockIdx.x * 256ll + threadIdx.x;
  if (grad && e < ngrad) grad[e] = 0.f;
  if (blockIdx.x) return;
  __shared__ double sh[256];
  double s = 0.0;
  for (int b = threadIdx.x; b < n; b += 256) s += (double)w[b];
  sh[threadIdx.x] = s;
  __syncthreads();
  for (int o = 128; o > 0; o >>= 1) {
    if (threadIdx.x < o) sh[threadIdx.x] += sh[threadIdx.x + o];
    __syncthreads();
  }
  if (threadIdx.x == 0) {
    *wsum = sh[0];
    if (loss) *loss = 0.0;
  }
}

// The slices' bias sums and, with `weights`, their parts of the weight gradients, added in the order of
// the slices: the last launch of a backward pass of 512 rows or more. (With it and the ordered sums in a
// CTA a BF16 gradient takes 136 us at 600 rows, 138 at 1024 and 177 at 4096, against 129, 136 and 175
// with every sum by atomics; the last CTA of a tile folding the slices took 136, 137 and 186.)
struct TailArgs {
  float* grad;
  const float* bpart;  // [slice][layer][kMaxHidden]
  const float* gpart;  // [slice][gstep]
  long long nparams, gstep, offW[kLayers], offB[kLayers];
  int ks[kLayers], rows[kLayers];
  int any, weights;
};

__global__ void __launch_bounds__(256) grad_tail_kernel(TailArgs a) {
  grid_wait_previous();
  const long long t = blockIdx.x * 256ll + threadIdx.x;
  const float* src;
  long long step, e;
  int l;
  if (t < kLayers * kMaxHidden) {
    l = (int)(t / kMaxHidden);
    const int m = (int)(t % kMaxHidden);
    if (m >= a.rows[l]) return;
    src = a.bpart + t;
    step = kLayers * kMaxHidden;
    e = a.offB[l] + m;
  } else {
    e = t - kLayers * kMaxHidden;
    if (e >= a.nparams) return;
    for (l = kLayers - 1; l > 0 && e < a.offW[l]; --l) {
    }
    if (e >= a.offB[l]) return;  // a bias
    src = a.gpart + e;
    step = a.gstep;
  }
  const int ks = a.ks[l];
  if (ks <= 2) return;  // it is in place
  float s = 0.f;
#pragma unroll 8
  for (int q = 0; q < ks; ++q) s += src[q * step];
  a.grad[e] = s;
}

// minibatch gather: rows perm[b] of F, Z, w
__global__ void gather_rows_kernel(const float* F, const float* Z, const float* w, const int64_t* perm,
                                   int nb, int din, int d2, float* Fb, float* Zb, float* wb, int round) {
  const int b = blockIdx.x;
  if (b >= nb) return;
  const long long r = perm[b];
  for (int c = threadIdx.x; c < din; c += blockDim.x) {
    const float v = F[r * din + c];
    Fb[(long long)b * din + c] = round ? round_bf16(v) : v;
  }
  for (int c = threadIdx.x; c < d2; c += blockDim.x) Zb[(long long)b * d2 + c] = Z[r * d2 + c];  // d2: row width
  if (threadIdx.x == 0) wb[b] = w[r];
}

struct AdamArgs {
  float* W;
  float* Wq;  // the weights the forward pass uses (bfloat16-rounded weight matrices)
  float* m;
  float* v;
  const float* g;
  long long n;
  long long wend[kLayers];  // [wbeg[l], wend[l]) is weight matrix l
  long long wbeg[kLayers];
  float lr, b1, b2, eps, c1, c2;  // c1 = 1 - b1^t, c2 = 1 - b2^t
  int round;
};

__global__ void adam_kernel(AdamArgs a) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= a.n) return;
  const float g = a.g[e];
  const float m = a.b1 * a.m[e] + (1.f - a.b1) * g;
  const float v = a.b2 * a.v[e] + (1.f - a.b2) * g * g;
  a.m[e] = m;
  a.v[e] = v;
  const float mh = m / a.c1, vh = v / a.c2;
  const float w = a.W[e] - a.lr * mh / (sqrtf(vh) + a.eps);
  a.W[e] = w;
  bool is_w = false;
  for (int l = 0; l < kLayers; ++l) is_w |= (e >= a.wbeg[l] && e < a.wend[l]);
  a.Wq[e] = (is_w && a.round) ? round_bf16(w) : w;
}

__global__ void quantize_params_kernel(const float* W, float* Wq, long long n, AdamArgs seg) {
  const long long e = blockIdx.x * (long long)blockDim.x + threadIdx.x;
  if (e >= n) return;
  bool is_w = false;
  for (int l = 0; l < kLayers; ++l) is_w |= (e >= seg.wbeg[l] && e < seg.wend[l]);
  Wq[e] = (is_w && seg.round) ? round_bf16(W[e]) : W[e];
}

// ---- host side ----
static dpf_status palloc(dpf_proposal& p, void** ptr, size_t bytes) {
  cudaError_t e = device_malloc(ptr, bytes < 16 ? 16 : bytes);
  if (e != cudaSuccess) {
    cudaGetLastError();
    *ptr = nullptr;
    return set_error(DPF_E_NOMEM, "proposal: device allocation failed");
  }
  p.allocs.push_back(*ptr);
  return DPF_OK;
}

int dpf_proposal_dout(const dpf_proposal* p) { return p->dout; }
int dpf_proposal_kind(const dpf_proposal* p) { return p->kind; }

static AdamArgs segments(const dpf_proposal& p) {
  AdamArgs a{};
  for (int l = 0; l < kLayers; ++l) {
    a.wbeg[l] = p.offW[l];
    a.wend[l] = p.offW[l] + (long long)p.rows[l] * p.cols[l];
  }
  a.round = p.bf16 ? 1 : 0;
  return a;
}

dpf_status proposal_requantize(dpf_proposal& p) {
  AdamArgs seg = segments(p);
  quantize_params_kernel<<<(unsigned)((p.nparams + 255) / 256), 256, 0, p.stream>>>(p.W, p.Wq, p.nparams, seg);
  p.packed_valid = false;
  return cuda_error(cudaGetLastError(), "proposal quantize");
}

// The buffers bufs[q] of nb x widths[q] floats, where they hold `rows` rows now: kept if that is
// enough, else given back and allocated anew (the sizes need not be held twice).
template <size_t NB>
static dpf_status hold_rows(dpf_proposal& p, int nb, int& rows, float** const (&bufs)[NB], const int (&widths)[NB]) {
  if (nb <= rows) return DPF_OK;
  cudaError_t e = cudaStreamSynchronize(p.stream);
  if (e != cudaSuccess) return cuda_error(e, "proposal workspace");
  rows = 0;
  for (float** b : bufs) {
    p.allocs.erase(std::remove(p.allocs.begin(), p.allocs.end(), (void*)*b), p.allocs.end());
    cudaFree(*b);
    *b = nullptr;
  }
  for (size_t q = 0; q < NB; ++q) {
    dpf_status st = palloc(p, (void**)bufs[q], sizeof(float) * (size_t)nb * widths[q]);
    if (st) return st;
  }
  rows = nb;
  return DPF_OK;
}

// Ensure the per-minibatch workspace holds nb rows; gather: training's gathered rows too.
static dpf_status workspace(dpf_proposal& p, int nb, bool gather) {
  const int H = p.hidden;
  dpf_status st = hold_rows(p, nb, p.ws_rows, {&p.h1, &p.h2, &p.h3, &p.ob, &p.dA, &p.dB, &p.dO},
                            {H, H, H, p.dout, H, H, p.dout});
  if (!st && gather) st = hold_rows(p, nb, p.gather_rows, {&p.Fb, &p.Zb, &p.wb}, {p.din, p.zw, 1});
  return st;
}

// Forward and backward over nb rows (features F, targets Z, weights w): loss into *loss_dev
// (accumulated, from zero when zero_loss), gradients into grad (nparams floats).
static dpf_status fwd_bwd(dpf_proposal& p, const float* F, const float* Z, const float* w, int nb, double* loss_dev,
                          bool zero_loss, float* grad) {
  cudaStream_t s = p.stream;
  const int H = p.hidden, din = p.din, dO = p.dout;
  const float* Wq = p.Wq;
  const bool bf = p.bf16;
  const int rd = bf ? 1 : 0;
  const float *W1 = Wq + p.offW[0], *W2 = Wq + p.offW[1], *W3 = Wq + p.offW[2], *W4 = Wq + p.offW[3];
  const float *b1 = Wq + p.offB[0], *b2 = Wq + p.offB[1], *b3 = Wq + p.offB[2], *b4 = Wq + p.offB[3];
  const unsigned zb = grad ? (unsigned)((p.nparams + 255) / 256) : 1u;
  batch_prologue_kernel<<<zb, 256, 0, s>>>(w, nb, p.wsum_d, grad, p.nparams, zero_loss ? loss_dev : nullptr);
  // forward: h_l = round(relu(h_{l-1} W_l^T + b_l)), out = h3 W4^T + b4
  tgemm(s, bf, true, p.err_d, tg_prob(false, true, 1, nb, H, din, F, din, W1, din, p.h1, H, b1, nullptr, rd));
  tgemm(s, bf, true, p.err_d, tg_prob(false, true, 1, nb, H, H, p.h1, H, W2, H, p.h2, H, b2, nullptr, rd));
  tgemm(s, bf, true, p.err_d, tg_prob(false, true, 1, nb, H, H, p.h2, H, W3, H, p.h3, H, b3, nullptr, rd));
  tgemm(s, bf, true, p.err_d, tg_prob(false, true, 2, nb, dO, H, p.h3, H, W4, H, p.ob, dO, b4));
  if (p.kind == 0) {
    HeadArgs ha{p.ob, Z, w, p.wsum_d, p.dO, loss_dev, nb, p.d2, p.C, dO};
    launch_after(s, true, (nb + 127) / 128, 128, 0, head_loss_kernel, ha);
  } else {
    AffineArgs aa{};
    aa.out = p.ob; aa.Z = Z; aa.w = w; aa.wsum = p.wsum_d; aa.dout = p.dO; aa.loss = loss_dev;
    aa.n = nb; aa.d2 = p.d2;
    aa.qinv = p.qinv_d;
    aa.half_logdet = p.half_logdet;
    launch_after(s, true, (nb + HA_WARPS - 1) / HA_WARPS, 32 * HA_WARPS, 0, head_affine_kernel, aa);
  }
  if (!grad) return cuda_error(cudaGetLastError(), "proposal forward");
  // layer l: dW_l = d_l^T h_{l-1} with db_l = colsum d_l from the same rows as they are staged,
  // and in the same launch d_{l-1} = (d_l W_l) * (h_{l-1} > 0), which reads the same d_l
  TailArgs tail{};
  tail.gstep = (p.nparams + 3) / 4 * 4;
  auto layer = [&](int l, int rows, int cols, const float* d, const float* h, const float* W, float* dprev) {
    TgProb gw = tg_prob(true, false, 0, rows, cols, nb, d, rows, h, cols, grad + p.offW[l], cols);
    gw.asum = grad + p.offB[l];
    if (gw.ks > 2) {
      gw.asum = p.bias_part + l * kMaxHidden;
      gw.apart = kLayers * kMaxHidden;
      if (nb < TG_REPEAT_ROWS) {
        gw.C = p.grad_part + p.offW[l];
        gw.cpart = tail.gstep;
        gw.vc = tg_rows16(gw.C, cols);  // (gstep is a multiple of 4)
        tail.weights = 1;
      }
      tail.any = 1;
    }
    tail.ks[l] = gw.ks;
    tail.rows[l] = rows;
    tail.offW[l] = p.offW[l];
    tail.offB[l] = p.offB[l];
    if (!dprev) return tgemm(s, bf, true, p.err_d, gw);
    const TgProb gd = tg_prob(false, false, 3, nb, cols, rows, d, rows, W, cols, dprev, cols, nullptr, h);
    tgemm(s, bf, true, p.err_d, gd, &gw);
  };
  layer(3, dO, H, p.dO, p.h3, W4, p.dA);
  layer(2, H, H, p.dA, p.h2, W3, p.dB);
  layer(1, H, H, p.dB, p.h1, W2, p.dA);
  layer(0, H, din, p.dA, F, W1, nullptr);
  if (tail.any) {
    tail.grad = grad;
    tail.bpart = p.bias_part;
    tail.gpart = p.grad_part;
    tail.nparams = p.nparams;
    const long long n = kLayers * kMaxHidden + (tail.weights ? p.nparams : 0);
    launch_after(s, true, (unsigned)((n + 255) / 256), 256, 0, grad_tail_kernel, tail);
  }
  return cuda_error(cudaGetLastError(), "proposal backward");
}

dpf_status proposal_forward_rows(dpf_proposal& p, const float* F, long long n, float* hidden, float* out, int* err,
                                 cudaStream_t s) {
  if (n < 1) return DPF_OK;
  if (n > (1LL << 30)) return set_error(DPF_E_INVALID, "proposal forward: too many rows");
  const int H = p.hidden, din = p.din, dO = p.dout, m = (int)n;
  const bool bf = p.bf16;
  const int rd = bf ? 1 : 0;
  const float* Wq = p.Wq;
  float* ha = hidden;
  float* hb = hidden + (size_t)n * H;
  tgemm(s, bf, false, err, tg_prob(false, true, 1, m, H, din, F, din, Wq + p.offW[0], din, ha, H, Wq + p.offB[0], nullptr, rd));
  tgemm(s, bf, true, err, tg_prob(false, true, 1, m, H, H, ha, H, Wq + p.offW[1], H, hb, H, Wq + p.offB[1], nullptr, rd));
  tgemm(s, bf, true, err, tg_prob(false, true, 1, m, H, H, hb, H, Wq + p.offW[2], H, ha, H, Wq + p.offB[2], nullptr, rd));
  tgemm(s, bf, true, err, tg_prob(false, true, 2, m, dO, H, ha, H, Wq + p.offW[3], H, out, dO, Wq + p.offB[3]));
  return cuda_error(cudaGetLastError(), "proposal forward");
}

static dpf_status adam(dpf_proposal& p, const float* grad, float lr) {
  p.adam_t += 1;
  AdamArgs a = segments(p);
  a.W = p.W;
  a.Wq = p.Wq;
  a.m = p.am;
  a.v = p.av;
  a.g = grad;
  a.n = p.nparams;
  a.lr = lr;
  a.b1 = 0.9f;
  a.b2 = 0.999f;
  a.eps = 1e-8f;
  a.c1 = (float)(1.0 - std::pow(0.9, (double)p.adam_t));
  a.c2 = (float)(1.0 - std::pow(0.999, (double)p.adam_t));
  adam_kernel<<<(unsigned)((p.nparams + 255) / 256), 256, 0, p.stream>>>(a);
  p.packed_valid = false;
  return cuda_error(cudaGetLastError(), "adam");
}

// splitmix64 (Steele, Lea and Flood 2014): the minibatch order of training.
static uint64_t splitmix64(uint64_t& s) {
  uint64_t z = (s += 0x9E3779B97F4A7C15ull);
  z = (z ^ (z >> 30)) * 0xBF58476D1CE4E5B9ull;
  z = (z ^ (z >> 27)) * 0x94D049BB133111EBull;
  return z ^ (z >> 31);
}

static dpf_status proposal_make(int kind, int32_t d1, int32_t d2, int32_t dy, int32_t hidden, int32_t components,
                                int din, int dout, int zw, void* stream, dpf_proposal** out) {
  const int max_din = kind == 1 ? kMaxDinAmortised : kMaxDin;
  const int max_d2 = kind == 1 ? kMaxD2Amortised : kMaxD2;
  if (d1 < 1 || d2 < 1 || dy < 1 || din > max_din || d2 > max_d2 || hidden < 16 || hidden > kMaxHidden ||
      hidden % 16 || components < 1 || components > kMaxComponents || dout > kMaxDout)
    return set_error(DPF_E_INVALID, "dpf_proposal_create: unsupported sizes (mixture: din <= 16, d2 <= 8; "
                                    "amortised: din <= 160, d2 <= 64; hidden a multiple of 16 up to 256, "
                                    "components 1..8, head <= 128)");
  dpf_proposal* p = new dpf_proposal();
  p->kind = kind;
  p->d1 = d1;
  p->d2 = d2;
  p->dy = dy;
  p->din = din;
  p->hidden = hidden;
  p->C = components;
  p->dout = dout;
  p->zw = zw;
  p->stream = (cudaStream_t)stream;
  const int H = hidden;
  p->rows[0] = H; p->cols[0] = din;
  p->rows[1] = H; p->cols[1] = H;
  p->rows[2] = H; p->cols[2] = H;
  p->rows[3] = p->dout; p->cols[3] = H;
  long long o = 0;
  for (int l = 0; l < kLayers; ++l) {
    p->offW[l] = o;
    o += (long long)p->rows[l] * p->cols[l];
    p->offB[l] = o;
    o += p->rows[l];
  }
  p->nparams = o;
  const size_t bytes = sizeof(float) * (size_t)o;
  if (palloc(*p, (void**)&p->W, bytes) || palloc(*p, (void**)&p->Wq, bytes) ||
      palloc(*p, (void**)&p->am, bytes) || palloc(*p, (void**)&p->av, bytes) ||
      palloc(*p, (void**)&p->grad, bytes) || palloc(*p, (void**)&p->loss_d, 2 * sizeof(double)) ||
      palloc(*p, (void**)&p->wsum_d, sizeof(double)) ||
      palloc(*p, (void**)&p->bias_part, sizeof(float) * TG_MAX_SLICES * kLayers * kMaxHidden) ||
      palloc(*p, (void**)&p->grad_part, (bytes + 16) * TG_REPEAT_SLICES)) {
    dpf_proposal_destroy(p);
    return DPF_E_NOMEM;
  }
  p->err_d = (int*)(p->loss_d + 1);  // after the loss: one copy reads both
  cudaMemsetAsync(p->err_d, 0, sizeof(int), p->stream);
  cudaMemsetAsync(p->W, 0, bytes, p->stream);
  cudaMemsetAsync(p->Wq, 0, bytes, p->stream);
  cudaMemsetAsync(p->am, 0, bytes, p->stream);
  cudaMemsetAsync(p->av, 0, bytes, p->stream);
  cudaError_t e = cudaStreamSynchronize(p->stream);
  if (e != cudaSuccess) {
    dpf_proposal_destroy(p);
    return cuda_error(e, "dpf_proposal_create");
  }
  *out = p;
  return DPF_OK;
}

}  // namespace dpf

using namespace dpf;

extern "C" {

dpf_status dpf_proposal_create(int32_t d1, int32_t d2, int32_t dy, int32_t hidden, int32_t components,
                               void* stream, dpf_proposal** out) {
  clear_error();
  if (!out) return set_error(DPF_E_INVALID, "dpf_proposal_create: null output");
  *out = nullptr;
  return dpf::proposal_make(0, d1, d2, dy, hidden, components, 2 * d1 + d2 + dy, components * (1 + 2 * d2), d2,
                            stream, out);
}

dpf_status dpf_proposal_create_amortised(int32_t d1, int32_t d2, int32_t dy, int32_t hidden, const double* Qz,
                                         void* stream, dpf_proposal** out) {
  clear_error();
  if (!out || !Qz) return set_error(DPF_E_INVALID, "dpf_proposal_create_amortised: null argument");
  *out = nullptr;
  if (d2 < 1 || d2 > kMaxD2Amortised)
    return set_error(DPF_E_INVALID, "dpf_proposal_create_amortised: d2 in 1..64");
  // Q_z^-1 and log det(2 pi Q_z) by a Cholesky factorisation on the host
  std::vector<double> Lc(d2 * d2, 0.0), inv(d2 * d2, 0.0);
  for (int r = 0; r < d2; ++r)
    for (int c = 0; c <= r; ++c) {
      double v = Qz[r * d2 + c];
      for (int k = 0; k < c; ++k) v -= Lc[r * d2 + k] * Lc[c * d2 + k];
      if (r == c) {
        if (!(v > 0)) return set_error(DPF_E_INVALID, "dpf_proposal_create_amortised: Q_z not positive definite");
        Lc[r * d2 + r] = std::sqrt(v);
      } else {
        Lc[r * d2 + c] = v / Lc[c * d2 + c];
      }
    }
  double logdet = 0.0;
  for (int r = 0; r < d2; ++r) logdet += 2.0 * std::log(Lc[r * d2 + r]);
  for (int col = 0; col < d2; ++col) {  // solve Q x = e_col
    std::vector<double> yv(d2), xv(d2);
    for (int r = 0; r < d2; ++r) {
      double v = (r == col) ? 1.0 : 0.0;
      for (int k = 0; k < r; ++k) v -= Lc[r * d2 + k] * yv[k];
      yv[r] = v / Lc[r * d2 + r];
    }
    for (int r = d2 - 1; r >= 0; --r) {
      double v = yv[r];
      for (int k = r + 1; k < d2; ++k) v -= Lc[k * d2 + r] * xv[k];
      xv[r] = v / Lc[r * d2 + r];
    }
    for (int r = 0; r < d2; ++r) inv[r * d2 + col] = xv[r];
  }
  dpf_status st = dpf::proposal_make(1, d1, d2, dy, hidden, 1, 2 * d1 + dy + 2 * d2, 2 * d2, 3 * d2, stream, out);
  if (st) return st;
  for (int q = 0; q < d2 * d2; ++q) (*out)->qinv[q] = (float)inv[q];
  dpf_proposal* p = *out;
  cudaError_t e = cudaErrorMemoryAllocation;
  if (palloc(*p, (void**)&p->qinv_d, sizeof(float) * (size_t)d2 * d2) == DPF_OK)
    e = cudaMemcpyAsync(p->qinv_d, p->qinv, sizeof(float) * (size_t)d2 * d2, cudaMemcpyHostToDevice, p->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(p->stream);
  if (e != cudaSuccess) {
    dpf_proposal_destroy(p);
    *out = nullptr;
    return e == cudaErrorMemoryAllocation ? DPF_E_NOMEM : cuda_error(e, "dpf_proposal_create_amortised");
  }
  (*out)->half_logdet = (float)(0.5 * (logdet + d2 * std::log(2.0 * M_PI)));
  return DPF_OK;
}

dpf_status dpf_proposal_set_centre(dpf_proposal* p, int32_t per_particle) {
  clear_error();
  if (!p || p->kind != 1 || (per_particle != 0 && per_particle != 1))
    return set_error(DPF_E_INVALID, "dpf_proposal_set_centre: an outer-amortised proposal and 0 or 1");
  p->centre = per_particle;
  return DPF_OK;
}

dpf_status dpf_proposal_num_params(const dpf_proposal* p, int64_t* n) {
  clear_error();
  if (!p || !n) return set_error(DPF_E_INVALID, "dpf_proposal_num_params: null argument");
  *n = p->nparams;
  return DPF_OK;
}

dpf_status dpf_proposal_set_bf16(dpf_proposal* p, int32_t enable) {
  clear_error();
  if (!p) return set_error(DPF_E_INVALID, "dpf_proposal_set_bf16: null proposal");
  p->bf16 = enable != 0;
  dpf_status st = proposal_requantize(*p);
  if (st) return st;
  return cuda_error(cudaStreamSynchronize(p->stream), "dpf_proposal_set_bf16");
}

dpf_status dpf_proposal_set_weights(dpf_proposal* p, const float* params, int64_t n) {
  clear_error();
  if (!p || !params || n != p->nparams)
    return set_error(DPF_E_INVALID, "dpf_proposal_set_weights: need exactly num_params floats");
  cudaError_t e = cudaMemcpyAsync(p->W, params, sizeof(float) * n, cudaMemcpyHostToDevice, p->stream);
  if (e != cudaSuccess) return cuda_error(e, "dpf_proposal_set_weights");
  cudaMemsetAsync(p->am, 0, sizeof(float) * n, p->stream);
  cudaMemsetAsync(p->av, 0, sizeof(float) * n, p->stream);
  p->adam_t = 0;
  dpf_status st = proposal_requantize(*p);
  if (st) return st;
  return cuda_error(cudaStreamSynchronize(p->stream), "dpf_proposal_set_weights");
}

dpf_status dpf_proposal_get_weights(const dpf_proposal* p, float* params, int64_t n) {
  clear_error();
  if (!p || !params || n != p->nparams)
    return set_error(DPF_E_INVALID, "dpf_proposal_get_weights: need exactly num_params floats");
  cudaError_t e = cudaMemcpyAsync(params, p->W, sizeof(float) * n, cudaMemcpyDeviceToHost, p->stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(p->stream);
  return cuda_error(e, "dpf_proposal_get_weights");
}

// The training products' error word: DPF_E_TIMEOUT (and cleared) if a wait gave up.
static dpf_status training_err(dpf_proposal& p, const char* what) {
  int h = 0;
  cudaError_t e = cudaMemcpyAsync(&h, p.err_d, sizeof(int), cudaMemcpyDeviceToHost, p.stream);
  if (e == cudaSuccess) e = cudaStreamSynchronize(p.stream);
  if (e != cudaSuccess) return cuda_error(e, what);
  if (h) {
    cudaMemsetAsync(p.err_d, 0, sizeof(int), p.stream);
    return set_error(DPF_E_TIMEOUT, std::string(what) + ": a tensor-core product did not complete in time");
  }
  return DPF_OK;
}

dpf_status dpf_proposal_loss_grad(dpf_proposal* p, const float* F, const float* Z, const float* w, int64_t n,
                                  double* loss, float* grad_dev) {
  clear_error();
  if (!p || !F || !Z || !w || n < 1 || n > (1 << 24))
    return set_error(DPF_E_INVALID, "dpf_proposal_loss_grad: bad arguments");
  dpf_status st = workspace(*p, (int)n, false);
  if (st) return st;
  cudaStream_t s = p->stream;
  // the caller's rows are read where they lie (the products round them as they stage them)
  st = fwd_bwd(*p, F, Z, w, (int)n, p->loss_d, true, grad_dev);
  if (st) return st;
  struct {
    double loss;
    int err;
  } h = {0.0, 0};
  cudaError_t e = cudaMemcpyAsync(&h, p->loss_d, sizeof(double) + sizeof(int), cudaMemcpyDeviceToHost, s);
  if (e == cudaSuccess) e = cudaStreamSynchronize(s);
  if (e != cudaSuccess) return cuda_error(e, "dpf_proposal_loss_grad");
  if (h.err) return training_err(*p, "dpf_proposal_loss_grad");
  if (loss) *loss = h.loss;
  return DPF_OK;
}

dpf_status dpf_proposal_adam_step(dpf_proposal* p, const float* grad_dev, float lr) {
  clear_error();
  if (!p || !grad_dev || !(lr > 0.f)) return set_error(DPF_E_INVALID, "dpf_proposal_adam_step: bad arguments");
  dpf_status st = adam(*p, grad_dev, lr);
  if (st) return st;
  return cuda_error(cudaStreamSynchronize(p->stream), "dpf_proposal_adam_step");
}

dpf_status dpf_proposal_train(dpf_proposal* p, const float* F, const float* Z, const float* w, int64_t n,
                              int32_t batch, int32_t epochs, float lr, uint64_t seed, double* losses) {
  clear_error();
  if (!p || !F || !Z || !w || n < 1 || batch < 1 || batch > (1 << 16) || epochs < 1 || !(lr > 0.f))
    return set_error(DPF_E_INVALID, "dpf_proposal_train: bad arguments");
  const int nb_max = (int)std::min<int64_t>(batch, n);
  dpf_status st = workspace(*p, nb_max, true);
  if (st) return st;
  cudaStream_t s = p->stream;
  const int rd = p->bf16 ? 1 : 0;
  std::vector<int64_t> perm(n);
  for (int64_t i = 0; i < n; ++i) perm[i] = i;
  uint64_t rs = seed;
  int64_t* perm_dev = nullptr;
  cudaError_t e = cudaMallocAsync((void**)&perm_dev, sizeof(int64_t) * n, s);
  if (e != cudaSuccess) return cuda_error(e, "dpf_proposal_train: allocation");
  std::vector<double> ep_loss(epochs, 0.0);
  double* eloss_d = nullptr;
  e = cudaMallocAsync((void**)&eloss_d, sizeof(double) * epochs, s);
  if (e != cudaSuccess) {
    cudaFreeAsync(perm_dev, s);
    return cuda_error(e, "dpf_proposal_train: allocation");
  }
  cudaMemsetAsync(eloss_d, 0, sizeof(double) * epochs, s);
  const int64_t nbatches = (n + nb_max - 1) / nb_max;
  for (int ep = 0; ep < epochs && !st; ++ep) {
    for (int64_t i = n - 1; i > 0; --i) {  // Fisher-Yates with splitmix64
      const int64_t j = (int64_t)(splitmix64(rs) % (uint64_t)(i + 1));
      std::swap(perm[i], perm[j]);
    }
    e = cudaMemcpyAsync(perm_dev, perm.data(), sizeof(int64_t) * n, cudaMemcpyHostToDevice, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);  // perm is rewritten next epoch
    if (e != cudaSuccess) {
      st = cuda_error(e, "dpf_proposal_train: permutation");
      break;
    }
    for (int64_t bi = 0; bi < nbatches && !st; ++bi) {
      const int64_t b0 = bi * nb_max;
      const int nb = (int)std::min<int64_t>(nb_max, n - b0);
      gather_rows_kernel<<<nb, 32, 0, s>>>(F, Z, w, perm_dev + b0, nb, p->din, p->zw, p->Fb, p->Zb, p->wb, rd);
      st = fwd_bwd(*p, p->Fb, p->Zb, p->wb, nb, eloss_d + ep, false, p->grad);
      if (!st) st = adam(*p, p->grad, lr);
    }
  }
  if (!st) {
    e = cudaMemcpyAsync(ep_loss.data(), eloss_d, sizeof(double) * epochs, cudaMemcpyDeviceToHost, s);
    if (e == cudaSuccess) e = cudaStreamSynchronize(s);
    if (e != cudaSuccess) st = cuda_error(e, "dpf_proposal_train");
  }
  cudaFreeAsync(perm_dev, s);
  cudaFreeAsync(eloss_d, s);
  if (!st) st = training_err(*p, "dpf_proposal_train");
  if (!st && losses)
    for (int ep = 0; ep < epochs; ++ep) losses[ep] = ep_loss[ep] / (double)nbatches;
  return st;
}

void dpf_proposal_destroy(dpf_proposal* p) {
  if (!p) return;
  if (p->stream) cudaStreamSynchronize(p->stream);
  for (void* q : p->allocs) cudaFree(q);
  delete p;
}

}  // extern "C"
