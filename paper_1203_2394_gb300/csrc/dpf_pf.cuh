// The bootstrap particle filter over the full state s = (x, z), the baseline the
// paper compares the decentralized filters with (Section 4.1, "PF"): every particle
// is propagated from its resampled ancestor by the model's transition and weighted
// by the likelihood of y_t. One thread a particle. The outer stages of the filter
// (the evidence, the weighted mean and the global systematic resampling) serve it
// unchanged, with one "group" a particle: lw is the particle's log-weight and its state the
// "means". The kernel also sums the weighted state as it goes, relative to the largest weight
// any particle can have (lognorm_y), so that the outer stage need not read the particles again
// (it still can, when every weight is far below that: sums_given in dpf_outer.cuh).
//
// Bound by memory: 56 bytes read and 52 written a particle at d = 10 (the x rows padded to 16
// bytes, z coordinate by coordinate, ancestors nearly in order); before, the
// state was written twice (144 bytes) and read again by the outer stage. 8,454,144 particles at
// d = 10: 472 us a step, 344 with the state written once, 275 with the outer stage's present scatter.
//
// Transition (no x/z cross-covariance in Q, as for the filter):
//   x_t = mu_x(x_{t-1}) + A_xz z_{t-1} + L_qx e_x,   z_t = A_zx x_{t-1} + A_zz z_{t-1} + L_qz e_z,
// with e_x the Philox normals of purpose PF_X and e_z those of PF_Z at counter
// (t, i, purpose, 0). Weight: log w_i = log N(y_t; h_x(x_t) + H_z z_t, R).
#pragma once

#include "dpf_step.cuh"

namespace dpf {

template <typename T>
struct PFArgs {
  const T* x_old;  // [N][xp]: the particles of step t-1 (t = 1: the initial draw)
  const T* z_old;  // [D2][N]
  T* x_new;
  T* z_new;
  T* lw;           // [N] log-weights of step t
  double* partials;  // one row a CTA: the sums of W', W'^2, W' x, W' z, W' = exp(lw - lognorm_y)
  const int32_t* anc;  // [N] ancestors from the last resampling (t >= 2)
  const T* y;          // [DY] y_t
  unsigned long long* lwmax_key;
  unsigned long long* Csum;  // reset here for this step's outer reduction
  long long N;
  uint32_t t;
  Key key;
  T gcos;     // growth cosine term of the transition into step t
  int first;  // t == 1: the particles are the initial draw, no ancestors yet
};

// A whole x row (16-byte units) at once.
template <typename T, int XP>
__device__ __forceinline__ void row_load(const T* src, T (&row)[XP]) {
#pragma unroll
  for (int q = 0; q < XP * (int)sizeof(T) / 16; ++q) {
    const uint4 v = reinterpret_cast<const uint4*>(src)[q];
    memcpy(&row[q * 16 / (int)sizeof(T)], &v, 16);
  }
}
template <typename T, int XP>
__device__ __forceinline__ void row_store(T* dst, const T (&row)[XP]) {
#pragma unroll
  for (int q = 0; q < XP * (int)sizeof(T) / 16; ++q) {
    uint4 v;
    memcpy(&v, &row[q * 16 / (int)sizeof(T)], 16);
    reinterpret_cast<uint4*>(dst)[q] = v;
  }
}

constexpr int PF_NT = 256;

template <typename T, int D1, int D2, int DY, bool XZ>
__global__ void __launch_bounds__(PF_NT)
    pf_kernel(const __grid_constant__ MC<T, D1, D2, DY> mc, const __grid_constant__ PFArgs<T> a) {
  constexpr int XP = (D1 * (int)sizeof(T) + 15) / 16 * 16 / (int)sizeof(T);  // elements of an x row
  constexpr int NV = 2 + D1 + D2, NW = PF_NT / 32;
  __shared__ T sv[NV][NW];
  __shared__ T smax[NW];
  const RoundKeys rk = round_keys(a.key);
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.Csum = 0ull;
  const long long N = a.N;
  const int lane = threadIdx.x & 31, w = threadIdx.x >> 5;
  T acc[NV], lmax = neg_inf<T>();
#pragma unroll
  for (int q = 0; q < NV; ++q) acc[q] = T(0);
  for (long long i = (long long)blockIdx.x * blockDim.x + threadIdx.x; i < N;
       i += (long long)gridDim.x * blockDim.x) {
    const long long s = a.first ? i : (long long)a.anc[i];
    T x[D1], z[D2];
    {
      T row[XP];
      row_load<T, XP>(a.x_old + s * XP, row);
#pragma unroll
      for (int c = 0; c < D1; ++c) x[c] = row[c];
    }
#pragma unroll
    for (int c = 0; c < D2; ++c) z[c] = a.z_old[c * N + s];
    T ex[D1], ez[D2];
    normals_rk<D1>(rk, a.t, (uint32_t)i, P_PF_X, 0u, ex);
    normals_rk<D2>(rk, a.t, (uint32_t)i, P_PF_Z, 0u, ez);
    // x_t = mu_x + L_qx (L_qx^-1 A_xz z + e_x)
    T mux[D1];
    mu_x(mc, x, a.gcos, mux);
    T wx[D1];
#pragma unroll
    for (int r = 0; r < D1; ++r) {
      T v = ex[r];
      if (XZ) {
#pragma unroll
        for (int c = 0; c < D2; ++c) v += mc.WAxz[r][c] * z[c];
      }
      wx[r] = v;
    }
    T xn[D1];
#pragma unroll
    for (int r = 0; r < D1; ++r) {
      T v = mux[r];
#pragma unroll
      for (int c = 0; c < D1; ++c)
        if (c <= r) v += mc.Lqx[r][c] * wx[c];
      xn[r] = v;
    }
    // z_t = A_zx x + A_zz z + L_qz e_z
    T zn[D2];
#pragma unroll
    for (int r = 0; r < D2; ++r) {
      T v = T(0);
#pragma unroll
      for (int c = 0; c < D1; ++c) v += mc.Azx[r][c] * x[c];
#pragma unroll
      for (int c = 0; c < D2; ++c) v += mc.Azz[r][c] * z[c];
      if (mc.diag_qz) {
        v += mc.Lqz[r][r] * ez[r];
      } else {
#pragma unroll
        for (int c = 0; c < D2; ++c)
          if (c <= r) v += mc.Lqz[r][c] * ez[c];
      }
      zn[r] = v;
    }
    // log N(y_t; h_x(x_t) + H_z z_t, R): whitened residual L_r^-1 (y - h_x) - L_r^-1 H_z z
    T hx[DY], res[DY];
    h_x(mc, xn, hx);
#pragma unroll
    for (int q = 0; q < DY; ++q) res[q] = a.y[q] - hx[q];
    T qf = T(0);
#pragma unroll
    for (int q = 0; q < DY; ++q) {
      T v = T(0);
#pragma unroll
      for (int c = 0; c < DY; ++c)
        if (c <= q) v += mc.LrInv[q][c] * res[c];
#pragma unroll
      for (int c = 0; c < D2; ++c) v -= mc.LrHz[q][c] * zn[c];
      qf += v * v;
    }
    const T lwi = mc.lognorm_y - T(0.5) * qf;
    {
      T row[XP];
#pragma unroll
      for (int c = 0; c < XP; ++c) row[c] = c < D1 ? xn[c < D1 ? c : 0] : T(0);
      row_store<T, XP>(a.x_new + i * XP, row);
    }
#pragma unroll
    for (int c = 0; c < D2; ++c) a.z_new[c * N + i] = zn[c];
    a.lw[i] = lwi;
    const T W = exp_t<T>(T(-0.5) * qf);
    acc[0] += W;
    acc[1] += W * W;
#pragma unroll
    for (int c = 0; c < D1; ++c) acc[2 + c] += W * xn[c];
#pragma unroll
    for (int c = 0; c < D2; ++c) acc[2 + D1 + c] += W * zn[c];
    lmax = fmax(lmax, lwi);
  }
  lmax = warp_max(lmax);
#pragma unroll
  for (int q = 0; q < NV; ++q) acc[q] = warp_sum(acc[q]);
  if (lane == 0) {
    smax[w] = lmax;
#pragma unroll
    for (int q = 0; q < NV; ++q) sv[q][w] = acc[q];
  }
  __syncthreads();
  for (int q = threadIdx.x; q < NV; q += PF_NT) {
    double t = 0.0;
#pragma unroll
    for (int r = 0; r < NW; ++r) t += (double)sv[q][r];
    a.partials[(long long)blockIdx.x * NV + q] = t;
  }
  if (threadIdx.x == 0) {
    T m = smax[0];
#pragma unroll
    for (int r = 1; r < NW; ++r) m = fmax(m, smax[r]);
    if (m > neg_inf<T>()) atomicMax(a.lwmax_key, order_key(m));
  }
}

}  // namespace dpf
