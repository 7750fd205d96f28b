// The decentralized particle filter without look-ahead (the paper's Fig. dpf, after
// Chen et al. 2011), with the prior as both proposals, the filter the LA-DPF extends.
// Call t, for each outer particle i (one CTA a group, one thread an inner particle):
//   a = the ancestor the outer resampling of call t-1 gave i (i itself at t = 1);
//   x_t^i ~ sum_j qbar^(a,j) p(x_t | x_{t-1}^a, z_{t-1}^(a,j))      (step 4: the mixture prior;
//          the component by the one-draw local systematic rule, the Gaussian draw after it);
//   q^(j) proportional to qbar^(a,j) p(x_t^i | x_{t-1}^a, z_{t-1}^(a,j))   (step 5);
//   b = local systematic resampling of j by q                          (step 6);
//   z_t^(i,j) = A_zx x_{t-1}^a + A_zz z_{t-1}^(a,b_j) + chol(Q_z) e     (step 7, r = 1);
//   ell^(i,j) = log p(y_t | x_t^i, z_t^(i,j)); log w^i = LSE_j ell - log M   (step 1);
//   qbar^(i,j) = exp(ell - LSE_j ell)                                  (step 3).
// The outer resampling of step 2 is the filter's global scan after the kernel, which
// also gives the evidence and the weighted mean. Random words: the component (t, i,
// LA_J, 0), the x noise (t, i, LA_X, 0), the local resampling (t, i, INNER, 0), the z
// noise (t, i, PROP, j). With the Gaussian approximation of the mixture (Section 4.2),
// step 4 draws x_t from the Gaussian with the mixture's mean and covariance instead, with
// the same normals.
#pragma once

#include "dpf_step_warp.cuh"

namespace dpf {

template <typename T>
struct StdArgs {
  const T* x_old;  // [N][xp]
  const T* z_old;  // [D2][N M]
  const T* lq_old;  // [N][M] normalised inner log-weights (log qbar)
  T* x_new;
  T* z_new;
  T* lq_new;
  T* lw;  // [N]
  T* xm;  // [D1][N]
  T* zm;  // [D2][N]: sum_j qbar z
  const int32_t* anc;
  const T* y;  // [DY] y_t
  unsigned long long* lwmax_key;
  unsigned long long* Csum;
  int* err;
  long long N;
  int M, xp;
  uint32_t t;
  Key key;
  T gcos;     // growth cosine term of the transition into step t
  T scaleM;   // 2^(31 - ceil(log2 M)): the local rule's quantisation
  T logM;
  int first;  // t == 1: no ancestors yet
  int gauss;  // draw x_t from the moment-matched Gaussian of the mixture (Section 4.2)
  int32_t* dbg_b;  // debug (or null): the local resampling indices, N x M
  int32_t* dbg_j;  // debug (or null): the mixture component of x_t (-1 for the Gaussian form), N
};

template <typename T, int D1, int D2, int DY, bool XZ>
__global__ void __launch_bounds__(1024)
    std_dpf_kernel(const __grid_constant__ MC<T, D1, D2, DY> mc, const __grid_constant__ StdArgs<T> a) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  const int M = a.M, tid = threadIdx.x, j = tid;
  const bool act = j < M;
  const long long N = a.N, NM = N * (long long)M;
  T* zs = (T*)smem_raw;                         // [D2][M] the ancestor group's z
  uint32_t* cum = (uint32_t*)(zs + D2 * M);     // [M]
  T* red = (T*)(cum + M + (M & 1));             // [32] block reductions
  uint32_t* redU = (uint32_t*)(red + 32);       // [64]
  const T NEG = neg_inf<T>();
  const T LOG2E = (T)LOG2E_D;
  if (blockIdx.x == 0 && tid == 0) *a.Csum = 0ull;
  for (long long i = blockIdx.x; i < N; i += gridDim.x) {
    const long long g = a.first ? i : (long long)a.anc[i];
    T xp_[D1];
#pragma unroll
    for (int c = 0; c < D1; ++c) xp_[c] = a.x_old[g * a.xp + c];
    T lqj = NEG;
    if (act) {
#pragma unroll
      for (int c = 0; c < D2; ++c) zs[c * M + j] = a.z_old[c * NM + g * M + j];
      lqj = a.lq_old[g * M + j];
    }
    // ---- x_t from the mixture: the component, then the Gaussian draw ----
    const T mx = bmax(lqj, red);
    {
      uint32_t cw[1] = {act ? (uint32_t)floor(exp2_t((lqj - mx) * LOG2E) * a.scaleM) : 0u}, incl[1];
      bscan_planes<1>(cw, incl, redU);
      if (act) cum[j] = incl[0];
    }
    __syncthreads();  // the staged rows and the component weights are complete
    const int jm = sys_local_pick(cum, M, cum[M - 1], 1, 0, rand_word(a.key, a.t, (uint32_t)i, P_LA_J, 0u));
    if (a.dbg_j && j == 0) a.dbg_j[i] = (XZ && a.gauss) ? -1 : jm;
    T e1[D1];
    normals<D1>(a.key, a.t, (uint32_t)i, P_LA_X, 0u, e1);
    T mux[D1];
    mu_x(mc, xp_, a.gcos, mux);
    T xt[D1];
    {
      T w[D1];
      if (XZ && a.gauss) {
        // the mixture's moment-matched Gaussian, in the coordinates whitened by L_qx: with
        // u_j = L_qx^-1 A_xz z_j, mean ubar = sum_j qbar_j u_j and covariance I + C,
        // C = sum_j qbar_j (u_j - ubar)(u_j - ubar)^T; w = ubar + chol(I + C) e
        T uj[D1];
#pragma unroll
        for (int r = 0; r < D1; ++r) {
          T v = T(0);
          if (act) {
#pragma unroll
            for (int c = 0; c < D2; ++c) v += mc.WAxz[r][c] * zs[c * M + j];
          }
          uj[r] = v;
        }
        const T qj = act ? exp_t<T>(lqj - mx) : T(0);
        const T qs = bsum(qj, red);
        T ub[D1];
#pragma unroll
        for (int r = 0; r < D1; ++r) ub[r] = bsum(qj * uj[r], red) / qs;
        T G[D1][D1];
#pragma unroll
        for (int r = 0; r < D1; ++r)
#pragma unroll
          for (int c = 0; c < D1; ++c)
            if (c <= r) G[r][c] = bsum(qj * (uj[r] - ub[r]) * (uj[c] - ub[c]), red) / qs + (r == c ? T(1) : T(0));
        // Cholesky of I + C in place (lower triangle), the same in every thread
#pragma unroll
        for (int c = 0; c < D1; ++c) {
          T d = G[c][c];
#pragma unroll
          for (int k = 0; k < D1; ++k)
            if (k < c) d -= G[c][k] * G[c][k];
          d = sqrt(d);
          G[c][c] = d;
#pragma unroll
          for (int r = 0; r < D1; ++r) {
            if (r > c) {
              T v = G[r][c];
#pragma unroll
              for (int k = 0; k < D1; ++k)
                if (k < c) v -= G[r][k] * G[c][k];
              G[r][c] = v / d;
            }
          }
        }
#pragma unroll
        for (int r = 0; r < D1; ++r) {
          T v = ub[r];
#pragma unroll
          for (int c = 0; c < D1; ++c)
            if (c <= r) v += G[r][c] * e1[c];
          w[r] = v;
        }
      } else {
#pragma unroll
        for (int r = 0; r < D1; ++r) {
          T v = e1[r];
          if (XZ) {
#pragma unroll
            for (int c = 0; c < D2; ++c) v += mc.WAxz[r][c] * zs[c * M + jm];
          }
          w[r] = v;
        }
      }
#pragma unroll
      for (int r = 0; r < D1; ++r) {
        T v = mux[r];
#pragma unroll
        for (int c = 0; c < D1; ++c)
          if (c <= r) v += mc.Lqx[r][c] * w[c];
        xt[r] = v;
      }
    }
    // ---- local resampling by q = qbar p(x_t | x_{t-1}, z) ----
    T alpha = lqj;
    if (XZ && act) {
      T wres[D1];  // L_qx^-1 (x_t - mu_x): the z-free part of the whitened residual
#pragma unroll
      for (int r = 0; r < D1; ++r) {
        T v = T(0);
#pragma unroll
        for (int c = 0; c < D1; ++c)
          if (c <= r) v += mc.LqxInv[r][c] * (xt[c] - mux[c]);
        wres[r] = v;
      }
      T q = T(0);
#pragma unroll
      for (int r = 0; r < D1; ++r) {
        T v = wres[r];
#pragma unroll
        for (int c = 0; c < D2; ++c) v -= mc.WAxz[r][c] * zs[c * M + j];
        q += v * v;
      }
      alpha -= T(0.5) * q;
    }
    const T amax = bmax(act ? alpha : NEG, red);  // its barriers also end every read of cum above
    {
      uint32_t cw[1] = {act ? (uint32_t)floor(exp2_t((alpha - amax) * LOG2E) * a.scaleM) : 0u}, incl[1];
      bscan_planes<1>(cw, incl, redU);
      if (act) cum[j] = incl[0];
    }
    __syncthreads();
    const uint32_t C = cum[M - 1];
    const uint32_t uin = rand_word(a.key, a.t, (uint32_t)i, P_INNER, 0u);
    // ---- propagation from the prior and the weights of y_t ----
    T yh[DY];
    {
      T hx[DY], res[DY];
      h_x(mc, xt, hx);
#pragma unroll
      for (int q = 0; q < DY; ++q) res[q] = a.y[q] - hx[q];
#pragma unroll
      for (int q = 0; q < DY; ++q) {
        T v = T(0);
#pragma unroll
        for (int c = 0; c < DY; ++c)
          if (c <= q) v += mc.LrInv[q][c] * res[c];
        yh[q] = v;
      }
    }
    T zn[D2];
    T ell = NEG;
    if (act) {
      const int b = sys_local_pick(cum, M, C, M, j, uin);
      if (a.dbg_b) a.dbg_b[i * M + j] = b;
      T eps[D2];
      normals<D2>(a.key, a.t, (uint32_t)i, P_PROP, (uint32_t)j, eps);
#pragma unroll
      for (int r = 0; r < D2; ++r) {
        T v = T(0);
#pragma unroll
        for (int c = 0; c < D1; ++c) v += mc.Azx[r][c] * xp_[c];
#pragma unroll
        for (int c = 0; c < D2; ++c) v += mc.Azz[r][c] * zs[c * M + b];
#pragma unroll
        for (int c = 0; c < D2; ++c)
          if (c <= r) v += mc.Lqz[r][c] * eps[c];
        zn[r] = v;
      }
      T qf = T(0);
#pragma unroll
      for (int q = 0; q < DY; ++q) {
        T v = yh[q];
#pragma unroll
        for (int c = 0; c < D2; ++c) v -= mc.LrHz[q][c] * zn[c];
        qf += v * v;
      }
      ell = mc.lognorm_y - T(0.5) * qf;
    }
    const T lmax = bmax(ell, red);
    const T lsum = bsum(act ? exp_t<T>(ell - lmax) : T(0), red);
    const T lse = lmax + log_t(lsum);
    const T lqn = ell - lse;
    T W = act ? exp_t<T>(lqn) : T(0);
    if (act) {
#pragma unroll
      for (int c = 0; c < D2; ++c) a.z_new[c * NM + i * M + j] = zn[c];
      a.lq_new[i * M + j] = lqn;
    }
    // the group's z-mean sum_j qbar z_t, one coordinate at a time
#pragma unroll
    for (int c = 0; c < D2; ++c) {
      const T s = bsum(act ? W * zn[c] : T(0), red);
      if (tid == 0) a.zm[c * N + i] = s;
    }
    if (tid == 0) {
      const T lwi = lse - a.logM;
#pragma unroll
      for (int c = 0; c < D1; ++c) {
        a.x_new[i * a.xp + c] = xt[c];
        a.xm[c * N + i] = xt[c];
      }
      a.lw[i] = lwi;
      if (lwi != lwi) atomicOr(a.err, ERR_NUMERIC);
      const unsigned long long key = order_key(lwi);
      if (lwi == lwi && key > *(volatile unsigned long long*)a.lwmax_key) atomicMax(a.lwmax_key, key);
    }
    __syncthreads();  // the staged rows are free for the next group
  }
}

// The same step with one warp a group (M <= 256, rows of whole 16-byte units): each lane owns
// PPL consecutive inner particles in registers, every reduction and scan is a warp shuffle, the
// local resampling takes the offspring ranges (no search), and the ancestor's rows of the next
// group are bulk-copied into the warp's stage while this one's are used. A group takes 1.9 k warp instructions, not 6.9 k; the growth model's step (N = 65536,
// M = 128) went from 581 to 194 us, 46% of the copy bandwidth; what bounds it now is the issue of
// the random numbers and the propagation at four warps a scheduler.
// The component draw of x_t is made only where it is read (an x transition that depends
// on z, or debug recording). The Gaussian form of the draw keeps the block kernel.
template <typename T, int D1, int D2>
inline size_t std_warp_smem(int M, int xp) {  // bytes a warp
  return (size_t)D2 * M * sizeof(T) + (size_t)M * sizeof(T) + (size_t)xp * sizeof(T) +
         ((size_t)M * sizeof(int) + 15) / 16 * 16 + 256 * sizeof(T);
}

// Sum over the warp of values held PPL consecutive ones a lane, added as a block of one thread a
// value adds them: 32 neighbours by a butterfly, then the groups of 32 in order (the block-wide
// form's bits, so that the weights, and every resampling decision after them, do not depend
// on which form ran). ws: 32 PPL elements of the warp's shared memory.
template <typename T, int PPL>
__device__ __forceinline__ T strided_sum(const T (&v)[PPL], T* ws, int k0, int lane) {
  if constexpr (PPL == 1) {
    return warp_sum(v[0]);
  } else {
    vst<T, PPL>(ws + k0, v);
    __syncwarp();
    T r = T(0);
#pragma unroll
    for (int p = 0; p < PPL; ++p) {
      const T s = warp_sum(ws[32 * p + lane]);
      r = p ? r + s : s;
    }
    __syncwarp();
    return r;
  }
}

template <typename T, int D1, int D2, int DY, bool XZ, int PPL>
__global__ void __launch_bounds__(WARPS_PER_CTA * 32, warp_min_blocks<PPL, D2>())
    std_warp_kernel(const __grid_constant__ MC<T, D1, D2, DY> mc, const __grid_constant__ StdArgs<T> a,
                    uint32_t warp_bytes) {
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bars[WARPS_PER_CTA];
  const int lane = threadIdx.x & 31, wib = threadIdx.x >> 5, nw = blockDim.x >> 5;
  const int M = a.M, k0 = PPL * lane;
  const bool act = k0 < M;
  const long long N = a.N, NM = N * (long long)M;
  T* sz = (T*)(smem_raw + (size_t)wib * warp_bytes);  // [D2][M] the ancestor group's z
  T* slq = sz + D2 * M;                               // [M]
  T* sx = slq + M;                                    // [xp]
  int* slot = (int*)(sx + a.xp);                      // [M] scratch of the local resampling
  T* ws = (T*)((unsigned char*)slot + ((size_t)M * sizeof(int) + 15) / 16 * 16);  // [32 PPL] sums
  uint64_t* bar = &bars[wib];
  uint32_t phase = 0;
  const T NEG = neg_inf<T>(), LOG2E = (T)LOG2E_D;
  const RoundKeys rk = round_keys(a.key);
  if (lane == 0) {
    mbar_init(bar, 1);
    mbar_fence_init();
  }
  __syncwarp();
  if (blockIdx.x == 0 && threadIdx.x == 0) *a.Csum = 0ull;
  const uint32_t row = (uint32_t)(M * sizeof(T));
  auto stage = [&](long long src) {
    if (lane == 0) mbar_arrive_tx(bar, (D2 + 1) * row + (uint32_t)(a.xp * sizeof(T)));
    for (int e = lane; e < D2 + 2; e += 32) {
      if (e < D2)
        bulk_load(sz + e * M, a.z_old + e * NM + src * M, row, bar);
      else if (e == D2)
        bulk_load(slq, a.lq_old + src * M, row, bar);
      else
        bulk_load(sx, a.x_old + src * a.xp, (uint32_t)(a.xp * sizeof(T)), bar);
    }
  };
  const long long W = (long long)gridDim.x * nw;
  long long i = (long long)blockIdx.x * nw + wib;
  long long src_next = -1;
  if (i < N) {
    stage(a.first ? i : (long long)a.anc[i]);
    if (i + W < N) src_next = a.first ? i + W : (long long)a.anc[i + W];
  }
  for (; i < N; i += W, phase ^= 1u) {
    if (!warp_rows_in(bar, phase, a.err, lane)) break;
    T xp_[D1], alpha[PPL];
#pragma unroll
    for (int c = 0; c < D1; ++c) xp_[c] = sx[c];
#pragma unroll
    for (int p = 0; p < PPL; ++p) alpha[p] = NEG;
    if (act) vld<T, PPL>(slq + k0, alpha);
    // inclusive cumulative counts of the lane's particles for the log-weights v, and the total
    auto counts = [&](const T (&v)[PPL], T mx, uint32_t (&loc)[PPL]) {
      uint32_t run = 0;
#pragma unroll
      for (int p = 0; p < PPL; ++p) {
        run += act ? (uint32_t)floor(exp2_t((v[p] - mx) * LOG2E) * a.scaleM) : 0u;
        loc[p] = run;
      }
      uint32_t s = run;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t n = __shfl_up_sync(FULL, s, o);
        if (lane >= o) s += n;
      }
#pragma unroll
      for (int p = 0; p < PPL; ++p) loc[p] += s - run;
      return __shfl_sync(FULL, s, 31);
    };
    auto lane_max = [&](const T (&v)[PPL]) {
      T m = v[0];
#pragma unroll
      for (int p = 1; p < PPL; ++p) m = fmax(m, v[p]);
      return warp_max_redux(m);
    };
    // ---- x_t from the mixture: the component, then the Gaussian draw ----
    T e1[D1], mux[D1], xt[D1];
    normals_rk<D1>(rk, a.t, (uint32_t)i, P_LA_X, 0u, e1);
    mu_x(mc, xp_, a.gcos, mux);
    T w[D1];
#pragma unroll
    for (int r = 0; r < D1; ++r) w[r] = e1[r];
    if (XZ || a.dbg_j) {
      // the one-draw local rule: the component is the number of particles whose cumulative
      // count c_k has c_k 2^32 <= u C
      uint32_t loc[PPL];
      const uint32_t C = counts(alpha, lane_max(alpha), loc);
      const uint64_t rhs = (uint64_t)philox_rk(ctr(a.t, (uint32_t)i, P_LA_J, 0u, 0u), rk).x * C;
      unsigned below = 0;
#pragma unroll
      for (int p = 0; p < PPL; ++p) below += act && ((uint64_t)loc[p] << 32) <= rhs ? 1u : 0u;
      const int jm = min((int)__reduce_add_sync(FULL, below), M - 1);
      if (a.dbg_j && lane == 0) a.dbg_j[i] = jm;
      if (XZ) {
#pragma unroll
        for (int r = 0; r < D1; ++r) {
#pragma unroll
          for (int c = 0; c < D2; ++c) w[r] += mc.WAxz[r][c] * sz[c * M + jm];
        }
      }
    }
#pragma unroll
    for (int r = 0; r < D1; ++r) {
      T v = mux[r];
#pragma unroll
      for (int c = 0; c < D1; ++c)
        if (c <= r) v += mc.Lqx[r][c] * w[c];
      xt[r] = v;
    }
    // ---- local resampling by q = qbar p(x_t | x_{t-1}, z) ----
    if (XZ && act) {
      T wres[D1], q[PPL];
#pragma unroll
      for (int r = 0; r < D1; ++r) {
        T v = T(0);
#pragma unroll
        for (int c = 0; c < D1; ++c)
          if (c <= r) v += mc.LqxInv[r][c] * (xt[c] - mux[c]);
        wres[r] = v;
      }
#pragma unroll
      for (int p = 0; p < PPL; ++p) q[p] = T(0);
#pragma unroll
      for (int r = 0; r < D1; ++r) {
        T v[PPL];
#pragma unroll
        for (int p = 0; p < PPL; ++p) v[p] = wres[r];
#pragma unroll
        for (int c = 0; c < D2; ++c) {
          T zc[PPL];
          vld<T, PPL>(sz + c * M + k0, zc);
          axpy<T, PPL>(-mc.WAxz[r][c], zc, v);
        }
#pragma unroll
        for (int p = 0; p < PPL; ++p) q[p] += v[p] * v[p];
      }
#pragma unroll
      for (int p = 0; p < PPL; ++p) alpha[p] -= T(0.5) * q[p];
    }
    int bidx[PPL];
    {
      uint32_t loc[PPL];
      const uint32_t C = counts(alpha, lane_max(alpha), loc);
      const uint32_t uin = philox_rk(ctr(a.t, (uint32_t)i, P_INNER, 0u, 0u), rk).x;
      sys_local_offspring<PPL>(loc, C, M, uin >> 16, k0, act, lane, slot, bidx);
    }
    if (a.dbg_b && act) vst<int, PPL>(a.dbg_b + i * M + k0, bidx);
    // ---- propagation from the prior and the weights of y_t ----
    T yh[DY];
    {
      T hx[DY], res[DY];
      h_x(mc, xt, hx);
#pragma unroll
      for (int q = 0; q < DY; ++q) res[q] = a.y[q] - hx[q];
#pragma unroll
      for (int q = 0; q < DY; ++q) {
        T v = T(0);
#pragma unroll
        for (int c = 0; c < DY; ++c)
          if (c <= q) v += mc.LrInv[q][c] * res[c];
        yh[q] = v;
      }
    }
    T zn[D2][PPL];
#pragma unroll
    for (int r = 0; r < D2; ++r) {
      T v = T(0);
#pragma unroll
      for (int c = 0; c < D1; ++c) v += mc.Azx[r][c] * xp_[c];
#pragma unroll
      for (int p = 0; p < PPL; ++p) zn[r][p] = v;
    }
#pragma unroll
    for (int c = 0; c < D2; ++c) {
      T zc[PPL];
#pragma unroll
      for (int p = 0; p < PPL; ++p) zc[p] = sz[c * M + bidx[p]];
#pragma unroll
      for (int r = 0; r < D2; ++r) axpy<T, PPL>(mc.Azz[r][c], zc, zn[r]);
    }
    // the stage is consumed: prefetch the next group's rows into it
    __syncwarp();
    if (i + W < N) {
      stage(src_next);
      if (i + 2 * W < N) src_next = a.first ? i + 2 * W : (long long)a.anc[i + 2 * W];
    }
#pragma unroll
    for (int b = 0; b < (D2 + 3) / 4; ++b) {
      T e4[4][PPL];
#pragma unroll
      for (int p = 0; p < PPL; ++p) {
        T e[4];
        normal_block_rk(rk, a.t, (uint32_t)i, P_PROP, (uint32_t)(k0 + p), b, D2 - 4 * b, e);
#pragma unroll
        for (int j = 0; j < 4; ++j) e4[j][p] = e[j];
      }
#pragma unroll
      for (int j = 0; j < 4; ++j) {
        const int c = 4 * b + j;
        if (c < D2) {
          if (mc.diag_qz) {
            axpy<T, PPL>(mc.Lqz[c][c], e4[j], zn[c]);
          } else {
#pragma unroll
            for (int r = 0; r < D2; ++r)
              if (r >= c) axpy<T, PPL>(mc.Lqz[r][c], e4[j], zn[r]);
          }
        }
      }
    }
    T ell[PPL], lmax = NEG;
    {
      T qf[PPL];
#pragma unroll
      for (int p = 0; p < PPL; ++p) qf[p] = T(0);
#pragma unroll
      for (int q = 0; q < DY; ++q) {
        T v[PPL];
#pragma unroll
        for (int p = 0; p < PPL; ++p) v[p] = yh[q];
#pragma unroll
        for (int c = 0; c < D2; ++c) axpy<T, PPL>(-mc.LrHz[q][c], zn[c], v);
#pragma unroll
        for (int p = 0; p < PPL; ++p) qf[p] += v[p] * v[p];
      }
#pragma unroll
      for (int p = 0; p < PPL; ++p) {
        ell[p] = act ? mc.lognorm_y - T(0.5) * qf[p] : NEG;
        lmax = fmax(lmax, ell[p]);
      }
    }
    lmax = warp_max_redux(lmax);
    T Wp[PPL];
#pragma unroll
    for (int p = 0; p < PPL; ++p) Wp[p] = act ? exp_t<T>(ell[p] - lmax) : T(0);
    const T lsum = strided_sum<T, PPL>(Wp, ws, k0, lane);
    const T lse = lmax + log_t(lsum);
    if (act) {
#pragma unroll
      for (int c = 0; c < D2; ++c) vst<T, PPL>(a.z_new + c * NM + i * M + k0, zn[c]);
      T lqn[PPL];
#pragma unroll
      for (int p = 0; p < PPL; ++p) lqn[p] = ell[p] - lse;
      vst<T, PPL>(a.lq_new + i * M + k0, lqn);
    }
    // the group's z-mean sum_j qbar z_t (lane c < D2 ends with coordinate c)
    {
      T acc[D2];
#pragma unroll
      for (int c = 0; c < D2; ++c) {
        T v = T(0);
#pragma unroll
        for (int p = 0; p < PPL; ++p) v += Wp[p] * zn[c][p];
        acc[c] = act ? v : T(0);
      }
      const T tot = warp_sum_vec<D2>(acc, lane) / lsum;
      if (lane < D2) a.zm[(long long)lane * N + i] = tot;
    }
    if (lane == 0) {
      const T lwi = lse - a.logM;
#pragma unroll
      for (int c = 0; c < D1; ++c) {
        a.x_new[i * a.xp + c] = xt[c];
        a.xm[(long long)c * N + i] = xt[c];
      }
      a.lw[i] = lwi;
      if (lwi != lwi) atomicOr(a.err, ERR_NUMERIC);
      const unsigned long long key = order_key(lwi);
      if (lwi == lwi && key > *(volatile unsigned long long*)a.lwmax_key) atomicMax(a.lwmax_key, key);
    }
    __syncwarp();
  }
}

}  // namespace dpf
