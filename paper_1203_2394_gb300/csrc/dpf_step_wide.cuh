// The steady-state step of the wide variant on the tensor cores (z of a few tens of coordinates,
// x transition free of z, diagonal Q_z, M = 128 or 256) with two threads an inner particle.
//
// The block step (step_body in dpf_step.cuh) gives a particle one thread, which at M = 256 is two
// warps a scheduler (a group fills the SM's shared memory) walking long chains between block
// barriers: 46 k cycles a group at 29% issue, 13 k of them drawing the noise beside the y and
// look-ahead projections, 6 k in sections that one warp runs while the others wait. Here thread
// (j, 0) and thread (j, 1) share particle j: each gathers, splits, draws the noise of and writes
// its half of the coordinates, then one accumulates the y residual and the other the look-ahead
// projection over all of them (in coordinate order, as the block step does). The noise and the
// look-ahead's draws are made while the MMAs run, the ancestor's selection beside the local
// resampling's scan, the MMAs are issued by a thread a tile (one thread took 4.6 k cycles for both),
// and what only one warp does (the next group's copies in, z_t's copies out, the outer weight) is
// given to warps of the half that then waits for the other. Every sum that feeds a weight keeps the
// block step's order, so the weights and every resampling decision keep their bits. Time steps of
// the 64-state growth model, N = 32768, M = 256, L = 16: 5007 -> 3343 us a step (the model read once a CTA from
// the context's own copy; with it copied into a constant bank before every launch 3389); what bounds it now is shared
// memory: the two projections read 56 rows of 8 weights for each particle (5 k cycles a group).
#pragma once

#include "dpf_step_warp.cuh"

namespace dpf {

// Bulk copy from shared to global memory (16-byte units), in the issuing thread's bulk group, and the
// wait until the group's copies have read their source.
__device__ __forceinline__ void bulk_store(void* dst, const void* src, uint32_t bytes) {
  asm volatile("cp.async.bulk.global.shared::cta.bulk_group [%0], [%1], %2;" ::"l"(dst), "r"(smem_addr(src)), "r"(bytes)
               : "memory");
}
__device__ __forceinline__ void bulk_store_commit() { asm volatile("cp.async.bulk.commit_group;" ::: "memory"); }
__device__ __forceinline__ void bulk_store_wait_read() {
  asm volatile("cp.async.bulk.wait_group.read 0;" ::: "memory");
}

// acc[0..N-1] += v * m[0..N-1] with m in shared memory (16-byte aligned): packed FMAs.
template <int N>
__device__ __forceinline__ void axpy_row(float v, const float* m, float (&acc)[N]) {
#pragma unroll
  for (int q = 0; q < N; q += 4) {
    const float4 x = *reinterpret_cast<const float4*>(m + q);
    const float2 a = __ffma2_rn(make_float2(x.x, x.y), make_float2(v, v), make_float2(acc[q], acc[q + 1]));
    const float2 b = __ffma2_rn(make_float2(x.z, x.w), make_float2(v, v), make_float2(acc[q + 2], acc[q + 3]));
    acc[q] = a.x;
    acc[q + 1] = a.y;
    acc[q + 2] = b.x;
    acc[q + 3] = b.y;
  }
}

// Barrier of the first `n` threads of the CTA (whole warps).
__device__ __forceinline__ void first_half_sync(int n) { asm volatile("bar.sync 1, %0;" ::"r"(n) : "memory"); }

template <int D1, int D2, int DY>
__device__ __forceinline__ void wide_pair_body(const MC<float, D1, D2, DY>& mc, const StepArgs<float>& a) {
  static_assert(D2 % 8 == 0 && D2 <= 64 && DY == 8 && D1 <= 32, "the compiled wide variant");
  // coordinates 0 .. 31 belong to a particle's first thread, the others to its second, which also
  // draws the look-ahead's DY inner normals: 8 Philox blocks each at d2 = 56, DY = 8
  constexpr int HC = 32, H1 = D2 - HC;
  static_assert(H1 == 24, "TMEM loads of 16 + 8 columns, and 8 more in the first half");
  constexpr int NP = (D2 + 15) / 16 * 16;  // MMA N: A_zz rows padded to 16
  constexpr int KC16 = D2 * 4 / 16;        // 16-byte chunks per operand row
  constexpr int REC = rec_len<float, D1, DY, false>();
  extern __shared__ __align__(128) unsigned char smem_raw[];
  __shared__ __align__(8) uint64_t bars[2];  // the stage's barrier (as stage_group takes it), spare
  __shared__ __align__(8) uint64_t tcbar;
  __shared__ uint32_t s_taddr, s_uin;
  __shared__ int s_ok;
  __shared__ float s_x[D1], s_mux[D1], s_ps, s_mx;
  __shared__ float s_model[6];  // growth (0 or 1), its a and b; h_x's quadratic part (0 or 1) and factor; log norm of R
  const int M = a.M, L = a.L;
  const long long N = a.N, NM = N * (long long)M;
  const int tid = threadIdx.x, lane = tid & 31, w = tid >> 5, nw = blockDim.x >> 5, hw = M >> 5;
  const int h = tid >= M ? 1 : 0, j = tid - h * M;
  unsigned char* const stage0 = smem_raw + a.off_stage;
  uint32_t* cum = (uint32_t*)(smem_raw + a.off_cum);
  float* kd = (float*)(smem_raw + a.off_kd);
  float* E = (float*)(smem_raw + a.off_E);
  float* cw = (float*)(smem_raw + a.off_cw);
  float* xbs = (float*)(smem_raw + a.off_xbs);
  float* rowS = (float*)(smem_raw + a.off_row);
  float* pm = rowS + L;    // the draws' weights relative to the largest
  float* shS = pm + L;
  float* coef = shS + 2 * L;
  float* red = (float*)(smem_raw + a.off_red);
  uint32_t* redU = (uint32_t*)(red + 32);
  float* part = (float*)(smem_raw + a.off_part);
  float* zmat = (float*)(smem_raw + a.off_zmat);
  float* sbs = (float*)(smem_raw + a.off_sb);
  float* pj = (float*)(smem_raw + a.off_proj);
  float* s_azx = part;  // A_zx x_a (free until the z-mean, which uses the first 32 DY floats of part)
  // the small matrices, by column where a thread accumulates a row after another: as constant-bank
  // operands they missed the constant cache anew for every group
  float* s_LsT = part + 512;         // [c][q] = L_s[q][c]
  float* s_LrInvT = s_LsT + DY * DY;  // [c][q] = L_r^-1[q][c]
  float* s_HzAzxT = s_LrInvT + DY * DY;  // [c][q] = (H_z A_zx)[q][c]
  float* s_HxT = s_HzAzxT + DY * D1;     // [c][q] = H_x[q][c]
  float* s_LqxT = s_HxT + DY * D1;       // [c][r] = L_qx[r][c]
  float* s_Axx = s_LqxT + D1 * D1;       // [r][c] = A_xx[r][c]
  static_assert(512 + 2 * DY * DY + 2 * DY * D1 + 2 * D1 * D1 <= 32 * (D2 + DY), "the matrices fit in part");
  const float* s_lqd = pj + D2 * (2 * DY + D1);
  const float* s_Azx = pj + D2 * 2 * DY;
  unsigned char* ahi = smem_raw + a.off_ahi;
  unsigned char* alo = smem_raw + a.off_alo;
  unsigned char* zlo = smem_raw + a.off_zlo;
  float* zsrc = (float*)zlo;  // z_t, once the MMAs have read the low parts
  float* sz = (float*)(stage0 + a.off_sz);
  float* slq = (float*)(stage0 + a.off_slq);
  float* sx = (float*)(stage0 + a.off_sx);
  float* slwh = (float*)(stage0 + a.off_slwh);
  float* sxbb = (float*)(stage0 + a.off_sxbb);
  const float NEG = neg_inf<float>(), LOG2E = (float)LOG2E_D, SQ = (float)SQ_D;
  const RoundKeys rk = round_keys(a.key);
  if (blockIdx.x == 0 && tid == 0) *a.Csum = 0ull;
  // ---- once a CTA: barriers, TMEM, the model's rows in shared memory (as the block step) ----
  if (tid == 0) {
    mbar_init(&bars[0], 1);
    mbar_init(&tcbar, (uint32_t)(M / 128));
    mbar_fence_init();
  }
  const int NT = blockDim.x;
  if (tid == 0) {
    s_model[0] = mc.growth ? 1.f : 0.f;
    s_model[1] = mc.ga;
    s_model[2] = mc.gb;
    s_model[3] = mc.quad ? 1.f : 0.f;
    s_model[4] = mc.qc;
    s_model[5] = mc.lognorm_y;
  }
  for (int e = tid; e < D2 * (D2 + DY); e += NT) {
    const int r = e / (D2 + DY), c = e % (D2 + DY);
    zmat[e] = c < D2 ? mc.Azz[r][c] : mc.K[r][c - D2];
  }
  for (int e = tid; e < D2 * 2 * DY; e += NT) {
    const int r = e / (2 * DY), q = e % (2 * DY);
    pj[e] = q < DY ? -mc.LrHz[q][r] : mc.HzAzz[q - DY][r];
  }
  for (int e = tid; e < DY * DY; e += NT) {
    const int c = e / DY, q = e % DY;
    s_LsT[e] = c <= q ? mc.Ls[q][c] : 0.f;
    s_LrInvT[e] = c <= q ? mc.LrInv[q][c] : 0.f;
  }
  for (int e = tid; e < DY * D1; e += NT) {
    s_HzAzxT[e] = mc.HzAzx[e % DY][e / DY];
    s_HxT[e] = mc.Hx[e % DY][e / DY];
  }
  for (int e = tid; e < D1 * D1; e += NT) {
    s_LqxT[e] = e / D1 <= e % D1 ? mc.Lqx[e % D1][e / D1] : 0.f;
    s_Axx[e] = mc.Axx[e / D1][e % D1];
  }
  for (int e = tid; e < D2 * D1; e += NT) pj[D2 * 2 * DY + e] = mc.Azx[e / D1][e % D1];
  for (int r = tid; r < D2; r += NT) pj[D2 * (2 * DY + D1) + r] = mc.Lqz[r][r];
  for (int e = tid; e < NP * D2; e += NT) {
    const int n = e / D2, k = e % D2;
    float hi = 0.f, lo = 0.f;
    if (n < D2) tc::split_tf32(mc.Azz[n][k], hi, lo);
    *(float*)(ahi + tc::kmajor_offset(n, 4 * k, KC16)) = hi;
    *(float*)(alo + tc::kmajor_offset(n, 4 * k, KC16)) = lo;
  }
  constexpr uint32_t TC_COLS = 2 * NP;
  tc::fence_proxy_async();
  if (w == 0) {
    tc::tmem_alloc(&s_taddr, TC_COLS);
    tc::tmem_relinquish();
  }
  tc::fence_before();
  __syncthreads();
  tc::fence_after();
  const uint32_t taddr = s_taddr;
  uint32_t tc_phase = 0;
  const uint32_t ta = taddr + ((uint32_t)(32 * (w & 3)) << 16) + (uint32_t)((j >> 7) * NP + HC * h);

  // out = L v for a lower-triangular L given by columns; out[q] sums c = 0 .. q in order
  auto tri = [&](const float* LT, const float (&v)[DY], float (&out)[DY]) {
#pragma unroll
    for (int q = 0; q < DY; ++q) out[q] = 0.f;
#pragma unroll
    for (int c = 0; c < DY; ++c) {
      const float4 m0 = *reinterpret_cast<const float4*>(LT + c * DY);
      const float4 m1 = *reinterpret_cast<const float4*>(LT + c * DY + 4);
      const float m[8] = {m0.x, m0.y, m0.z, m0.w, m1.x, m1.y, m1.z, m1.w};
#pragma unroll
      for (int q = 0; q < DY; ++q)
        if (c <= q) out[q] = fmaf(m[q], v[c], out[q]);
    }
  };
  // h_x(x) = qc x.^2 + H_x x, as h_x in dpf_step.cuh
  auto obs_x = [&](const float (&xv)[D1], float (&out)[DY]) {
#pragma unroll
    for (int q = 0; q < DY; ++q) out[q] = s_model[3] != 0.f ? s_model[4] * xv[q < D1 ? q : 0] * xv[q < D1 ? q : 0] : 0.f;
#pragma unroll
    for (int c = 0; c < D1; ++c) axpy_row<DY>(xv[c], s_HxT + c * DY, out);
  };
  const long long G = group_count(a);
  auto source_of = [&](long long q) {
    const long long iq = group_at(a, q);
    return a.first ? iq : (long long)a.anc[iq];
  };
  long long g = blockIdx.x;
  if (g < G && w == 0) stage_group<float, D1, D2, true, true>(a, stage0, &bars[0], source_of(g));
  for (int k = 0; g < G; g += gridDim.x, ++k) {
    const long long i = group_at(a, g);
    // one thread polls; the barrier releases the rest
    if (!__syncthreads_and(tid || tc::bar_wait(&bars[0], (uint32_t)(k & 1), MBAR_SPIN_LIMIT))) {
      if (tid == 0) {
        atomicOr(a.err, ERR_TIMEOUT);
        tc::bar_wait(&bars[0], (uint32_t)(k & 1), MBAR_SPIN_LIMIT);
      }
      break;
    }
    if (a.gskip && a.gskip[i]) {
      __syncthreads();
      if (w == 0 && g + gridDim.x < G)
        stage_group<float, D1, D2, true, true>(a, stage0, &bars[0], source_of(g + gridDim.x));
      continue;
    }
    // ---- local resampling's cumulative counts (first half), beside the selection of
    // x_{t-1}^(i) among the ancestor's look-ahead draws (first warp of the second half) ----
    if (h == 0) {
      const float al = slq[j];
      float amax = warp_max(al);
      if (lane == 0) red[w] = amax;
      first_half_sync(M);
      amax = red[0];
      for (int q = 1; q < hw; ++q) amax = fmaxf(amax, red[q]);
      uint32_t v = (uint32_t)floor(exp2_t((al - amax) * LOG2E) * a.scaleM);
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t n = __shfl_up_sync(FULL, v, o);
        if (lane >= o) v += n;
      }
      if (lane == 31) redU[w] = v;
      first_half_sync(M);
      for (int q = 0; q < w; ++q) v += redU[q];
      cum[j] = v;
    } else if (w == hw) {
      const float l0 = lane < L ? slwh[lane] : NEG;
      const float l1 = lane + 32 < L ? slwh[lane + 32] : NEG;
      const float mx = warp_max(fmaxf(l0, l1));
      const uint32_t c0 = lane < L ? (uint32_t)floor(exp2_t((l0 - mx) * LOG2E) * a.scaleL) : 0u;
      const uint32_t c1 = lane + 32 < L ? (uint32_t)floor(exp2_t((l1 - mx) * LOG2E) * a.scaleL) : 0u;
      uint32_t s0 = c0, s1 = c1;
#pragma unroll
      for (int o = 1; o < 32; o <<= 1) {
        const uint32_t n0 = __shfl_up_sync(FULL, s0, o), n1 = __shfl_up_sync(FULL, s1, o);
        if (lane >= o) {
          s0 += n0;
          s1 += n1;
        }
      }
      const uint32_t tot0 = __shfl_sync(FULL, s0, 31), tot1 = __shfl_sync(FULL, s1, 31);
      const uint64_t C = (uint64_t)tot0 + tot1;
      const uint32_t word = philox_rk(ctr(a.t - 1, (uint32_t)i, lane == 0 ? P_SEL : P_INNER, 0u, 0u), rk).x;
      const uint64_t rhs = (uint64_t)__shfl_sync(FULL, word, 0) * C;
      const unsigned b0 = __ballot_sync(FULL, ((uint64_t)s0 << 32) > rhs);
      const unsigned b1 = __ballot_sync(FULL, ((uint64_t)(s1 + tot0) << 32) > rhs);
      int m = b0 ? __ffs(b0) - 1 : (b1 ? 32 + __ffs(b1) - 1 : L - 1);
      if (C == 0 || m >= L) {  // no positive weight (NaN or -inf look-ahead weights)
        if (lane == 0) atomicOr(a.err, ERR_NUMERIC);
        m = L - 1;
      }
      if (lane == 0) a.sel[i] = m;
      if (lane == 1) s_uin = word;
      if (lane < D1) s_x[lane] = sxbb[m * D1 + lane];
    }
    __syncthreads();
    // ---- gather, split and product A_zz z_b (each thread its half of the coordinates) ----
    const uint32_t C = cum[M - 1];
    const int b = sys_local_pick(cum, M, C, M, j, s_uin);
    if (a.dbg_b && h == 0) a.dbg_b[i * M + j] = b;
    {
      float zb[HC];
#pragma unroll
      for (int c = 0; c < HC; ++c) zb[c] = c < H1 || h == 0 ? sz[(HC * h + c) * M + b] : 0.f;
      if (tid < D2) {
        const float* azr = s_Azx + tid * D1;
        float v = 0.f;
#pragma unroll
        for (int c = 0; c < D1; ++c) v += azr[c] * sx[c];
        s_azx[tid] = v;
      }
      if (w == hw && lane < D1) {  // mean of x_t without the z part, as mu_x in dpf_step.cuh
        float v = 0.f;
        const float xl = s_x[lane];
        if (s_model[0] != 0.f) v = s_model[1] * xl + s_model[2] * xl / (1.f + xl * xl) + a.gcos_cur;
#pragma unroll
        for (int c = 0; c < D1; ++c) v += s_Axx[lane * D1 + c] * s_x[c];
        s_mux[lane] = v;
      }
      if (w == hw + 1) bulk_store_wait_read();  // the last group's z_t has left its buffer (zlo)
      __syncthreads();  // every gather is done: the staged z rows become the A operand
      const uint32_t tb = (uint32_t)(j >> 7) * 128u * (uint32_t)(D2 * 4);
      const int rr = j & 127;
#pragma unroll
      for (int c = 0; c < HC; c += 4) {
        if (c >= H1 && h) break;
        float4 hi, lo;
        tc::split_tf32(zb[c + 0], hi.x, lo.x);
        tc::split_tf32(zb[c + 1], hi.y, lo.y);
        tc::split_tf32(zb[c + 2], hi.z, lo.z);
        tc::split_tf32(zb[c + 3], hi.w, lo.w);
        const uint32_t o = tb + tc::kmajor_offset(rr, 4 * (HC * h + c), KC16);
        *(float4*)((unsigned char*)sz + o) = hi;
        *(float4*)(zlo + o) = lo;
      }
    }
    tc::fence_proxy_async();
    tc::fence_before();
    __syncthreads();
    if (w < M / 128 && lane == 0) {  // a thread a tile of 128 particles
      tc::fence_after();
      constexpr uint32_t idesc = tc::instr_desc(tc::FMT_TF32, 128, NP);
      const uint32_t s_zhi = smem_addr(sz), s_zlo = smem_addr(zlo), s_ahi = smem_addr(ahi), s_alo = smem_addr(alo);
      const uint32_t d = taddr + (uint32_t)(w * NP), ob = (uint32_t)w * 128u * (uint32_t)(D2 * 4);
#pragma unroll
      for (int ks = 0; ks < D2 / 8; ++ks) {
        const uint32_t o = (uint32_t)ks * 256u;
        tc::mma_tf32(d, tc::smem_desc(s_zlo + ob + o, KC16), tc::smem_desc(s_ahi + o, KC16), idesc, ks > 0);
        tc::mma_tf32(d, tc::smem_desc(s_zhi + ob + o, KC16), tc::smem_desc(s_alo + o, KC16), idesc, 1);
        tc::mma_tf32(d, tc::smem_desc(s_zhi + ob + o, KC16), tc::smem_desc(s_ahi + o, KC16), idesc, 1);
      }
      tc::commit(&tcbar);
    }
    __syncwarp();
    // ---- while the MMAs run: the propagation noise, the look-ahead's inner noise (second half),
    // the whitened y_{t-1} - h_x(x_{t-1}) (first half), and the L draws (one warp) ----
    float x[D1];
#pragma unroll
    for (int c = 0; c < D1; ++c) x[c] = s_x[c];
    float eps[HC];
#pragma unroll
    for (int c = H1; c < HC; ++c) eps[c] = 0.f;
#pragma unroll
    for (int q = 0; q < HC / 4; ++q) {
      if (4 * q >= H1 && h) break;
      float e[4];
      normal_block_rk(rk, a.t - 1, (uint32_t)i, P_PROP, (uint32_t)j, HC / 4 * h + q, 4, e);
#pragma unroll
      for (int u = 0; u < 4; ++u) eps[4 * q + u] = e[u];
    }
    float vq[DY];  // first half: the y residual; second half: the look-ahead's inner noise
    if (h == 0) {
      float res[DY];
      obs_x(x, res);
#pragma unroll
      for (int q = 0; q < DY; ++q) res[q] = a.y_prev[q] - res[q];
      tri(s_LrInvT, res, vq);
    } else {
      float e2[DY];
      normals_rk<DY>(rk, a.t, (uint32_t)i, P_LA_Z, (uint32_t)j, e2);
      tri(s_LsT, e2, vq);
    }
    if (w == nw - 1) {
      float mux[D1];
#pragma unroll
      for (int c = 0; c < D1; ++c) mux[c] = s_mux[c];
      for (int m = lane; m < L; m += 32) {
        float e1[D1], xb[D1], res[DY], cv[DY];
        normals_rk<D1>(rk, a.t, (uint32_t)i, P_LA_X, (uint32_t)m, e1);
#pragma unroll
        for (int r = 0; r < D1; ++r) xb[r] = mux[r];
#pragma unroll
        for (int c = 0; c < D1; ++c) {
#pragma unroll
          for (int r = 0; r < D1; ++r)
            if (c <= r) xb[r] = fmaf(s_LqxT[c * D1 + r], e1[c], xb[r]);
        }
        static_assert(D1 % 4 == 0, "vector stores of a draw");
#pragma unroll
        for (int r = 0; r < D1; r += 4) {
          const float4 v = make_float4(xb[r], xb[r + 1], xb[r + 2], xb[r + 3]);
          *reinterpret_cast<float4*>(a.xbb_new + ((long long)i * L + m) * D1 + r) = v;
          *reinterpret_cast<float4*>(xbs + m * D1 + r) = v;
        }
        obs_x(xb, res);
#pragma unroll
        for (int q = 0; q < DY; ++q) res[q] = a.y_cur[q] - res[q];
        tri(s_LrInvT, res, cv);
#pragma unroll
        for (int q = 0; q < DY; ++q) cw[m * DY + q] = SQ * cv[q];
      }
    }
    if (tid == 0) {
      s_ok = tc::bar_wait(&tcbar, tc_phase, TC_SPIN);
    }
    tc_phase ^= 1u;
    __syncwarp();
    tc::fence_before();
    __syncthreads();
    tc::fence_after();
    if (!s_ok) {  // (no copy is in flight here; the MMAs get a second wait)
      if (tid == 0) {
        atomicOr(a.err, ERR_TIMEOUT);
        tc::bar_wait(&tcbar, tc_phase ^ 1u, MBAR_SPIN_LIMIT);
      }
      break;
    }
    {
      float az[HC];
      tc::ld16(ta, *reinterpret_cast<float(*)[16]>(az));
      tc::ld8(ta + 16, *reinterpret_cast<float(*)[8]>(az + 16));
      if (h == 0) {
        tc::ld8(ta + 24, *reinterpret_cast<float(*)[8]>(az + 24));
      } else {
#pragma unroll
        for (int c = H1; c < HC; ++c) az[c] = 0.f;
      }
#pragma unroll
      for (int c = 0; c < HC; c += 4) {
        if (c >= H1 && h) break;
        const float4 za = *reinterpret_cast<const float4*>(s_azx + HC * h + c);
        const float4 lq = *reinterpret_cast<const float4*>(s_lqd + HC * h + c);
        const float azv[4] = {za.x, za.y, za.z, za.w}, lqv[4] = {lq.x, lq.y, lq.z, lq.w};
#pragma unroll
        for (int u = 0; u < 4; ++u) {
          const int r = HC * h + c + u;
          const float v = (az[c + u] + azv[u]) + lqv[u] * eps[c + u];
          zsrc[r * M + j] = v;
        }
      }
    }
    tc::fence_proxy_async();
    tc::fence_before();
    __syncthreads();  // z_t is in shared memory; it goes to the state by bulk copies, a row each
    if (w == hw + 1) {
      for (int r = lane; r < D2; r += 32)
        bulk_store(a.z_new + r * NM + i * M, zsrc + r * M, (uint32_t)(M * sizeof(float)));
      bulk_store_commit();
    }
    // the MMAs have read the stage: the next group's rows may come in
    if (w == hw && g + gridDim.x < G)
      stage_group<float, D1, D2, true, true>(a, stage0, &bars[0], source_of(g + gridDim.x));
    float lsum = 0.f;
    if (h == 0) {
      // ---- the y_{t-1} update (eq. qbar): the whitened residual over the coordinates in order ----
#pragma unroll 8
      for (int r = 0; r < D2; ++r) axpy_row<DY>(zsrc[r * M + j], pj + r * 2 * DY, vq);
      float qf = 0.f;
#pragma unroll
      for (int q = 0; q < DY; ++q) qf += vq[q] * vq[q];
      const float ell = -0.5f * qf;
      float lmax = warp_max(ell);
      if (lane == 0) red[w] = lmax;
      first_half_sync(M);
      lmax = red[0];
      for (int q = 1; q < hw; ++q) lmax = fmaxf(lmax, red[q]);
      const float ls = warp_sum(exp2_t((ell - lmax) * LOG2E));
      if (lane == 0) red[16 + w] = ls;
      first_half_sync(M);
      lsum = red[16];
      for (int q = 1; q < hw; ++q) lsum += red[16 + q];
      const float llsum = log_t(lsum);
      const float lqr = ell - lmax - llsum;
      a.lq_new[i * M + j] = lqr;
      kd[j * REC] = (lqr - -llsum) * LOG2E;  // relative to the largest, whose ell is lmax
      if (tid < D1) a.x_new[i * a.xp + tid] = s_x[tid];
    } else {
      // ---- the look-ahead's projected draw H_z (A_zx x + A_zz z) + noise, whitened ----
      float gz[DY];
#pragma unroll
      for (int q = 0; q < DY; ++q) gz[q] = 0.f;
#pragma unroll 8
      for (int r = 0; r < D2; ++r) axpy_row<DY>(zsrc[r * M + j], pj + r * 2 * DY + DY, gz);
      float gv[DY], rv[DY];
#pragma unroll
      for (int q = 0; q < DY; ++q) gv[q] = vq[q];
#pragma unroll
      for (int c = 0; c < D1; ++c) axpy_row<DY>(x[c], s_HzAzxT + c * DY, gv);
#pragma unroll
      for (int q = 0; q < DY; ++q) gv[q] += gz[q];
      tri(s_LrInvT, gv, rv);
      float* rec = kd + j * REC;
#pragma unroll
      for (int q = 0; q < DY; ++q) rec[1 + q] = SQ * rv[q];
    }
    __syncthreads();
    // ---- the L x M weights (eq. weightsMC), log2 units: a thread keeps its particle's record and
    // walks every other draw; then the row sums, tpm threads a row, in the block step's order ----
    const int tpm = a.tpm, rows = a.rows, stride = a.stride;
    const float tiny = 1e-30f;
    static_assert(REC % 4 == 0 && 1 + DY <= 12, "a record is three 16-byte units");
    float rec0, gk[DY];
    {
      const float4* rp = reinterpret_cast<const float4*>(kd + j * REC);
      const float4 r0 = rp[0], r1 = rp[1], r2 = rp[2];
      rec0 = r0.x;
      gk[0] = r0.y; gk[1] = r0.z; gk[2] = r0.w;
      gk[3] = r1.x; gk[4] = r1.y; gk[5] = r1.z; gk[6] = r1.w;
      gk[7] = r2.x;
    }
    auto exponent = [&](int m) {
      const float4 c0 = *reinterpret_cast<const float4*>(cw + m * DY);
      const float4 c1 = *reinterpret_cast<const float4*>(cw + m * DY + 4);
      const float cm[8] = {c0.x, c0.y, c0.z, c0.w, c1.x, c1.y, c1.z, c1.w};
      float v = rec0;
#pragma unroll
      for (int q = 0; q < DY; ++q) {
        const float d = cm[q] - gk[q];
        v = fmaf(-d, d, v);
      }
      return v;
    };
    auto row_sums = [&](bool redo) {  // redo: only the rows whose sums underflowed
      if (h) return;
      for (int m0 = 0; m0 < L; m0 += rows) {
        const int m = m0 + tid / tpm, s = tid % tpm;
        const bool need = m < L && (!redo || rowS[m] < tiny);
        float Sal = 0.f;
        if (need) {
          const float* Erow = E + m * stride;
#pragma unroll 8
          for (int k2 = s; k2 < M; k2 += tpm) Sal += Erow[k2];
        }
        for (int o = tpm >> 1; o > 0; o >>= 1) Sal += __shfl_xor_sync(FULL, Sal, o);
        if (need && s == 0) {
          rowS[m] = Sal;
          if (!redo) shS[m] = 0.f;
        }
      }
    };
#pragma unroll 4
    for (int m = h; m < L; m += 2) E[m * stride + j] = exp2_t(exponent(m));
    __syncthreads();
    row_sums(false);
    __syncthreads();
    // Rows whose sums fell below the normal range are redone with their own maxima.
    if (__any_sync(FULL, (lane < L && rowS[lane] < tiny) || (lane + 32 < L && rowS[lane + 32] < tiny))) {
      // the exponents of the flagged rows, their maxima a warp a row, then the exponentials
      for (int m = h; m < L; m += 2)
        if (rowS[m] < tiny) E[m * stride + j] = exponent(m);
      __syncthreads();
      for (int m = w; m < L; m += nw) {
        if (!(rowS[m] < tiny)) continue;
        float mx = NEG;
        for (int k2 = lane; k2 < M; k2 += 32) mx = fmaxf(mx, E[m * stride + k2]);
        mx = warp_max(mx);
        for (int k2 = lane; k2 < M; k2 += 32) E[m * stride + k2] = exp2_t(E[m * stride + k2] - mx);
        if (lane == 0) shS[m] = mx;
      }
      __syncthreads();
      row_sums(true);
      __syncthreads();
    }
    // ---- per-draw weights, the outer weight and the estimator coefficients ----
    if (w == 0) {
      const float LN2 = (float)LN2_D;
      const float lA = log2_t(lsum);
      float lw0 = NEG, lw1 = NEG;
      if (lane < L) lw0 = s_model[5] + LN2 * ((log2_t(rowS[lane]) + shS[lane]) - lA);
      if (lane + 32 < L) lw1 = s_model[5] + LN2 * ((log2_t(rowS[lane + 32]) + shS[lane + 32]) - lA);
      if (lane < L) a.lwh_new[i * L + lane] = lw0;
      if (lane + 32 < L) a.lwh_new[i * L + lane + 32] = lw1;
      const float mx = warp_max(fmaxf(lw0, lw1));
      const float p0 = lane < L ? exp_t<float>(lw0 - mx) : 0.f;
      const float p1 = lane + 32 < L ? exp_t<float>(lw1 - mx) : 0.f;
      const float ps = warp_sum(p0 + p1);
      if (lane < L) {
        coef[lane] = p0 / ps / rowS[lane];
        pm[lane] = p0;
      }
      if (lane + 32 < L) {
        coef[lane + 32] = p1 / ps / rowS[lane + 32];
        pm[lane + 32] = p1;
      }
      if (lane == 0) {
        s_ps = ps;
        s_mx = mx;
      }
    }
    __syncthreads();
    // ---- the filtered mean: the x part (first half), beta and the noise sums (second half), then
    // the z sums, four columns a warp, and the rows of [A_zz K] . sums, four rows a warp ----
    float* sbeta = kd;  // (the records are no longer read)
    if (h == 0) {
      for (int c = w; c < D1; c += hw) {
        float v = lane < L ? pm[lane] * xbs[lane * D1 + c] : 0.f;
        if (lane + 32 < L) v += pm[lane + 32] * xbs[(lane + 32) * D1 + c];
        v = warp_sum(v) / s_ps;
        if (lane == 0) a.xm[(long long)c * N + i] = v;
      }
      if (tid == M - 32) {  // the outer weight, off the other warps' path
        const float lwi = s_mx + log_t(s_ps) - log_t((float)L);
        a.lw[i] = lwi;
        if (lwi != lwi) atomicOr(a.err, ERR_NUMERIC);
        const unsigned long long key = order_key(lwi);
        if (lwi == lwi && key > *(volatile unsigned long long*)a.lwmax_key) atomicMax(a.lwmax_key, key);
      }
    } else {
      float beta = 0.f;
#pragma unroll 8
      for (int m = 0; m < L; ++m) beta += coef[m] * E[m * stride + j];
      sbeta[j] = beta;
      float acc[DY];
#pragma unroll
      for (int q = 0; q < DY; ++q) acc[q] = beta * vq[q];
      const float t = warp_sum_vec<DY>(acc, lane);
      if (lane < DY) part[lane * 32 + w - hw] = t;
    }
    __syncthreads();
    for (int c0 = 4 * w; c0 < D2; c0 += 4 * nw) {
      float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll 4
      for (int k2 = lane; k2 < M; k2 += 32) {
        const float bk = sbeta[k2];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] += bk * zsrc[(c0 + u) * M + k2];
      }
      const float t = warp_sum_vec<4>(v, lane);
      if (lane < 4) sbs[c0 + lane] = t;
    }
    if (w == nw - 1 && lane < DY) {
      float v = 0.f;
      for (int q = 0; q < hw; ++q) v += part[lane * 32 + q];
      sbs[D2 + lane] = v;
    }
    __syncthreads();
    for (int r0 = 4 * w; r0 < D2; r0 += 4 * nw) {
      float v[4] = {0.f, 0.f, 0.f, 0.f};
#pragma unroll
      for (int c = lane; c < D2 + DY; c += 32) {
        const float sc = sbs[c];
#pragma unroll
        for (int u = 0; u < 4; ++u) v[u] += zmat[(r0 + u) * (D2 + DY) + c] * sc;
      }
      float t = warp_sum_vec<4>(v, lane);
      if (lane < 4) {
        const int r = r0 + lane;
#pragma unroll
        for (int c = 0; c < D1; ++c) t += s_Azx[r * D1 + c] * x[c];
        a.zm[(long long)r * N + i] = t;
      }
    }
    // (the next group's first barrier ends every read of this one's buffers)
  }
  if (w == hw + 1) bulk_store_wait_read();  // shared memory outlives its last copies
  tc::fence_before();
  __syncthreads();
  if (w == 0) tc::tmem_dealloc(taddr, TC_COLS);
}

}  // namespace dpf
