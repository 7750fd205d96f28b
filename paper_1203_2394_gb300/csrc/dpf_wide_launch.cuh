// The step launch of a wide variant (see dpf_variant_wide.cuh): the block kernel
// with the model constants in device memory, one inner particle a thread.
#pragma once

#include "dpf_step_wide.cuh"
#include "dpf_variant_wide.cuh"

namespace dpf {

// The model constants of the (float, 8, 56, 8) variant, in this translation unit's
// constant bank (52 KB of the 64 KB): uniform reads become constant-bank operands. They
// are copied from the context's device copy before every launch of the block form, inside a
// ConstantBankUse, which keeps a copy for one filter from overtaking another's kernel on
// another stream. The two-thread form reads the context's own copy and shares nothing.
static __constant__ MC<float, 8, 56, 8> c_wide_mc;

template <bool TC>
__global__ void __launch_bounds__(256)
    step_kernel_wide(const __grid_constant__ StepArgs<float> a) {
  step_body<float, 8, 56, 8, false, 1, false, TC>(c_wide_mc, a);
}

// Two threads an inner particle (dpf_step_wide.cuh).
template <int D1, int D2, int DY>
__global__ void __launch_bounds__(512)
    step_kernel_wide_pair(const __grid_constant__ StepArgs<float> a, const MC<float, D1, D2, DY>* __restrict__ mc) {
  wide_pair_body<D1, D2, DY>(*mc, a);
}

template <typename T, int D1, int D2, int DY, bool TC>
dpf_status wide_launch(Ctx& x, StepArgs<T>& a, cudaStream_t s) {
  static_assert(sizeof(T) == 4 && D1 == 8 && D2 == 56 && DY == 8, "the compiled wide variant");
  constexpr int MAX_M = WideVariantImpl<T, D1, D2, DY>::MAX_M;
  static_assert(MAX_M == 256, "launch bounds of step_kernel_wide");
  const void* k = (const void*)step_kernel_wide<TC>;
  int nt = threads_for(x.M);
  const size_t sm = step_geometry<T, D1, D2, DY, false>(x.M, x.L, nt, &a, a.first != 0, 1, TC);
  // With the tensor cores and a diagonal Q_z, every step that has an inner update runs with two
  // threads a particle; the first step, a look-ahead alone and a full Q_z keep the block form.
  bool pair = false;
  if constexpr (TC) {
    pair = !a.first && reinterpret_cast<const MC<T, D1, D2, DY>*>(x.mconst.data())->diag_qz;
    if (pair) {
      k = (const void*)step_kernel_wide_pair<D1, D2, DY>;
      nt = 2 * x.M;
    }
  }
  static size_t attrs[2] = {0, 0};  // the largest dynamic shared memory requested so far, a kernel
  size_t& attr = attrs[pair];
  if (sm > attr) {
    cudaError_t e = cudaFuncSetAttribute(k, cudaFuncAttributeMaxDynamicSharedMemorySize, (int)sm);
    if (e != cudaSuccess) return cuda_error(e, "cudaFuncSetAttribute");
    attr = sm;
  }
  if (x.grid_step == 0 || x.grid_kernel != k) {  // persistent grid: as many CTAs as fit on the device at once
    int nb = 0, dev = 0, nsm = 0;
    cudaError_t e = cudaOccupancyMaxActiveBlocksPerMultiprocessor(&nb, k, nt, sm);
    if (e == cudaSuccess) e = cudaGetDevice(&dev);
    if (e == cudaSuccess) e = cudaDeviceGetAttribute(&nsm, cudaDevAttrMultiProcessorCount, dev);
    if (e != cudaSuccess) return cuda_error(e, "step kernel occupancy");
    x.grid_step = (nb > 0 ? nb : 1) * nsm;
    x.grid_kernel = k;
  }
  const long long grid = std::min<long long>(x.N, x.grid_step);
  if constexpr (TC) {
    if (pair) {
      step_kernel_wide_pair<D1, D2, DY><<<(unsigned)grid, nt, sm, s>>>(a, (const MC<T, D1, D2, DY>*)x.d_mconst);
      return cuda_error(cudaGetLastError(), "step kernel launch");
    }
  }
  ConstantBankUse use(s);
  if (use.error() != cudaSuccess) return cuda_error(use.error(), "model constants to the constant bank");
  cudaError_t e = cudaMemcpyToSymbolAsync(c_wide_mc, x.d_mconst, sizeof(MC<float, 8, 56, 8>), 0,
                                          cudaMemcpyDeviceToDevice, s);
  if (e != cudaSuccess) return cuda_error(e, "model constants to the constant bank");
  step_kernel_wide<TC><<<(unsigned)grid, nt, sm, s>>>(a);
  return cuda_error(cudaGetLastError(), "step kernel launch");
}

}  // namespace dpf
