// tp_rows_poisson_launch.cuh - launches of the inverse row pass of a Poisson solve
// (the three inverses of one spectrum as one batch), shared by the translation
// units of its plain and its exact kernels (Dct2dArgs::exact).
#pragma once

#include "tp_rows_launch.cuh"

namespace gbdct {
namespace {

template <int L, bool NARROW, bool STAGED, bool EXACT>
cudaError_t launch_k(const Dct2dArgs& a, const PoissonArgs& ps, int batch, cudaStream_t s, bool prepare) {
  using R = TpRows<L, NARROW>;
  constexpr size_t SMEM = !STAGED ? R::SMEM : tp_den_staged<L, NARROW>() ? R::SMEM_DEN : R::SMEM_STAGED;
  const auto k = k_tp_rows_inv<L, true, STAGED, NARROW, true, EXACT>;
  if (prepare) return tp_smem_limit(reinterpret_cast<const void*>(k), SMEM);
  if ((a.n1 / 4) % R::NP) return cudaErrorInvalidValue;
  return pdl::launch(k, dim3(a.n1 / 4 / R::NP, 1, batch), dim3(R::THREADS), SMEM, s, a, ps);
}

template <int L, bool NARROW, bool EXACT>
cudaError_t launch_n(const Dct2dArgs& a, const PoissonArgs& ps, cudaStream_t s, bool prepare) {
  if (prepare) {
    const cudaError_t e = launch_k<L, NARROW, false, EXACT>(a, ps, 3, s, true);
    return e == cudaSuccess ? launch_k<L, NARROW, true, EXACT>(a, ps, 3, s, true) : e;
  }
  return a.io_dev ? launch_k<L, NARROW, true, EXACT>(a, ps, 3, s, false)
                  : launch_k<L, NARROW, false, EXACT>(a, ps, 3, s, false);
}

template <int L, bool EXACT>
cudaError_t launch_e(const Dct2dArgs& a, const PoissonArgs& ps, cudaStream_t s, bool prepare) {
  if constexpr (L == 64 && !EXACT) {
    return cudaErrorInvalidValue;  // rows of 64 are always exact
  } else {
    return tp_rows_narrow<L>(a, 3) ? launch_n<L, true, EXACT>(a, ps, s, prepare) : launch_n<L, false, EXACT>(a, ps, s, prepare);
  }
}

}  // namespace
}  // namespace gbdct
