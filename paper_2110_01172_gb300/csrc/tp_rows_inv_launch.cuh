// tp_rows_inv_launch.cuh - launches of the inverse row pass of the two-pass family
// (radix-2 column step folded into the stores), shared by the translation units of
// its plain and its exact kernels (Dct2dArgs::exact).
#pragma once

#include "tp_rows_launch.cuh"

namespace gbdct {
namespace {

template <int L, bool NARROW, bool MAPPED, bool STAGED, bool EXACT>
cudaError_t launch_k(const Dct2dArgs& a, const PoissonArgs& ps, int batch, cudaStream_t s, bool prepare) {
  using R = TpRows<L, NARROW>;
  constexpr size_t SMEM = STAGED ? R::SMEM_STAGED : R::SMEM;
  const auto k = k_tp_rows_inv<L, MAPPED, STAGED, NARROW, false, EXACT>;
  if (prepare) return tp_smem_limit(reinterpret_cast<const void*>(k), SMEM);
  if ((a.n1 / 4) % R::NP) return cudaErrorInvalidValue;
  return pdl::launch(k, dim3(a.n1 / 4 / R::NP, 1, batch), dim3(R::THREADS), SMEM, s, a, ps);
}

template <int L, bool NARROW, bool MAPPED, bool EXACT>
cudaError_t launch_m(const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  const PoissonArgs none{};
  if constexpr (tp_inv_staged<L>()) {
    if (prepare) {
      const cudaError_t e = launch_k<L, NARROW, MAPPED, true, EXACT>(a, none, batch, s, true);
      if (e != cudaSuccess) return e;
    } else if (a.io_dev) {
      return launch_k<L, NARROW, MAPPED, true, EXACT>(a, none, batch, s, false);
    }
  }
  return launch_k<L, NARROW, MAPPED, false, EXACT>(a, none, batch, s, prepare);
}

template <int L, bool NARROW, bool EXACT>
cudaError_t launch_n(const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  return (a.vkind == 1 || a.vkind == 2) ? launch_m<L, NARROW, true, EXACT>(a, batch, s, prepare)
                                        : launch_m<L, NARROW, false, EXACT>(a, batch, s, prepare);
}

// `prepare` readies the kernels that a call with the same arguments may run
// (device and host-mapped buffers).
template <int L, bool EXACT>
cudaError_t launch_e(const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  if constexpr (L == 64 && !EXACT) {
    return cudaErrorInvalidValue;  // rows of 64 are always exact
  } else {
    return tp_rows_narrow<L>(a, batch) ? launch_n<L, true, EXACT>(a, batch, s, prepare) : launch_n<L, false, EXACT>(a, batch, s, prepare);
  }
}

}  // namespace
}  // namespace gbdct
