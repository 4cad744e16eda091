// pass_tp_rows_fwd.cu - forward row pass of the two-pass family (radix-2 column
// step folded into the loads).
#include "tp_rows_launch.cuh"

namespace gbdct {
namespace {

template <int L, bool NARROW, bool GENERAL, bool EXACT, bool HOST = false>
cudaError_t launch_k(const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  using R = TpRows<L, NARROW>;
  const auto k = k_tp_rows_fwd<L, NARROW, GENERAL, EXACT, HOST>;
  if (prepare) return tp_smem_limit(reinterpret_cast<const void*>(k), R::SMEM);
  if ((a.n1 / 4) % R::NP) return cudaErrorInvalidValue;
  return pdl::launch(k, dim3(a.n1 / 4 / R::NP, 1, batch), dim3(R::THREADS), R::SMEM, s, a);
}

template <int L, bool EXACT>
cudaError_t launch_e(const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  if (prepare) {
    const cudaError_t e = launch_k<L, true, true, EXACT, true>(a, batch, s, true);
    if (e != cudaSuccess) return e;
  } else if (!a.io_dev) {
    return launch_k<L, true, true, EXACT, true>(a, batch, s, false);
  }
  const bool general = a.vkind == 1 || a.thresh > 0.f;
  if (tp_rows_narrow<L>(a, batch))
    return general ? launch_k<L, true, true, EXACT>(a, batch, s, prepare)
                   : launch_k<L, true, false, EXACT>(a, batch, s, prepare);
  return general ? launch_k<L, false, true, EXACT>(a, batch, s, prepare)
                 : launch_k<L, false, false, EXACT>(a, batch, s, prepare);
}

// `prepare` readies the variants that a call with the same arguments runs (device
// and host-mapped buffers).
template <int L>
cudaError_t launch(const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  if (a.exact) return launch_e<L, true>(a, batch, s, prepare);
  if constexpr (L == 64) {
    return cudaErrorInvalidValue;  // rows of 64 are always exact
  } else {
    return launch_e<L, false>(a, batch, s, prepare);
  }
}

}  // namespace

cudaError_t run_tp_rows_fwd(int lg2, const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  GBDCT_TP_ROWS_SWITCH(lg2, launch, a, batch, s, prepare);
}

}  // namespace gbdct
