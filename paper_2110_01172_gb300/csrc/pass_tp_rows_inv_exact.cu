// pass_tp_rows_inv_exact.cu - inverse row pass of the two-pass family (radix-2
// column step folded into the stores):
// its exact kernels (Dct2dArgs::exact).
#include "tp_rows_inv_launch.cuh"

namespace gbdct {
namespace {

template <int L>
cudaError_t launch(const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  return launch_e<L, true>(a, batch, s, prepare);
}

}  // namespace

cudaError_t run_tp_rows_inv_exact(int lg2, const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  GBDCT_TP_ROWS_SWITCH(lg2, launch, a, batch, s, prepare);
}

}  // namespace gbdct
