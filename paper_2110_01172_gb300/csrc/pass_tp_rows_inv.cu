// pass_tp_rows_inv.cu - inverse row pass of the two-pass family (radix-2
// column step folded into the stores).
#include "tp_rows_inv_launch.cuh"

namespace gbdct {
namespace {

template <int L>
cudaError_t launch(const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  return launch_e<L, false>(a, batch, s, prepare);
}

}  // namespace

cudaError_t run_tp_rows_inv(int lg2, const Dct2dArgs& a, int batch, cudaStream_t s, bool prepare) {
  if (a.exact) return run_tp_rows_inv_exact(lg2, a, batch, s, prepare);
  GBDCT_TP_ROWS_SWITCH(lg2, launch, a, batch, s, prepare);
}

}  // namespace gbdct
